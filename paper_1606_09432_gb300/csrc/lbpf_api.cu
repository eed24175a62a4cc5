// Host side of the lbpf C ABI: context, device buffers, launches and the
// lagged/synchronised state of the heat populations.  See include/lbpf.h.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>

#include <sys/stat.h>
#include <vector>

#include "lbpf_internal.cuh"

using namespace lbpf;

namespace {

thread_local std::string t_err;

// Planes per z-segment of a work item of the step kernel.
// (0: chosen from the work size and the resident block count.)
#ifndef LBPF_SEGMENT
#define LBPF_SEGMENT 0
#endif

constexpr int kHistCap = 64;

// a2 of the thin-interface relations, Eq. (Kinetic-Coeff); lambda* cancels beta.
constexpr double kA2 = 0.6267;

}  // namespace

struct lbpf_ctx {
    int lattice = 0, grad = 0, precision = 0, dim = 2;
    int Qg = 0, Qu = 0, Sg = 0, Su = 0;
    size_t rsize = 8, ssize = 8;
    int n_domains = 0;
    std::vector<lbpf_domain> in;
    std::vector<DomainDev> dd;
    DomainDev* d_dd = nullptr;
    WorkItem* d_items = nullptr;
    int* d_counters = nullptr;
    int n_items = 0, n_blocks = 0, items_cap = 0;
    int tile_v = 0, seg_len = 0, sms = 1;
    bool staged = false;  // step kernel with bulk-copy staging (staged_kernel.cuh)
    bool vec = false;     // vector step: two launches, four sites a thread (vec_kernel.cuh)
    bool tile = false;    // one-tile step (tile_kernel.cuh)
    int kind = 0;         // step kernel kind: kStepWalls (some domain has walls) | kStepAdvect
    // graphs of kGraphSteps steady-state launches, keyed by (cur, fcur, acur)
    cudaGraphExec_t graphs[8] = {};
    bool graphs_off = false;
    std::string tuned;  // how the schedule was chosen
    bool tune_pending = false;  // time the schedules at the first step (on the seeded state)
    // measurement history: per domain a ring of kHistCap entries (t, tip6)
    double* d_hist = nullptr;
    std::vector<int> hist_count, hist_last;
    cudaStream_t stream = nullptr;
    int device = 0;
    const Launchers* L = nullptr;
    size_t smem = 0;
    int cur = 0, fcur = 0, acur = 0, lagged = 0;
    long long steps = 0, kernels = 0;
    void* scratch = nullptr;
    size_t scratch_bytes = 0;
    double* red = nullptr;
    double* d_seeds = nullptr;
    int seeds_cap = 0;
    size_t dev_bytes = 0;
    std::vector<void*> allocs;
    std::string err;
};

static int fail(lbpf_ctx* c, int code, const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    if (c)
        c->err = buf;
    else
        t_err = buf;
    return code;
}

#define CK(call)                                                                                  \
    do {                                                                                          \
        cudaError_t e_ = (call);                                                                  \
        if (e_ != cudaSuccess) return fail(c, LBPF_ECUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
    } while (0)

static int dev_alloc(lbpf_ctx* c, void** p, size_t bytes)
{
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        return fail(c, e == cudaErrorMemoryAllocation ? LBPF_ENOMEM : LBPF_ECUDA, "cudaMalloc(%zu bytes): %s", bytes,
                    cudaGetErrorString(e));
    }
    c->allocs.push_back(*p);
    c->dev_bytes += bytes;
    return LBPF_OK;
}

static const Launchers* pick(int lattice, int precision) { return launchers_for_pair(lattice, precision); }

static bool finite_pos(double v) { return std::isfinite(v) && v > 0.0; }

static void free_all(lbpf_ctx* c)
{
    for (void* p : c->allocs) cudaFree(p);
    c->allocs.clear();
}


// ---------------------------------------------------------------------------
// Work schedule of the step kernel.  Items are columns of tile_x x tile_y
// sites over segments of the marched axis (z in 3D, y in 2D), listed segment
// by segment; the kernel runs as many blocks as fit on the GPU and takes items
// in order (see step_kernel).
// ---------------------------------------------------------------------------
static long long column_units(const lbpf_ctx* c, int v)
{
    const int tx = c->vec ? kVecTX : tile_x(c->dim, v), ty = c->vec ? kVecTY : tile_y(c->dim, v);
    long long units = 0;
    for (const DomainDev& d : c->dd) {
        const int ny = c->dim == 3 ? d.ny : 1, nz = c->dim == 3 ? d.nz : d.ny;
        units += (long long)((d.nx + tx - 1) / tx) * ((ny + ty - 1) / ty) * nz;
    }
    return units;
}

static int blocks_per_sm(const lbpf_ctx* c, int v)
{
    if (c->vec) return c->L->vec_blocks_per_sm(c->kind & kStepWalls);
    return c->staged ? c->L->staged_blocks_per_sm() : c->L->blocks_per_sm(v, c->kind);
}

// Segment length balancing the per-item prologue (two extra planes) against
// the tail of the dynamic schedule: L ~ sqrt(5 units / resident blocks).
static int default_segment(const lbpf_ctx* c, int v)
{
    if (LBPF_SEGMENT > 0) return LBPF_SEGMENT;
    const double G = (double)blocks_per_sm(c, v) * c->sms;
    // vector step: below 64 planes a block the waves of equal items do not fill
    // (64^3: 53.6 us a step in segments, 28.2 balanced), above they do and share
    // their halo rims better (352^3: 1597 us in segments, 1681 balanced)
    if (c->vec && (double)column_units(c, v) < 64.0 * G) return 0;
    // small contexts: one wave of the shortest items that all blocks hold at
    // once, since a step then costs the latency of one item (us a step, 8 planes
    // an item / this rule: 2D 128^2 22.1 / 9.1, 256^2 25.8 / 12.3, 512^2 26.6 /
    // 20.4; 3D 64^3 FP32 37.3 / 27.3)
    const double units = (double)column_units(c, v);
    if (units <= 8.0 * G) return (int)std::ceil(units / G);
    int L = (int)std::lround(std::sqrt(5.0 * units / G));
    return L < 8 ? 8 : (L > 256 ? 256 : L);
}

// Items of equal total work per block: as many whole columns as go round all
// G blocks evenly, each marched in one piece (neighbouring columns advance
// together, so their halo rims meet in L2), then the remaining columns, laid
// end to end, in G runs of equal length (a run that crosses from one column to
// the next becomes two items), longest first.
static void balanced_items(const lbpf_ctx* c, int wx, int wy, long long G, std::vector<WorkItem>& items)
{
    std::vector<WorkItem> cols;
    for (int k = 0; k < c->n_domains; ++k) {
        const DomainDev& d = c->dd[k];
        const int ny = c->dim == 3 ? d.ny : 1, nz = c->dim == 3 ? d.nz : d.ny;
        for (int y = 0; y < ny; y += wy)
            for (int x = 0; x < d.nx; x += wx) cols.push_back(WorkItem{k, x, y, 0, nz, 0});
    }
    const size_t whole = c->n_domains == 1 ? cols.size() / (size_t)G * (size_t)G : 0;
    items.assign(cols.begin(), cols.begin() + whole);
    long long rest = 0;
    for (size_t j = whole; j < cols.size(); ++j) rest += cols[j].z1;
    if (rest > 0) {
        const long long run = (rest + G - 1) / G < 4 ? 4 : (rest + G - 1) / G;
        long long left = run;  // of the current run
        for (size_t j = whole; j < cols.size(); ++j) {
            const int nz = cols[j].z1;
            for (int z = 0; z < nz;) {
                int len = (int)(left < nz - z ? left : nz - z);
                if (nz - z - len > 0 && nz - z - len < 3) len = nz - z;  // no slivers
                WorkItem w = cols[j];
                w.z0 = z;
                w.z1 = z + len;
                items.push_back(w);
                z += len;
                left -= len;
                if (left < 3) left = run;
            }
        }
        std::stable_sort(items.begin() + whole, items.end(),
                         [](const WorkItem& a, const WorkItem& b) { return a.z1 - a.z0 > b.z1 - b.z0; });
    }
}

// seg: planes per item, 0 the balanced partition (vector step).
static int set_schedule(lbpf_ctx* c, int v, int seg)
{
    if (seg > 0) c->tile = false;  // a segment length asks for the march
    const int wx = c->vec ? kVecTX : tile_x(c->dim, v), wy = c->vec ? kVecTY : tile_y(c->dim, v);
    const long long G = (long long)blocks_per_sm(c, v) * c->sms;
    std::vector<WorkItem> items;
    if (c->tile) {
        for (int k = 0; k < c->n_domains; ++k)
            for (int y = 0; y < c->dd[k].ny; y += kTileRY - 2)
                for (int x = 0; x < c->dd[k].nx; x += kTileRX - 2) items.push_back(WorkItem{k, x, y, 0, c->dd[k].ny, 0});
        seg = kTileRY - 2;
    } else if (seg == 0) {
        balanced_items(c, wx, wy, G, items);
        seg = (int)(column_units(c, v) / (long long)items.size());
    } else
    for (int k = 0; k < c->n_domains; ++k) {
        const DomainDev& d = c->dd[k];
        // 2D: the kernel marches the y axis (its z) with one-row tiles
        const int ny = c->dim == 3 ? d.ny : 1, nz = c->dim == 3 ? d.nz : d.ny;
        const int tx = (d.nx + wx - 1) / wx, tyn = (ny + wy - 1) / wy;
        const int nseg = (nz + seg - 1) / seg;
        for (int sg = 0; sg < nseg; ++sg) {
            const int z0 = (int)((long long)sg * nz / nseg), z1 = (int)((long long)(sg + 1) * nz / nseg);
            for (int by = 0; by < tyn; ++by)
                for (int bx = 0; bx < tx; ++bx) {
                    WorkItem w;
                    w.dom = k;
                    w.x0 = bx * wx;
                    w.y0 = by * wy;
                    w.z0 = z0;
                    w.z1 = z1;
                    w.pad = 0;
                    items.push_back(w);
                }
        }
    }
    if ((int)items.size() > c->items_cap) {
        int rc;
        void* p = nullptr;
        if ((rc = dev_alloc(c, &p, sizeof(WorkItem) * items.size()))) return rc;
        c->d_items = static_cast<WorkItem*>(p);  // the old table stays in the context's allocation list
        c->items_cap = (int)items.size();
    }
    CK(cudaMemcpyAsync(c->d_items, items.data(), sizeof(WorkItem) * items.size(), cudaMemcpyHostToDevice, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    c->n_items = (int)items.size();
    c->n_blocks = c->tile ? c->n_items : (int)(G < c->n_items ? G : c->n_items);
    c->tile_v = v;
    c->seg_len = seg;
    for (cudaGraphExec_t& g : c->graphs)
        if (g) {
            cudaGraphExecDestroy(g);
            g = nullptr;
        }
    return LBPF_OK;
}

// Whether the one-tile step (tile_kernel.cuh) replaces the march: 2D, no
// advection, up to a few million sites.  us a step, march (its best schedule) /
// tile: FP32 128^2 8.9 / 3.2, 256^2 10.9 / 4.1, 512^2 18.5 / 10.2, 1024^2 45.2 /
// 37.0, 2048^2 148 / 137, 3000^2 289 / 288, 4096^2 522 / 535, 8000^2 1859 / 2030;
// with walls 1000^2 49.0 / 45.8, 3000^2 330 / 373; FP16 512^2 19.5 / 10.9, 2048^2
// 166 / 156, 4096^2 554 / 606; FP64 (bound by FP64 arithmetic) with walls 128^2 28
// / 14, 800^2 240 / 193, 2000^2 1080 / 1146, periodic 1500^2 612 / 534.
// Within that, where its estimated time is the shorter one, since domains that
// fill neither the tiles' 30 x 6 sites nor the march's 128-site strips cost each
// form differently.  A tile costs FP32 5.95 ns, 16 bits 6.9, FP64 41 (with walls 1.3
// times that), whatever its columns, up to a quarter less with fewer rows.  The
// march costs its rows (an item's and three before them) on all resident blocks,
// each the more the more warps of the strip have sites (FP32 1.9 + 0.6 us a warp, 16
// bits 1.8 + 0.8, FP64 4 + 7.5; with walls 1.25 times that), and at least one item.
// Batches, march / tile: FP32 3000 of 128 x 7 102 / 164, 200 of 128^2 124 / 132, 1000
// of 64^2 191 / 197, 60 of 256^2 143 / 138, 1000 of 32^2 93 / 71; FP16 107 / 195, 130 /
// 151, 203 / 231, 158 / 160, 84 / 69; FP64 1500 of 128 x 7 427 / 453, 500 of 64^2 612 /
// 701, 1000 of 32^2 416 / 481, 100 of 128^2 491 / 471; FP32 31 x 100000 247 / 178,
// 100000 x 7 38 / 30; with walls FP32 1200^2 80 / 64, 1400^2 90 / 85, 30 of 256^2 94 /
// 92, FP16 1400^2 97 / 78.
static bool tile_applies(const lbpf_ctx* c)
{
    const char *kenv = getenv("LBPF_KERNEL"), *tenv = getenv("LBPF_AUTOTUNE");
    if (!c->L->tile_step || (c->kind & kStepAdvect) || (kenv && *kenv) || (tenv && atoi(tenv))) return false;
    const bool walls = (c->kind & kStepWalls) != 0;
    const int type = c->rsize == 8 ? 0 : c->ssize == 4 ? 1 : 2;
    const double tile_us[3] = {0.041, 0.00595, 0.0069}, row_us[3] = {4.0, 1.9, 1.8}, warp_us[3] = {7.5, 0.6, 0.77};
    const int seg = default_segment(c, 0), TX = kTileRX - 2, TY = kTileRY - 2, SX = kStripX[0];
    auto strip_row = [&](int w) { return w > 0 ? row_us[type] + (w + 31) / 32 * warp_us[type] : 0.0; };
    double sites = 0, tile = 0, march = 0, item = 0;
    for (const DomainDev& d : c->dd) {
        sites += (double)d.n;
        // full tile rows, and the last one
        const int th = d.ny % TY;
        tile += (d.nx + TX - 1) / TX * (d.ny / TY + (th ? 0.6 + 0.4 * (th + 2) / kTileRY : 0.0));
        march += (d.ny + 3.0 * ((d.ny + seg - 1) / seg)) * (d.nx / SX * strip_row(SX) + strip_row(d.nx % SX));
        item = std::max(item, (std::min(seg, d.ny) + 3) * strip_row(std::min(d.nx, SX)));
    }
    if (sites > (c->rsize == 8 ? 2.5e6 : walls ? 2.0e6 : 4.5e6)) return false;
    tile *= tile_us[type] * (walls ? 1.3 : 1.0);
    march = std::max(march / ((double)blocks_per_sm(c, 0) * c->sms), item) * (walls ? 1.25 : 1.0);
    return tile <= march;
}

static std::string tune_key(const lbpf_ctx* c)
{
    char buf[160];
    // FNV-1a over the domain sizes and the build time of this library, so
    // that a rebuilt kernel is timed again instead of taking a stale choice
    unsigned long long h = 1469598103934665603ULL;
    for (const DomainDev& d : c->dd)
        for (int v : {d.nx, d.ny, d.nz, d.use_index}) {
            h ^= (unsigned long long)(unsigned)v;
            h *= 1099511628211ULL;
        }
    for (const char* p = __DATE__ " " __TIME__; *p; ++p) {
        h ^= (unsigned char)*p;
        h *= 1099511628211ULL;
    }
    snprintf(buf, sizeof(buf), "s2-lat%d-prec%d-grad%d-dom%d-%016llx-sm%d-k%d", c->lattice, c->precision, c->grad,
             c->n_domains, h, c->sms, (c->staged ? 1 : 0) | (c->kind << 1) | (c->vec ? 8 : 0));
    return buf;
}

static std::string tune_cache_path()
{
    const char* p = getenv("LBPF_TUNE_CACHE");
    if (p) return p;
    const char* home = getenv("HOME");
    return std::string(home ? home : "/tmp") + "/.cache/lbpf_tune.txt";
}

static StepArgs step_args(const lbpf_ctx* c)
{
    StepArgs a;
    a.doms = c->d_dd;
    a.items = c->d_items;
    a.n_items = c->n_items;
    a.counters = c->d_counters;
    a.cur = c->cur;
    a.fcur = c->fcur;
    a.acur = c->acur;
    a.collide = c->lagged;
    a.grad = c->grad;
    a.index = 0;
    for (const DomainDev& d : c->dd) a.index |= d.use_index;
    return a;
}

static long long launches_per_step(const lbpf_ctx* c)
{
    return c->vec ? c->L->heat_vec_launches(c->dd.data(), c->n_domains) + 1 : 1;
}

// The launches of one time step.
static cudaError_t issue_step(lbpf_ctx* c, const StepArgs& a)
{
    if (c->staged) return c->L->step_staged(a, c->n_blocks, c->stream);
    if (c->tile) return c->L->tile_step(c->kind & kStepWalls, a, c->stream);
    if (!c->vec) return c->L->step(c->tile_v, c->kind, a, c->n_blocks, c->stream);
    const cudaError_t e = c->L->heat_vec(c->dd.data(), c->d_dd, c->n_domains, a, c->stream);
    if (e != cudaSuccess) return e;
    return c->L->phi_vec(c->kind & kStepWalls, a, c->n_blocks, c->stream);
}

// Time a few launches of the current schedule on the live state.  Every trial
// reads the current buffers (cur, fcur, acur) and writes the other ones,
// which the next real step overwrites, so the state is left as it was.
static double time_schedule(lbpf_ctx* c, int launches)
{
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        cudaGetLastError();
        return 1e30;
    }
    StepArgs a = step_args(c);
    a.collide = 1;
    double best = 1e30;
    for (int k = 0; k < launches + 2; ++k) {
        if (cudaMemsetAsync(c->d_counters + c->cur, 0, sizeof(int), c->stream) != cudaSuccess) break;
        cudaEventRecord(e0, c->stream);
        if (issue_step(c, a) != cudaSuccess) break;
        cudaEventRecord(e1, c->stream);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (k >= 2 && ms < best) best = ms;
    }
    cudaGetLastError();
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return best;
}

// Schedule at context creation: a cached choice for this configuration, else
// the rule (tile variant 0, default segment); large configurations (or
// LBPF_AUTOTUNE=1) are then timed at the first step, on the seeded state.
static int initial_schedule(lbpf_ctx* c)
{
    if ((c->tile = tile_applies(c))) {
        c->tuned = "rule";
        return set_schedule(c, 0, 0);
    }
    const std::string key = tune_key(c);
    if (FILE* f = fopen(tune_cache_path().c_str(), "r")) {
        char k[200];
        int v, seg;
        while (fscanf(f, "%199s %d %d", k, &v, &seg) == 3)
            if (key == k && v >= 0 && v < (c->staged || c->vec || c->kind ? 1 : kNumTileVariants) && seg >= (c->vec ? 0 : 1)) {
                fclose(f);
                c->tuned = "cache";
                return set_schedule(c, v, seg);
            }
        fclose(f);
    }
    double sites = 0;
    for (const DomainDev& d : c->dd) sites += (double)d.n;
    const char* env = getenv("LBPF_AUTOTUNE");
    c->tune_pending = env ? atoi(env) != 0 : sites >= 4e6;
    c->tuned = "rule";
    return set_schedule(c, 0, default_segment(c, 0));
}

// Time tile variants x segments {L, L/2, 2L} and keep (and cache) the
// fastest, but leave the rule's schedule (variant 0, segment L) only for one
// at least 3 % faster: short trials at the first step are noisy, and a
// wrong switch has cost up to 10 % in steady state.
static int autotune(lbpf_ctx* c)
{
    CK(cudaStreamSynchronize(c->stream));
    double best_t = 1e30, rule_t = 1e30;
    int best_v = 0, best_seg = default_segment(c, 0);
    for (int v = 0; v < (c->staged || c->vec || c->kind ? 1 : kNumTileVariants); ++v) {
        const int L0 = default_segment(c, v);
        const int segs[3] = {L0, L0 / 2 > 8 ? L0 / 2 : 8, L0 ? L0 * 2 : 32};
        for (int j = 0; j < 3; ++j) {
            int rc = set_schedule(c, v, segs[j]);
            if (rc) return rc;
            const double t = time_schedule(c, 6);
            if (v == 0 && j == 0) rule_t = t;
            if (t < best_t) {
                best_t = t;
                best_v = v;
                best_seg = segs[j];
            }
        }
    }
    if (!(best_t < 0.97 * rule_t)) {
        best_v = 0;
        best_seg = default_segment(c, 0);
    }
    CK(cudaMemsetAsync(c->d_counters, 0, sizeof(int) * 2, c->stream));
    c->tuned = "timed";
    const std::string path = tune_cache_path();
    const size_t slash = path.find_last_of('/');
    if (slash != std::string::npos && slash > 0) mkdir(path.substr(0, slash).c_str(), 0755);  // e.g. ~/.cache
    if (FILE* f = fopen(path.c_str(), "a")) {
        fprintf(f, "%s %d %d\n", tune_key(c).c_str(), best_v, best_seg);
        fclose(f);
    }
    return set_schedule(c, best_v, best_seg);
}

// Whether the context takes the vector step.  It can where every domain is 3D
// with 16-bit deviations, one crystal, no advection, site indices in 31 bits and
// rows and planes within a launch grid's limits; it pays where its 64-site row
// segments are at least 0.6 full and its 64 x 12 tiles 0.5, and there is work for
// more than a wave of blocks (FP16, us a step, one launch / vector: 32^3 14.5
// / 25.1, 64^3 29.7 / 29.1, 96^3 56.0 / 52.8, 128^3 115 / 85, 207x174x190 397 /
// 296, 351^3 walls 2307 / 1682; nx = 24, 24x400x400, 266 / 325; nx = 40 271 / 201;
// rows in y: 512x2x500 55 / 71, 128x2x1000 D3Q27 45 / 73, 512x4x500 71 / 80, 512x6x500
// 94 / 86, 256x13x256 62 / 56),
// and where the domains share their heat launches (heat_grid): one more launch a
// step costs 3 to 6 us, which takes half a million sites to earn (one launch /
// vector with a heat launch a domain, walls alternating: 64 domains of 48^3 549 /
// 547, 64 of 64^3 902 / 983, 16 of 96^3 755 / 746, 8 of 128^3 866 / 674).
// LBPF_KERNEL: "vector" wherever it can, any other value never.
static bool vec_applies(const Launchers* L, const lbpf_domain* domains, int n_domains)
{
    const char* kenv = getenv("LBPF_KERNEL");
    const bool forced = kenv && strcmp(kenv, "vector") == 0;
    if (!L->heat_vec || (kenv && *kenv && !forced)) return false;
    double sites = 0, slots = 0, tiles = 0;
    std::vector<DomainDev> sizes(n_domains);  // what heat_grid looks at
    for (int k = 0; k < n_domains; ++k) {
        const lbpf_domain& d = domains[k];
        if (d.nx < 8 || (long long)((d.nx + 3) / 4 * 4) * d.ny * d.nz >= (1LL << 31) || d.n_crystals > 1 ||
            d.adv[0] != 0.0 || d.adv[1] != 0.0 || d.adv[2] != 0.0 || d.ny > 65535 * kHeatY || d.nz > 65535)
            return false;
        sites += (double)d.nx * d.ny * d.nz;
        const double segments = (double)((d.nx + kVecTX - 1) / kVecTX) * d.nz;
        slots += segments * kVecTX * d.ny;
        tiles += segments * ((d.ny + kVecTY - 1) / kVecTY);
        sizes[k].px = (d.nx + 3) / 4 * 4;
        sizes[k].ny = d.ny;
        sizes[k].nz = d.nz;
        sizes[k].bc = d.bc;
    }
    return forced || (sites >= 2e5 && sites >= 0.6 * slots && sites >= 0.5 * kVecTX * kVecTY * tiles &&
                      L->heat_vec_launches(sizes.data(), n_domains) - 1 <= sites / 5e5);
}

// lbpf_create with the vector step where it applies, or (vec false) never.
// *vec: whether the context was to take it.
static int create(const lbpf_domain* domains, int n_domains, int lattice, int grad, int precision, void* stream,
                  bool* vec, lbpf_ctx** out)
{
    lbpf_ctx* c = nullptr;
    if (!out) return fail(nullptr, LBPF_EINVAL, "lbpf_create: out is NULL");
    *out = nullptr;
    if (!domains || n_domains < 1) return fail(nullptr, LBPF_EINVAL, "lbpf_create: need at least one domain");
    if (grad != LBPF_GRAD_DD && grad != LBPF_GRAD_FD) return fail(nullptr, LBPF_EINVAL, "lbpf_create: bad grad %d", grad);
    const Launchers* L = pick(lattice, precision);
    if (!L) return fail(nullptr, LBPF_EINVAL, "lbpf_create: bad lattice %d or precision %d", lattice, precision);
    const int dim = L->D;
    for (int k = 0; k < n_domains; ++k) {
        const lbpf_domain& d = domains[k];
        if (d.nx < 2 || d.ny < 2 || (dim == 2 && d.nz != 1) || (dim == 3 && d.nz < 2))
            return fail(nullptr, LBPF_EINVAL, "domain %d: sizes %d x %d x %d invalid for a %dD lattice (each >= 2; nz = 1 in 2D)",
                        k, d.nx, d.ny, d.nz, dim);
        if (d.bc < 0 || d.bc > 7 || (dim == 2 && (d.bc & LBPF_BC_WALL_Z)) ||
            ((d.bc & LBPF_BC_WALL_X) && d.nx < 3) || ((d.bc & LBPF_BC_WALL_Y) && d.ny < 3) ||
            ((d.bc & LBPF_BC_WALL_Z) && d.nz < 3))
            return fail(nullptr, LBPF_EINVAL,
                        "domain %d: bc %d invalid (LBPF_BC_WALL_* bits, no z wall in 2D, >= 3 sites on a walled axis)",
                        k, d.bc);
        if ((long long)d.nx * d.ny > (1LL << 31) || (long long)d.nx * d.ny * d.nz > (1LL << 40))
            return fail(nullptr, LBPF_EINVAL, "domain %d: too many sites", k);
        if (!finite_pos(d.dx) || !finite_pos(d.dt) || !finite_pos(d.W0) || !finite_pos(d.tau0) || !finite_pos(d.kappa))
            return fail(nullptr, LBPF_EINVAL, "domain %d: dx, dt, W0, tau0, kappa must be finite and > 0", k);
        if (!std::isfinite(d.lambda) || !std::isfinite(d.delta) || !std::isfinite(d.xi) || d.xi < 0)
            return fail(nullptr, LBPF_EINVAL, "domain %d: lambda, delta, xi must be finite (xi >= 0)", k);
        if (!std::isfinite(d.adv[0]) || !std::isfinite(d.adv[1]) || !std::isfinite(d.adv[2]))
            return fail(nullptr, LBPF_EINVAL, "domain %d: adv must be finite", k);
        if (d.adv[0] != 0.0 || d.adv[1] != 0.0 || d.adv[2] != 0.0) {
            if (dim == 2 && d.adv[2] != 0.0)
                return fail(nullptr, LBPF_EINVAL, "domain %d: adv[2] must be 0 on a 2D lattice", k);
            if (((d.bc & LBPF_BC_WALL_X) && d.adv[0] != 0.0) || ((d.bc & LBPF_BC_WALL_Y) && d.adv[1] != 0.0) ||
                ((d.bc & LBPF_BC_WALL_Z) && d.adv[2] != 0.0))
                return fail(nullptr, LBPF_EINVAL, "domain %d: the velocity must be tangential to the walls", k);
        }
        if (d.n_crystals < 1 || d.n_crystals > LBPF_MAX_CRYSTALS)
            return fail(nullptr, LBPF_EINVAL, "domain %d: n_crystals %d not in 1..%d", k, d.n_crystals, LBPF_MAX_CRYSTALS);
        for (int j = 0; j < d.n_crystals; ++j) {
            const lbpf_crystal& cr = d.crystals[j];
            if (cr.kind < LBPF_AS_CUBIC100 || cr.kind > LBPF_AS_S111)
                return fail(nullptr, LBPF_EINVAL, "domain %d crystal %d: unknown anisotropy kind %d", k, j, cr.kind);
            if (cr.kind == LBPF_AS_ANGLE && (dim != 2 || cr.q < 1))
                return fail(nullptr, LBPF_EINVAL, "domain %d crystal %d: the angle form needs a 2D lattice and q >= 1", k, j);
            if (!std::isfinite(cr.eps) || !std::isfinite(cr.gamma) || !std::isfinite(cr.phi0))
                return fail(nullptr, LBPF_EINVAL, "domain %d crystal %d: non-finite parameter", k, j);
        }
    }

    c = new (std::nothrow) lbpf_ctx();
    if (!c) return fail(nullptr, LBPF_ENOMEM, "lbpf_create: out of host memory");
    c->lattice = lattice;
    c->grad = grad;
    c->precision = precision;
    c->dim = dim;
    c->L = L;
    c->Qg = L->Qphi;
    c->Qu = L->Qu;
    const bool dev = precision >= LBPF_FP32_FP16DEV;
    c->Sg = dev ? c->Qg - 1 : c->Qg;
    c->Su = dev ? c->Qu - 1 : c->Qu;
    c->rsize = precision == LBPF_FP64 ? 8 : 4;
    c->ssize = precision == LBPF_FP64 ? 8 : (precision == LBPF_FP32 ? 4 : 2);
    c->n_domains = n_domains;
    c->in.assign(domains, domains + n_domains);
    c->stream = static_cast<cudaStream_t>(stream);
    if (cudaGetDevice(&c->device) != cudaSuccess) {
        cudaGetLastError();
        delete c;
        return fail(nullptr, LBPF_ECUDA, "lbpf_create: no CUDA device");
    }
    const double e2u = (dim == 2) ? 1.0 / 3.0 : 1.0 / 4.0;

    const char* kenv = getenv("LBPF_KERNEL");
    c->vec = *vec = *vec && vec_applies(L, domains, n_domains);

    int rc = LBPF_OK;
    long long max_n = 0;
    c->dd.resize(n_domains);
    for (int k = 0; k < n_domains && rc == LBPF_OK; ++k) {
        const lbpf_domain& d = domains[k];
        DomainDev& h = c->dd[k];
        memset(&h, 0, sizeof(h));
        h.nx = d.nx;
        h.ny = d.ny;
        h.nz = d.nz;
        h.bc = d.bc;
        if (d.bc) c->kind |= kStepWalls;
        h.px = c->vec ? (d.nx + 3) / 4 * 4 : d.nx;  // rows of whole vectors
        h.n = (long long)h.px * d.ny * d.nz;
        max_n = h.n > max_n ? h.n : max_n;
        // D_phi = (W0^2/tau0)(dt/dx^2), Eq. (LBE_RelaxationTime)
        h.Dphi = (d.W0 * d.W0 / d.tau0) * (d.dt / (d.dx * d.dx));
        h.qphi = d.dt / d.tau0;
        h.lambda = d.lambda > 0.0 ? d.lambda : d.kappa * d.tau0 / (kA2 * d.W0 * d.W0);
        // kappa = e^2 (eta_u - 1/2) dx^2 / dt, Eq. (ThermalDiffusivity)
        h.inv_eta_u = 1.0 / (d.kappa * d.dt / (e2u * d.dx * d.dx) + 0.5);
        h.xi_lu = d.xi * d.dx;
        const double De2 = h.Dphi / D2Q9::E2, xi32 = std::max(h.xi_lu, 1e-6);
        h.r64 = {De2, 1.0 / (De2 + 0.5), h.qphi, h.lambda, h.inv_eta_u, h.xi_lu * h.xi_lu};
        h.r32 = {(float)De2, (float)h.r64.ieta1, (float)h.qphi, (float)h.lambda, (float)h.inv_eta_u, (float)(xi32 * xi32)};
        // advective heat equilibrium: a = v dt / (dx e^2)
        h.advect = d.adv[0] != 0.0 || d.adv[1] != 0.0 || d.adv[2] != 0.0;
        if (h.advect) c->kind |= kStepAdvect;
        for (int a = 0; a < 3; ++a) h.adv[a] = d.adv[a] * d.dt / (d.dx * e2u);
        h.n_crystals = d.n_crystals;
        h.use_index = d.n_crystals > 1;
        for (int j = 0; j < d.n_crystals; ++j) {
            h.cr[j].kind = d.crystals[j].kind;
            h.cr[j].q = d.crystals[j].q;
            const lbpf_crystal& cr = d.crystals[j];
            h.cr[j].r64 = {cr.eps, cr.gamma, cr.phi0};
            h.cr[j].r32 = {(float)cr.eps, (float)cr.gamma, (float)cr.phi0};
        }
        for (int b = 0; b < 2 && rc == LBPF_OK; ++b) {
            rc = dev_alloc(c, &h.g[b], (size_t)c->Sg * h.n * c->ssize);
            if (rc == LBPF_OK) rc = dev_alloc(c, &h.f[b], (size_t)c->Su * h.n * c->ssize);
            if (rc == LBPF_OK) rc = dev_alloc(c, &h.phi[b], (size_t)h.n * c->rsize);
            if (rc == LBPF_OK) rc = dev_alloc(c, &h.aux[b], (size_t)h.n * c->rsize);
            if (rc == LBPF_OK && h.use_index) rc = dev_alloc(c, reinterpret_cast<void**>(&h.I[b]), (size_t)h.n);
            if (rc == LBPF_OK && h.advect) rc = dev_alloc(c, &h.U[b], (size_t)h.n * c->rsize);
        }
        if (rc == LBPF_OK && c->vec) rc = dev_alloc(c, &h.u_work, (size_t)h.n * c->rsize);
        // zero state so that an unseeded domain holds finite values
        for (int b = 0; b < 2 && rc == LBPF_OK; ++b) {
            if (cudaMemsetAsync(h.g[b], 0, (size_t)c->Sg * h.n * c->ssize, c->stream) != cudaSuccess ||
                cudaMemsetAsync(h.f[b], 0, (size_t)c->Su * h.n * c->ssize, c->stream) != cudaSuccess ||
                cudaMemsetAsync(h.phi[b], 0, (size_t)h.n * c->rsize, c->stream) != cudaSuccess ||
                cudaMemsetAsync(h.aux[b], 0, (size_t)h.n * c->rsize, c->stream) != cudaSuccess ||
                (h.use_index && cudaMemsetAsync(h.I[b], 0, (size_t)h.n, c->stream) != cudaSuccess) ||
                (h.advect && cudaMemsetAsync(h.U[b], 0, (size_t)h.n * c->rsize, c->stream) != cudaSuccess))
                rc = fail(c, LBPF_ECUDA, "lbpf_create: cudaMemsetAsync failed");
        }
    }
    if (rc == LBPF_OK) {
        // the staged kernel (opt-in: it measured slower than the generic one,
        // see staged_kernel.cuh) needs 16-byte aligned row copies (nx a
        // multiple of 8), rows wider than the staged 48-site window, one crystal
        c->staged = L->step_staged != nullptr && kenv && strcmp(kenv, "staged") == 0;
        for (const DomainDev& h : c->dd)
            if (h.nx % 8 != 0 || h.nx < 64 || h.use_index || h.bc || h.advect) c->staged = false;
        if (cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess || c->sms < 1)
            c->sms = 1;
        for (int v = 0; v < kNumTileVariants && rc == LBPF_OK; ++v) {
            cudaError_t e = L->prepare(v);
            if (e != cudaSuccess) rc = fail(c, LBPF_ECUDA, "lbpf_create: kernel attribute: %s", cudaGetErrorString(e));
        }
    }
    if (rc == LBPF_OK) rc = dev_alloc(c, reinterpret_cast<void**>(&c->d_counters), sizeof(int) * 8);
    if (rc == LBPF_OK && cudaMemsetAsync(c->d_counters, 0, sizeof(int) * 8, c->stream) != cudaSuccess)
        rc = fail(c, LBPF_ECUDA, "lbpf_create: cudaMemsetAsync failed");
    if (rc == LBPF_OK) rc = dev_alloc(c, reinterpret_cast<void**>(&c->d_dd), sizeof(DomainDev) * n_domains);
    if (rc == LBPF_OK) {
        c->scratch_bytes = (size_t)max_n * (c->rsize > 4 ? c->rsize : 4);
        rc = dev_alloc(c, &c->scratch, c->scratch_bytes);
    }
    if (rc == LBPF_OK) rc = dev_alloc(c, reinterpret_cast<void**>(&c->red), sizeof(double) * (3 * kReduceBlocks + 16));
    if (rc == LBPF_OK) {
        rc = dev_alloc(c, reinterpret_cast<void**>(&c->d_hist), sizeof(double) * 7 * kHistCap * n_domains);
        c->hist_count.assign(n_domains, 0);
        c->hist_last.assign(n_domains, kHistCap - 1);
    }
    if (rc == LBPF_OK) {
        if (cudaMemcpyAsync(c->d_dd, c->dd.data(), sizeof(DomainDev) * n_domains, cudaMemcpyHostToDevice, c->stream) !=
            cudaSuccess)
            rc = fail(c, LBPF_ECUDA, "lbpf_create: copying the domain table failed");
    }
    if (rc == LBPF_OK && cudaStreamSynchronize(c->stream) != cudaSuccess)
        rc = fail(c, LBPF_ECUDA, "lbpf_create: stream synchronisation failed");
    if (rc == LBPF_OK) rc = initial_schedule(c);
    if (rc != LBPF_OK) {
        t_err = c->err;
        free_all(c);
        delete c;
        return rc;
    }
    *out = c;
    return LBPF_OK;
}

extern "C" int lbpf_create(const lbpf_domain* domains, int n_domains, int lattice, int grad, int precision,
                           void* stream, lbpf_ctx** out)
{
    bool vec = true;
    int rc = create(domains, n_domains, lattice, grad, precision, stream, &vec, out);
    if (rc == LBPF_ENOMEM && vec) {  // its work field (4 B a site) and row padding may be what does not fit
        vec = false;
        rc = create(domains, n_domains, lattice, grad, precision, stream, &vec, out);
    }
    return rc;
}

static int check_ctx(lbpf_ctx* c, int domain)
{
    if (!c) return fail(nullptr, LBPF_EINVAL, "context is NULL");
    if (domain < 0 || domain >= c->n_domains) return fail(c, LBPF_EINVAL, "domain %d out of range", domain);
    if (cudaSetDevice(c->device) != cudaSuccess) return fail(c, LBPF_ECUDA, "cudaSetDevice(%d) failed", c->device);
    return LBPF_OK;
}

// The device error word (set by a bounded wait of the staged kernel that
// gave up); read after the stream has been synchronised.
static int device_error(lbpf_ctx* c)
{
    if (!c->staged) return LBPF_OK;  // no other kernel sets it
    int w = 0;
    CK(cudaMemcpy(&w, c->d_counters + 4, sizeof(int), cudaMemcpyDeviceToHost));
    if (w) return fail(c, LBPF_ETIMEOUT, "a bounded wait in the step kernel gave up (device error word %d)", w);
    return LBPF_OK;
}

// Lagged -> synchronised: the heat update of the last step on every domain.
static int sync_state(lbpf_ctx* c)
{
    if (!c->lagged) return LBPF_OK;
    if (c->vec && c->precision != LBPF_FP32_FP16DEV_SR) {
        // the vector step's heat launch is this update (it also fills its work
        // field; the stochastic form rounds differently here)
        StepArgs a = step_args(c);
        a.collide = 1;
        CK(c->L->heat_vec(c->dd.data(), c->d_dd, c->n_domains, a, c->stream));
    } else {
        CK(c->L->heat_sync(c->dd.data(), c->d_dd, c->n_domains, c->cur, c->fcur, c->acur, c->stream));
    }
    c->fcur ^= 1;
    if (c->Sg != c->Qg) c->acur ^= 1;
    c->lagged = 0;
    return LBPF_OK;
}

extern "C" int lbpf_seed(lbpf_ctx* c, int domain, const lbpf_seed_t* seeds, int n_seeds)
{
    int rc = check_ctx(c, domain);
    if (rc) return rc;
    if (!seeds || n_seeds < 1 || n_seeds > 4096) return fail(c, LBPF_EINVAL, "lbpf_seed: need 1..4096 seeds");
    const lbpf_domain& d = c->in[domain];
    std::vector<double> h(5 * (size_t)n_seeds);
    for (int j = 0; j < n_seeds; ++j) {
        const lbpf_seed_t& s = seeds[j];
        if (s.crystal < 0 || s.crystal >= d.n_crystals)
            return fail(c, LBPF_EINVAL, "lbpf_seed: seed %d crystal %d out of range", j, s.crystal);
        if (!std::isfinite(s.x) || !std::isfinite(s.y) || !std::isfinite(s.z) || !std::isfinite(s.radius))
            return fail(c, LBPF_EINVAL, "lbpf_seed: seed %d not finite", j);
        h[5 * j + 0] = s.x;
        h[5 * j + 1] = s.y;
        h[5 * j + 2] = s.z;
        h[5 * j + 3] = s.radius;
        h[5 * j + 4] = s.crystal;
    }
    if ((rc = sync_state(c))) return rc;
    if (n_seeds > c->seeds_cap) {
        void* p = nullptr;
        if ((rc = dev_alloc(c, &p, sizeof(double) * 5 * n_seeds))) return rc;
        c->d_seeds = static_cast<double*>(p);
        c->seeds_cap = n_seeds;
    }
    CK(cudaMemcpyAsync(c->d_seeds, h.data(), sizeof(double) * h.size(), cudaMemcpyHostToDevice, c->stream));
    CK(launch_seed(c->d_dd + domain, c->dd[domain].n, c->cur, c->acur, c->precision, c->d_seeds, n_seeds, c->dim,
                   d.dx / (std::sqrt(2.0) * d.W0), -d.delta, c->stream));
    CK(c->L->equilibrate(c->d_dd + domain, c->cur, c->fcur, c->acur, c->grad, 1, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    c->steps = 0;
    c->hist_count[domain] = 0;
    return LBPF_OK;
}

// Sites of a domain (its arrays may hold row padding besides).
static long long sites_of(const DomainDev& h) { return (long long)h.nx * h.ny * h.nz; }

// A field of the arithmetic type between an array of the context (own, row pitch
// h.px) and a dense one of the caller's, host or device.  Padded rows (only with
// FP32 arithmetic) go through the context's scratch on their way from or to the
// host, in one dense copy.
static cudaError_t put_field(lbpf_ctx* c, const DomainDev& h, void* own, const void* from, cudaMemcpyKind kind)
{
    const size_t bytes = (size_t)sites_of(h) * c->rsize;
    if (h.px == h.nx) return cudaMemcpyAsync(own, from, bytes, kind, c->stream);
    if (kind == cudaMemcpyHostToDevice || ((uintptr_t)from & 3)) {
        const cudaError_t e = cudaMemcpyAsync(c->scratch, from, bytes, kind, c->stream);
        if (e != cudaSuccess) return e;
        from = c->scratch;
    }
    return launch_copy_rows(static_cast<float*>(own), h.px, static_cast<const float*>(from), h.nx, h.nx,
                            (long long)h.ny * h.nz, c->stream);
}
static cudaError_t get_field(lbpf_ctx* c, const DomainDev& h, void* to, const void* own, cudaMemcpyKind kind)
{
    const size_t bytes = (size_t)sites_of(h) * c->rsize;
    if (h.px == h.nx) return cudaMemcpyAsync(to, own, bytes, kind, c->stream);
    const bool direct = kind == cudaMemcpyDeviceToDevice && !((uintptr_t)to & 3);
    const cudaError_t e = launch_copy_rows(static_cast<float*>(direct ? to : c->scratch), h.nx,
                                           static_cast<const float*>(own), h.px, h.nx, (long long)h.ny * h.nz, c->stream);
    if (e != cudaSuccess || direct) return e;
    return cudaMemcpyAsync(to, c->scratch, bytes, kind, c->stream);
}

extern "C" int lbpf_write_fields(lbpf_ctx* c, int domain, const void* phi, const void* u, const int* index,
                                 int on_device)
{
    int rc = check_ctx(c, domain);
    if (rc) return rc;
    if (!phi || !u) return fail(c, LBPF_EINVAL, "lbpf_write_fields: phi and u are required");
    if ((rc = sync_state(c))) return rc;
    const DomainDev& h = c->dd[domain];
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    CK(put_field(c, h, h.phi[c->cur], phi, kind));
    CK(put_field(c, h, h.aux[c->acur], u, kind));
    if (h.use_index) {
        if (index) {
            CK(cudaMemcpyAsync(c->scratch, index, sizeof(int) * h.n, kind, c->stream));
            CK(launch_index_from_i32(static_cast<const int*>(c->scratch), h.I[c->cur], h.n, h.n_crystals, c->stream));
        } else {
            CK(launch_fill_i8(h.I[c->cur], 0, h.n, c->stream));
        }
    }
    CK(c->L->equilibrate(c->d_dd + domain, c->cur, c->fcur, c->acur, c->grad, 0, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    c->steps = 0;
    c->hist_count[domain] = 0;
    return LBPF_OK;
}

// One launch of the fused step on the context's stream.
static int launch_step(lbpf_ctx* c)
{
    const StepArgs a = step_args(c);
    CK(issue_step(c, a));
    c->cur ^= 1;
    c->acur ^= 1;
    if (c->lagged) c->fcur ^= 1;
    c->lagged = 1;
    c->steps += 1;
    c->kernels += launches_per_step(c);
    return LBPF_OK;
}

// Steady-state launches come in batches of kGraphSteps replayed from a CUDA
// graph; the launch arguments of a batch depend only on the buffer parities
// (cur, fcur, acur), which return to their start after an even batch.
constexpr int kGraphSteps = 16;

static int graph_batch(lbpf_ctx* c)
{
    const int key = c->cur | (c->fcur << 1) | (c->acur << 2);
    cudaGraphExec_t& ex = c->graphs[key];
    if (!ex) {
        const int cur = c->cur, fcur = c->fcur, acur = c->acur;
        const long long steps = c->steps, kernels = c->kernels;
        cudaGraph_t g = nullptr;
        if (cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
            cudaGetLastError();
            c->graphs_off = true;
            return LBPF_OK;
        }
        int rc = LBPF_OK;
        for (int k = 0; k < kGraphSteps && rc == LBPF_OK; ++k) rc = launch_step(c);
        cudaError_t e = cudaStreamEndCapture(c->stream, &g);
        c->cur = cur;  // capture recorded the launches without running them
        c->fcur = fcur;
        c->acur = acur;
        c->steps = steps;
        c->kernels = kernels;
        if (rc != LBPF_OK || e != cudaSuccess || cudaGraphInstantiate(&ex, g, 0) != cudaSuccess) {
            cudaGetLastError();
            if (g) cudaGraphDestroy(g);
            ex = nullptr;
            c->graphs_off = true;
            return LBPF_OK;
        }
        cudaGraphDestroy(g);
    }
    CK(cudaGraphLaunch(ex, c->stream));
    c->steps += kGraphSteps;
    c->kernels += kGraphSteps * launches_per_step(c);
    return LBPF_OK;
}

extern "C" int lbpf_step(lbpf_ctx* c, int n_steps)
{
    int rc = check_ctx(c, 0);
    if (rc) return rc;
    if (n_steps < 0) return fail(c, LBPF_EINVAL, "lbpf_step: n_steps < 0");
    if (c->tune_pending && n_steps > 0) {
        c->tune_pending = false;
        if ((rc = autotune(c))) return rc;
    }
    // graphs need a capturable stream (not the legacy default stream)
    const bool graphs = c->stream != nullptr && !c->graphs_off;
    while (n_steps > 0) {
        if (graphs && c->lagged && n_steps >= kGraphSteps && !c->graphs_off) {
            if ((rc = graph_batch(c))) return rc;
            if (!c->graphs_off) {
                n_steps -= kGraphSteps;
                continue;
            }
        }
        if ((rc = launch_step(c))) return rc;
        n_steps -= 1;
    }
    return LBPF_OK;
}

// Element size of a field selected by one LBPF_READ_* bit.
static size_t field_esize(const lbpf_ctx* c, unsigned bit) { return bit == LBPF_READ_INDEX ? sizeof(int) : c->rsize; }

extern "C" int lbpf_read_fields(lbpf_ctx* c, int domain, unsigned mask, void* out, int out_on_device, size_t out_bytes)
{
    int rc = check_ctx(c, domain);
    if (rc) return rc;
    constexpr unsigned kAll = LBPF_READ_PHI | LBPF_READ_U | LBPF_READ_AS | LBPF_READ_INDEX;
    if (!out) return fail(c, LBPF_EINVAL, "lbpf_read_fields: out is NULL");
    if (mask == 0 || (mask & ~kAll)) return fail(c, LBPF_EINVAL, "lbpf_read_fields: bad mask 0x%x", mask);
    const DomainDev& h = c->dd[domain];
    size_t need = 0;
    for (unsigned bit = 1; bit <= LBPF_READ_INDEX; bit <<= 1)
        if (mask & bit) need += (size_t)sites_of(h) * field_esize(c, bit);
    if (out_bytes < need) return fail(c, LBPF_ERANGE, "lbpf_read_fields: need %zu bytes, got %zu", need, out_bytes);
    if (mask & LBPF_READ_U)
        if ((rc = sync_state(c))) return rc;
    const cudaMemcpyKind kind = out_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    char* o = static_cast<char*>(out);
    for (unsigned bit = 1; bit <= LBPF_READ_INDEX; bit <<= 1) {
        if (!(mask & bit)) continue;
        const size_t bytes = (size_t)sites_of(h) * field_esize(c, bit);
        // fields that need a kernel are written in place (device output) or
        // into the context's scratch and copied from there (host output); the
        // copies run in stream order, so the scratch is free again for the
        // next field without a synchronisation
        void* dst = out_on_device ? static_cast<void*>(o) : c->scratch;
        switch (bit) {
        case LBPF_READ_PHI:
            CK(get_field(c, h, o, h.phi[c->cur], kind));
            dst = nullptr;
            break;
        case LBPF_READ_U: CK(c->L->read_u(c->d_dd + domain, c->cur, c->fcur, c->acur, dst, c->stream)); break;
        case LBPF_READ_AS: CK(c->L->read_as(c->d_dd + domain, c->cur, c->grad, dst, c->stream)); break;
        case LBPF_READ_INDEX:
            if (h.use_index)
                CK(launch_index_to_i32(h.I[c->cur], static_cast<int*>(dst), sites_of(h), c->stream));
            else
                CK(launch_fill_i32(static_cast<int*>(dst), 1, sites_of(h), c->stream));
            break;
        }
        if (dst && !out_on_device) CK(cudaMemcpyAsync(o, dst, bytes, cudaMemcpyDeviceToHost, c->stream));
        o += bytes;
    }
    CK(cudaStreamSynchronize(c->stream));
    return device_error(c);
}

extern "C" int lbpf_read_field(lbpf_ctx* c, int domain, int field, void* out, int out_on_device, size_t out_bytes)
{
    static const unsigned bits[4] = {LBPF_READ_PHI, LBPF_READ_U, LBPF_READ_INDEX, LBPF_READ_AS};
    if (field < LBPF_FIELD_PHI || field > LBPF_FIELD_AS) {
        int rc = check_ctx(c, domain);
        return rc ? rc : fail(c, LBPF_EINVAL, "lbpf_read_field: bad field %d", field);
    }
    return lbpf_read_fields(c, domain, bits[field], out, out_on_device, out_bytes);
}

extern "C" int lbpf_read_populations(lbpf_ctx* c, int domain, int which, void* out, int out_on_device, size_t out_bytes)
{
    int rc = check_ctx(c, domain);
    if (rc) return rc;
    if (!out || (which != 0 && which != 1)) return fail(c, LBPF_EINVAL, "lbpf_read_populations: bad arguments");
    const DomainDev& h = c->dd[domain];
    const int Q = which == 0 ? c->Qg : c->Qu;
    const size_t one = (size_t)sites_of(h) * c->rsize, bytes = (size_t)Q * one;
    if (out_bytes < bytes) return fail(c, LBPF_ERANGE, "lbpf_read_populations: need %zu bytes, got %zu", bytes, out_bytes);
    if ((rc = sync_state(c))) return rc;
    // one population at a time, host reads through the context's scratch
    for (int i = 0; i < Q; ++i) {
        char* o = static_cast<char*>(out) + (size_t)i * one;
        void* dst = out_on_device ? static_cast<void*>(o) : c->scratch;
        CK(c->L->read_pop(c->d_dd + domain, which, i, c->cur, c->fcur, c->acur, dst, c->stream));
        if (!out_on_device) CK(cudaMemcpyAsync(o, dst, one, cudaMemcpyDeviceToHost, c->stream));
    }
    CK(cudaStreamSynchronize(c->stream));
    return LBPF_OK;
}

extern "C" int lbpf_measure(lbpf_ctx* c, int domain, int cx, int cy, int cz, double* tip6, double* solid_fraction,
                            double* conserved)
{
    int rc = check_ctx(c, domain);
    if (rc) return rc;
    const DomainDev& h = c->dd[domain];
    if (cx < 0 || cx >= h.nx || cy < 0 || cy >= h.ny || cz < 0 || cz >= h.nz)
        return fail(c, LBPF_EINVAL, "lbpf_measure: centre (%d, %d, %d) outside the domain", cx, cy, cz);
    if ((rc = sync_state(c))) return rc;
    CK(c->L->read_u(c->d_dd + domain, c->cur, c->fcur, c->acur, c->scratch, c->stream));
    double* outp = c->red + 3 * kReduceBlocks;
    CK(launch_reduce(h.phi[c->cur], c->scratch, sites_of(h), c->precision, c->red, outp, c->stream, h.nx, h.ny, h.nz,
                     h.bc, c->dim, h.px));
    CK(launch_tips(h.phi[c->cur], h.nx, h.ny, h.nz, cx, cy, cz, c->dim, c->precision, outp + 3, c->stream, h.bc,
                   h.px));
    {
        const int slot = (c->hist_last[domain] + 1) % kHistCap;
        CK(launch_hist_append(outp + 3, (double)c->steps * c->in[domain].dt,
                              c->d_hist + 7 * ((size_t)domain * kHistCap + slot), c->stream));
        c->hist_last[domain] = slot;
        if (c->hist_count[domain] < kHistCap) c->hist_count[domain] += 1;
    }
    double hv[9];
    CK(cudaMemcpyAsync(hv, outp, sizeof(hv), cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    if (tip6)
        for (int k = 0; k < 6; ++k) tip6[k] = hv[3 + k];
    if ((rc = device_error(c))) return rc;
    if (solid_fraction) *solid_fraction = hv[0] / (double)sites_of(h);
    if (conserved) *conserved = hv[1];
    if (hv[2] > 0) return fail(c, LBPF_ENONFINITE, "lbpf_measure: %.0f non-finite values in phi or u", hv[2]);
    return LBPF_OK;
}

extern "C" int lbpf_tip_velocity(lbpf_ctx* c, int domain, int window, double* v6)
{
    int rc = check_ctx(c, domain);
    if (rc) return rc;
    if (!v6 || window < 2) return fail(c, LBPF_EINVAL, "lbpf_tip_velocity: need v6 and window >= 2");
    if (c->hist_count[domain] < 2)
        return fail(c, LBPF_EINVAL, "lbpf_tip_velocity: fewer than two measurements since the last seed");
    double* out = c->red + 3 * kReduceBlocks + 9;
    CK(launch_tip_velocity(c->d_hist + 7 * (size_t)domain * kHistCap, kHistCap, c->hist_last[domain],
                           c->hist_count[domain], window, c->in[domain].dx, out, c->stream));
    CK(cudaMemcpyAsync(v6, out, 6 * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    return LBPF_OK;
}

extern "C" int lbpf_tip_radius(lbpf_ctx* c, int domain, int cx, int cy, int cz, int dir, int J, double* rho)
{
    int rc = check_ctx(c, domain);
    if (rc) return rc;
    const DomainDev& h = c->dd[domain];
    if (!rho || dir < 0 || dir >= 2 * c->dim || J < 1 || (2 * J + 1) * (c->dim - 1) > 32)
        return fail(c, LBPF_EINVAL, "lbpf_tip_radius: bad direction or J (1..15 in 2D, 1..7 in 3D)");
    if (cx < 0 || cx >= h.nx || cy < 0 || cy >= h.ny || cz < 0 || cz >= h.nz)
        return fail(c, LBPF_EINVAL, "lbpf_tip_radius: centre outside the domain");
    double* out = c->red + 3 * kReduceBlocks + 15;
    CK(launch_tip_radius(h.phi[c->cur], h.nx, h.ny, h.nz, cx, cy, cz, dir, J, c->dim, c->precision, out, c->stream,
                         h.bc, h.px));
    CK(cudaMemcpyAsync(rho, out, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    return LBPF_OK;
}

extern "C" int lbpf_set_schedule(lbpf_ctx* c, int tile_rows, int segment)
{
    int rc = check_ctx(c, 0);
    if (rc) return rc;
    int v = -1;
    for (int k = 0; k < kNumTileVariants; ++k)
        if (kTileRows[k] == tile_rows) v = k;
    if (v < 0 || segment < 1) return fail(c, LBPF_EINVAL, "lbpf_set_schedule: tile_rows must be 8 or 16, segment >= 1");
    if ((c->staged || c->kind) && v != 0)
        return fail(c, LBPF_EINVAL,
                    "lbpf_set_schedule: 16-row tiles exist only for periodic domains without advection (generic kernel)");
    CK(cudaStreamSynchronize(c->stream));
    c->tune_pending = false;
    c->tuned = "set";
    return set_schedule(c, v, segment);
}

extern "C" int lbpf_query(const lbpf_ctx* c, int what, double* value)
{
    if (!c || !value) return fail(nullptr, LBPF_EINVAL, "lbpf_query: NULL argument");
    double v = 0;
    switch (what) {
    case LBPF_Q_SITES:
        for (const DomainDev& h : c->dd) v += (double)sites_of(h);
        break;
    case LBPF_Q_STEPS: v = (double)c->steps; break;
    case LBPF_Q_BYTES_PER_SITE: {
        // read + write of every stored population, of phi and of aux (and of
        // the index field when it is used)
        double idx_sites = 0, all_sites = 0;
        for (const DomainDev& h : c->dd) {
            all_sites += (double)sites_of(h);
            if (h.use_index) idx_sites += (double)sites_of(h);
        }
        v = 2.0 * (c->Sg + c->Su) * c->ssize + 4.0 * c->rsize + 2.0 * idx_sites / all_sites;
        break;
    }
    case LBPF_Q_DEVICE_BYTES: v = (double)c->dev_bytes; break;
    case LBPF_Q_LAMBDA: v = c->dd[0].lambda; break;
    case LBPF_Q_STEP_KERNELS: v = (double)c->kernels; break;
    case LBPF_Q_TILE_ROWS: v = kTileRows[c->tile_v]; break;
    case LBPF_Q_SEGMENT: v = c->seg_len; break;
    case LBPF_Q_BLOCKS: v = c->n_blocks; break;
    case LBPF_Q_KERNEL: v = c->staged ? 1 : 0; break;
    case LBPF_Q_STEP_FORM: v = c->staged ? 1 : c->vec ? 2 : c->tile ? 3 : 0; break;
    default: return fail(const_cast<lbpf_ctx*>(c), LBPF_EINVAL, "lbpf_query: unknown property %d", what);
    }
    *value = v;
    return LBPF_OK;
}

extern "C" int lbpf_destroy(lbpf_ctx* c)
{
    if (!c) return LBPF_OK;
    cudaSetDevice(c->device);
    cudaStreamSynchronize(c->stream);
    for (cudaGraphExec_t g : c->graphs)
        if (g) cudaGraphExecDestroy(g);
    free_all(c);
    delete c;
    return LBPF_OK;
}

extern "C" const char* lbpf_last_error(const lbpf_ctx* c) { return c ? c->err.c_str() : t_err.c_str(); }
