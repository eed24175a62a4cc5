// Kernels of the learned surrogate: a 2D U-Net on periodic fields, NHWC
// activations in FP32, 3x3 convolutions on the 5th-generation tensor cores
// (tcgen05.mma, BF16 operands, FP32 accumulation in tensor memory), the small
// layers on the CUDA cores in FP32.
//
// Layouts:
//   activations  x[n][h][w][c]            (c fastest), FP32
//   3x3 weights  w[tap][cout][cin]        BF16 (tap = 3 * (dy + 1) + (dx + 1))
//   weight grads dw[tap][cout][cin]       FP32
//   1x1 weights  w[cout][cin]             FP32
// Convolutions are periodic ("same" size, wrap-around), matching the periodic
// lattice Boltzmann domains.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "lbpf_nn.cuh"

namespace lbpf_nn {

// ---- 3x3 convolution as an implicit GEMM on the 5th-generation tensor cores
//
// y[p][co] = act(sum_tap sum_ci x[p + tap][ci] w[tap][co][ci] + b[co]):
// D (M = 128 pixels of the flattened (n, h, w) order) x (N = a tile of at
// most 256 output channels, grid y) with K = 9 cin, one
// tcgen05.mma.kind::f16 (BF16 x BF16 -> FP32, M = 128, N = the tile, K = 16)
// per 16 input channels of one tap, the accumulator in tensor memory (TMEM).  The K loop runs over stages (tap, block of KC input channels), two
// stage buffers in shared memory: while the tensor core works on stage s - 1,
// the 128 threads gather stage s — each thread one pixel row of A (the tap's
// neighbour, periodic in h and w, FP32 -> BF16) and the weight pieces of B
// (cp.async) — into the no-swizzle K-major layout: 8-row x 16-byte core
// matrices, rows of a core matrix 16 bytes apart, 8-row groups 128 bytes
// apart (SBO), 8-channel K slices one matrix apart (LBO).  One thread issues
// the MMAs of a stage and commits them to the stage buffer's mbarrier, which
// the gatherers of stage s + 2 wait on before they overwrite the buffer.
// The epilogue reads the accumulator rows with tcgen05.ld (warp w owns TMEM
// lanes 32w .. 32w + 31 = pixels), adds the bias, applies the ReLU and
// stores FP32.  Waits are bounded (2 s by %globaltimer); on expiry the block
// sets the error word and stops (conv_error()).

__device__ int g_conv_error;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start, LBO, SBO (bytes, multiples of 16),
// no swizzle, descriptor version 1 (bits 46-48 = 0b001)
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void umma_commit(uint64_t* mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar))
                 : "memory");
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for the completion of phase `parity` of an mbarrier, at most ~2 s (each
// try suspends for at most 0.1 ms);
// false on expiry.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* mbar, uint32_t parity)
{
    const uint32_t a = smem_u32(mbar);
    unsigned long long t0 = 0;  // the clock is read only once the first waits fail
    for (int n = 0;; ++n) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(a), "r"(parity), "r"(100000u)
            : "memory");
        if (ok) return true;
        if (n < 4) continue;
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 > 2000000000ull) return false;
    }
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

constexpr int kConvM = 128;  // pixels per block (one TMEM lane each)

__global__ void __launch_bounds__(kConvM) conv3x3_tc_kernel(const float* __restrict__ x,
                                                            const __nv_bfloat16* __restrict__ w,
                                                            const float* __restrict__ bias, float* __restrict__ y,
                                                            long long P, int H, int W, int cin, int cout_all,
                                                            int cout, int KC, int relu, uint32_t tmem_cols)
{
    // output channels co0 .. co0 + cout of cout_all (grid y: channel tile)
    const int co0 = blockIdx.y * cout;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_mbar[2];
    const int tid = threadIdx.x, warp = tid >> 5;
    const size_t a_bytes = (size_t)kConvM * KC * 2, b_bytes = (size_t)cout * KC * 2;
    auto sA = [&](int b) { return smem_raw + b * a_bytes; };
    auto sB = [&](int b) { return smem_raw + 2 * a_bytes + b * b_bytes; };

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_mbar[0])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_mbar[1])));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;

    // this thread's pixel row
    const long long p = (long long)blockIdx.x * kConvM + tid;
    const bool valid = p < P;
    const long long HW = (long long)H * W;
    const long long img = valid ? p / HW : 0;
    const int rem = valid ? (int)(p - img * HW) : 0;
    const int py = rem / W, px = rem - py * W;
    const float* ximg = x + img * HW * cin;

    const int nkb = cin / KC, S = 9 * nkb;
    const uint32_t idesc = umma_idesc_bf16(kConvM, cout);
    bool ok = true;
    int issued = 0;  // stages committed
    for (int s = 0; s < S && ok; ++s) {
        const int buf = s & 1, tap = s / nkb, c0 = (s - tap * nkb) * KC;
        if (s >= 2 && !mbar_wait_bounded(&s_mbar[buf], ((s - 2) >> 1) & 1)) {
            atomicOr(&g_conv_error, 1);
            ok = false;  // the buffer stays as it is; the block leaves together below
        }
        // A: row tid = x at the tap's neighbour, channels c0 .. c0 + KC
        if (ok) {
            const int dy = tap / 3 - 1, dx = tap % 3 - 1;
            int yy = py + dy, xx = px + dx;
            yy = yy < 0 ? yy + H : (yy >= H ? yy - H : yy);
            xx = xx < 0 ? xx + W : (xx >= W ? xx - W : xx);
            const float4* src = reinterpret_cast<const float4*>(ximg + ((long long)yy * W + xx) * cin + c0);
            unsigned char* dst = sA(buf) + tid * 16;
            for (int k8 = 0; k8 < KC / 8; ++k8) {
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (valid) {
                    const float4 f0 = __ldg(src + 2 * k8), f1 = __ldg(src + 2 * k8 + 1);
                    v = make_uint4(pack_bf16(f0.x, f0.y), pack_bf16(f0.z, f0.w), pack_bf16(f1.x, f1.y),
                                   pack_bf16(f1.z, f1.w));
                }
                *reinterpret_cast<uint4*>(dst + (size_t)k8 * kConvM * 16) = v;
            }
        }
        // B: 16-byte pieces w[tap][co][c0 + 8 k8 ..] -> [k8][co]
        for (int e = tid; ok && e < cout * (KC / 8); e += kConvM) {
            const int co = e % cout, k8 = e / cout;
            const __nv_bfloat16* g = w + ((size_t)tap * cout_all + co0 + co) * cin + c0 + 8 * k8;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             smem_u32(sB(buf) + (size_t)k8 * cout * 16 + co * 16)),
                         "l"(g));
        }
        asm volatile("cp.async.commit_group;");
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        ok = __syncthreads_and(ok) != 0;
        if (!ok) break;
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t a0 = smem_u32(sA(buf)), b0 = smem_u32(sB(buf));
            for (int k16 = 0; k16 < KC / 16; ++k16) {
                const uint64_t ad = umma_desc(a0 + k16 * 2 * kConvM * 16, kConvM * 16, 128);
                const uint64_t bd = umma_desc(b0 + k16 * 2 * cout * 16, cout * 16, 128);
                umma_bf16(tmem, ad, bd, idesc, (s > 0 || k16 > 0) ? 1u : 0u);
            }
            umma_commit(&s_mbar[buf]);
        }
        issued = s + 1;
    }
    // the last committed stage covers every MMA issued before it
    bool done = false;
    if (issued > 0) {
        const int last = issued - 1;
        done = mbar_wait_bounded(&s_mbar[last & 1], (last >> 1) & 1);
        if (!done) atomicOr(&g_conv_error, 2);
    }
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (__all_sync(0xffffffffu, ok && done)) {  // the loads below are the whole warp's
        float* out = y + p * cout_all + co0;
        for (int c = 0; c < cout; c += 8) {
            uint32_t r[8];
            __syncwarp();
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                           "=r"(r[7])
                         : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (valid) {
                float v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    v[j] = __uint_as_float(r[j]) + (bias ? bias[co0 + c + j] : 0.f);
                    if (relu) v[j] = fmaxf(v[j], 0.f);
                }
                reinterpret_cast<float4*>(out + c)[0] = make_float4(v[0], v[1], v[2], v[3]);
                reinterpret_cast<float4*>(out + c)[1] = make_float4(v[4], v[5], v[6], v[7]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols));
}

// Halo form of the same convolution for images whose H is a multiple of 16
// and W of 8, and layers whose halo fits in shared memory beside two stages of
// weights (halo_plan).  A tile is 16 x 8 pixels (M = 128: tile row = 8-row group, pixel
// in the row = row of the core matrix); its 18 x 10 halo of all cin channels
// is converted to BF16 once (layout [8-channel slice][halo pixel][8]), and
// every tap is a matrix descriptor over it: start at the tap's offset, SBO =
// one halo row (10 pixels x 16 bytes), LBO = one slice.  A slice is 181 pixels
// long (180 used): at 181 x 16 bytes the eight slices a quarter-warp stores
// fall into different banks (at 180, into two: 4-way conflicts).
//
// A block is persistent over tiles and its warps take different parts:
// warps 0-3 the epilogue (bias, ReLU, coalesced stores), 4-11 load and convert
// halos (two buffers where they fit), warp 12 issues the MMAs (two
// accumulators where they fit), 13-20 stream the weights through a ring where
// they don't all stay resident, a stage (KC channels of one tap) per warp, or,
// where KC is 64 channels, warp 13 alone by one TMA load a stage (rows of 64
// channels in the 128-byte swizzle; the per-piece copies of the eight warps
// kept the load/store pipe busy for 1800 cycles a stage: 256^2 128 -> 128 65 us,
// 29 us by TMA).  Every hand-over is an mbarrier with a bounded
// wait; on expiry a role sets the error word and leaves, the others follow.
// MMAs are issued tap by tap, 16 channels at a time, for every tile: the sum's
// order is that of the gather kernel.
//
// Measured, us (a block a tile, loads exposed / this): 1024^2 32 -> 32 190 / 64,
// 512^2 64 -> 64 129 / 52, 256^2 128 -> 128 97 / 29, 128^2 256 -> 256 95 / 25,
// 8 x 128^2 32 -> 32 32 / 18.  What bounds it: with few channels the halo loads'
// latency and their conversion (1024^2: 21 % of the DRAM rate, long_scoreboard
// 10 stalls an issue; other operand strides change nothing), with many the MMA
// issue of one thread (42 % of the BF16 peak at 256 channels).
constexpr int kHaloY = 18, kHaloX = 10, kHaloP = kHaloY * kHaloX, kHaloS = kHaloP + 1;
constexpr int kEpiT = 128, kLoadT = 256, kWtT = 256;
constexpr int kMaxWStages = kWtT / 32;  // a warp a slot
constexpr int kOutPitch = 36;  // floats a pixel of the store staging (32 + 4)

// Channels of the convolution's input: all cin from a, or (b set) the first ca
// from a at half the resolution (nearest 2x upsampling), the others from b.
// near: offsets of a tile's halo pixels fit in 32 bits (fill_halo_table).
struct ConvSrc {
    const float* a;
    const float* b;
    int ca, cb;
    bool near;
};
static ConvSrc conv_src(const float* a, const float* b, int ca, int cb, int W)
{
    return ConvSrc{a, b, ca, cb, (long long)W * (ca > cb ? ca : cb) <= 0x7fffffff / kHaloY};
}

__device__ __forceinline__ const float* src_at(const ConvSrc& s, int img, int y, int x, int H, int W, int c)
{
    if (!s.b) return s.a + (((size_t)img * H + y) * W + x) * s.ca + c;
    if (c < s.ca) return s.a + (((size_t)img * (H >> 1) + (y >> 1)) * (W >> 1) + (x >> 1)) * s.ca + c;
    return s.b + (((size_t)img * H + y) * W + x) * s.cb + (c - s.ca);
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}

// Offsets (floats) of the halo pixels from the tile's first pixel in the full
// resolution source and in the half resolution one, for tiles whose halo does
// not wrap: filled once a block, so that a piece's address is one table entry.
// Images so wide that an offset may not fit (rows of 1.2e8 floats) go without.
__device__ __forceinline__ void fill_halo_table(int* tab, const ConvSrc& s, int W, int t, int nt)
{
    if (!s.near) return;
    for (int hp = t; hp < kHaloP; hp += nt) {
        const int hy = hp / kHaloX - 1, hx = hp % kHaloX - 1;
        tab[hp] = (hy * W + hx) * (s.b ? s.cb : s.ca);
        tab[kHaloP + hp] = s.b ? ((hy >> 1) * (W >> 1) + (hx >> 1)) * s.ca : 0;
    }
}

// Halo pixels [r0, r0 + rows) x 10 of tile (img, ty0, tx0), channels c0 ..
// c0 + 8 k8n, as BF16 into dst ([slice][kHaloS pixels][8]), by threads t of nt:
// a thread keeps one 8-channel slice and takes every dq-th pixel, six 32-byte
// pieces in flight.  tab: fill_halo_table of the source.
__device__ __forceinline__ void load_halo(const ConvSrc& src, const int* tab, unsigned char* dst, int img, int ty0,
                                          int tx0, int H, int W, int c0, int k8n, int r0, int rows, int t, int nt)
{
    constexpr int B = 6;
    const int dq = nt / k8n;
    if (t >= dq * k8n) return;
    const int p0 = t / k8n, k8 = t - p0 * k8n, c = c0 + 8 * k8, end = rows * kHaloX;
    const bool inside = src.near && ty0 > 0 && tx0 > 0 && ty0 + 16 < H && tx0 + 8 < W;
    const bool half = src.b && c < src.ca;
    const float* base;
    if (!src.b)
        base = src.a + (((size_t)img * H + ty0) * W + tx0) * src.ca + c;
    else if (half)
        base = src.a + (((size_t)img * (H >> 1) + (ty0 >> 1)) * (W >> 1) + (tx0 >> 1)) * src.ca + c;
    else
        base = src.b + (((size_t)img * H + ty0) * W + tx0) * src.cb + (c - src.ca);
    const int* tb = tab + (half ? kHaloP : 0) + r0 * kHaloX;
    unsigned char* o = dst + ((size_t)k8 * kHaloS + p0) * 16;
    for (int hp = p0; hp < end; hp += B * dq, o += B * dq * 16) {
        float4 f[B][2];
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const int p = hp + j * dq;
            if (p < end) {
                const float* g;
                if (inside) {
                    g = base + tb[p];
                } else {
                    const int hy = p / kHaloX, hx = p - hy * kHaloX;
                    int gy = ty0 + r0 + hy - 1, gx = tx0 + hx - 1;
                    gy = gy < 0 ? gy + H : (gy >= H ? gy - H : gy);
                    gx = gx < 0 ? gx + W : (gx >= W ? gx - W : gx);
                    g = src_at(src, img, gy, gx, H, W, c);
                }
                f[j][0] = __ldg(reinterpret_cast<const float4*>(g));
                f[j][1] = __ldg(reinterpret_cast<const float4*>(g) + 1);
            }
        }
#pragma unroll
        for (int j = 0; j < B; ++j)
            if (hp + j * dq < end)
                *reinterpret_cast<uint4*>(o + j * dq * 16) =
                    make_uint4(pack_bf16(f[j][0].x, f[j][0].y), pack_bf16(f[j][0].z, f[j][0].w),
                               pack_bf16(f[j][1].x, f[j][1].y), pack_bf16(f[j][1].z, f[j][1].w));
    }
}

struct HaloArgs {
    ConvSrc src;
    const __nv_bfloat16* w;
    const float* bias;
    float* y;
    int H, W, n_tiles, cin, cout_all, cout, KC, relu;
    int nbuf, nacc, wst;  // halo buffers, accumulators, weight ring stages (0: resident)
    uint32_t tmem_cols;
};

// MMAs of one K block (16 k16n channels of one tap), K16 = k16n where it is known
// at compile time.
template <int K16>
__device__ __forceinline__ void umma_block(uint32_t d, uint64_t ad, uint64_t bd, uint32_t bstep, uint32_t idesc, int k16n,
                                           uint32_t more)
{
    if constexpr (K16 > 0) {
#pragma unroll
        for (int k = 0; k < K16; ++k) umma_bf16(d, ad + k * (2 * kHaloS), bd + k * bstep, idesc, k > 0 ? 1u : more);
    } else {
        for (int k = 0; k < k16n; ++k)
            umma_bf16(d, ad + k * (2 * kHaloS), bd + (uint64_t)k * bstep, idesc, k > 0 ? 1u : more);
    }
}

// MODE: the weights stay resident, or go through the ring.  K16: 16-channel steps of a K block
// (KC / 16; resident weights: cin / 16), 0 = any.  One thread issues a tile's
// MMAs in straight-line code: with a loop over taps and a warp-wide branch in
// each, an MMA took 150-300 cycles to issue, several times its execution.
enum { kResident, kStream, kTma };  // where the weights come from
constexpr int halo_threads(int mode) { return kEpiT + kLoadT + 32 + (mode == kStream ? kWtT : mode == kTma ? 32 : 0); }

template <int K16, int MODE>
__global__ void __launch_bounds__(halo_threads(MODE), MODE == kResident ? 2 : 1)
    conv3x3_halo_tc_kernel(const HaloArgs q, const __grid_constant__ CUtensorMap wmap)
{
    constexpr bool STREAM = MODE != kResident;
    constexpr int kHaloThreads = halo_threads(MODE);
    const int co0 = blockIdx.y * q.cout;  // output channel tile
    const int cin = q.cin, cout = q.cout, k8n = cin / 8;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_hfull[4], s_hempty[4], s_afull[2], s_aempty[2], s_wfull[kMaxWStages],
        s_wempty[kMaxWStages];
    __shared__ int s_tab[2 * kHaloP];
    __shared__ __align__(16) float s_bias[256];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const size_t halo_b = (size_t)kHaloS * 16 * k8n;
    // a stage: slices of cout + 1 rows (conflict-free copies); TMA: cout rows of
    // 128 bytes, at a multiple of 1024
    const size_t wst_b = MODE == kTma ? (size_t)cout * 128 : (size_t)(cout + 1) * q.KC * 2;
    unsigned char* sH = smem_raw;
    unsigned char* sW = smem_raw + q.nbuf * halo_b;
    if (MODE == kTma) sW += (1024 - (smem_u32(sW) & 1023)) & 1023;
    float* sO = reinterpret_cast<float*>(sW + (STREAM ? q.wst * wst_b : (size_t)9 * cin * (cout + 1) * 2));

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(q.tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int k = 0; k < 4; ++k) {
            mbar_init(&s_hfull[k], kLoadT / q.nbuf);
            mbar_init(&s_hempty[k], 1);
        }
        for (int k = 0; k < 2; ++k) {
            mbar_init(&s_afull[k], 1);
            mbar_init(&s_aempty[k], kEpiT);
        }
        for (int k = 0; k < kMaxWStages; ++k) {
            mbar_init(&s_wfull[k], MODE == kTma ? 1 : 32);
            mbar_init(&s_wempty[k], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    fill_halo_table(s_tab, q.src, q.W, tid, kHaloThreads);
    for (int c = tid; c < cout; c += kHaloThreads) s_bias[c] = q.bias ? q.bias[co0 + c] : 0.f;
    if (!STREAM) {  // every tap's weights, [tap][slice][co][8], once per block
        for (int e = tid; e < 9 * k8n * cout; e += kHaloThreads) {
            const int co = e % cout, r = e / cout, k8 = r % k8n, tap = r / k8n;
            const __nv_bfloat16* g = q.w + ((size_t)tap * q.cout_all + co0 + co) * cin + 8 * k8;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(sW + ((size_t)r * (cout + 1) + co) * 16)),
                         "l"(g));
        }
        asm volatile("cp.async.commit_group;");
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;
    const int tiles_x = q.W / 8, tiles_img = tiles_x * (q.H / 16);
    const int nkb = cin / q.KC;
    auto split = [&](int t, int& img, int& ty0, int& tx0) {
        img = t / tiles_img;
        const int r = t - img * tiles_img, by = r / tiles_x;
        ty0 = by * 16;
        tx0 = (r - by * tiles_x) * 8;
    };

    if (warp < 4) {  // epilogue: TMEM lanes 32 warp .. are the warp's 32 pixels (4 tile rows)
        float* st = sO + warp * 32 * kOutPitch;
        int k = 0;
        for (int t = blockIdx.x; t < q.n_tiles; t += gridDim.x, ++k) {
            const int acc = k % q.nacc;
            // (the loads below are the whole warp's: its lanes go on or leave together)
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(&s_afull[acc], (k / q.nacc) & 1))) {
                atomicOr(&g_conv_error, 32);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            int img, ty0, tx0;
            split(t, img, ty0, tx0);
            const uint32_t ta = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(acc * cout);
            float* yt = q.y + (((size_t)img * q.H + ty0 + 4 * warp) * q.W + tx0) * q.cout_all;
            for (int c0 = 0; c0 < cout; c0 += 32) {
                const int cw = cout - c0 < 32 ? cout - c0 : 32;  // 16 or 32 channels
                for (int c = 0; c < cw; c += 16) {
                    uint32_t r[16];
                    __syncwarp();
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                        "[%16];"
                        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                          "=r"(r[15])
                        : "r"(ta + (uint32_t)(c0 + c)));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < 16; j += 4) {
                        const float4 bq = *reinterpret_cast<const float4*>(s_bias + c0 + c + j);
                        float4 v = make_float4(__uint_as_float(r[j]) + bq.x, __uint_as_float(r[j + 1]) + bq.y,
                                               __uint_as_float(r[j + 2]) + bq.z, __uint_as_float(r[j + 3]) + bq.w);
                        if (q.relu)
                            v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
                        *reinterpret_cast<float4*>(st + lane * kOutPitch + c + j) = v;
                    }
                }
                if (c0 + 32 >= cout) {  // the accumulator is read: the next tile may overwrite it
                    asm volatile("tcgen05.fence::before_thread_sync;");
                    mbar_arrive(&s_aempty[acc]);
                }
                __syncwarp();
                // the warp's 32 pixels, four tile rows, cw channels each: whole
                // 64- or 128-byte pieces per pixel
                const int sh = cw == 32 ? 3 : 2, ppi = 32 >> sh;  // pixels a pass
                float* og = yt + co0 + c0 + 4 * (lane & ((1 << sh) - 1));
                const float* sg = st + 4 * (lane & ((1 << sh) - 1));
#pragma unroll 4
                for (int px = lane >> sh; px < 32; px += ppi)
                    *reinterpret_cast<float4*>(og + (size_t)((px >> 3) * q.W + (px & 7)) * q.cout_all) =
                        *reinterpret_cast<const float4*>(sg + px * kOutPitch);
                __syncwarp();
            }
        }
    } else if (warp < 12) {
        // halo loaders: one group of warps per buffer, each on its own tiles, so
        // that the loads of nbuf tiles are in flight
        const int gt = kLoadT / q.nbuf, buf = (tid - kEpiT) / gt, g = (tid - kEpiT) - buf * gt;
        int use = 0;
        for (long long t = blockIdx.x + (long long)buf * gridDim.x; t < q.n_tiles; t += (long long)q.nbuf * gridDim.x, ++use) {
            if (use > 0 && !mbar_wait_bounded(&s_hempty[buf], (use - 1) & 1)) {
                atomicOr(&g_conv_error, 16);
                break;
            }
            int img, ty0, tx0;
            split((int)t, img, ty0, tx0);
            load_halo(q.src, s_tab, sH + buf * halo_b, img, ty0, tx0, q.H, q.W, 0, k8n, 0, kHaloY, g, gt);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(&s_hfull[buf]);
        }
    } else if (warp == 12) {
        if (elect_one()) {
            const uint32_t idesc = umma_idesc_bf16(kConvM, cout), bstep = 2 * (cout + 1);
            const int k16n = q.KC / 16;
            const uint64_t w0 = umma_desc(smem_u32(sW), (cout + 1) * 16, 128);
            // K-major with the 128-byte swizzle (layout 2 at bit 61): 8-row groups
            // 1024 bytes apart, 16 channels 32 bytes along the row
            const uint64_t w128 = umma_desc(smem_u32(sW), 16, 1024) | (2ull << 61);
            int buf = 0, acc = 0, st = 0;  // halo buffer, accumulator and weight slot, with their phases
            uint32_t hpar = 0, apar = 1, wpar = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < q.n_tiles && ok; t += gridDim.x) {
                if (!mbar_wait_bounded(&s_aempty[acc], apar) || !mbar_wait_bounded(&s_hfull[buf], hpar)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                // descriptors advance by adding to their address field (16-byte units)
                const uint32_t d = tmem + (uint32_t)(acc * cout);
                const uint64_t a0 = umma_desc(smem_u32(sH + buf * halo_b), kHaloS * 16, kHaloX * 16);
                if constexpr (!STREAM) {
                    const int n16 = K16 ? K16 : cin / 16;
                    uint64_t bd = w0;
#pragma unroll
                    for (int tap = 0; tap < 9; ++tap) {
                        umma_block<K16>(d, a0 + (tap / 3) * kHaloX + tap % 3, bd, bstep, idesc, n16, tap > 0 ? 1u : 0u);
                        bd += (uint64_t)n16 * bstep;
                    }
                } else {
                    for (int tap = 0; tap < 9 && ok; ++tap) {
                        uint64_t ad = a0 + (uint64_t)((tap / 3) * kHaloX + tap % 3);
                        for (int kb = 0; kb < nkb; ++kb) {
                            if (!mbar_wait_bounded(&s_wfull[st], wpar)) {
                                ok = false;
                                break;
                            }
                            asm volatile("tcgen05.fence::after_thread_sync;");
                            const uint64_t bd = (MODE == kTma ? w128 : w0) + (uint64_t)st * (wst_b >> 4);
                            umma_block<K16>(d, ad, bd, MODE == kTma ? 2 : bstep, idesc, k16n, (tap | kb) ? 1u : 0u);
                            umma_commit(&s_wempty[st]);
                            ad += (uint64_t)k16n * (2 * kHaloS);
                            if (++st == q.wst) {
                                st = 0;
                                wpar ^= 1;
                            }
                        }
                    }
                }
                umma_commit(&s_hempty[buf]);
                umma_commit(&s_afull[acc]);
                if (++buf == q.nbuf) {
                    buf = 0;
                    hpar ^= 1;
                }
                if (++acc == q.nacc) {
                    acc = 0;
                    apar ^= 1;
                }
            }
            if (!ok) atomicOr(&g_conv_error, 64);
        }
        __syncwarp();
    } else if (MODE == kTma) {
        if (lane == 0) {
            int my_tiles = 0;
            for (int t = blockIdx.x; t < q.n_tiles; t += gridDim.x) ++my_tiles;
            int st = 0, s = 0, sent = 0;
            uint32_t par = 1;
            bool ok = true;
            for (int k = 0; k < my_tiles && ok; ++k)
                for (int tap = 0; tap < 9 && ok; ++tap)
                    for (int kb = 0; kb < nkb; ++kb, ++sent) {
                        if (!mbar_wait_bounded(&s_wempty[st], par)) {
                            atomicOr(&g_conv_error, 128);
                            ok = false;
                            break;
                        }
                        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&s_wfull[st])),
                                     "r"((uint32_t)wst_b)
                                     : "memory");
                        asm volatile(
                            "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
                            "%3}], [%4];" ::"r"(smem_u32(sW + st * wst_b)),
                            "l"(&wmap), "r"(kb * 64), "r"(tap * q.cout_all + co0), "r"(smem_u32(&s_wfull[st]))
                            : "memory");
                        if (++st == q.wst) {
                            st = 0;
                            par ^= 1;
                        }
                    }
            // on expiry: the copies in flight land before the block ends
            if (!ok)
                for (s = sent > q.wst ? sent - q.wst : 0; s < sent; ++s)
                    mbar_wait_bounded(&s_wfull[s % q.wst], (s / q.wst) & 1);
        }
        __syncwarp();
    } else if (MODE == kStream && warp - 13 < q.wst) {
        // weight stream: warp j owns ring slot j and fills the stages j, j + wst,
        // ... (one owner a slot: a slot's phases are waited for in order)
        const int st = warp - 13;
        int my_tiles = 0;
        for (int t = blockIdx.x; t < q.n_tiles; t += gridDim.x) ++my_tiles;
        const int S = 9 * nkb, total = my_tiles * S, k8s = q.KC / 8;
        // the lanes' pieces: k8s slices of a row, rpp rows a pass (k8s = 2, 4, 8;
        // 6 leaves two lanes idle)
        const int rpp = 32 / k8s, k8 = lane % k8s, r0 = lane / k8s;
        int use = 0;
        for (int ws = st; ws < total; ws += q.wst, ++use) {
            if (use > 0 && !mbar_wait_bounded(&s_wempty[st], (use - 1) & 1)) {
                if (lane == 0) atomicOr(&g_conv_error, 128);
                break;
            }
            const int s = ws % S, tap = s / nkb, c0 = (s - tap * nkb) * q.KC;
            const __nv_bfloat16* g = q.w + ((size_t)tap * q.cout_all + co0 + r0) * cin + c0 + 8 * k8;
            uint32_t o = smem_u32(sW + st * wst_b) + (k8 * (cout + 1) + r0) * 16;
            if (r0 < rpp) {
#pragma unroll 4
                for (int co = r0; co < cout; co += rpp) {
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(o), "l"(g));
                    o += rpp * 16;
                    g += (size_t)rpp * cin;
                }
            }
            asm volatile("cp.async.commit_group;");
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(&s_wfull[st]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(q.tmem_cols));
}

// Input channels a stage: all of them up to 64, else the largest of 64, 48,
// 32, 16 dividing cin.
static int conv_kc(int cin)
{
    if (cin <= 64) return cin;
    for (int kc : {64, 48, 32, 16})
        if (cin % kc == 0) return kc;
    return 16;
}

// Largest dynamic shared memory a block may opt into, less the kernels' own
// static part.
constexpr size_t kSmemMax = 224 * 1024;

// Raises a kernel's dynamic shared memory limit, once per device (done: the
// kernel's own flags).
constexpr int kMaxDevices = 64;
template <class K>
static cudaError_t opt_in(K kernel, std::atomic<bool> (&done)[kMaxDevices])
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool known = dev >= 0 && dev < kMaxDevices;
    if (known && done[dev].load(std::memory_order_relaxed)) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    if (e == cudaSuccess && known) done[dev].store(true, std::memory_order_relaxed);
    return e;
}
static std::atomic<bool> g_gather_ready[kMaxDevices], g_wgrad_ready[kMaxDevices],
    g_wgrad9_ready[kMaxDevices], g_wgrad3_ready[kMaxDevices];

template <int K16, int MODE>
static cudaError_t launch_halo(const HaloArgs& q, const CUtensorMap& wmap, dim3 grid, size_t smem, cudaStream_t s)
{
    static std::atomic<bool> ready[kMaxDevices];
    const cudaError_t e = opt_in(conv3x3_halo_tc_kernel<K16, MODE>, ready);
    if (e != cudaSuccess) return e;
    conv3x3_halo_tc_kernel<K16, MODE><<<grid, halo_threads(MODE), smem, s>>>(q, wmap);
    return cudaGetLastError();
}

// Tensor map of the weights as rows of cin channels, boxes of cout rows by 64
// channels; false where it cannot be had (the piecewise stream takes over).
static bool weight_map(const HaloArgs& q, CUtensorMap& map)
{
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static std::atomic<void*> fn{nullptr};
    void* f = fn.load(std::memory_order_relaxed);
    if (!f) {
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &r) != cudaSuccess ||
            r != cudaDriverEntryPointSuccess || !f) {
            cudaGetLastError();
            return false;
        }
        fn.store(f, std::memory_order_relaxed);
    }
    const cuuint64_t dims[2] = {(cuuint64_t)q.cin, (cuuint64_t)9 * q.cout_all}, stride[1] = {(cuuint64_t)q.cin * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)q.cout}, one[2] = {1, 1};
    return reinterpret_cast<Encode>(f)(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                                       const_cast<__nv_bfloat16*>(q.w), dims, stride, box, one,
                                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Plan of the halo kernel: false where it does not apply.
static bool halo_plan(HaloArgs& q, size_t& smem, int& per_sm)
{
    if (q.H % 16 || q.W % 8) return false;
    const size_t halo = (size_t)kHaloS * 16 * (q.cin / 8), out = (size_t)4 * 32 * kOutPitch * 4;
    const size_t all_w = (size_t)9 * q.cin * (q.cout + 1) * 2, st = (size_t)(q.cout + 1) * q.KC * 2;
    q.nacc = q.cout <= 128 ? 2 : 1;
    // four halo buffers where two blocks an SM hold them, else two
    q.nbuf = 4 * halo + all_w + out <= 110 * 1024 ? 4 : 2;
    q.wst = 0;
    smem = q.nbuf * halo + all_w + out;
    if (smem > kSmemMax) {
        // the weights stream; a second halo buffer only beside four stages (and
        // 1 KB for the TMA form's alignment).  Two stages of a wide tile beside one
        // halo are enough (us at 256^2, gather kernel / this: 384 -> 256 565 / 135,
        // 320 -> 256 478 / 117, 384 -> 512 1033 / 224, 448 -> 128 559 / 125, 512 -> 64
        // 670 / 121); below that only the gather kernel's small stages fit
        const size_t rest = kSmemMax - out - 1024;
        q.nbuf = 2 * halo + 4 * st <= rest ? 2 : 1;
        if (q.nbuf * halo + 2 * st > rest) return false;
        const size_t n = (rest - q.nbuf * halo) / st;
        q.wst = (int)(n < kMaxWStages ? n : kMaxWStages);
        smem = q.nbuf * halo + q.wst * st + out + 1024;
    }
    q.tmem_cols = 32;
    while ((int)q.tmem_cols < q.nacc * q.cout) q.tmem_cols <<= 1;
    // blocks an SM: shared memory, and 512 columns of tensor memory between them
    per_sm = (int)(228 * 1024 / (smem + 2048));
    const int by_tmem = 512 / (int)q.tmem_cols;
    if (per_sm > by_tmem) per_sm = by_tmem;
    if (per_sm > 2) per_sm = 2;  // registers
    if (per_sm < 1 || q.wst) per_sm = 1;
    const size_t least = (size_t)(228 * 1024) / (per_sm + 1) - 1024;  // no more blocks than that fit
    if (smem < least) smem = least;
    return true;
}

int conv3x3_form(int H, int W, int cin, int cout_all)
{
    const int n_tiles = (cout_all + 255) / 256;
    HaloArgs q;
    q.H = H;
    q.W = W;
    q.cin = cin;
    q.cout = cout_all / n_tiles;
    q.KC = conv_kc(cin);
    size_t smem = 0;
    int per_sm = 1;
    return !halo_plan(q, smem, per_sm) ? 0 : q.wst ? 2 : 1;
}

cudaError_t conv3x3_fwd_src(const float* a, const float* b, int ca, int cb, const __nv_bfloat16* w, const float* bias,
                            float* y, int N, int H, int W, int cout_all, int relu, cudaStream_t s)
{
    const int cin = ca + cb;
    // output channels in equal tiles of at most 256 (one MMA's N), multiples of 16
    const int n_tiles = (cout_all + 255) / 256;
    if (cin % 16 || ca % 8 || cout_all % (16 * n_tiles) || cin < 16 || cout_all < 16 || H < 1 || W < 1)
        return cudaErrorInvalidValue;
    HaloArgs q;
    q.src = conv_src(a, b, ca, cb, W);
    q.w = w;
    q.bias = bias;
    q.y = y;
    q.H = H;
    q.W = W;
    q.cin = cin;
    q.cout_all = cout_all;
    q.cout = cout_all / n_tiles;
    q.KC = conv_kc(cin);
    q.relu = relu;
    size_t smem = 0;
    int per_sm = 1;
    if (halo_plan(q, smem, per_sm)) {
        const long long tiles = (long long)N * (H / 16) * (W / 8);
        if (tiles > 0x7fffffff) return cudaErrorInvalidValue;
        q.n_tiles = (int)tiles;
        long long blocks = 152LL * per_sm / n_tiles;
        if (blocks < 1) blocks = 1;
        if (blocks > tiles) blocks = tiles;
        const dim3 grid((unsigned)blocks, n_tiles);
        CUtensorMap map = {};
        if (q.wst) {
            if (q.KC == 64 && weight_map(q, map)) return launch_halo<4, kTma>(q, map, grid, smem, s);
            // (blocks of 64 channels by pieces: only where the driver has no tensor-map
            // encoder, which no test meets)
            return q.KC == 64 ? launch_halo<4, kStream>(q, map, grid, smem, s)
                              : launch_halo<0, kStream>(q, map, grid, smem, s);
        }
        switch (cin / 16) {
        case 1: return launch_halo<1, kResident>(q, map, grid, smem, s);
        case 2: return launch_halo<2, kResident>(q, map, grid, smem, s);
        case 3: return launch_halo<3, kResident>(q, map, grid, smem, s);
        case 4: return launch_halo<4, kResident>(q, map, grid, smem, s);
        case 6: return launch_halo<6, kResident>(q, map, grid, smem, s);
        default: return launch_halo<0, kResident>(q, map, grid, smem, s);
        }
    }
    if (b) return cudaErrorInvalidValue;
    const int cout = q.cout, KC = q.KC;
    smem = 2 * ((size_t)kConvM * KC * 2 + (size_t)cout * KC * 2);
    cudaError_t e = opt_in(conv3x3_tc_kernel, g_gather_ready);
    if (e != cudaSuccess) return e;
    uint32_t cols = 32;
    while ((int)cols < cout) cols <<= 1;
    const long long P = (long long)N * H * W;
    const long long blocks = (P + kConvM - 1) / kConvM;
    conv3x3_tc_kernel<<<dim3((unsigned)blocks, n_tiles), kConvM, smem, s>>>(a, w, bias, y, P, H, W, cin, cout_all, cout,
                                                                            KC, relu, cols);
    return cudaGetLastError();
}

cudaError_t conv3x3_fwd(const float* x, const __nv_bfloat16* w, const float* bias, float* y, int N, int H, int W,
                        int cin, int cout_all, int relu, cudaStream_t s)
{
    return conv3x3_fwd_src(x, nullptr, cin, 0, w, bias, y, N, H, W, cout_all, relu, s);
}

int conv_error()
{
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_conv_error, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return v;
}

// Weights for the data gradient: dX = conv3x3(dY, wt) with
// wt[tap][ci][co] = w[8 - tap][co][ci] (taps flipped, channels swapped).
__global__ void flip_weights_kernel(const __nv_bfloat16* w, __nv_bfloat16* wt, int cin, int cout)
{
    const int total = 9 * cin * cout;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int co = e % cout, r = e / cout;  // e indexes wt[tap][ci][co]
        const int ci = r % cin, tap = r / cin;
        wt[e] = w[((size_t)(8 - tap) * cout + co) * cin + ci];
    }
}

cudaError_t flip_weights(const __nv_bfloat16* w, __nv_bfloat16* wt, int cin, int cout, cudaStream_t s)
{
    flip_weights_kernel<<<64, 256, 0, s>>>(w, wt, cin, cout);
    return cudaGetLastError();
}

// ---- weight gradient on the tensor cores
//
// dw[tap][co][ci] += sum_p dy[p][co] x[p + tap][ci]: per block one tap, one
// tile of 128 output channels (M; rows beyond cout are zero) and one tile of
// nci input channels (N), over a range of pixels (K) in stages of 64:
// A[co][p] = dy (BF16), B[ci][p] = x at the tap's neighbour (BF16), both
// gathered transposed into the no-swizzle K-major layout (8 pixels of one
// channel per 16-byte row of a core matrix).  Double-buffered stages,
// mbarrier completion and bounded waits as in conv3x3_tc_kernel; the block's
// partial sums leave tensor memory through tcgen05.ld and are added to dw
// with FP32 atomics.
constexpr int kWgK = 64;  // pixels a stage

__global__ void __launch_bounds__(kConvM) conv3x3_wgrad_tc_kernel(const float* __restrict__ x,
                                                                  const float* __restrict__ dy, float* dw, long long P,
                                                                  int H, int W, int cin, int cout, int nci,
                                                                  long long KP, uint32_t tmem_cols)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_mbar[2];
    __shared__ long long s_q[2][kWgK];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int tap = blockIdx.z;
    const int n_ntiles = cin / nci;
    const int co0 = (blockIdx.y / n_ntiles) * kConvM, ci0 = (blockIdx.y % n_ntiles) * nci;
    const long long p0 = (long long)blockIdx.x * KP, p1 = p0 + KP < P ? p0 + KP : P;
    const size_t a_bytes = (size_t)kConvM * kWgK * 2, b_bytes = (size_t)nci * kWgK * 2;
    auto sA = [&](int b) { return smem_raw + b * a_bytes; };
    auto sB = [&](int b) { return smem_raw + 2 * a_bytes + b * b_bytes; };

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_mbar[0])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_mbar[1])));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;

    const int dyy = tap / 3 - 1, dxx = tap % 3 - 1;
    const long long HW = (long long)H * W;
    // A rows beyond cout stay zero: clear both A buffers once
    const int mv = cout - co0 < kConvM ? cout - co0 : kConvM;  // valid A rows
    for (int e = tid; e < (int)(2 * a_bytes / 16); e += kConvM)
        reinterpret_cast<uint4*>(smem_raw)[e] = make_uint4(0u, 0u, 0u, 0u);
    const uint32_t idesc = umma_idesc_bf16(kConvM, nci);
    const int S = (int)((p1 - p0 + kWgK - 1) / kWgK);
    bool ok = true;
    int issued = 0;
    for (int s = 0; s < S && ok; ++s) {
        const int buf = s & 1;
        const long long pb = p0 + (long long)s * kWgK;
        if (s >= 2 && !mbar_wait_bounded(&s_mbar[buf], ((s - 2) >> 1) & 1)) {
            atomicOr(&g_conv_error, 4);
            ok = false;  // the block leaves together below
        }
        if (tid < kWgK) {  // the stage's pixels and their neighbours at the tap
            const long long pp = pb + tid;
            long long q = -1;
            if (pp < p1) {
                const long long img = pp / HW;
                const int rem = (int)(pp - img * HW), py = rem / W, px = rem - py * W;
                int yy = py + dyy, xx = px + dxx;
                yy = yy < 0 ? yy + H : (yy >= H ? yy - H : yy);
                xx = xx < 0 ? xx + W : (xx >= W ? xx - W : xx);
                q = img * HW + (long long)yy * W + xx;
            }
            s_q[buf][tid] = q;
        }
        ok = __syncthreads_and(ok) != 0;
        if (!ok) break;
        // 16-byte pieces (channel row, 8 pixels) of A = dy and B = x at the
        // tap's neighbours.  Tiles of at least 128 channels: one row a thread,
        // its 64 pixels unrolled (more loads in flight); narrower tiles
        // spread the pieces over all threads, consecutive threads on
        // consecutive channels (measured 2.4x on 32 channels, 8-27 % slower
        // than one row a thread at 128-384)
        auto pieceA = [&](int m, int k8) {
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const long long pp = pb + 8 * k8 + j;
                v[j] = pp < p1 ? __ldg(dy + pp * cout + co0 + m) : 0.f;
            }
            *reinterpret_cast<uint4*>(sA(buf) + (size_t)k8 * kConvM * 16 + m * 16) =
                make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
        };
        auto pieceB = [&](int n, int k8) {
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const long long q = s_q[buf][8 * k8 + j];
                v[j] = q >= 0 ? __ldg(x + q * cin + ci0 + n) : 0.f;
            }
            *reinterpret_cast<uint4*>(sB(buf) + (size_t)k8 * nci * 16 + n * 16) = make_uint4(
                pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
        };
        if (mv == kConvM) {
#pragma unroll
            for (int k8 = 0; k8 < kWgK / 8; ++k8) pieceA(tid, k8);
        } else {
            for (int e = tid; e < mv * (kWgK / 8); e += kConvM) pieceA(e % mv, e / mv);
        }
        if (nci >= kConvM) {
            for (int n = tid; n < nci; n += kConvM)
#pragma unroll
                for (int k8 = 0; k8 < kWgK / 8; ++k8) pieceB(n, k8);
        } else {
            for (int e = tid; e < nci * (kWgK / 8); e += kConvM) pieceB(e % nci, e / nci);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t a0 = smem_u32(sA(buf)), b0 = smem_u32(sB(buf));
            for (int k16 = 0; k16 < kWgK / 16; ++k16) {
                const uint64_t ad = umma_desc(a0 + k16 * 2 * kConvM * 16, kConvM * 16, 128);
                const uint64_t bd = umma_desc(b0 + k16 * 2 * nci * 16, nci * 16, 128);
                umma_bf16(tmem, ad, bd, idesc, (s > 0 || k16 > 0) ? 1u : 0u);
            }
            umma_commit(&s_mbar[buf]);
        }
        issued = s + 1;
    }
    bool done = false;
    if (issued > 0) {
        const int last = issued - 1;
        done = mbar_wait_bounded(&s_mbar[last & 1], (last >> 1) & 1);
        if (!done) atomicOr(&g_conv_error, 8);
    }
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (__all_sync(0xffffffffu, ok && done)) {  // the loads below are the whole warp's
        for (int c = 0; c < nci; c += 8) {
            uint32_t r[8];
            __syncwarp();
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                           "=r"(r[7])
                         : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            const int co = co0 + tid;  // this thread's TMEM lane = D row
            if (co < cout) {
                float* d = dw + ((size_t)tap * cout + co) * cin + ci0 + c;
#pragma unroll
                for (int j = 0; j < 8; ++j) atomicAdd(d + j, __uint_as_float(r[j]));
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols));
}

// Halo form of the weight gradient (H a multiple of 16, W of 8): no transposed
// gathers.  Both operands are MN-major in shared memory as they lie in the
// image: A = dy of a 16 x 8 tile, [8-channel slice][pixel][8] (M = 128 output
// channels; rows beyond cout read whatever follows and are never stored), B =
// x of the tile's halo in the same layout, a tap's pixels being a start offset
// as in the forward kernel; K = 16 pixels, two tile rows, a call (K groups of 8
// pixels: 128 bytes apart in A, one halo row apart in B; slices are the M and N
// groups).  A block takes TAPS taps (all nine, or the three of one row dy) of
// one output-channel tile and nci input channels, keeps their accumulators in
// tensor memory (TAPS x nci <= 512 columns) over all its tiles and adds them to
// dw once at the end, four floats an atomic.  Warps 0-3 load and convert dy,
// warps 4-11 x (two buffers), warp 12 issues the MMAs, warps 0-3 store.
// Measured, us (gathered transposed / this): 1024^2 32 -> 32 929 / 117, 512^2
// 64 -> 64 438 / 98, 256^2 128 -> 128 295 / 44, 128^2 256 -> 256 262 / 41.
// Bound by the loads' latency at one block an SM (27 % of the DRAM rate, tensor
// pipe 25 %, of which M = 128 rows for 32 channels waste three quarters).
constexpr int kWgDyT = 128, kWgXT = 256, kWgLoadT = kWgDyT + kWgXT, kWgThreads = kWgLoadT + 32;
constexpr int kDyS = kConvM + 1;  // pixels a dy slice (129 x 16 bytes: conflict-free stores)

struct WgradArgs {
    ConvSrc src;
    const float* dy;
    float* dw;
    int H, W, n_tiles, cin, cout, nci, vec;
    size_t buf_b;  // bytes of one buffer (dy, then x)
    uint32_t tmem_cols;
};

template <int TAPS>
__global__ void __launch_bounds__(kWgThreads) conv3x3_wgrad_halo_kernel(const WgradArgs q)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_full[2], s_empty[2], s_done;
    __shared__ int s_tab[2 * kHaloP];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int n_ntiles = q.cin / q.nci;
    const int co0 = ((int)blockIdx.y / n_ntiles) * kConvM, ci0 = ((int)blockIdx.y % n_ntiles) * q.nci;
    const int tap0 = blockIdx.z * TAPS;
    const int mco = min(kConvM, q.cout - co0), m8 = mco / 8, n8 = q.nci / 8;
    const size_t dy_b = (size_t)kDyS * 16 * m8;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(q.tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int k = 0; k < 2; ++k) {
            mbar_init(&s_full[k], kWgLoadT);
            mbar_init(&s_empty[k], 1);
        }
        mbar_init(&s_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    fill_halo_table(s_tab, q.src, q.W, tid, kWgThreads);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;
    const int tiles_x = q.W / 8, tiles_img = tiles_x * (q.H / 16);
    // taps of one row dy need the halo rows 1 + dy .. 16 + dy only
    const int r0 = TAPS == 3 ? tap0 / 3 : 0, rows = TAPS == 3 ? 16 : kHaloY;

    bool ok = true;
    if (warp < kWgLoadT / 32) {
        int k = 0;
        for (int t = blockIdx.x; t < q.n_tiles; t += gridDim.x, ++k) {
            const int buf = k & 1, use = k >> 1;
            if (use > 0 && !mbar_wait_bounded(&s_empty[buf], (use - 1) & 1)) {
                atomicOr(&g_conv_error, 4);
                ok = false;
                break;
            }
            const int img = t / tiles_img, r = t - img * tiles_img, by = r / tiles_x;
            const int ty0 = by * 16, tx0 = (r - by * tiles_x) * 8;
            unsigned char* sA = smem_raw + buf * q.buf_b;
            if (warp < 4) {
                // dy of the tile: a thread keeps one 8-channel slice, six pieces in flight
                constexpr int B = 6;
                const int dq = kWgDyT / m8, p0 = tid / m8, c8 = tid - p0 * m8;
                const float* base = q.dy + (((size_t)img * q.H + ty0) * q.W + tx0) * q.cout + co0 + 8 * c8;
                unsigned char* o = sA + ((size_t)c8 * kDyS + p0) * 16;
                for (int px = p0; px < kConvM && p0 < dq; px += B * dq, o += B * dq * 16) {
                    float4 f[B][2];
#pragma unroll
                    for (int j = 0; j < B; ++j) {
                        const int p = px + j * dq;
                        if (p < kConvM) {
                            const float4* g = reinterpret_cast<const float4*>(
                                base + (size_t)((p >> 3) * q.W + (p & 7)) * q.cout);
                            f[j][0] = __ldg(g);
                            f[j][1] = __ldg(g + 1);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < B; ++j)
                        if (px + j * dq < kConvM)
                            *reinterpret_cast<uint4*>(o + j * dq * 16) =
                                make_uint4(pack_bf16(f[j][0].x, f[j][0].y), pack_bf16(f[j][0].z, f[j][0].w),
                                           pack_bf16(f[j][1].x, f[j][1].y), pack_bf16(f[j][1].z, f[j][1].w));
                }
            } else {
                load_halo(q.src, s_tab, sA + dy_b, img, ty0, tx0, q.H, q.W, ci0, n8, r0, rows, tid - kWgDyT, kWgXT);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(&s_full[buf]);
        }
    } else {
        if (elect_one()) {
            // as umma_idesc_bf16, A and B MN-major (bits 15, 16)
            const uint32_t idesc = umma_idesc_bf16(kConvM, q.nci) | (1u << 15) | (1u << 16);
            int k = 0;
            for (int t = blockIdx.x; t < q.n_tiles; t += gridDim.x, ++k) {
                const int buf = k & 1;
                if (!mbar_wait_bounded(&s_full[buf], (k >> 1) & 1)) {
                    atomicOr(&g_conv_error, 256);
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t sa = smem_u32(smem_raw + buf * q.buf_b);
                const uint64_t a0 = umma_desc(sa, 128, kDyS * 16);
                const uint32_t more = k > 0 ? 1u : 0u;
                // halo rows start at r0: a row of taps (TAPS = 3) reads rows 0 .. 15
                const uint64_t b0 = umma_desc(sa + (uint32_t)dy_b, kHaloX * 16, kHaloS * 16);
#pragma unroll
                for (int tp = 0; tp < TAPS; ++tp) {
                    const uint64_t bt = b0 + (TAPS == 9 ? (tp / 3) * kHaloX + tp % 3 : tp);
                    const uint32_t d = tmem + (uint32_t)(tp * q.nci);
#pragma unroll
                    for (int k16 = 0; k16 < 8; ++k16)
                        umma_bf16(d, a0 + k16 * 16, bt + k16 * 2 * kHaloX, idesc, k16 > 0 ? 1u : more);
                }
                umma_commit(&s_empty[buf]);
            }
            umma_commit(&s_done);
        }
        __syncwarp();
    }
    if (warp < 4) {
        const bool any = (int)blockIdx.x < q.n_tiles;
        const bool done = mbar_wait_bounded(&s_done, 0);
        if (!done) atomicOr(&g_conv_error, 8);
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (__all_sync(0xffffffffu, ok && done && any)) {  // the loads below are the whole warp's
            const int co = co0 + tid;  // this thread's TMEM lane = D row
            for (int tp = 0; tp < TAPS; ++tp)
                for (int c = 0; c < q.nci; c += 16) {
                    uint32_t r[16];
                    __syncwarp();
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                        "[%16];"
                        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                          "=r"(r[15])
                        : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(tp * q.nci + c)));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (tid < mco) {
                        float* d = q.dw + ((size_t)(tap0 + tp) * q.cout + co) * q.cin + ci0 + c;
#pragma unroll
                        for (int j = 0; j < 16; j += 4) {
                            const float4 v = make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                                                         __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
                            if (q.vec) {
                                atomicAdd(reinterpret_cast<float4*>(d + j), v);
                            } else {
                                atomicAdd(d + j, v.x);
                                atomicAdd(d + j + 1, v.y);
                                atomicAdd(d + j + 2, v.z);
                                atomicAdd(d + j + 3, v.w);
                            }
                        }
                    }
                }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(q.tmem_cols));
}

// Launches the halo form where it applies; false otherwise.
static bool wgrad_halo(const ConvSrc& src, const float* dy, float* dw, int N, int H, int W, int cin, int cout,
                       cudaStream_t s, cudaError_t& err)
{
    const uintptr_t al = (uintptr_t)src.a | (uintptr_t)src.b | (uintptr_t)dy;
    if (H % 16 || W % 8 || src.ca % 8 || (al & 15)) return false;
    WgradArgs q;
    q.src = src;
    q.dy = dy;
    q.dw = dw;
    q.H = H;
    q.W = W;
    q.cin = cin;
    q.cout = cout;
    q.vec = ((uintptr_t)dw & 15) == 0;
    // all nine taps where their accumulators fit, else one row of three
    const int taps = cin <= 48 ? 9 : 3;
    int nt = 1;
    while (cin % (16 * nt) || cin / nt > 160) {
        if (++nt > cin / 16) return false;
    }
    q.nci = cin / nt;
    const int n_mtiles = (cout + kConvM - 1) / kConvM, mco = cout < kConvM ? cout : kConvM;
    q.buf_b = (size_t)kDyS * 16 * (mco / 8) + (size_t)kHaloS * 16 * (q.nci / 8);
    // an A descriptor spans the slices of 128 channels, valid or not
    size_t smem = 2 * q.buf_b;
    const size_t span = q.buf_b + (size_t)kDyS * 16 * 16;
    if (smem < span) smem = span;
    if (smem > kSmemMax) return false;
    q.tmem_cols = 32;
    while ((int)q.tmem_cols < taps * q.nci) q.tmem_cols <<= 1;
    int per_sm = (int)(228 * 1024 / (smem + 2048));
    const int by_tmem = 512 / (int)q.tmem_cols;
    if (per_sm > by_tmem) per_sm = by_tmem;
    if (per_sm > 2) per_sm = 2;  // registers
    if (per_sm < 1) per_sm = 1;
    const size_t least = (size_t)(228 * 1024) / (per_sm + 1) - 1024;  // no more blocks than that fit
    if (smem < least) smem = least;
    const long long tiles = (long long)N * (H / 16) * (W / 8);
    if (tiles > 0x7fffffff) return false;
    q.n_tiles = (int)tiles;
    const int groups = n_mtiles * nt * (9 / taps);
    long long chunks = 152LL * per_sm / groups;
    if (chunks < 1) chunks = 1;
    if (chunks > tiles) chunks = tiles;
    const dim3 grid((unsigned)chunks, n_mtiles * nt, 9 / taps);
    err = taps == 9 ? opt_in(conv3x3_wgrad_halo_kernel<9>, g_wgrad9_ready)
                    : opt_in(conv3x3_wgrad_halo_kernel<3>, g_wgrad3_ready);
    if (err != cudaSuccess) return true;
    if (taps == 9)
        conv3x3_wgrad_halo_kernel<9><<<grid, kWgThreads, smem, s>>>(q);
    else
        conv3x3_wgrad_halo_kernel<3><<<grid, kWgThreads, smem, s>>>(q);
    err = cudaGetLastError();
    return true;
}

cudaError_t conv3x3_wgrad_src(const float* a, const float* b, int ca, int cb, const float* dy, float* dw, int N, int H,
                              int W, int cout, cudaStream_t s)
{
    const int cin = ca + cb;
    const int n_ntiles = (cin + 255) / 256;
    if (cin % 16 || cout % 16 || cin < 16 || cout < 16 || cin % (16 * n_ntiles)) return cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
    if (wgrad_halo(conv_src(a, b, ca, cb, W), dy, dw, N, H, W, cin, cout, s, e)) return e;
    if (b) return cudaErrorInvalidValue;
    const int nci = cin / n_ntiles, n_mtiles = (cout + kConvM - 1) / kConvM;
    const long long P = (long long)N * H * W;
    // about four blocks an SM in all: pixel chunks of a multiple of 64
    long long chunks = (4LL * 152 + 9 * n_mtiles * n_ntiles - 1) / (9 * n_mtiles * n_ntiles);
    long long KP = (P + chunks - 1) / chunks;
    KP = ((KP + kWgK - 1) / kWgK) * kWgK;
    chunks = (P + KP - 1) / KP;
    const size_t smem = 2 * ((size_t)kConvM * kWgK * 2 + (size_t)nci * kWgK * 2);
    e = opt_in(conv3x3_wgrad_tc_kernel, g_wgrad_ready);
    if (e != cudaSuccess) return e;
    uint32_t cols = 32;
    while ((int)cols < nci) cols <<= 1;
    dim3 grid((unsigned)chunks, (unsigned)(n_mtiles * n_ntiles), 9);
    conv3x3_wgrad_tc_kernel<<<grid, kConvM, smem, s>>>(a, dy, dw, P, H, W, cin, cout, nci, KP, cols);
    return cudaGetLastError();
}

cudaError_t conv3x3_wgrad(const float* x, const float* dy, float* dw, int N, int H, int W, int cin, int cout,
                          cudaStream_t s)
{
    return conv3x3_wgrad_src(x, nullptr, cin, 0, dy, dw, N, H, W, cout, s);
}

// Elementwise and small kernels -------------------------------------------------

static int eblocks(long long n)
{
    long long b = (n + 255) / 256;
    return (int)(b < 1 ? 1 : (b > 152 * 32 ? 152 * 32 : b));
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

// Sum of v over the block's threads with the same tid % q4 (q4 a power of two
// dividing 256) into out[4 (tid % q4) ..], by the first q4 threads.
__device__ __forceinline__ void block_sum4(float4 v, int q4, float* out, float4* red)
{
    __syncthreads();
    red[threadIdx.x] = v;
    __syncthreads();
    for (int o = 128; o >= q4; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] = add4(red[threadIdx.x], red[threadIdx.x + o]);
        __syncthreads();
    }
    if ((int)threadIdx.x < q4) {
        const float4 t = red[threadIdx.x];
        out[4 * threadIdx.x] = t.x;
        out[4 * threadIdx.x + 1] = t.y;
        out[4 * threadIdx.x + 2] = t.z;
        out[4 * threadIdx.x + 3] = t.w;
    }
}

// Bias and head gradients repeat bit for bit: each block of the backward element
// passes writes its sums as a row of partials, and one launch at the end of the
// backward pass adds the rows of every gradient in a fixed order, a block per 32
// columns, 32 rows at a time.  (Float atomics of up to 608 blocks on each value,
// besides leaving the order open, took longer: the backward pass of 8 x 128^2 with
// its forward 612 us, 576 this way.)
__global__ void __launch_bounds__(1024) sum_partials_kernel(const PartialSums q)
{
    __shared__ float red[32][33];
    int k = 0, b = blockIdx.x;
    while (b >= (q.s[k].width + 31) / 32) b -= (q.s[k++].width + 31) / 32;
    const PartialSums::Sum m = q.s[k];
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5, col = 32 * b + l;
    float t = 0.f;
    if (col < m.width) {
#pragma unroll 4
        for (int r = w; r < m.rows; r += 32) t += m.part[(size_t)r * m.pitch + col];
    }
    red[w][l] = t;
    __syncthreads();
    if (w > 0 || col >= m.width) return;
    t = red[0][l];
#pragma unroll
    for (int r = 1; r < 32; ++r) t += red[r][l];
    m.out[col] += t;
}

cudaError_t sum_partials(const PartialSums& q, cudaStream_t s)
{
    int blocks = 0;
    for (int k = 0; k < q.n; ++k) blocks += (q.s[k].width + 31) / 32;
    if (blocks > 0) sum_partials_kernel<<<blocks, 1024, 0, s>>>(q);
    return cudaGetLastError();
}

// Gradient before a layer's ReLU and the layer's bias gradient, in one pass:
//   dst[p][ch] = y[p][ch] > 0 ? g[p][ch] : 0,   db[ch] += sum_p dst[p][ch]
// (the block's part of the sum: part[block][ch], added up by sum_partials),
// where g is, by `from`:
//   kFromSame   src[p][ch] (dst may be src);
//   kFromUp     the sum over the pixel's 2 x 2 children in src (N, 2H, 2W, sc),
//               channel ch (backward of the nearest upsampling);
//   kFromPool   0.25 src[parent][ch] (N, H/2, W/2, c: backward of the pooling)
//               + skip[p][so + ch] (N, H, W, sc: the decoder's skip gradient).
// Bound by memory: 12 to 17 bytes an element.  A thread keeps one channel quad
// (c / 4 a power of two) and sums it over its pixels.
// Replaces a ReLU, a pooling or upsampling, an addition and a one-block-a-channel
// sum (for 16 channels at 8 x 128^2: 76 us of 90, now 8 in all).
enum { kFromSame, kFromUp, kFromPool };
template <int FROM>
__global__ void __launch_bounds__(256) act_bwd_kernel(const float* y, const float* src, const float* skip, float* dst,
                                                      float* part, long long P, int H, int W, int c, int sc, int so)
{
    __shared__ float4 red[256];
    const int q4 = c / 4, ch = 4 * ((int)threadIdx.x % q4), ppb = 256 / q4;
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    for (long long p = (long long)blockIdx.x * ppb + threadIdx.x / q4; p < P; p += (long long)gridDim.x * ppb) {
        float4 g;
        if (FROM == kFromSame) {
            g = ld4(src + p * c + ch);
        } else {
            const int x = (int)(p % W);
            const long long r = p / W;
            const int yy = (int)(r % H);
            const long long n = r / H;
            if (FROM == kFromUp) {
                const float* b = src + ((n * 2 * H + 2 * yy) * 2 * W + 2 * x) * sc + ch;
                const size_t row = (size_t)2 * W * sc;
                g = add4(add4(add4(ld4(b), ld4(b + sc)), ld4(b + row)), ld4(b + row + sc));
            } else {
                const float4 a = ld4(src + ((n * (H / 2) + yy / 2) * (W / 2) + x / 2) * c + ch);
                g = make_float4(0.25f * a.x, 0.25f * a.y, 0.25f * a.z, 0.25f * a.w);
                if (skip) g = add4(g, ld4(skip + p * sc + so + ch));
            }
        }
        const float4 v = ld4(y + p * c + ch);
        if (!(v.x > 0.f)) g.x = 0.f;
        if (!(v.y > 0.f)) g.y = 0.f;
        if (!(v.z > 0.f)) g.z = 0.f;
        if (!(v.w > 0.f)) g.w = 0.f;
        st4(dst + p * c + ch, g);
        sum = add4(sum, g);
    }
    block_sum4(sum, q4, part + (size_t)blockIdx.x * c, red);
}

int act_blocks(long long P, int c)
{
    const long long b = (P + 256 / (c / 4) - 1) / (256 / (c / 4));
    return (int)(b < 1 ? 1 : (b > 152 * 4 ? 152 * 4 : b));
}

cudaError_t act_bwd(const float* y, float* dy, float* part, long long P, int c, cudaStream_t s)
{
    act_bwd_kernel<kFromSame><<<act_blocks(P, c), 256, 0, s>>>(y, dy, nullptr, dy, part, P, 1, 1, c, 0, 0);
    return cudaGetLastError();
}
cudaError_t act_bwd_up(const float* y, const float* src, float* dst, float* part, int N, int H, int W, int c, int sc,
                       cudaStream_t s)
{
    const long long P = (long long)N * H * W;
    act_bwd_kernel<kFromUp><<<act_blocks(P, c), 256, 0, s>>>(y, src, nullptr, dst, part, P, H, W, c, sc, 0);
    return cudaGetLastError();
}
cudaError_t act_bwd_pool(const float* y, const float* src, const float* skip, float* dst, float* part, int N, int H, int W,
                         int c, int sc, int so, cudaStream_t s)
{
    const long long P = (long long)N * H * W;
    act_bwd_kernel<kFromPool><<<act_blocks(P, c), 256, 0, s>>>(y, src, skip, dst, part, P, H, W, c, sc, so);
    return cudaGetLastError();
}

// 2 x 2 average pool (NHWC), a channel quad a thread.
__global__ void pool_fwd_kernel(const float* x, float* y, int N, int H, int W, int c)
{
    const int Ho = H / 2, Wo = W / 2, q4 = c / 4;
    const long long total = (long long)N * Ho * Wo * q4;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int ch = 4 * (int)(i % q4);
        long long r = i / q4;
        const int xo = (int)(r % Wo);
        r /= Wo;
        const int yo = (int)(r % Ho);
        const long long n = r / Ho;
        const float* b = x + ((n * H + 2 * yo) * W + 2 * xo) * c + ch;
        const float4 t = add4(add4(add4(ld4(b), ld4(b + c)), ld4(b + (size_t)W * c)), ld4(b + (size_t)W * c + c));
        st4(y + 4 * i, make_float4(0.25f * t.x, 0.25f * t.y, 0.25f * t.z, 0.25f * t.w));
    }
}

cudaError_t pool_fwd(const float* x, float* y, int N, int H, int W, int c, cudaStream_t s)
{
    pool_fwd_kernel<<<eblocks((long long)N * H * W * c / 16), 256, 0, s>>>(x, y, N, H, W, c);
    return cudaGetLastError();
}

// The head, forward: out[p] = b + w x[p] (2 outputs, FP32), the first times the
// interface gate 1 - phi^2 (xin[p][0] = phi), so that the network changes phi
// only in the diffuse interface.  Written to out, and to y when given.
__global__ void head_fwd_kernel(const float* x, const float* w, const float* b, const float* xin, int cx, float* out,
                                float* y, long long P, int c)
{
    __shared__ float sw[2 * 64];
    for (int k = threadIdx.x; k < 2 * c; k += blockDim.x) sw[k] = w[k];
    __syncthreads();
    const float b0 = b[0], b1 = b[1];
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        float a0 = b0, a1 = b1;
        for (int k = 0; k < c; k += 4) {
            const float4 v = ld4(x + p * c + k);
            a0 += sw[k] * v.x;
            a1 += sw[c + k] * v.x;
            a0 += sw[k + 1] * v.y;
            a1 += sw[c + k + 1] * v.y;
            a0 += sw[k + 2] * v.z;
            a1 += sw[c + k + 2] * v.z;
            a0 += sw[k + 3] * v.w;
            a1 += sw[c + k + 3] * v.w;
        }
        const float ph = xin[p * cx];
        a0 *= (1.f - ph) * (1.f + ph);
        const float2 o = make_float2(a0, a1);
        reinterpret_cast<float2*>(out)[p] = o;
        if (y) {  // y: the caller's, any alignment
            y[2 * p] = a0;
            y[2 * p + 1] = a1;
        }
    }
}

cudaError_t head_fwd(const float* x, const float* w, const float* b, const float* xin, int cx, float* out, float* y,
                     long long P, int c, cudaStream_t s)
{
    if (c > 64 || c % 4) return cudaErrorInvalidValue;
    head_fwd_kernel<<<eblocks(P), 256, 0, s>>>(x, w, b, xin, cx, out, y, P, c);
    return cudaGetLastError();
}

// The head, backward, with the gate and the last layer's ReLU and bias in the
// same pass: g = (dy0 (1 - phi^2), dy1); dw += g x^T, db += g; dx = w^T g where
// x > 0 (x is that layer's output), else 0; db_last += sum dx.  The block's parts
// of the sums are a row of 3 c + 2 partials: dw, db, db_last.
__global__ void __launch_bounds__(256) head_bwd_kernel(const float* x, const float* dy, const float* w, const float* xin,
                                                       int cx, float* dx, float* part, long long P, int c)
{
    __shared__ float4 red[256];
    const int q4 = c / 4, ch = 4 * ((int)threadIdx.x % q4), ppb = 256 / q4;
    float w0[4], w1[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        w0[k] = w[ch + k];
        w1[k] = w[c + ch + k];
    }
    float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0, sl = s0, sb = s0;
    for (long long p = (long long)blockIdx.x * ppb + threadIdx.x / q4; p < P; p += (long long)gridDim.x * ppb) {
        const float ph = __ldg(xin + p * cx);
        const float g0 = __ldg(dy + 2 * p) * ((1.f - ph) * (1.f + ph)), g1 = __ldg(dy + 2 * p + 1);
        const float4 v = ld4(x + p * c + ch);
        float4 d = make_float4(__fmaf_rn(w1[0], g1, w0[0] * g0), __fmaf_rn(w1[1], g1, w0[1] * g0),
                               __fmaf_rn(w1[2], g1, w0[2] * g0), __fmaf_rn(w1[3], g1, w0[3] * g0));
        if (!(v.x > 0.f)) d.x = 0.f;
        if (!(v.y > 0.f)) d.y = 0.f;
        if (!(v.z > 0.f)) d.z = 0.f;
        if (!(v.w > 0.f)) d.w = 0.f;
        st4(dx + p * c + ch, d);
        sl = add4(sl, d);
        s0 = add4(s0, make_float4(g0 * v.x, g0 * v.y, g0 * v.z, g0 * v.w));
        s1 = add4(s1, make_float4(g1 * v.x, g1 * v.y, g1 * v.z, g1 * v.w));
        if (ch == 0) {
            sb.x += g0;
            sb.y += g1;
        }
    }
    float* row = part + (size_t)blockIdx.x * (3 * c + 2);
    block_sum4(s0, q4, row, red);
    block_sum4(s1, q4, row + c, red);
    block_sum4(sl, q4, row + 2 * c + 2, red);
    // db: the first quad's threads hold the two sums
    __syncthreads();
    red[threadIdx.x] = sb;
    __syncthreads();
    for (int o = 128; o >= 1; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] = add4(red[threadIdx.x], red[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        row[2 * c] = red[0].x;
        row[2 * c + 1] = red[0].y;
    }
}

cudaError_t head_bwd(const float* x, const float* dy, const float* w, const float* xin, int cx, float* dx, float* part,
                     long long P, int c, cudaStream_t s)
{
    head_bwd_kernel<<<act_blocks(P, c), 256, 0, s>>>(x, dy, w, xin, cx, dx, part, P, c);
    return cudaGetLastError();
}

// Weighted mean squared error over n values (cout per site): loss[0] +=
// sum w (p - t)^2 / n (FP64 atomics per block), dp = 2 w (p - t) / n, with
// w = 1 + alpha max(0, 1 - phi^2) and phi = x[site * cin] the input phase
// field of the value's site (alpha = 0: plain mean squared error).
__global__ void mse_kernel(const float* p, const float* t, const float* x, int cin, int cout, float alpha, float* dp,
                           double* loss, long long n)
{
    double acc = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float d = p[i] - t[i];
        float w = 1.f;
        if (alpha > 0.f) {
            const float ph = x[(i / cout) * cin];
            w += alpha * fmaxf(0.f, 1.f - ph * ph);
        }
        dp[i] = 2.f * w * d / (float)n;
        acc += (double)w * d * d;
    }
    __shared__ double red[256];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, red[0] / (double)n);
}

cudaError_t mse(const float* p, const float* t, const float* x, int cin, int cout, float alpha, float* dp, double* loss,
                long long n, cudaStream_t s)
{
    mse_kernel<<<eblocks(n) < 304 ? eblocks(n) : 304, 256, 0, s>>>(p, t, x, cin, cout, alpha, dp, loss, n);
    return cudaGetLastError();
}

// Adam update of FP32 master weights; refreshes the BF16 copy when given.
__global__ void adam_kernel(float* w, const float* g, float* m, float* v, __nv_bfloat16* wb, long long n, float lr,
                            float b1, float b2, float eps, float c1, float c2)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        w[i] = wi;
        if (wb) wb[i] = __float2bfloat16_rn(wi);
    }
}

cudaError_t adam(float* w, const float* g, float* m, float* v, __nv_bfloat16* wb, long long n, float lr, float b1,
                 float b2, float eps, int t, cudaStream_t s)
{
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    adam_kernel<<<eblocks(n), 256, 0, s>>>(w, g, m, v, wb, n, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

__global__ void to_bf16_kernel(const float* a, __nv_bfloat16* b, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        b[i] = __float2bfloat16_rn(a[i]);
}

cudaError_t to_bf16(const float* a, __nv_bfloat16* b, long long n, cudaStream_t s)
{
    to_bf16_kernel<<<eblocks(n), 256, 0, s>>>(a, b, n);
    return cudaGetLastError();
}

// The network input's cin <= 8 channels into the first 8 of 16 (the others were
// cleared when y was allocated and stay zero): two threads a pixel.
__global__ void pad_channels_kernel(const float* x, float* y, long long P, int cin, int cout)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < 2 * P; i += (long long)gridDim.x * blockDim.x) {
        const int c = 4 * (int)(i & 1);
        const float* b = x + (i >> 1) * cin;
        float v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = c + k < cin ? b[c + k] : 0.f;
        st4(y + (i >> 1) * cout + c, make_float4(v[0], v[1], v[2], v[3]));
    }
}

cudaError_t pad_channels(const float* x, float* y, long long P, int cin, int cout, cudaStream_t s)
{
    if (cin > 8 || cout % 4) return cudaErrorInvalidValue;
    pad_channels_kernel<<<eblocks(2 * P), 256, 0, s>>>(x, y, P, cin, cout);
    return cudaGetLastError();
}

}  // namespace lbpf_nn

namespace lbpf_nn {

// x[p] = (phi, u, cos 4 theta, sin 4 theta, eps) of the site's crystal
// (crystal table tab[2 * (I - 1)] = eps, tab[2 * (I - 1) + 1] = theta; I from
// the index field, 1 everywhere when index is NULL; zeros where I = 0).
__global__ void assemble_kernel(const float* phi, const float* u, const int* index, const float* tab, int nc, float* x,
                                long long P)
{
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        const int I = index ? index[p] : 1;
        float c = 0.f, sn = 0.f, e = 0.f;
        if (I >= 1 && I <= nc) {
            e = tab[2 * (I - 1)];
            sincosf(4.f * tab[2 * (I - 1) + 1], &sn, &c);
        }
        float* o = x + p * 5;
        o[0] = phi[p];
        o[1] = u[p];
        o[2] = c;
        o[3] = sn;
        o[4] = e;
    }
}

cudaError_t assemble(const float* phi, const float* u, const int* index, const float* tab, int nc, float* x, long long P,
                     cudaStream_t s)
{
    assemble_kernel<<<eblocks(P), 256, 0, s>>>(phi, u, index, tab, nc, x, P);
    return cudaGetLastError();
}

// phi += y[p][0], u += y[p][1]
__global__ void apply_kernel(const float* y, float* phi, float* u, long long P)
{
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        phi[p] += y[2 * p];
        u[p] += y[2 * p + 1];
    }
}

cudaError_t apply(const float* y, float* phi, float* u, long long P, cudaStream_t s)
{
    apply_kernel<<<eblocks(P), 256, 0, s>>>(y, phi, u, P);
    return cudaGetLastError();
}

}  // namespace lbpf_nn

namespace lbpf_nn {

// y[p] = (phi1 - phi0, u1 - u0): training target of a jump.
__global__ void delta_kernel(const float* phi0, const float* u0, const float* phi1, const float* u1, float* y,
                             long long P)
{
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        y[2 * p] = phi1[p] - phi0[p];
        y[2 * p + 1] = u1[p] - u0[p];
    }
}

cudaError_t delta(const float* phi0, const float* u0, const float* phi1, const float* u1, float* y, long long P,
                  cudaStream_t s)
{
    delta_kernel<<<eblocks(P), 256, 0, s>>>(phi0, u0, phi1, u1, y, P);
    return cudaGetLastError();
}

// count[0] += number of phi values outside [lo, hi] (or not finite).
__global__ void range_kernel(const float* phi, long long P, float lo, float hi, unsigned int* count)
{
    unsigned int c = 0;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x)
        if (!(phi[p] >= lo && phi[p] <= hi)) ++c;
    if (c) atomicAdd(count, c);
}

cudaError_t range_count(const float* phi, long long P, float lo, float hi, unsigned int* count, cudaStream_t s)
{
    range_kernel<<<eblocks(P) < 608 ? eblocks(P) : 608, 256, 0, s>>>(phi, P, lo, hi, count);
    return cudaGetLastError();
}

}  // namespace lbpf_nn
