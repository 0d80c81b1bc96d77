// Steps a6-a8 at FP32 accuracy on the tensor cores: Green's function synthesis and the two
// complex contractions of an FP32 job (and the plain adjoint of every job), and the same with
// split BF16 (hi + lo).
//
//  forward (Eqs. perturb1, derivative):  D[e,r] = sum_x G_e[x] G_r[x] v[x]
//  back-projection (Eq. sound_speed_update2), exact two-term factorisation:
//     W_er = 2 (1 + s cos(gamma_e - gamma_r)) = 2 + s (kappa_e conj(kappa_r) + conj(kappa_e) kappa_r),
//     kappa = e^{i gamma}, s = -1 (printed scattering angle) or +1 (isochron); since W and
//     u_e u_r are symmetric in (e, r) the residual may be replaced by R_s = (R + R^T)/2, so
//     grad[x] = 2 sum_e u_e P0[x,e] + 2 s sum_e kappa_e u_e P1[x,e],
//     P0 = U^T R_s, P1 = (conj(kappa) U)^T R_s,
//  i.e. a complex GEMM with the two stacks as rows and a fused row-dot epilogue.
//
// An FP32 operand is held as three BF16 parts, v = hi + mid + lo, which together carry its 24
// bits exactly while its size lies between 2^-110 (1e-33; below, the last part would be less than BF16's
// smallest number, and the lowest bits go) and BF16's largest, 3.39e38 (a larger one, an infinity and not a number
// all give not a number). The six products hi hi, hi mid, mid hi, mid mid, hi lo, lo hi leave out terms of
// 2^-26 of the product. tcgen05 adds to its FP32 accumulators in tensor memory without rounding
// to nearest, so a long sum there drifts; here a sum in tensor memory covers 32 terms of K (one
// pipeline stage, the five small products before hi hi so that only four additions meet the
// full-size sum) and is then added to FP32 registers, rounded to nearest, by the epilogue warps.
// Two accumulator buffers alternate, so the MMAs do not wait for that. Split BF16 takes two parts
// and three products in the same way. Sums over 16 terms gave
// no smaller error (twice as many FP32 additions follow) and ran 7 % slower.
#include "rbx_internal.cuh"
#include "tc_sm100.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

namespace rbx {
using namespace tc;

namespace {

constexpr int BM = 128, BN = 128, BK = 32;
constexpr uint32_t PLANE = BM * BK * 2;                    // 8 KB: one part of one operand tile
// NP parts per real number: planes re hi (, mid), lo, im hi (, mid), lo
template <int NP>
struct Form {
    static constexpr int PLANES = 2 * NP;
    static constexpr uint32_t OPER = PLANES * PLANE;       // an operand's tile, all parts: 48 or 32 KB
    static constexpr int STAGES = NP == 3 ? 2 : 3;
    static constexpr size_t SMEM = 1024 + (size_t)STAGES * 2 * OPER + 2304;
    static constexpr int PRODUCTS = NP == 3 ? 6 : 3;
};
constexpr int EPI = 256;                                   // epilogue threads (warps 2..9)
constexpr int THREADS = 64 + EPI;

__device__ __forceinline__ float phase_cycles_(float T, int K, float fhi, float flo)
{
    float p = fhi * T;
    float err = fmaf(fhi, T, -p) + flo * T;
    float r = (p - rintf(p)) + err;
    return r + 0.125f - 0.25f * (float)K;
}

// Box of `planes` parts: with a 128-row box the K-major tile [part][row][32] (64-byte swizzle),
// with a 32-row box the M-major half tile [part][k][64] (128-byte swizzle).
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *m, uint64_t *bar, int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
        : "memory");
}

// K-major, 64-byte swizzle (rows of 32 BF16, 8-row groups 512 B apart).
__device__ __forceinline__ uint64_t desc_k64(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}
// M-major, 128-byte swizzle: 64 rows of M contiguous, the next 64 rows half an operand on, groups
// of 8 K 1024 B apart.
template <int NP>
__device__ __forceinline__ uint64_t desc_m128(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((Form<NP>::OPER / 2) >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// sin and cos of g in [-pi, pi] to about 1 ulp: sincospif of g / pi with the rounding of the
// quotient carried as a first-order correction.
__device__ __forceinline__ float2 unit_of(float g)
{
    const float IPI = 0.318309886183790672f, IPI_LO = 1.28412766e-8f, PI = 3.14159265358979f;
    const float r = g * IPI, d = PI * (fmaf(g, IPI, -r) + g * IPI_LO);
    float s, c;
    sincospif(r, &s, &c);
    return make_float2(fmaf(-s, d, c), fmaf(c, d, s));
}

struct GemmArgs {
    CUtensorMap a, b;
    int N, ntile, nk, kper;         // tiles of transducers, K chunks; forward: chunks per split
    float2 *part;                   // forward: [split][N][N] partial D
    const TabEntry *tab;            // back-projection: directions of stack 1
    int X;                          // back-projection: nodes
    float2 *bpart;                  // back-projection: [stack][e tile][X] partial row-dots
    unsigned *err;
};

// BP false: the forward's upper tile pair (te, tr) over the K chunks of one split.
// BP true: for 128 nodes, 128 emitters and one stack, P = A^T R_s over all receivers and the
// row-dot with the weights. CONJ: the plain adjoint, A = W = conj(G).
// NP = 3: FP32 accuracy, six products. NP = 2 (split BF16): hi hi + hi lo + lo hi; against kernels
// that drained long sums to global memory (forward) or stopped for the drain (back-projection),
// 768 transducers, 59,800 nodes: an update from tables 3.24 -> 2.60 ms (2.35 with the row-dot as it
// is now), forward error 2.7e-6 -> 1.1e-6.
//
// Bound: shared-memory bandwidth of the tensor cores. A 128 x 128 x 16 MMA reads 8 KB in the 64
// clocks it takes at the peak rate (128 B per clock, all an SM has), the tile loads write 31 B
// per clock besides, so 0.7-0.8 of the BF16 peak over the six products is what the form allows (tensor
// pipes busy, ncu: plain adjoint of 768 transducers 65 % of the launch; of 256, forward 53 %, back-projection 49 %:
// there the start of each CTA, its last drain and the row-dot weigh more).
// K chunks of 32 because a 64-term stage of both operands' parts (192 KB) leaves no second one.
// Against FP32 multiply-adds on the CUDA cores (64 x 64 tiles, 0.5 of their peak), ncu: 256
// transducers, 48,120 nodes: forward 437 -> 89 us, back-projection 1297 -> 321 us (its row-dot as it
// is now takes another 75 us off the update); 768 transducers, 19,760 nodes: plain adjoint 2915 -> 384
// us, 364 now. Error against 64 bits smaller at
// every size from 5 transducers on (N = 1024, 20,000 nodes: forward 6.0e-7 -> 2.2e-7, plain adjoint
// 6.1e-7 -> 1.7e-7; N = 8, mean of six tables: forward 2.7e-7 -> 1.2e-7, plain 1.42e-7 -> 1.36e-7,
// preconditioned 1.9e-7 -> 1.7e-7); with 3 transducers the plain adjoint's is 1.30e-7 -> 1.37e-7.
template <int NP, bool BP, bool CONJ>
__global__ __launch_bounds__(THREADS, 1) void k_cgemm_f32(const __grid_constant__ GemmArgs g)
{
    constexpr int STAGES = Form<NP>::STAGES, PLANES = Form<NP>::PLANES;
    constexpr uint32_t OPER = Form<NP>::OPER;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *full = reinterpret_cast<uint64_t *>(tiles + (size_t)STAGES * 2 * OPER);
    uint64_t *empty = full + STAGES;
    uint64_t *accf = empty + STAGES;       // [2] accumulator buffer ready to drain
    uint64_t *acce = accf + 2;             // [2] accumulator buffer drained
    uint64_t *wfull = acce + 2;            // [2] weights of the tile's emitters 0-63, 64-127 landed
    float2 *half_sum = reinterpret_cast<float2 *>(wfull + 2);   // [2][128]
    uint32_t *tslot = reinterpret_cast<uint32_t *>(half_sum + 2 * BM);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int N = g.N;

    int ta, tb, c0 = 0, nc;                // tile of A (rows of D), tile of B (columns), K chunks
    if (BP) {
        tb = blockIdx.x % g.ntile;         // one grid dimension: any number of nodes
        ta = blockIdx.x / g.ntile;
        nc = g.nk;
    } else {
        int b = blockIdx.x, te = 0;
        while (b >= g.ntile - te) { b -= g.ntile - te; te++; }
        ta = te;
        tb = te + b;
        c0 = blockIdx.y * g.kper;
        nc = min(g.nk, c0 + g.kper) - c0;
    }
    const int stack = BP ? blockIdx.y : 0;
    const int ncol = min(BN, (N - tb * BN + 15) & ~15);   // columns of the MMAs (a ragged last tile)

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; s++) { mbar_init(full + s, 1); mbar_init(empty + s, 1); }
        for (int q = 0; q < 2; q++) { mbar_init(accf + q, 1); mbar_init(acce + q, EPI); mbar_init(wfull + q, 1); }
        fence_mbar_init();
    }
    if (warp == 1) tmem_alloc(tslot, 512);
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;

    if (warp == 0 && lane == 0) {
        prefetch_tmap(&g.a);
        if (BP) prefetch_tmap(&g.b);
        int issued = 0;
        for (int c = 0; c < nc; c++) {
            const int s = c % STAGES;
            if (c >= STAGES && !mbar_wait(empty + s, ((c / STAGES) - 1) & 1)) { atomicOr(g.err, 1u); break; }
            mbar_arrive_expect_tx(full + s, 2 * OPER);
            const uint32_t base = smem_u32(tiles + (size_t)s * 2 * OPER);
            const int k = (c0 + c) * BK;
            if (BP) {
                tma_load_3d(base, &g.a, full + s, ta * BM, k, PLANES * stack);
                tma_load_3d(base + OPER / 2, &g.a, full + s, ta * BM + 64, k, PLANES * stack);
                tma_load_3d(base + OPER, &g.b, full + s, k, tb * BN, 0);
            } else {
                tma_load_3d(base, &g.a, full + s, k, ta * BM, 0);
                tma_load_3d(base + OPER, &g.a, full + s, k, tb * BN, PLANES);
            }
            issued++;
        }
        // the row-dot's weights (the first operand's rows of the tile's emitters), 64 emitters to
        // each of the first two stages that the MMAs leave
        int halves = 0;
        for (; BP && issued == nc && halves < 2; halves++) {
            const int s = (nc + halves) % STAGES, c = nc - STAGES + halves;
            if (c >= 0 && !mbar_wait(empty + s, (c / STAGES) & 1)) { atomicOr(g.err, 64u); break; }
            mbar_arrive_expect_tx(wfull + halves, 2 * OPER);
            for (int q = 0; q < 4; q++)
                tma_load_3d(smem_u32(tiles + (size_t)s * 2 * OPER + q * (OPER / 2)), &g.a, wfull + halves,
                            ta * BM + (q & 1) * 64, tb * BN + halves * 64 + (q >> 1) * BK, 0);
        }
        // no copy may still be in flight when the CTA retires
        for (int h = 0; h < halves; h++)
            if (!mbar_wait(wfull + h, 0)) atomicOr(g.err, 4u);
        for (int c = (issued > STAGES ? issued - STAGES : 0); c < issued; c++)
            if (!mbar_wait(full + (c % STAGES), (c / STAGES) & 1)) atomicOr(g.err, 4u);
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t mn = BP ? (1u << 15) : 0u;      // A is M-major
            const uint32_t ip = idesc_bf16(BM, ncol, 0) | mn, in = idesc_bf16(BM, ncol, 1) | mn;
            const uint32_t i_re = CONJ ? ip : in, i_im = CONJ ? in : ip;   // signs of A_im B_im and A_im B_re
            bool ok = true;
            for (int c = 0; c < nc && ok; c++) {
                const int buf = c & 1, s = c % STAGES;
                if (c >= 2 && !mbar_wait(acce + buf, ((c >> 1) - 1) & 1)) { atomicOr(g.err, 32u); ok = false; break; }
                if (!mbar_wait(full + s, (c / STAGES) & 1)) { atomicOr(g.err, 2u); ok = false; break; }
                fence_after();
                const uint32_t dre = tmem + buf * 2 * BN, dim = dre + BN;
                const uint32_t a = smem_u32(tiles + (size_t)s * 2 * OPER), b = a + OPER;
                constexpr uint32_t APART = BP ? PLANE / 2 : PLANE, AK = BP ? 2048 : 32;
#pragma unroll
                for (int p = 6 - Form<NP>::PRODUCTS; p < 6; p++) {
                    // three parts: (hi, lo), (lo, hi), (mid, mid), (hi, mid), (mid, hi), (hi, hi); of
                    // two parts, hi and lo, the last three
                    constexpr int PA[6] = {0, 2, 1, 0, 1, 0}, PB[6] = {2, 0, 1, 1, 0, 0};
#pragma unroll
                    for (int k = 0; k < BK / 16; k++) {
                        const uint32_t ar = a + PA[p] * APART + k * AK, br = b + PB[p] * PLANE + k * 32;
                        const uint64_t a0 = BP ? desc_m128<NP>(ar) : desc_k64(ar);
                        const uint64_t a1 = BP ? desc_m128<NP>(ar + NP * APART) : desc_k64(ar + NP * APART);
                        const uint64_t b0 = desc_k64(br), b1 = desc_k64(br + NP * PLANE);
                        const uint32_t acc = (p > 6 - Form<NP>::PRODUCTS || k > 0) ? 1u : 0u;
                        mma_bf16(dre, a0, b0, ip, acc);
                        mma_bf16(dre, a1, b1, i_re, 1u);
                        mma_bf16(dim, a0, b1, ip, acc);
                        mma_bf16(dim, a1, b0, i_im, 1u);
                    }
                }
                mma_commit(empty + s);
                mma_commit(accf + buf);
            }
            // every MMA of this CTA has completed once the last buffer is signalled
            if (ok && !mbar_wait(accf + ((nc - 1) & 1), ((nc - 1) >> 1) & 1)) atomicOr(g.err, 8u);
        }
        __syncwarp();
    } else if (warp >= 2) {
        // warp w reads TMEM lanes 32 (w mod 4) .. + 31; warps 2-5 columns 0-63, warps 6-9 the rest
        const int sub = warp & 3, row = sub * 32 + lane, half = (warp - 2) >> 2;
        const uint32_t at = tmem + ((uint32_t)(sub * 32) << 16) + half * 64;
        float re[64], im[64];
#pragma unroll
        for (int i = 0; i < 64; i++) re[i] = im[i] = 0.f;
        bool ok = true;
        for (int c = 0; c < nc; c++) {
            const int buf = c & 1;
            ok = __all_sync(0xffffffffu, mbar_wait(accf + buf, (c >> 1) & 1));
            if (!ok) {
                if (lane == 0) atomicOr(g.err, 16u);
                break;
            }
            fence_after();
            if (half * 64 < ncol) {
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    float t[32];
                    tmem_ld32(at + buf * 2 * BN + (q >> 1) * BN + (q & 1) * 32, t);
                    float *d = (q < 2 ? re : im) + (q & 1) * 32;
#pragma unroll
                    for (int i = 0; i < 32; i++) d[i] += t[i];
                }
            }
            fence_before();
            mbar_arrive(acce + buf);
        }
        if (!BP) {
            const int e = ta * BM + row;
            float2 *P = g.part + ((size_t)blockIdx.y * N + e) * N;
            if (e < N) {
#pragma unroll
                for (int i = 0; i < 64; i++) {
                    const int r = tb * BN + half * 64 + i;
                    if (r < N) P[r] = make_float2(re[i], im[i]);
                }
            }
        } else {
            // The row-dot: a thread's node and 64 emitters. P goes back to tensor memory, so that a
            // loop over eight emitters at a time can index it; the weights come by TMA into the
            // stages, in the layout of the first operand, two of them while the last products run
            // (loaded from global memory into registers, eight emitters at a time: 768 transducers,
            // 59,800 nodes, split: an update from tables 2.58 -> 2.35 ms; 256, 48,120 nodes, FP32:
            // an update 75 us less).
            const int xl = min(ta * BM + row, g.X - 1), e0 = tb * BN + half * 64, ne = min(64, N - e0);
            const TabEntry *tab = g.tab + (size_t)e0 * g.X + xl;
            const uint8_t *wt = tiles + (size_t)((nc + half) % STAGES) * 2 * OPER + (row >> 6) * (OPER / 2);
            const uint32_t chunk = (uint32_t)(row & 63) >> 3, in_chunk = (uint32_t)(row & 7) * 2;
            float2 s[8];   // partial sums, of every eighth emitter
#pragma unroll
            for (int k = 0; k < 8; k++) s[k] = make_float2(0.f, 0.f);
            // directions of the weights kappa u, loaded eight emitters ahead
            uint32_t idk[8];
            float gam[8];
            auto directions = [&](int i0) {
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    const TabEntry *t = tab + (size_t)min(i0 + k, ne - 1) * g.X;
                    idk[k] = __ldg(&t->idk);
                    gam[k] = __ldg(&t->gam);
                }
            };
            if (!CONJ && stack == 1 && ne > 0) directions(0);
            const bool have = __all_sync(0xffffffffu, ok && mbar_wait(wfull + half, 0));
            if (!have && lane == 0) atomicOr(g.err, 64u);
            if (have) {
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    tmem_st32(at + q * 32, re + q * 32);
                    tmem_st32(at + BN + q * 32, im + q * 32);
                }
            }
#pragma unroll 1
            for (int i0 = 0; have && i0 < ne; i0 += 8) {
                float2 kap[8];
                if (!CONJ && stack == 1) {
                    // an uncovered entry's weight is zero and its direction not a number
#pragma unroll
                    for (int k = 0; k < 8; k++) kap[k] = unit_of(idk[k] == kUncovered ? 0.f : gam[k]);
                    if (i0 + 8 < ne) directions(i0 + 8);
                }
                float pr[8], pi[8];
                tmem_ld8(at + i0, pr);
                tmem_ld8(at + BN + i0, pi);
                const uint8_t *wk = wt + (size_t)(i0 >> 5) * OPER + (i0 & 31) * 128;
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    const uint8_t *z = wk + k * 128 + ((chunk ^ (uint32_t)k) << 4) + in_chunk;
                    // the parts add up to the weight (three: the FP32 weight) exactly
                    float wr = 0.f, wi = 0.f;
#pragma unroll
                    for (int m = 0; m < NP; m++) {
                        wr += __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(z + m * (PLANE / 2)));
                        wi += __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(z + (NP + m) * (PLANE / 2)));
                    }
                    if (CONJ) wi = -wi;
                    if (!CONJ && stack == 1) {
                        const float ur = wr;
                        wr = kap[k].x * ur - kap[k].y * wi;
                        wi = kap[k].x * wi + kap[k].y * ur;
                    }
                    s[k].x = fmaf(wr, pr[k], s[k].x);
                    s[k].x = fmaf(-wi, pi[k], s[k].x);
                    s[k].y = fmaf(wr, pi[k], s[k].y);
                    s[k].y = fmaf(wi, pr[k], s[k].y);
                }
            }
#pragma unroll
            for (int d = 4; d > 0; d >>= 1)
#pragma unroll
                for (int k = 0; k < d; k++) {
                    s[k].x += s[k + d].x;
                    s[k].y += s[k + d].y;
                }
            half_sum[half * BM + row] = s[0];
            asm volatile("bar.sync 1, 256;" ::: "memory");   // the epilogue warps
            const int t = threadIdx.x - 64;
            const int xo = ta * BM + t;
            if (t < BM && xo < g.X) {
                const float2 a = half_sum[t], b = half_sum[BM + t];
                g.bpart[((size_t)stack * g.ntile + tb) * g.X + xo] = make_float2(a.x + b.x, a.y + b.y);
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// v = hi (+ mid) + lo, each BF16
template <int NP>
__device__ __forceinline__ void split(float v, __nv_bfloat16 *q)
{
#pragma unroll
    for (int k = 0; k < NP; k++) {
        q[k] = __float2bfloat16_rn(v);
        v -= __bfloat162float(q[k]);
    }
}

// The parts of two neighbouring complex values to [plane][N][xld]
template <int NP>
__device__ __forceinline__ void put_parts(__nv_bfloat16 *planes, size_t pstride, size_t at, const float2 *z)
{
    __nv_bfloat16 a[2 * NP], b[2 * NP];
    split<NP>(z[0].x, a);
    split<NP>(z[0].y, a + NP);
    split<NP>(z[1].x, b);
    split<NP>(z[1].y, b + NP);
#pragma unroll
    for (int k = 0; k < 2 * NP; k++)
        *reinterpret_cast<__nv_bfloat162 *>(planes + k * pstride + at) = __halves2bfloat162(a[k], b[k]);
}

// Operands of the contractions from the tables, two nodes and `walk` transducers per thread, as
// parts in [plane][N][xld].
//  KIND 0: first operand G_e[x] = (8 pi omega/c0)^(-1/2) a exp(i 2 pi (f T - K/4 + 1/8)) (Eq. 2D_greens)
//  KIND 1: first G, second G v (the forward)
//  KIND 2: first u_e[x] = dgamma / ((8 pi omega/c0)^(-1/2) a) exp(-i 2 pi (...)) (Eq.
//          greens-time-reversed), second conj(kappa) u. The angular density dgamma (step a4)
//          comes from the direction angles of the neighbouring transducers, kept in registers as
//          the thread walks its transducers: the tables are read 1 + 2 / walk times and no
//          array of dgamma is written or read.
// Bound: HBM. Per entry 16 B are read and 8 NP B (4 NP for KIND 0) written; 512 transducers, 47,660
// nodes, NP = 3: 0.98 GB in 147 us.
template <int KIND, int NP>
__global__ __launch_bounds__(128) void k_synth_parts(const TabEntry *__restrict__ tab, const float2 *__restrict__ v, int N,
                                                     int X, int xld, size_t pstride, float fhi, float flo,
                                                     float C, __nv_bfloat16 *__restrict__ planes, int walk)
{
    const int xl = 2 * (blockIdx.x * blockDim.x + threadIdx.x), e0 = blockIdx.y * walk;
    if (xl >= X) return;
    const bool two = xl + 1 < X;
    const TabEntry *t = tab + xl;
    TabEntry none;
    none.idk = kUncovered;
    none.T = none.a = none.gam = 0.f;
    TabEntry prev[2], cur[2], next[2];
    auto row = [&](int e, TabEntry *o) {
        o[0] = t[(size_t)e * X];
        o[1] = two ? t[(size_t)e * X + 1] : none;
    };
    if (KIND == 2) row((e0 + N - 1) % N, prev);
    row(e0, cur);
    float2 w[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    if (KIND == 1) {
        w[0] = v[xl];
        if (two) w[1] = v[xl + 1];
    }
    const int e1 = min(N, e0 + walk);
    for (int e = e0; e < e1; e++) {
        if (KIND == 2 || e + 1 < e1) row((e + 1) % N, next);
        float2 z[2], z2[2];
#pragma unroll
        for (int q = 0; q < 2; q++) {
            z[q] = z2[q] = make_float2(0.f, 0.f);
            if (cur[q].idk == kUncovered) continue;
            float s, c;
            sincospif(2.f * phase_cycles_(cur[q].T, (int)(cur[q].idk & 0xffu), fhi, flo), &s, &c);
            if (KIND == 2) {
                const float dg = (next[q].idk == kUncovered || prev[q].idk == kUncovered)
                                     ? 0.f : dgamma_of(next[q].gam, prev[q].gam);
                const float A = dg / (C * cur[q].a);
                z[q] = make_float2(A * c, -A * s);
                const float2 k = unit_of(cur[q].gam);
                z2[q] = make_float2(k.x * z[q].x + k.y * z[q].y, k.x * z[q].y - k.y * z[q].x);
            } else {
                const float A = C * cur[q].a;
                z[q] = make_float2(A * c, A * s);
                if (KIND == 1)
                    z2[q] = make_float2(z[q].x * w[q].x - z[q].y * w[q].y, z[q].x * w[q].y + z[q].y * w[q].x);
            }
        }
        const size_t at = (size_t)e * xld + xl;
        put_parts<NP>(planes, pstride, at, z);
        if (KIND != 0) put_parts<NP>(planes + 2 * NP * pstride, pstride, at, z2);
#pragma unroll
        for (int q = 0; q < 2; q++) {
            prev[q] = cur[q];
            cur[q] = next[q];
        }
    }
}

// R_s (complex N x N; SYM: R, from which R_s = (R + R^T)/2 is formed here, one launch less in an
// adjoint) -> parts [2 NP][N][rld]
template <int NP, bool SYM>
__global__ void k_rs_parts(const float2 *__restrict__ Rs, int N, int rld, __nv_bfloat16 *__restrict__ planes)
{
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= (size_t)N * N) return;
    const size_t o = (i / N) * rld + i % N, P = (size_t)N * rld;
    __nv_bfloat16 q[2 * NP];
    float2 v = Rs[i];
    if (SYM) {
        const float2 t = Rs[(i % N) * N + i / N];
        v = make_float2(0.5f * (v.x + t.x), 0.5f * (v.y + t.y));
    }
    split<NP>(v.x, q);
    split<NP>(v.y, q + NP);
#pragma unroll
    for (int k = 0; k < 2 * NP; k++) planes[k * P + o] = q[k];
}

// gpart[stack][x] = sum over emitter tiles, in order
__global__ void k_bp_sum(const float2 *__restrict__ bpart, int ET, int X, float2 *__restrict__ gpart)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= X) return;
    float2 s = make_float2(0.f, 0.f);
    for (int t = 0; t < ET; t++) {
        const float2 p = bpart[((size_t)blockIdx.y * ET + t) * X + x];
        s.x += p.x;
        s.y += p.y;
    }
    gpart[(size_t)blockIdx.y * X + x] = s;
}

void fsplit(double f, float &fhi, float &flo)
{
    fhi = (float)f;
    flo = (float)(f - (double)fhi);
}

float green_const(double f, double c0)
{
    return (float)(1.0 / sqrt(8.0 * 3.14159265358979323846 * (2.0 * 3.14159265358979323846 * f) / c0));
}

// BF16 planes [planes][rows][cols], rows ld elements apart, read in boxes of `inner` columns,
// `outer` rows and `deep` planes
bool make_map(CUtensorMap *m, void *base, size_t cols, size_t rows, size_t planes, size_t ld, unsigned inner,
              unsigned outer, unsigned deep)
{
    cuuint64_t dims[3] = {cols, rows, planes};
    cuuint64_t strides[2] = {ld * 2, ld * rows * 2};
    cuuint32_t box[3] = {inner, outer, deep}, estr[3] = {1, 1, 1};
    return encode_tiled(m, base, 3, dims, strides, box, estr,
                        inner * 2 == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B);
}

template <int KIND>
void synth(const F32Planes &p, const TabEntry *tab, const float2 *v, double f, double c0, cudaStream_t s)
{
    float fhi, flo;
    fsplit(f, fhi, flo);
    // a walk of 8 once that still gives every SM a full set of blocks; short ones on small
    // problems, which a long walk leaves waiting on its chain of loads
    const unsigned bx = (unsigned)((p.X + 255) / 256);
    const int walk = (size_t)bx * ((p.N + 7) / 8) >= 152 * 16 ? 8 : 2;
    const dim3 grd(bx, (unsigned)((p.N + walk - 1) / walk));
    __nv_bfloat16 *planes = static_cast<__nv_bfloat16 *>(p.planes);
    auto go = [&](auto parts) {
        k_synth_parts<KIND, decltype(parts)::value><<<grd, 128, 0, s>>>(tab, v, p.N, p.X, p.xld, p.pstride, fhi, flo,
                                                                        green_const(f, c0), planes, walk);
    };
    if constexpr (KIND != 0) {   // the plain adjoint always takes three parts
        if (p.parts == 2) return go(std::integral_constant<int, 2>{});
    }
    go(std::integral_constant<int, 3>{});
}

}  // namespace

// Splits of the forward's K loop: the tile pairs fill the GPU once, at most 64 partials (the
// bound of the job's memory estimate) and no split below three K chunks (the start of a CTA
// and its drain cost about as much).
int forward_splits(int N, int X)
{
    const int T = (N + BM - 1) / BM, pairs = T * (T + 1) / 2, nk = (X + BK - 1) / BK;
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int s = std::max(1, sms / pairs);
    s = std::min(s, std::min(64, (nk + 2) / 3));
    const int kper = (nk + s - 1) / s;
    return (nk + kper - 1) / kper;
}

template <int NP>
static bool allow_smem()
{
    return cudaFuncSetAttribute(k_cgemm_f32<NP, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Form<NP>::SMEM) == cudaSuccess &&
           cudaFuncSetAttribute(k_cgemm_f32<NP, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Form<NP>::SMEM) == cudaSuccess &&
           (NP != 3 ||   // the plain adjoint always takes three parts
            cudaFuncSetAttribute(k_cgemm_f32<3, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)Form<3>::SMEM) == cudaSuccess);
}

bool f32_setup(F32Planes &p, int N, int X, int parts, bool full, unsigned *err, cudaStream_t st)
{
    p.err = err;
    p.N = N;
    p.X = X;
    p.parts = parts;
    // all nodes' forward or back-projection operands (24 or 16 B an entry), or on a BF16 or split
    // BF16 job the plain adjoint's alone (12 B)
    p.xld = (X + 7) / 8 * 8;
    p.pstride = (size_t)N * p.xld;
    p.rld = (N + 7) / 8 * 8;
    const size_t deep = 2 * parts, planes = full ? 2 * deep : deep;
    const size_t ET = (N + BN - 1) / BN;
    if (cudaMallocAsync(&p.planes, planes * p.pstride * sizeof(__nv_bfloat16), st) != cudaSuccess) return false;
    if (cudaMallocAsync(&p.rs, deep * N * p.rld * sizeof(__nv_bfloat16), st) != cudaSuccess) return false;
    if (ET > 1 &&   // with one emitter tile the partial row-dots are the result
        cudaMallocAsync(reinterpret_cast<void **>(&p.bpart), (full ? 2 : 1) * ET * X * sizeof(float2), st) != cudaSuccess)
        return false;
    return make_map(&p.fmap, p.planes, X, N, planes, p.xld, BK, BM, deep) &&
           make_map(&p.amap, p.planes, X, N, planes, p.xld, 64, BK, deep) &&
           make_map(&p.rmap, p.rs, N, N, deep, p.rld, BK, BN, deep) && (parts == 3 ? allow_smem<3>() : allow_smem<2>());
}

void f32_free(F32Planes &p, cudaStream_t st)
{
    void *ps[] = {p.planes, p.rs, p.bpart};
    for (void *q : ps)
        if (q) cudaFreeAsync(q, st);
    p = F32Planes{};
}

void launch_synth_fwd(F32Planes &p, const TabEntry *tab, const float2 *v, double f, double c0, cudaStream_t s)
{
    synth<1>(p, tab, v, f, c0, s);
}

void launch_synth_bp(F32Planes &p, const TabEntry *tab, double f, double c0, cudaStream_t s)
{
    synth<2>(p, tab, nullptr, f, c0, s);
}

void launch_forward_f32(F32Planes &p, int splits, float2 *part, cudaStream_t s)
{
    const int T = (p.N + BM - 1) / BM, nk = (p.X + BK - 1) / BK;
    GemmArgs g{};
    g.a = g.b = p.fmap;
    g.N = p.N;
    g.ntile = T;
    g.nk = nk;
    g.kper = (nk + splits - 1) / splits;
    g.part = part;
    g.err = p.err;
    const dim3 grd(T * (T + 1) / 2, splits);
    if (p.parts == 3)
        k_cgemm_f32<3, false, false><<<grd, THREADS, Form<3>::SMEM, s>>>(g);
    else
        k_cgemm_f32<2, false, false><<<grd, THREADS, Form<2>::SMEM, s>>>(g);
}

static GemmArgs bp_args(F32Planes &p, const TabEntry *tab, float2 *gpart)
{
    GemmArgs g{};
    g.a = p.amap;
    g.b = p.rmap;
    g.N = p.N;
    g.ntile = (p.N + BN - 1) / BN;
    g.nk = (p.N + BK - 1) / BK;
    g.tab = tab;
    g.X = p.X;
    g.bpart = p.bpart ? p.bpart : gpart;
    g.err = p.err;
    return g;
}

template <bool SYM>
static void rs_parts(F32Planes &p, const float2 *Rs, cudaStream_t s)
{
    const size_t nn = (size_t)p.N * p.N;
    const unsigned nb = (unsigned)((nn + 255) / 256);
    if (p.parts == 3)
        k_rs_parts<3, SYM><<<nb, 256, 0, s>>>(Rs, p.N, p.rld, static_cast<__nv_bfloat16 *>(p.rs));
    else
        k_rs_parts<2, SYM><<<nb, 256, 0, s>>>(Rs, p.N, p.rld, static_cast<__nv_bfloat16 *>(p.rs));
}

// The preconditioned back-projection from the operands of launch_synth_bp: gpart[2][X].
int launch_backproject_f32(F32Planes &p, const TabEntry *tab, const float2 *R, bool symmetric, float2 *gpart,
                           cudaStream_t s)
{
    const int ET = (p.N + BN - 1) / BN;
    if (symmetric)
        rs_parts<false>(p, R, s);
    else
        rs_parts<true>(p, R, s);
    const GemmArgs g = bp_args(p, tab, gpart);
    const dim3 grd((unsigned)ET * ((p.X + BM - 1) / BM), 2);
    if (p.parts == 3)
        k_cgemm_f32<3, true, false><<<grd, THREADS, Form<3>::SMEM, s>>>(g);
    else
        k_cgemm_f32<2, true, false><<<grd, THREADS, Form<2>::SMEM, s>>>(g);
    if (ET == 1) return 2;
    k_bp_sum<<<dim3((p.X + 255) / 256, 2), 256, 0, s>>>(p.bpart, ET, p.X, gpart);
    return 3;
}

// The plain adjoint's sum_{e,r} conj(G_e G_r) R_s: synthesis and contraction, all nodes at once (BF16
// job, 48 transducers, 2,828 nodes: 22.6 us, 37 in two slabs of nodes; 24.7 as FP32 multiply-adds).
int launch_adjoint_f32(F32Planes &p, const TabEntry *tab, const float2 *R, double f, double c0, float2 *gpart,
                       cudaStream_t s)
{
    const int ET = (p.N + BN - 1) / BN;
    rs_parts<true>(p, R, s);
    synth<0>(p, tab, nullptr, f, c0, s);
    k_cgemm_f32<3, true, true><<<(unsigned)ET * ((p.X + BM - 1) / BM), THREADS, Form<3>::SMEM, s>>>(bp_args(p, tab, gpart));
    if (ET == 1) return 3;
    k_bp_sum<<<dim3((p.X + 255) / 256, 1), 256, 0, s>>>(p.bpart, ET, p.X, gpart);
    return 4;
}

}  // namespace rbx
