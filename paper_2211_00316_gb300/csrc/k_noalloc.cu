// Born forward for callers that cannot allocate device memory.
//
// Some callers cannot call cudaMalloc at all: code running inside a CUDA-graph capture
// that must not add allocation nodes, plug-ins hosted by a framework whose caching
// allocator owns the whole device, or real-time services that forbid allocation after
// start-up. rbx_forward_noalloc serves them: it computes the same D as rbx_forward but
// takes the tables straight from the caller, synthesises the Green's functions inside
// the contraction (no N x X operand buffer), and keeps its only scratch -- the split
// partial sums -- in one fixed array in this library's device memory.
//
// The scratch is a file-scope __device__ array of kScratchElems float2 (8 MiB). Every GPU
// that loads the library holds it until the process exits. All calls share it, and each
// call overwrites every element it later reads, so nothing needs clearing between calls;
// calls whose work overlaps on the GPU (different streams, or different host threads on
// one device) race on it and must be serialised by the caller.
//
// In host code the array's name is only a stand-in for the device object, so the device
// address is fetched with cudaGetSymbolAddress once per device, with that device current,
// on the first call made on it. That first call may load the module; make it before any
// stream capture.
#include "rbx_internal.cuh"
#include "tc_sm100.cuh"

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <cmath>
#include <cstdio>
#include <mutex>

namespace rbx {
using namespace tc;
namespace cg = cooperative_groups;

constexpr size_t kScratchElems = 1u << 20;   // float2 elements: 8 MiB
static __device__ __align__(256) float2 g_fwd_scratch[kScratchElems];

namespace {

constexpr int BM = 128, BK = 32, STAGES = 2;
constexpr uint32_t PLANE = BM * BK * 2, OPER = 6 * PLANE;   // an operand's tile: re hi, mid, lo, im hi, mid, lo
constexpr size_t NA_SMEM = 1024 + (size_t)STAGES * 2 * OPER + 256;
constexpr int THREADS = 512;

__device__ __forceinline__ float phase_cycles_na(float T, int K, float fhi, float flo)
{
    float p = fhi * T;
    float err = fmaf(fhi, T, -p) + flo * T;
    float r = (p - rintf(p)) + err;
    return r + 0.125f - 0.25f * (float)K;
}

// K-major, 64-byte swizzle (rows of 32 BF16, 8-row groups 512 B apart).
__device__ __forceinline__ uint64_t desc_k64(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

// The three BF16 parts of four neighbouring values to the planes at `at` (8 bytes each).
__device__ __forceinline__ void put3(uint8_t *at, float4 v)
{
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
        uint2 u;
        u.x = *reinterpret_cast<const uint32_t *>(&a);
        u.y = *reinterpret_cast<const uint32_t *>(&b);
        *reinterpret_cast<uint2 *>(at + k * PLANE) = u;
        v.x -= __low2float(a);
        v.y -= __high2float(a);
        v.z -= __low2float(b);
        v.w -= __high2float(b);
    }
}

struct NaArgs {
    const float *T, *a, *v;
    const uint8_t *K;
    int N, X, ntile, nk, kper;   // nk K chunks of 32 nodes, kper per CTA
    float fhi, flo, C;
    float2 *part;
};

// D = sum_x G_e G_r v for an upper 128 x 128 tile pair over a range of nodes, on the tensor
// cores at FP32 accuracy (three BF16 parts per operand, six products, 32-node sums in tensor
// memory added to FP32 registers), the operands formed from the tables where the MMAs read
// them. Sixteen warps form the tiles (128-byte rows of the tables, four nodes per thread, stored in
// the 64-byte-swizzled K-major layout of the MMA descriptors) and, between two tiles, add the
// finished sums to their registers; one thread of the first issues the MMAs.
// The CTAs of a cluster take parts of the same tile's nodes and add their sums up through
// distributed shared memory in rank order, because the fixed scratch holds few partial sums
// (one at 1024 transducers, which would leave 116 SMs idle).
// Bound: the synthesis, about 65 instructions for each of a chunk's 8192 entries (4096 on the
// diagonal) and the latency of their loads (issue port busy 42 % of cycles), against 3100 clocks
// of MMAs.
// 256 transducers, 48,120 nodes: 1.52 -> 0.21 ms; 1024, 152,088: 69.3 -> 7.1 ms; 64, 5,140: 87 -> 40 us (FP32
// multiply-adds in 64 x 64 tiles, with the hardware sine and cosine; error against 64 bits 1.1e-6
// -> 1.3e-7 at 256, 3.3e-6 -> 2.3e-7 at 1024). Prefetching the next tables' lines into L2 cost 8 %.
__global__ __launch_bounds__(THREADS, 1) void k_forward_tables(const __grid_constant__ NaArgs g)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *full = reinterpret_cast<uint64_t *>(tiles + (size_t)STAGES * 2 * OPER);
    uint64_t *empty = full + STAGES;
    uint64_t *accf = empty + STAGES;       // [2] accumulator buffer ready to drain
    uint32_t *tslot = reinterpret_cast<uint32_t *>(accf + 2);
    cg::cluster_group cluster = cg::this_cluster();
    const int cs = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, N = g.N, X = g.X;
    int b = blockIdx.x / cs, te = 0;
    while (b >= g.ntile - te) { b -= g.ntile - te; te++; }
    const int tr = te + b;
    const int c0 = ((int)blockIdx.y * cs + rank) * g.kper, nc = max(0, min(g.nk, c0 + g.kper) - c0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; s++) { mbar_init(full + s, THREADS); mbar_init(empty + s, 1); }
        for (int q = 0; q < 2; q++) mbar_init(accf + q, 1);
        fence_mbar_init();
    }
    if (warp == 0) tmem_alloc(tslot, 512);
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;
    float re[32], im[32];
#pragma unroll
    for (int i = 0; i < 32; i++) re[i] = im[i] = 0.f;

    {
        const int sub = warp & 3, col0 = (warp >> 2) * 32;
        const int q4 = threadIdx.x & 7, r0 = threadIdx.x >> 3;   // four nodes of rows r0 and r0 + 64
        bool ok = true;
        // tile rows `tile` (both halves) at chunk kx: G, times v too when with_v
        auto form = [&](int tile, int kx, uint8_t *to, uint8_t *to_v, const float4 &w) {
            float T[2][4], a[2][4];
            int K[2][4];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int row = tile * BM + r0 + 64 * h;
                const size_t at = (size_t)row * X + kx + 4 * q4;
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const bool in = row < N && kx + 4 * q4 + i < X;
                    T[h][i] = in ? g.T[at + i] : 0.f;
                    a[h][i] = in ? g.a[at + i] : 0.f;
                    K[h][i] = in ? (int)g.K[at + i] : 0;
                }
            }
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int r = r0 + 64 * h;
                const uint32_t off = (uint32_t)r * 64u + ((((uint32_t)q4 >> 1) ^ (((uint32_t)r >> 1) & 3u)) << 4) +
                                     (((uint32_t)q4 & 1u) << 3);
                float zr[4], zi[4];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    float s, c;
                    sincospif(2.f * phase_cycles_na(T[h][i], K[h][i], g.fhi, g.flo), &s, &c);
                    const float A = a[h][i] > 0.f ? g.C * a[h][i] : 0.f;   // 0: uncovered
                    zr[i] = a[h][i] > 0.f ? A * c : 0.f;
                    zi[i] = a[h][i] > 0.f ? A * s : 0.f;
                }
                if (to) {
                    put3(to + off, make_float4(zr[0], zr[1], zr[2], zr[3]));
                    put3(to + 3 * PLANE + off, make_float4(zi[0], zi[1], zi[2], zi[3]));
                }
                if (to_v) {
                    put3(to_v + off, make_float4(zr[0] * w.x, zr[1] * w.y, zr[2] * w.z, zr[3] * w.w));
                    put3(to_v + 3 * PLANE + off, make_float4(zi[0] * w.x, zi[1] * w.y, zi[2] * w.z, zi[3] * w.w));
                }
            }
        };
        auto drain = [&](int c) {
            const int s = c & 1;
            if (!__all_sync(0xffffffffu, mbar_wait(accf + s, (c >> 1) & 1))) return false;
            fence_after();
            const uint32_t at = tmem + ((uint32_t)(sub * 32) << 16) + s * 2 * BM + col0;
            float t[32];
            tmem_ld32(at, t);
#pragma unroll
            for (int i = 0; i < 32; i++) re[i] += t[i];
            tmem_ld32(at + BM, t);
#pragma unroll
            for (int i = 0; i < 32; i++) im[i] += t[i];
            fence_before();
            return true;
        };
        // the chunk's products, from the thread that saw all of its tile stored; that thread's
        // warp arrived after draining buffer s, as all others did
        auto products = [&](int c) {
            const int s = c & 1;
            if (!mbar_wait(full + s, (c >> 1) & 1)) return false;
            fence_after();
            const uint32_t ip = idesc_bf16(BM, BM, 0), in = idesc_bf16(BM, BM, 1);
            const uint32_t dre = tmem + s * 2 * BM, dim = dre + BM;
            const uint32_t a = smem_u32(tiles + (size_t)s * 2 * OPER), bb = a + OPER;
#pragma unroll
            for (int p = 0; p < 6; p++) {
                // (hi, lo), (lo, hi), (mid, mid), (hi, mid), (mid, hi), (hi, hi)
                constexpr int PA[6] = {0, 2, 1, 0, 1, 0}, PB[6] = {2, 0, 1, 1, 0, 0};
#pragma unroll
                for (int k = 0; k < BK / 16; k++) {
                    const uint32_t ar = a + PA[p] * PLANE + k * 32, br = bb + PB[p] * PLANE + k * 32;
                    const uint64_t a0 = desc_k64(ar), a1 = desc_k64(ar + 3 * PLANE);
                    const uint64_t b0 = desc_k64(br), b1 = desc_k64(br + 3 * PLANE);
                    const uint32_t acc = (p > 0 || k > 0) ? 1u : 0u;
                    mma_bf16(dre, a0, b0, ip, acc);
                    mma_bf16(dre, a1, b1, in, 1u);
                    mma_bf16(dim, a0, b1, ip, acc);
                    mma_bf16(dim, a1, b0, ip, 1u);
                }
            }
            mma_commit(empty + s);
            mma_commit(accf + s);
            return true;
        };
        for (int c = 0; c < nc; c++) {
            const int s = c & 1, kx = (c0 + c) * BK, x = kx + 4 * q4;
            ok = c < 2 || __all_sync(0xffffffffu, mbar_wait(empty + s, ((c >> 1) - 1) & 1));
            if (!ok) break;
            uint8_t *A = tiles + (size_t)s * 2 * OPER, *B = A + OPER;
            const float4 w = make_float4(x < X ? g.v[x] : 0.f, x + 1 < X ? g.v[x + 1] : 0.f, x + 2 < X ? g.v[x + 2] : 0.f,
                                         x + 3 < X ? g.v[x + 3] : 0.f);
            if (te == tr) {
                form(te, kx, A, B, w);
            } else {
                form(te, kx, A, nullptr, w);
                form(tr, kx, nullptr, B, w);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(full + s);
            if (warp == 0) ok = __all_sync(0xffffffffu, lane != 0 || products(c));
            if (!ok || (c > 0 && !(ok = drain(c - 1)))) break;
        }
        if (ok && nc > 0) ok = drain(nc - 1);
        if (!ok) {   // a wait gave up: the caller sees it in D
            const float nan = __int_as_float(0x7fffffff);
#pragma unroll
            for (int i = 0; i < 32; i++) re[i] = im[i] = nan;
        }
        const int row = sub * 32 + lane, e = te * BM + row;
        if (cs == 1) {
            if (e < N) {
                float2 *P = g.part + ((size_t)blockIdx.y * N + e) * N;
#pragma unroll
                for (int i = 0; i < 32; i++) {
                    const int r = tr * BM + col0 + i;
                    if (r < N) P[r] = make_float2(re[i], im[i]);
                }
            }
        } else {
            // the stages are free: every MMA has read them
            float2 *S = reinterpret_cast<float2 *>(tiles);
#pragma unroll
            for (int i = 0; i < 32; i++) S[(col0 + i) * BM + row] = make_float2(re[i], im[i]);
        }
    }
    if (cs > 1) {
        cluster.sync();
        {   // this CTA's share of the columns, over the ranks in order
            const int row = threadIdx.x & (BM - 1), per = BM / cs, e = te * BM + row;
            for (int i = threadIdx.x / BM; i < per; i += THREADS / BM) {
                const int col = rank * per + i, r = tr * BM + col;
                float2 sum = make_float2(0.f, 0.f);
                for (int q = 0; q < cs; q++) {
                    const float2 z = cluster.map_shared_rank(reinterpret_cast<float2 *>(tiles), q)[col * BM + row];
                    sum.x += z.x;
                    sum.y += z.y;
                }
                if (e < N && r < N) g.part[((size_t)blockIdx.y * N + e) * N + r] = sum;
            }
        }
        cluster.sync();   // no CTA retires while another reads its sums
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// CTAs per tile pair: splits (partial sums in the scratch, at most cap) times the cluster's
// size, the most that fill the GPU once with at least three K chunks each.
void noalloc_shape(int N, int X, int cap, int sms, int *splits, int *cs)
{
    const int T = (N + BM - 1) / BM, pairs = T * (T + 1) / 2, nk = (X + BK - 1) / BK;
    *splits = *cs = 1;
    int best = 1;
    for (int c = 1; c <= 4; c *= 2) {
        int s = sms / (pairs * c);
        if (s > cap) s = cap;
        if (s > (nk + 2) / 3 / c) s = (nk + 2) / 3 / c;
        if (s >= 1 && s * c > best) {
            best = s * c;
            *splits = s;
            *cs = c;
        }
    }
}

std::mutex g_scratch_mu;
float2 *g_scratch_ptr[64] = {};

void seterr(char *err, size_t errlen, const char *msg)
{
    if (err && errlen) snprintf(err, errlen, "%s", msg);
}

}  // namespace
}  // namespace rbx

using namespace rbx;

extern "C" rbx_status rbx_forward_noalloc(const float *T_dev, const float *a_dev, const uint8_t *K_dev,
                                          const float *v_dev, int n_xducers, int n_nodes, double freq_hz, double c0,
                                          void *D_dev, void *cuda_stream, char *err, size_t errlen)
{
    if (!T_dev || !a_dev || !K_dev || !v_dev || !D_dev) {
        seterr(err, errlen, "null pointer argument");
        return RBX_EINVAL;
    }
    const int N = n_xducers, X = n_nodes;
    if (N < 3 || X < 1 || !(freq_hz > 0) || !std::isfinite(freq_hz) || !(c0 > 0) || !std::isfinite(c0)) {
        seterr(err, errlen, "need n_xducers >= 3, n_nodes >= 1, finite freq_hz > 0 and c0 > 0");
        return RBX_EINVAL;
    }
    if ((size_t)N * (size_t)N > kScratchElems) {
        seterr(err, errlen, "n_xducers exceeds 1024: N*N partial sums must fit the 8 MiB fixed scratch");
        return RBX_EINVAL;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        seterr(err, errlen, "no current CUDA device (or device index >= 64)");
        return RBX_ECUDA;
    }
    float2 *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_scratch_mu);
        if (!g_scratch_ptr[dev]) {
            void *p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_fwd_scratch);
            if (e != cudaSuccess || !p) {
                char buf[256];
                snprintf(buf, sizeof buf, "cudaGetSymbolAddress of the forward scratch failed: %s",
                         cudaGetErrorString(e));
                seterr(err, errlen, buf);
                return RBX_ECUDA;
            }
            g_scratch_ptr[dev] = static_cast<float2 *>(p);
        }
        scratch = g_scratch_ptr[dev];
    }
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int splits = 1, cs = 1;
    noalloc_shape(N, X, (int)(kScratchElems / ((size_t)N * N)), sms, &splits, &cs);
    NaArgs g{};
    g.T = T_dev;
    g.a = a_dev;
    g.v = v_dev;
    g.K = K_dev;
    g.N = N;
    g.X = X;
    g.ntile = (N + BM - 1) / BM;
    g.nk = (X + BK - 1) / BK;
    g.kper = (g.nk + splits * cs - 1) / (splits * cs);
    g.fhi = (float)freq_hz;
    g.flo = (float)(freq_hz - (double)g.fhi);
    g.C = (float)(1.0 / std::sqrt(8.0 * 3.14159265358979323846 * (2.0 * 3.14159265358979323846 * freq_hz) / c0));
    g.part = scratch;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cs;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(g.ntile * (g.ntile + 1) / 2 * cs), (unsigned)splits);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = NA_SMEM;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaError_t e = cudaFuncSetAttribute(k_forward_tables, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)NA_SMEM);
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, k_forward_tables, g);
    if (e != cudaSuccess) {
        char buf[256];
        snprintf(buf, sizeof buf, "kernel launch failed: %s", cudaGetErrorString(e));
        cudaGetLastError();
        seterr(err, errlen, buf);
        return RBX_ECUDA;
    }
    launch_forward_reduce(scratch, N, splits, nullptr, static_cast<float2 *>(D_dev), s);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        char buf[256];
        snprintf(buf, sizeof buf, "kernel launch failed: %s", cudaGetErrorString(e));
        seterr(err, errlen, buf);
        return RBX_ECUDA;
    }
    seterr(err, errlen, "");
    return RBX_OK;
}
