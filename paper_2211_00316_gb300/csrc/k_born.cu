// Born weights of the forward (Eq. scattering-potential) and the reduction of its partial sums,
// shared by every precision.
#include "rbx_internal.cuh"

namespace rbx {

// Scattering potential Upsilon_m = omega c k~ (Eq. scattering-potential), with
// k~ = omega/c + alpha0 omega^y (tan(pi y/2) + i) (Eq. szabo_dispersion_equation):
// (omega^2 + omega c alpha tan(pi y/2), omega c alpha), alpha = alpha0 omega^y; omega^2 lossless.
__device__ __forceinline__ double2 upsilon_m(double w, double c, double alpha, double tn)
{
    return make_double2(w * w + w * c * alpha * tn, w * c * alpha);
}

// v[x] = Upsilon_m dA (m - m_s) on the mask: Born weight of the rough part of the model.
__global__ void k_born_rough(const float *__restrict__ c, const double *__restrict__ ns, const int *__restrict__ idx,
                             int X, double w, double dA, const float *__restrict__ alpha0, double wy, double tn,
                             float2 *__restrict__ v)
{
    int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= X) return;
    int k = idx[q];
    double cc = c[k], n = ns[k];
    double2 u = upsilon_m(w, cc, alpha0 ? wy * (double)alpha0[k] : 0.0, tn);
    double d = dA * (1.0 / (cc * cc) - n * n);
    v[q] = make_float2((float)(u.x * d), (float)(u.y * d));
}

__global__ void k_born_dm(const float *__restrict__ dm, const float *__restrict__ c, const int *__restrict__ idx, int X,
                          double w, double dA, const float *__restrict__ alpha0, double wy, double tn,
                          float2 *__restrict__ v)
{
    int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= X) return;
    int k = idx[q];
    double2 u = alpha0 ? upsilon_m(w, (double)c[k], wy * (double)alpha0[k], tn) : make_double2(w * w, 0.0);
    double d = dA * (double)dm[k];
    v[q] = make_float2((float)(u.x * d), (float)(u.y * d));
}

static void lossy_factors(const Lossy &ab, double w, double &wy, double &tn)
{
    wy = tn = 0.0;
    if (ab.alpha0) {
        wy = pow(w, ab.y);
        tn = tan(3.14159265358979323846 * ab.y / 2.0);
    }
}

void launch_born_weights_rough(const float *c, const double *ns64, const int *idx, int X, double f, double dA,
                               const Lossy &ab, float2 *v, cudaStream_t s)
{
    double w = 2.0 * 3.14159265358979323846 * f, wy, tn;
    lossy_factors(ab, w, wy, tn);
    k_born_rough<<<(X + 255) / 256, 256, 0, s>>>(c, ns64, idx, X, w, dA, ab.alpha0, wy, tn, v);
}

void launch_born_weights_dm(const float *dm, const float *c, const int *idx, int X, double f, double dA,
                            const Lossy &ab, float2 *v, cudaStream_t s)
{
    double w = 2.0 * 3.14159265358979323846 * f, wy, tn;
    lossy_factors(ab, w, wy, tn);
    k_born_dm<<<(X + 255) / 256, 256, 0, s>>>(dm, c, idx, X, w, dA, ab.alpha0, wy, tn, v);
}

// The timeout word (no word: 0) through L1 and in flight beside the sums' loads: read where it is used, after
// them, it cost the reduction another 1.7 us; past L1, where all blocks ask one L2 slice for it, 1 us.
__device__ __forceinline__ unsigned timeout_word(const unsigned *err)
{
    unsigned v = 0u;
    if (err) asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(err));
    return v;
}

// D[e,r] = D[r,e] = sum over splits (fixed order) of the upper-triangle partials; not a number when a wait
// of the contraction gave up (*err), so that a call whose status is not waited for shows it.
__global__ void k_forward_reduce(const float2 *__restrict__ part, int N, int splits, const unsigned *__restrict__ err,
                                 float2 *__restrict__ D)
{
    size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= (size_t)N * N) return;
    int e = (int)(i / N), r = (int)(i % N);
    if (e > r) return;
    const unsigned lost = timeout_word(err);
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int q = 0; q < splits; q++) {
        float2 p = part[(size_t)q * N * N + i];
        acc.x += p.x;
        acc.y += p.y;
    }
    if (lost) acc.x = acc.y = __int_as_float(0x7fffffff);
    D[(size_t)e * N + r] = acc;
    D[(size_t)r * N + e] = acc;
}

// The same with four lanes per entry, each summing every fourth split: a small D with many splits
// is one chain of loads otherwise (64 transducers, 54 splits: 15 -> 7 us).
__global__ void k_forward_reduce4(const float2 *__restrict__ part, int N, int splits, const unsigned *__restrict__ err,
                                  float2 *__restrict__ D)
{
    const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x, i = t >> 2;
    const int e = (int)(i / N), r = (int)(i % N);
    const unsigned lost = timeout_word(err);
    float2 acc = make_float2(0.f, 0.f);
    if (i < (size_t)N * N && e <= r) {
#pragma unroll 8
        for (int q = (int)(t & 3); q < splits; q += 4) {
            const float2 p = part[(size_t)q * N * N + i];
            acc.x += p.x;
            acc.y += p.y;
        }
    }
#pragma unroll
    for (int d = 1; d < 4; d <<= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, d);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, d);
    }
    if ((t & 3) == 0 && i < (size_t)N * N && e <= r) {
        if (lost) acc.x = acc.y = __int_as_float(0x7fffffff);
        D[(size_t)e * N + r] = acc;
        D[(size_t)r * N + e] = acc;
    }
}

void launch_forward_reduce(const float2 *part, int N, int splits, const unsigned *err, float2 *D, cudaStream_t s)
{
    size_t n = (size_t)N * N;
    if (splits > 16 && n <= 65536)   // beyond, one lane per entry fills the GPU by itself
        k_forward_reduce4<<<(unsigned)((4 * n + 255) / 256), 256, 0, s>>>(part, N, splits, err, D);
    else
        k_forward_reduce<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(part, N, splits, err, D);
}

}  // namespace rbx
