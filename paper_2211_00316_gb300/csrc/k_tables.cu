// Import and export of the ray tables (rbx_set_tables, rbx_get_tables). A file of their own: beside them the
// compiler gave the linking step of k_rays.cu three registers more and it ran 2.8 % slower.
#include "rbx_internal.cuh"

namespace rbx {

// counters[0] gains the number of covered entries (a > 0).
__global__ void k_set_tables(const float *T, const float *a, const float *gam, const uint8_t *K, TabEntry *tab,
                             size_t n, unsigned long long *counters)
{
    size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    bool cov = false;
    if (i < n) {
        TabEntry t;
        float av = a[i];
        cov = av > 0.f;
        t.idk = cov ? (uint32_t)K[i] : kUncovered;
        t.T = T[i];
        t.a = av;
        t.gam = gam[i];
        tab[i] = t;
    }
    const unsigned b = __ballot_sync(0xffffffffu, cov);
    if ((threadIdx.x & 31) == 0 && b) atomicAdd(&counters[0], (unsigned long long)__popc(b));
}

void launch_set_tables(const float *T, const float *a, const float *gam, const uint8_t *K, TabEntry *tab, size_t n,
                       unsigned long long *counters, cudaStream_t s)
{
    k_set_tables<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(T, a, gam, K, tab, n, counters);
}

// dg: the angular density (step a4), the values that the operand syntheses form, from the direction angles of
// the neighbouring transducers. A thread walks eight transducers of a node, so the tables are read 1.25 times
// for all arrays.
constexpr int kGetWalk = 8;

__global__ void k_get_tables(const TabEntry *__restrict__ tab, float *T, float *a, float *gam, uint8_t *K, float *dg, int N,
                             int X)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, e0 = blockIdx.y * kGetWalk, e1 = min(N, e0 + kGetWalk);
    if (x >= X) return;
    auto row = [&](int e) { return tab[(size_t)e * X + x]; };
    TabEntry prev{}, t = row(e0), next{};
    if (dg) prev = row(e0 > 0 ? e0 - 1 : N - 1);
    for (int e = e0; e < e1; e++) {
        if (dg || e + 1 < e1) next = row(e + 1 < N ? e + 1 : 0);
        const size_t i = (size_t)e * X + x;
        const bool cov = t.idk != kUncovered;
        if (T) T[i] = cov ? t.T : 0.f;
        if (a) a[i] = cov ? t.a : 0.f;
        if (gam) gam[i] = cov ? t.gam : 0.f;
        if (K) K[i] = cov ? (uint8_t)(t.idk & 0xffu) : 0;
        if (dg) dg[i] = (next.idk == kUncovered || prev.idk == kUncovered) ? 0.f : dgamma_of(next.gam, prev.gam);
        prev = t;
        t = next;
    }
}

void launch_get_tables(const TabEntry *tab, float *T, float *a, float *gam, uint8_t *K, float *dg, int N, int X,
                       cudaStream_t s)
{
    const dim3 grd((X + 255) / 256, (N + kGetWalk - 1) / kGetWalk);
    k_get_tables<<<grd, 256, 0, s>>>(tab, T, a, gam, K, dg, N, X);
}

}  // namespace rbx
