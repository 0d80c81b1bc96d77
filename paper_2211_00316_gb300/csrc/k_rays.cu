// Steps a2-a5: paraxial ray tracing, ray-to-grid tables, angular density and the
// direct Green's function at the receivers.
//
// Ray fan (reading of the paper's ray linking for a full ring, Sec. 4.4 / 6.3): from
// transducer e, N-1 rays j = 1..N-1 leave at gamma0 = beta_e + pi/2 + pi j / N, so that in
// water ray j reaches receiver e + j. Each ray is integrated by Heun's method with the
// normalisations of Alg. 1 and the paraxial system of Eq. ray-equation-paraxial, in
// slowness variables (p = k / omega, the path does not depend on omega), with step ds and
// a final partial step that lands on the ring (Def. ray-parameterisation).
//
// GB300 mapping: one thread per ray, 32 adjacent rays of one fan per warp stepping in
// lockstep; a block's four warps take the same rays of four neighbouring transducers, the warps
// with the longest rays first (a small ring gives each ray several lanes: k_trace_wide). At
// each step a lane fetches its neighbour's new sample with a shuffle and rasterises the
// ray-tube quad (rays j, j+1; samples i, i+1) as two triangles straight
// into the fan's table (Sec. 4.4: triangulation of the ray samples). Overlapping triangles
// keep the first arrival: the 16-byte table entry starts with the key (T bits, triangle
// id, K) and a 128-bit compare-and-swap keeps the smallest key, so the table does not
// depend on the order in which warps finish. The ray samples are never stored.
//
// Fields are bilinearly interpolated from the field map (L1/L2 cached; a lossless trace on
// the smoothed map reads 24 B per node, 6 MB at 512^2). Travel time uses compensated (Kahan)
// summation.
#include <climits>
#include <type_traits>

#include "rbx_internal.cuh"

namespace rbx {

// 1/v by the hardware approximation alone (within about 1 ulp): the Heun stages' 1/n, which
// scales the direction and the paraxial terms; the refined rcp_nr serves the rest.
__device__ __forceinline__ float rcp_ap(float v)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ int clampi_(int i, int lo, int hi) { return i < lo ? lo : (i > hi ? hi : i); }

struct Fv {
    float n, gx, gy, hxx, hxy, hyy, al;   // al: absorption coefficient alpha (lossy media only)
    float nr;                              // slowness integrated along the ray (n, or the non-smoothed one)
};

// s += inc with compensation term c (Kahan): the ray state is a sum of ~10^3 small steps
__device__ __forceinline__ void kadd(float &s, float &c, float inc)
{
    const float y = inc - c, t = s + y;
    c = (t - s) - y;
    s = t;
}

// The four nodes of a grid cell (i, j), (i + 1, j), (i, j + 1), (i + 1, j + 1): every field.
template <bool LOSSY, bool RAW>
struct Cell {
    float i, j;
    float4 a0, b0, c0, d0;   // n, n_x, n_y, n_xx
    float2 a1, b1, c1, d1;   // n_xy, n_yy
    float2 a2, b2, c2, d2;   // alpha, n_raw (lossy or non-smoothed integration only)
};

// The cell of grid position (u, v) (the outermost one beyond the grid).
template <bool LOSSY, bool RAW>
__device__ __forceinline__ void cell_load(const float *__restrict__ F, const RayParams &p, float u, float v,
                                          Cell<LOSSY, RAW> &c)
{
    const int i = clampi_((int)floorf(u), 0, p.nx - 2), j = clampi_((int)floorf(v), 0, p.ny - 2);
    c.i = (float)i;
    c.j = (float)j;
    const size_t nxy = (size_t)p.nx * p.ny, k00 = (size_t)j * p.nx + i, k01 = k00 + p.nx;
    const float4 *F4 = reinterpret_cast<const float4 *>(F);
    const float2 *F2 = reinterpret_cast<const float2 *>(F4 + nxy);
    c.a0 = __ldg(F4 + k00); c.b0 = __ldg(F4 + k00 + 1); c.c0 = __ldg(F4 + k01); c.d0 = __ldg(F4 + k01 + 1);
    c.a1 = __ldg(F2 + k00); c.b1 = __ldg(F2 + k00 + 1); c.c1 = __ldg(F2 + k01); c.d1 = __ldg(F2 + k01 + 1);
    if (LOSSY || RAW) {
        const float2 *F3 = F2 + nxy;
        c.a2 = __ldg(F3 + k00); c.b2 = __ldg(F3 + k00 + 1); c.c2 = __ldg(F3 + k01); c.d2 = __ldg(F3 + k01 + 1);
    }
}

template <bool LOSSY, bool RAW>
__device__ __forceinline__ void cell_eval(const Cell<LOSSY, RAW> &c, float tx, float ty, Fv &o)
{
    const float w00 = (1.f - tx) * (1.f - ty), w10 = tx * (1.f - ty), w01 = (1.f - tx) * ty, w11 = tx * ty;
    o.n = w00 * c.a0.x + w10 * c.b0.x + w01 * c.c0.x + w11 * c.d0.x;
    o.gx = w00 * c.a0.y + w10 * c.b0.y + w01 * c.c0.y + w11 * c.d0.y;
    o.gy = w00 * c.a0.z + w10 * c.b0.z + w01 * c.c0.z + w11 * c.d0.z;
    o.hxx = w00 * c.a0.w + w10 * c.b0.w + w01 * c.c0.w + w11 * c.d0.w;
    o.hxy = w00 * c.a1.x + w10 * c.b1.x + w01 * c.c1.x + w11 * c.d1.x;
    o.hyy = w00 * c.a1.y + w10 * c.b1.y + w01 * c.c1.y + w11 * c.d1.y;
    o.al = LOSSY ? w00 * c.a2.x + w10 * c.b2.x + w01 * c.c2.x + w11 * c.d2.x : 0.f;
    o.nr = RAW ? w00 * c.a2.y + w10 * c.b2.y + w01 * c.c2.y + w11 * c.d2.y : o.n;
}

template <bool LOSSY, bool RAW>
__device__ __forceinline__ void field_eval(const float *__restrict__ F, const RayParams &p, float px, float py, Fv &o)
{
    const float u = (px - p.x0) * p.inv_dx, v = (py - p.y0) * p.inv_dx;
    Cell<LOSSY, RAW> c;
    cell_load<LOSSY, RAW>(F, p, u, v, c);
    cell_eval<LOSSY, RAW>(c, u - c.i, v - c.j, o);
}

// r2 - R^2 with its rounding fixed (R^2 not rounded by itself), so every kernel that takes a ray
// straight to the ring ends it on the same sample, bit for bit, however R^2 is kept.
__device__ __forceinline__ float over_ring(float r2, float R) { return __fmaf_rn(-R, R, r2); }

// A ray sample as a triangle vertex.
struct Vtx {
    float x, y, T, a, kx, ky;
    int K;
};

__device__ __forceinline__ void cas128(unsigned long long *addr, unsigned long long clo, unsigned long long chi,
                                       unsigned long long nlo, unsigned long long nhi, unsigned long long &olo,
                                       unsigned long long &ohi)
{
    asm volatile(
        "{\n\t.reg .b128 d, b, c;\n\t"
        "mov.b128 b, {%2, %3};\n\t"
        "mov.b128 c, {%4, %5};\n\t"
        "atom.global.cas.b128 d, [%6], b, c;\n\t"
        "mov.b128 {%0, %1}, d;\n\t}"
        : "=l"(olo), "=l"(ohi)
        : "l"(clo), "l"(chi), "l"(nlo), "l"(nhi), "l"(addr)
        : "memory");
}

// Keep the entry with the smaller key, starting from a known content (lo, hi) of the
// entry. Every successful exchange lowers the stored key, so the loop ends after at most as
// many rounds as there are competing triangles (the bound only reports a broken invariant).
__device__ __forceinline__ void cas_min_from(TabEntry *e, unsigned long long key, unsigned long long pay,
                                             unsigned long long lo, unsigned long long hi,
                                             unsigned long long *counters)
{
    unsigned long long *a = reinterpret_cast<unsigned long long *>(e);
    for (int it = 0; it < 1 << 16; ++it) {
        if (key >= lo) return;
        unsigned long long plo, phi;
        cas128(a, lo, hi, key, pay, plo, phi);
        if (plo == lo && phi == hi) return;
        lo = plo;
        hi = phi;
    }
    atomicAdd(&counters[3], 1ull);
}

// Per-warp queue of table hits in shared memory, drained 32 at a time (one per lane): the
// entry's low key word, T, and the interpolated amplitude and direction (the direction angle
// is formed at the drain, where all 32 lanes are busy).
struct HitQueue {
    uint4 *v;        // (triangle id << 8 | K, T, a, kappa_x)
    float2 *w;       // (kappa_y, mask node)
    unsigned *cov;   // entries this warp found untouched (each entry is found so exactly once)
    int n;           // warp-uniform
};

// Returns true when this exchange was the entry's first write.
__device__ __forceinline__ bool drain_one(const HitQueue &hq, int q, TabEntry *fan, unsigned long long *counters)
{
    const uint4 v = hq.v[q];
    const float2 w = hq.w[q];
    const unsigned long long key = ((unsigned long long)v.y << 32) | v.x;
    const unsigned long long pay = ((unsigned long long)__float_as_uint(atan2f(w.x, __uint_as_float(v.w))) << 32) | v.z;
    TabEntry *addr = fan + __float_as_int(w.y);
    // most entries are still untouched (all ones): try that first, then take the minimum
    unsigned long long lo, hi;
    cas128(reinterpret_cast<unsigned long long *>(addr), ~0ull, ~0ull, key, pay, lo, hi);
    if (lo == ~0ull && hi == ~0ull) return true;
    cas_min_from(addr, key, pay, lo, hi, counters);
    return false;
}

// Adds the warp's first writes to its count of covered entries (all lanes take part).
__device__ __forceinline__ void count_first(const HitQueue &hq, bool first)
{
    const unsigned b = __ballot_sync(0xffffffffu, first);
    if ((threadIdx.x & 31) == 0) *hq.cov += __popc(b);
}

// Edge function of P -> Q at (px, py), always evaluated from the vertex with the smaller
// id (ids order P[j,i] < P[j,i+1] < P[j+1,i] < P[j+1,i+1]), so the triangles on both sides
// of an edge see exactly opposite values and no node falls between them.
__device__ __forceinline__ float edge_fn(const Vtx &P, const Vtx &Q, float px, float py)
{
    return __fmaf_rn(Q.x - P.x, py - P.y, -__fmul_rn(Q.y - P.y, px - P.x));
}

__device__ __forceinline__ bool tri_inside(float eA, float eB, float eC, float &sum)
{
    sum = eA + eB + eC;
    bool in = sum > 0.f ? (eA >= 0.f && eB >= 0.f && eC >= 0.f) : (eA <= 0.f && eB <= 0.f && eC <= 0.f);
    return in && sum != 0.f;
}

__device__ __forceinline__ unsigned long long tri_key(const Vtx &A, const Vtx &B, const Vtx &C, float lb, float lc,
                                                      uint32_t tid)
{
    float T = A.T + lb * (B.T - A.T) + lc * (C.T - A.T);
    int K = max(A.K, max(B.K, C.K));
    return ((unsigned long long)__float_as_uint(T) << 32) | ((unsigned long long)tid << 8) |
           (unsigned long long)min(K, 255);
}

// Queue the hits of the lanes in `hit` (the whole warp calls); a full batch of 32 is drained.
__device__ __forceinline__ void push_hits(bool hit, uint4 v, float2 w, TabEntry *fan, HitQueue &hq,
                                          unsigned long long *counters)
{
    const int lane = threadIdx.x & 31;
    const unsigned b = __ballot_sync(0xffffffffu, hit);
    if (!b) return;
    const int slot = hq.n + __popc(b & ((1u << lane) - 1));
    if (hit) {
        hq.v[slot] = v;
        hq.w[slot] = w;
    }
    hq.n += __popc(b);
    __syncwarp();
    if (hq.n >= 32) {
        count_first(hq, drain_one(hq, hq.n - 32 + lane, fan, counters));
        hq.n -= 32;
        __syncwarp();
    }
}

// A node of a ray-tube quad against both of its triangles: the hit with the smaller key.
__device__ __forceinline__ bool test_both(const Vtx &P00, const Vtx &P01, const Vtx &P10, const Vtx &P11, bool ok0,
                                          bool ok1, uint32_t tid0, float px, float py, int xi, uint4 &v, float2 &u)
{
    const float e1 = edge_fn(P00, P10, px, py), e2 = edge_fn(P10, P11, px, py);
    const float e3 = edge_fn(P00, P11, px, py);
    const float e4 = edge_fn(P01, P11, px, py), e5 = edge_fn(P00, P01, px, py);
    float s0, s1, lb0 = 0.f, lc0 = 0.f, lb1 = 0.f, lc1 = 0.f;
    unsigned long long k0 = ~0ull, k1 = ~0ull;
    if (ok0 && tri_inside(e2, -e3, e1, s0)) {
        float inv = rcp_nr(s0);
        lb0 = -e3 * inv;
        lc0 = e1 * inv;
        k0 = tri_key(P00, P10, P11, lb0, lc0, tid0);
    }
    if (ok1 && tri_inside(-e4, -e5, e3, s1)) {
        float inv = rcp_nr(s1);
        lb1 = -e5 * inv;
        lc1 = e3 * inv;
        k1 = tri_key(P00, P11, P01, lb1, lc1, tid0 + 1);
    }
    if (k0 == ~0ull && k1 == ~0ull) return false;
    const bool use0 = k0 < k1;
    const float lb = use0 ? lb0 : lb1, lc = use0 ? lc0 : lc1, la = 1.f - lb - lc;
    const float Ba = use0 ? P10.a : P11.a, Ca = use0 ? P11.a : P01.a;
    const float Bkx = use0 ? P10.kx : P11.kx, Ckx = use0 ? P11.kx : P01.kx;
    const float Bky = use0 ? P10.ky : P11.ky, Cky = use0 ? P11.ky : P01.ky;
    const unsigned long long key = use0 ? k0 : k1;
    v = make_uint4((uint32_t)key, (uint32_t)(key >> 32), __float_as_uint(la * P00.a + lb * Ba + lc * Ca),
                   __float_as_uint(la * P00.kx + lb * Bkx + lc * Ckx));
    u = make_float2(la * P00.ky + lb * Bky + lc * Cky, __int_as_float(xi));
    return true;
}

// Rasterise the ray-tube quad P00 = P[j,i], P01 = P[j,i+1], P10 = P[j+1,i], P11 = P[j+1,i+1]
// of every valid lane as triangles t0 = (P00, P10, P11) and t1 = (P00, P11, P01) (ids
// tid0, tid0 + 1). Called by the whole warp; a ray's `lpr` lanes share out its quad's candidate
// nodes, sub = 0 .. lpr - 1. Hits go to the warp's queue. rows[iy] gives the mask nodes of grid
// row iy: (first compact index, first ix, last ix).
//
// A regular quad (both triangles of the same orientation and not slivers) holds a node in one
// triangle only, that on the node's side of the diagonal P00-P11. Its lanes run through their
// candidates with the edge functions alone (about 30 instructions each) until one is a hit, and
// the interpolation, mask look-up and queueing (three times that) run once for the hits of all
// lanes. Testing and interpolating candidate by candidate took 160 instructions for each of the
// 1.2 (1024 transducers) to 5 (64) candidates of the warp's fullest quad per step, where a
// quad holds 0.3 to 1.1 nodes (trace of 64 transducers 0.63 -> 0.50 ms, 256: 2.50 -> 1.90).
// Folded quads, slivers (near a caustic) and nodes on the diagonal take the two-triangle test, the
// smaller key winning.
__device__ __forceinline__ void raster_quad_warp(bool valid, const Vtx &P00, const Vtx &P01, const Vtx &P10,
                                                 const Vtx &P11, uint32_t tid0, const RayParams &p, float inv_dx,
                                                 int sub, int lpr, const int4 *rows, TabEntry *fan, HitQueue &hq,
                                                 unsigned long long *counters)
{
    const unsigned FULL = 0xffffffffu;
    bool regular = false, odd = false, ok0 = false, ok1 = false;
    float ar1 = 0.f, fx0 = 0.f, fx1 = -1.f, fy1 = -1.f, fx = 0.f, fy = 0.f;
    if (valid) {
        const float tiny = 1e-9f * p.ds * p.ds, thin = 1e-3f * p.ds * p.ds;
        const float ar0 = (P10.x - P00.x) * (P11.y - P00.y) - (P10.y - P00.y) * (P11.x - P00.x);
        ar1 = (P11.x - P00.x) * (P01.y - P00.y) - (P11.y - P00.y) * (P01.x - P00.x);
        ok0 = fabsf(ar0) > tiny;
        ok1 = fabsf(ar1) > tiny;
        regular = fminf(fabsf(ar0), fabsf(ar1)) > thin && ((ar0 > 0.f) == (ar1 > 0.f));
        odd = !regular && (ok0 || ok1);
        const float minx = fminf(fminf(P00.x, P01.x), fminf(P10.x, P11.x));
        const float maxx = fmaxf(fmaxf(P00.x, P01.x), fmaxf(P10.x, P11.x));
        const float miny = fminf(fminf(P00.y, P01.y), fminf(P10.y, P11.y));
        const float maxy = fmaxf(fmaxf(P00.y, P01.y), fmaxf(P10.y, P11.y));
        // candidate nodes of the bounding box, widened by 1e-3 cells: in FP32 the box's grid
        // coordinates carry ~2e-5 cells of rounding, and a node that lies on a box edge (at a
        // triangle's tip) must stay a candidate of every quad that may hold it; the edge
        // functions below decide which does
        const float slack = 1e-3f;
        fx0 = fmaxf(0.f, ceilf((minx - p.x0) * inv_dx - slack));
        fx1 = fminf((float)(p.nx - 1), floorf((maxx - p.x0) * inv_dx + slack));
        fy = fmaxf(0.f, ceilf((miny - p.y0) * inv_dx - slack));
        fy1 = fminf((float)(p.ny - 1), floorf((maxy - p.y0) * inv_dx + slack));
        if (fx0 > fx1) fy1 = -1.f;   // no column: no candidate
    }
    const float w = fx1 - fx0 + 1.f;
    // candidates row by row, lpr apart
    auto wrap = [&]() {
        if (lpr == 1) {
            if (fx > fx1) { fx = fx0; fy += 1.f; }
        } else {
            while (fx > fx1 && fy <= fy1) { fx -= w; fy += 1.f; }
        }
    };
    const float fy0 = fy;
    fx = fx0 + (float)sub;
    wrap();
    bool more = regular && fy <= fy1;
    while (__any_sync(FULL, more)) {
        float hx = 0.f, hy = 0.f, e3 = 0.f, x1 = 0.f, x2 = 0.f;
        bool hit = false, use1 = false;
        while (more && !hit) {
            hx = fx;
            hy = fy;
            const float px = p.x0 + fx * p.dx, py = p.y0 + fy * p.dx;
            e3 = edge_fn(P00, P11, px, py);
            // t1 = (P00, P11, P01) where e3 has t1's orientation, else t0 = (P00, P10, P11); with
            // M = P01 (t1) or P10 (t0) the other edges are M -> P11 and P00 -> M
            use1 = (e3 > 0.f) == (ar1 > 0.f);
            const float mx = use1 ? P01.x : P10.x, my = use1 ? P01.y : P10.y;
            x1 = __fmaf_rn(P11.x - mx, py - my, -__fmul_rn(P11.y - my, px - mx));
            x2 = __fmaf_rn(mx - P00.x, py - P00.y, -__fmul_rn(my - P00.y, px - P00.x));
            hit = use1 != (ar1 > 0.f) ? fminf(x1, x2) >= 0.f : fmaxf(x1, x2) <= 0.f;
            hit = hit || e3 == 0.f;
            fx += (float)lpr;
            wrap();
            more = fy <= fy1;
        }
        __syncwarp();
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        float2 u = make_float2(0.f, 0.f);
        if (hit) {
            const int4 ro = rows[(int)hy];
            const int ix = (int)hx, xi = ro.x + ix - ro.y;
            hit = ix >= ro.y && ix <= ro.z;
            if (e3 == 0.f) {
                hit = hit && test_both(P00, P01, P10, P11, ok0, ok1, tid0, p.x0 + hx * p.dx, p.y0 + hy * p.dx, xi, v, u);
            } else {
                // barycentric weights of the second and third vertex, (P10, P11) or (P11, P01)
                const float eBC = use1 ? -x1 : x1, eCA = use1 ? -x2 : -e3, eAB = use1 ? e3 : x2;
                const float sum = eBC + eCA + eAB;
                hit = hit && sum != 0.f;
                const float inv = rcp_nr(sum), lb = eCA * inv, lc = eAB * inv, la = 1.f - lb - lc;
                const Vtx &B = use1 ? P11 : P10, &C = use1 ? P01 : P11;
                const unsigned long long key = tri_key(P00, B, C, lb, lc, tid0 + (use1 ? 1u : 0u));
                v = make_uint4((uint32_t)key, (uint32_t)(key >> 32), __float_as_uint(la * P00.a + lb * B.a + lc * C.a),
                               __float_as_uint(la * P00.kx + lb * B.kx + lc * C.kx));
                u = make_float2(la * P00.ky + lb * B.ky + lc * C.ky, __int_as_float(xi));
            }
        }
        push_hits(hit, v, u, fan, hq, counters);
    }
    if (!__any_sync(FULL, odd)) return;
    fx = fx0 + (float)sub;
    fy = fy0;
    wrap();
    more = odd && fy <= fy1;
    while (__any_sync(FULL, more)) {
        bool hit = false;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        float2 u = make_float2(0.f, 0.f);
        if (more) {
            const int4 ro = rows[(int)fy];
            const int ix = (int)fx;
            if (ix >= ro.y && ix <= ro.z) {
                hit = test_both(P00, P01, P10, P11, ok0, ok1, tid0, p.x0 + fx * p.dx, p.y0 + fy * p.dx, ro.x + ix - ro.y, v, u);
            }
            fx += (float)lpr;
            wrap();
            more = fy <= fy1;
        }
        push_hits(hit, v, u, fan, hq, counters);
    }
}

// Warps per block, each tracing the same rays of a neighbouring transducer.
constexpr int kFansPerBlock = 4;

// The per-warp hit queues of a block (shared memory).
struct BlockQueues {
    uint4 v[kFansPerBlock][64];
    float2 w[kFansPerBlock][64];
    unsigned cov[kFansPerBlock];
};

// The rank-th longest warp of a fan: rays near the middle of the fan cross the whole ring.
__device__ __forceinline__ int warp_of_rank(int rank, int nwarps)
{
    const int mid = (nwarps - 1) / 2, d = (rank + 1) >> 1;
    return rank & 1 ? mid + d : mid - d;
}

// One block's work: warp `warp` of the fans of fan block `eblk` (fans 4 eblk .. 4 eblk + 3),
// one warp per fan; `rows` (the mask's row ranges) and the queues' coverage counts are set up
// by the caller. No block-wide barrier inside: a warp may return early.
template <bool LOSSY, bool RAW>
__device__ __forceinline__ void trace_block(const float *__restrict__ F, const int4 *rows, TabEntry *__restrict__ tab,
                                            float4 *__restrict__ exits, const RayParams &p,
                                            unsigned long long *counters, int warp, int eblk, BlockQueues &bq)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    // the warps of a block trace the same 32 rays of neighbouring transducers: rotated by one
    // ring step, those rays stay within about a cell of one another, so their field gathers
    // share L1 lines
    const int e = eblk * kFansPerBlock + wib;
    const int N = p.N;
    const int nwarps = (N - 2 + 30) / 31;
    if (warp >= nwarps || e >= N) return;  // whole warp leaves together
    const int j = 1 + 31 * warp + lane;      // this lane's ray
    const bool has_ray = j <= N - 1;
    TabEntry *fan = tab + (size_t)e * p.X;
    const float ds = p.ds, hds = 0.5f * p.ds, inv_dx = p.inv_dx, R2 = p.R * p.R;
    HitQueue hq{bq.v[wib], bq.w[wib], &bq.cov[wib], 0};

    const double be = p.beta ? p.beta[e] : 2.0 * 3.14159265358979323846 * e / N;
    float x = (float)(p.R * cos(be)), y = (float)(p.R * sin(be));
    const float gam0 = (float)(be + 3.14159265358979323846 / 2 + 3.14159265358979323846 * j / N);

    // reference ray (x, p) and paraxial ray (dx, dp); F1 caches the fields at x
    Fv F1;
    field_eval<LOSSY, RAW>(F, p, x, y, F1);
    float px, py, dpx, dpy, dxx = 0.f, dxy = 0.f, T = 0.f, Tc = 0.f;
    float B = 0.f, Bc = 0.f;   // lossy media: B = int alpha ds by the rule of T; a gains exp(-B)
    // compensation terms of the position and of the paraxial ray's closed-form steps (T has
    // Tc). In the Heun steps the momentum, renormalised to n(x) at every step, and the
    // paraxial ray, which only sets the amplitude, take plain sums: compensated too, the
    // tables met the same parity bars against the FP64 oracle (T 1e-9 s, a 1e-5) and the
    // trace took 1.6 % longer.
    float cx = 0.f, cy = 0.f, cdx = 0.f, cdy = 0.f;

    // Uniform water near the ring (exact up to rounding). Beyond radius rho every cell that a
    // sample or an auxiliary point can touch holds the same medium with zero derivatives (rho
    // exceeds the largest radius of a non-uniform node by a cell diagonal and a step), so there
    // a ray is a straight line with constant n and a linearly growing paraxial deviation; rho
    // also stays two cells outside the mask, so a quad with all vertices beyond rho holds no
    // mask node. Up to its entry step kin (its last sample beyond rho on the way in) a ray
    // takes the closed form of the step; kin depends on the ray alone, so the ray shared by two
    // warps has identical samples in both. The warp rasterises nothing before its smallest kin.
    const float ru = __uint_as_float((unsigned)counters[7]);
    const float rho = fmaxf(ru + 1.5f * p.dx + ds, p.rmask + 2.f * p.dx), rho2 = rho * rho;
    int kin = 0;
    {
        float s0, c0;
        sincosf(gam0, &s0, &c0);
        px = F1.n * c0; py = F1.n * s0;
        dpx = -F1.n * s0; dpy = F1.n * c0;
        if (has_ray && R2 > rho2) {
            const float b = x * c0 + y * s0, disc = b * b - (fmaf(x, x, y * y) - rho2);
            const float s_in = disc >= 0.f ? -b - sqrtf(disc) : -b;   // entry, or closest approach
            kin = max(0, (int)floorf(s_in / ds) - 1);
        }
    }
    const int i0 = __reduce_min_sync(FULL, has_ray ? kin : 0x7fffffff);
    const float rm = p.rmask + 2.f * p.dx, rm2 = rm * rm;
    float sc1 = 0.f, Jlast = 0.f;   // sc1 = sqrt(n_1 |J_1| / ds): a_i = sc1 / sqrt(n_i |J_i|)
    int K = 0;
    bool alive = has_ray;
    Vtx prev{}, nprev{};

    for (int i = 0; i < p.maxs; i++) {
        Vtx cur{};
        bool have = false;
        if (alive && i < kin) {
            // the step below in a uniform medium: straight, p constant, dx += ds dp / n
            const float n = F1.n, in = rcp_nr(n);
            const float rp = rsqrtf(px * px + py * py), tx = px * rp, ty = py * rp;
            kadd(x, cx, ds * tx); kadd(y, cy, ds * ty);
            kadd(dxx, cdx, ds * (dpx * in)); kadd(dxy, cdy, ds * (dpy * in));
            kadd(T, Tc, hds * (F1.nr + F1.nr));
            if (LOSSY) kadd(B, Bc, hds * (F1.al + F1.al));
            const float J = dxx * ty - dxy * tx;
            if (i == 0) { sc1 = sqrtf(F1.nr * fabsf(J) / ds); Jlast = J; }
            else if (J * Jlast < 0.f) K++;
            if (J != 0.f) Jlast = J;
            cur.x = x; cur.y = y; cur.T = T; cur.kx = tx; cur.ky = ty; cur.K = K;
            cur.a = sc1 * rsqrtf(F1.nr * fabsf(J));
            if (LOSSY) cur.a *= expf(-B);
            have = true;
        } else if (alive) {
            // stage 1 at x: normalise p to n(x), q_x = p/n, q_p = grad n
            const float n = F1.n, in = rcp_ap(n);
            const float sc = n * rsqrtf(px * px + py * py);
            px *= sc; py *= sc;
            const float qx = px * in, qy = py * in;
            // stage 2 at the auxiliary point x + ds q_x
            Fv F2;
            // The new sample lies within ds times half the step's bend of the auxiliary point
            // (about 1e-4 cells), so the nodes of one cell serve both but where a grid line runs
            // between them: half the loads and their address arithmetic (16.4 -> 15.6 ms at 1024
            // transducers on 512 x 512).
            Cell<LOSSY, RAW> cell;
            {
                const float ax = x + ds * qx, ay = y + ds * qy;
                const float u = (ax - p.x0) * p.inv_dx, v = (ay - p.y0) * p.inv_dx;
                cell_load<LOSSY, RAW>(F, p, u, v, cell);
                cell_eval<LOSSY, RAW>(cell, u - cell.i, v - cell.j, F2);
            }
            const float na = F2.n, ina = rcp_ap(na);
            float pax = px + ds * F1.gx, pay = py + ds * F1.gy;
            const float sca = na * rsqrtf(pax * pax + pay * pay);
            pax *= sca; pay *= sca;
            const float qax = pax * ina, qay = pay * ina;
            const float sx = qx + qax, sy = qy + qay, rs = rsqrtf(sx * sx + sy * sy);
            const float dirx = sx * rs, diry = sy * rs;
            const float ddpx = hds * (F1.gx + F2.gx), ddpy = hds * (F1.gy + F2.gy);
            // paraxial system, both stages at the reference ray's stage values:
            // q_dx = (dp - p (g.dx)/n)/n, q_dp = H dx + g ((p.dp)/n - g.dx)/n
            const float gd = F1.gx * dxx + F1.gy * dxy, pd = px * dpx + py * dpy;
            const float qdxx = in * (dpx - px * gd * in), qdxy = in * (dpy - py * gd * in);
            const float w1 = in * (pd * in - gd);
            const float qdpx = F1.hxx * dxx + F1.hxy * dxy + F1.gx * w1;
            const float qdpy = F1.hxy * dxx + F1.hyy * dxy + F1.gy * w1;
            const float dpax = dpx + ds * qdpx, dpay = dpy + ds * qdpy;
            const float dxax = dxx + ds * qdxx, dxay = dxy + ds * qdxy;
            const float gda = F2.gx * dxax + F2.gy * dxay, pda = pax * dpax + pay * dpay;
            const float qdxax = ina * (dpax - pax * gda * ina), qdxay = ina * (dpay - pay * gda * ina);
            const float w2 = ina * (pda * ina - gda);
            const float qdpax = F2.hxx * dxax + F2.hxy * dxay + F2.gx * w2;
            const float qdpay = F2.hxy * dxax + F2.hyy * dxay + F2.gy * w2;
            const float ddxx = hds * (qdxx + qdxax), ddxy = hds * (qdxy + qdxay);
            const float ddpx2 = hds * (qdpx + qdpax), ddpy2 = hds * (qdpy + qdpay);
            const float xn = x + ds * dirx, yn = y + ds * diry;
            Fv Fn;
            {
                const float u = (xn - p.x0) * p.inv_dx, v = (yn - p.y0) * p.inv_dx;
                float tx = u - cell.i, ty = v - cell.j;
                if (!(tx >= 0.f && tx < 1.f && ty >= 0.f && ty < 1.f)) {
                    cell_load<LOSSY, RAW>(F, p, u, v, cell);
                    tx = u - cell.i; ty = v - cell.j;
                }
                cell_eval<LOSSY, RAW>(cell, tx, ty, Fn);
            }
            float inc = hds * (F1.nr + Fn.nr), incB = LOSSY ? hds * (F1.al + Fn.al) : 0.f;
            const bool last = xn * xn + yn * yn >= R2;
            if (last) {
                // final partial step: crossing of the step's chord with the ring; the other
                // quantities interpolated linearly along the chord. A first step starts at the
                // transducer, on the ring: |x|^2 - R^2 is 0 there, and its FP32 rounding residue
                // (~R ulp(R)) would swamp b^2 for the near-tangent rays that end within a step
                float b = x * dirx + y * diry, cc = i == 0 ? 0.f : x * x + y * y - R2;
                float disc = b * b - cc;
                float t = -b + sqrtf(disc > 0.f ? disc : 0.f);
                t = fminf(fmaxf(t, 0.f), ds);
                float fr = t / ds;
                x = x + t * dirx; y = y + t * diry;
                inc *= fr;
                incB *= fr;
                dxx += fr * ddxx; dxy += fr * ddxy;
                dpx += fr * ddpx2; dpy += fr * ddpy2;
                px += fr * ddpx; py += fr * ddpy;
                field_eval<LOSSY, RAW>(F, p, x, y, Fn);
            } else {
                kadd(x, cx, ds * dirx); kadd(y, cy, ds * diry);
                px += ddpx; py += ddpy;
                dxx += ddxx; dxy += ddxy;
                dpx += ddpx2; dpy += ddpy2;
            }
            kadd(T, Tc, inc);   // trapezoid of n along the samples
            if (LOSSY) kadd(B, Bc, incB);
            F1 = Fn;
            const float rp = rsqrtf(px * px + py * py), tx = px * rp, ty = py * rp;
            const float J = dxx * ty - dxy * tx;
            if (i == 0) { sc1 = sqrtf(F1.nr * fabsf(J) / ds); Jlast = J; }
            else if (J * Jlast < 0.f) K++;   // caustic: sign change of the ray Jacobian
            if (J != 0.f) Jlast = J;
            cur.x = x; cur.y = y; cur.T = T; cur.kx = tx; cur.ky = ty; cur.K = K;
            cur.a = sc1 * rsqrtf(F1.nr * fabsf(J));
            if (LOSSY) cur.a *= expf(-B);
            have = true;
            if (last) {
                alive = false;
                if (lane < 31 || j == N - 1)
                    exits[(size_t)e * (N - 1) + (j - 1)] = make_float4(atan2f(y, x), T, cur.a, (float)K);
            }
        }
        // neighbour ray j+1 (lane + 1): its sample i+1
        Vtx ncur;
        ncur.x = __shfl_down_sync(FULL, cur.x, 1);
        ncur.y = __shfl_down_sync(FULL, cur.y, 1);
        ncur.T = __shfl_down_sync(FULL, cur.T, 1);
        ncur.a = __shfl_down_sync(FULL, cur.a, 1);
        ncur.kx = __shfl_down_sync(FULL, cur.kx, 1);
        ncur.ky = __shfl_down_sync(FULL, cur.ky, 1);
        ncur.K = __shfl_down_sync(FULL, cur.K, 1);
        const bool nhave = __shfl_down_sync(FULL, (int)have, 1) != 0;
        const bool valid = i >= 1 && i >= i0 && have && nhave && lane < 31 && j + 1 <= N - 1;
        // A quad beyond a line two cells outside the mask holds no mask node, in any medium:
        // the edge functions accept only points of its two triangles, which lie in the convex
        // hull of its corners, so when every corner q has u.q > rm for u the direction of the
        // corners' sum, so does every accepted point, and |q| > rm. The warp skips the step's
        // rasterisation when that holds for all its quads. The corners' own radii beyond rm
        // are necessary for it and cheap, so the line test runs only when they hold for the
        // whole warp (radii alone would not do: the cross edge of a wide tube can be a chord
        // through the mask).
        const bool ob = fmaf(cur.x, cur.x, cur.y * cur.y) > rm2 && fmaf(prev.x, prev.x, prev.y * prev.y) > rm2;
        const bool nb = __shfl_down_sync(FULL, (int)ob, 1) != 0;
        bool skip = __all_sync(FULL, !valid || (ob && nb));
        if (skip) {
            bool hs = true;
            if (valid) {
                const float gx = (prev.x + cur.x) + (nprev.x + ncur.x), gy = (prev.y + cur.y) + (nprev.y + ncur.y);
                const float h = fminf(fminf(fmaf(gx, prev.x, gy * prev.y), fmaf(gx, cur.x, gy * cur.y)),
                                      fminf(fmaf(gx, nprev.x, gy * nprev.y), fmaf(gx, ncur.x, gy * ncur.y)));
                hs = h > 0.f && h * h > rm2 * fmaf(gx, gx, gy * gy);
            }
            skip = __all_sync(FULL, hs);
        }
        if (!skip)
            raster_quad_warp(valid, prev, cur, nprev, ncur, ((uint32_t)j << 11 | (uint32_t)i) << 1, p, inv_dx, 0, 1, rows,
                             fan, hq, counters);
        prev = cur;
        nprev = ncur;
        // Leaving through the uniform water: once a ray is beyond rho, moving outward, and so
        // are (or have ended) the rays it forms quads with in this warp, no later quad of it
        // can hold a mask node, and it goes straight to the ring in closed form (the chord's
        // crossing as in the last step above; J is linear in s there, so at most one caustic).
        {
            const bool out = alive && i >= kin && fmaf(x, x, y * y) > rho2 && fmaf(x, px, y * py) > 0.f;
            if (__any_sync(FULL, out)) {
                const bool okself = !alive || out;
                bool okL = __shfl_up_sync(FULL, okself, 1), okR = __shfl_down_sync(FULL, okself, 1);
                const bool aL = __shfl_up_sync(FULL, alive, 1), aR = __shfl_down_sync(FULL, alive, 1);
                const float xl = __shfl_up_sync(FULL, x, 1), yl = __shfl_up_sync(FULL, y, 1);
                const float xr = __shfl_down_sync(FULL, x, 1), yr = __shfl_down_sync(FULL, y, 1);
                const float gap = rho - p.rmask, gap2 = gap * gap;
                if (lane == 0) okL = true;
                else if (aL) okL = okL && (x - xl) * (x - xl) + (y - yl) * (y - yl) < gap2;
                if (lane == 31) okR = true;
                else if (aR) okR = okR && (x - xr) * (x - xr) + (y - yr) * (y - yr) < gap2;
                if (out && okL && okR) {
                    const float n = F1.n, in = rcp_nr(n), inc = hds * (F1.nr + F1.nr);
                    const float rp = rsqrtf(px * px + py * py), tx = px * rp, ty = py * rp;
                    const float b = x * tx + y * ty, se = -b + sqrtf(fmaxf(b * b - over_ring(fmaf(x, x, y * y), p.R), 0.f));
                    const int m = max(0, (int)floorf(se / ds));
                    const float sm = (float)m * ds;
                    const float xm = fmaf(sm, tx, x), ym = fmaf(sm, ty, y);
                    const float b2 = xm * tx + ym * ty, disc = b2 * b2 - over_ring(fmaf(xm, xm, ym * ym), p.R);
                    float t = -b2 + sqrtf(disc > 0.f ? disc : 0.f);
                    t = fminf(fmaxf(t, 0.f), ds);
                    x = fmaf(t, tx, xm); y = fmaf(t, ty, ym);
                    kadd(T, Tc, (float)m * inc);
                    kadd(T, Tc, (t / ds) * inc);
                    if (LOSSY) {
                        const float incB = hds * (F1.al + F1.al);
                        kadd(B, Bc, (float)m * incB);
                        kadd(B, Bc, (t / ds) * incB);
                    }
                    dxx = fmaf(sm + t, dpx * in, dxx); dxy = fmaf(sm + t, dpy * in, dxy);
                    field_eval<LOSSY, RAW>(F, p, x, y, F1);
                    const float J = dxx * ty - dxy * tx;
                    if (J * Jlast < 0.f) K++;
                    const float a = sc1 * rsqrtf(F1.nr * fabsf(J)) * (LOSSY ? expf(-B) : 1.f);
                    if (lane < 31 || j == N - 1)
                        exits[(size_t)e * (N - 1) + (j - 1)] = make_float4(atan2f(y, x), T, a, (float)K);
                    alive = false;
                }
            }
        }
        if (!__any_sync(FULL, alive)) break;
        if (i == p.maxs - 1 && alive) atomicAdd(&counters[2], 1ull);   // ray never reached the ring
    }
    // drain the rest of the queue; the covered-entry count goes to counters[0]
    count_first(hq, lane < hq.n && drain_one(hq, lane, fan, counters));
    __syncwarp();
    if (lane == 0 && *hq.cov) atomicAdd(&counters[0], (unsigned long long)*hq.cov);
}

template <bool LOSSY, bool RAW, int WARPS>
__global__ __launch_bounds__(32 * kFansPerBlock, WARPS / kFansPerBlock) void k_trace_raster(const float *__restrict__ F, const int4 *__restrict__ rows_g,
                                                         TabEntry *__restrict__ tab, float4 *__restrict__ exits,
                                                         RayParams p, unsigned long long *counters)
{
    extern __shared__ int4 rows[];                          // [ny] mask row ranges
    __shared__ BlockQueues bq;
    for (int q = threadIdx.x; q < p.ny; q += blockDim.x) rows[q] = rows_g[q];
    if (threadIdx.x < kFansPerBlock) bq.cov[threadIdx.x] = 0u;
    __syncthreads();
    trace_block<LOSSY, RAW>(F, rows, tab, exits, p, counters, warp_of_rank(blockIdx.y, gridDim.y), blockIdx.x, bq);
}

// The trace of a small ring, whose rays are too few to fill the GPU with one lane each: a block
// takes the 32 rays of one warp of k_trace_raster with LPR lanes per ray, which carry the same ray and share out
// the candidate nodes of its tube (most of a step's time there). The rays' samples go to their
// neighbours through shared memory, one barrier per step. Same arithmetic, ray groups and
// table as k_trace_raster.
// Against one lane per ray (rbx_trace_rays): 64 transducers (96 x 96), eight lanes: 0.453 -> 0.351 ms; 128
// (160 x 160), four: 0.805 -> 0.755; 192 (217 x 217), two: 1.139 -> 1.112 (200 x 200: 0.99, 1.00). Bound: a ray's
// chain of steps and the barrier between them (64 transducers: issue port busy 27 % of the cycles of
// the SMs at work, a third of the stalled time at the barrier).
template <int LPR>
struct WideShared {
    uint4 v[LPR][64];
    float2 w[LPR][64];
    unsigned cov[LPR];
    float4 a[2][32];   // x, y, T, a of the rays' samples, by parity of the step
    float4 b[2][32];   // kx, ky, K, flags
    int i0;
};

template <bool LOSSY, bool RAW, int LPR>
__global__ __launch_bounds__(32 * LPR, 16 / LPR) void k_trace_wide(const float *__restrict__ F,
                                                                  const int4 *__restrict__ rows_g,
                                                                  TabEntry *__restrict__ tab, float4 *__restrict__ exits,
                                                                  RayParams p, unsigned long long *counters)
{
    extern __shared__ int4 rows[];                          // [ny] mask row ranges
    __shared__ WideShared<LPR> sh;
    for (int q = threadIdx.x; q < p.ny; q += blockDim.x) rows[q] = rows_g[q];
    if (threadIdx.x < LPR) sh.cov[threadIdx.x] = 0u;
    if (threadIdx.x == 0) sh.i0 = 0x7fffffff;
    __syncthreads();
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int e = blockIdx.x, N = p.N;
    const int ray = threadIdx.x / LPR, sub = threadIdx.x % LPR;
    const int j = 1 + 31 * warp_of_rank(blockIdx.y, gridDim.y) + ray;   // this lane's ray
    const bool has_ray = j <= N - 1;
    TabEntry *fan = tab + (size_t)e * p.X;
    const float ds = p.ds, hds = 0.5f * p.ds, inv_dx = p.inv_dx, R2 = p.R * p.R;
    HitQueue hq{sh.v[wib], sh.w[wib], &sh.cov[wib], 0};

    const double be = p.beta ? p.beta[e] : 2.0 * 3.14159265358979323846 * e / N;
    float x = (float)(p.R * cos(be)), y = (float)(p.R * sin(be));
    const float gam0 = (float)(be + 3.14159265358979323846 / 2 + 3.14159265358979323846 * j / N);

    // reference ray (x, p) and paraxial ray (dx, dp); F1 caches the fields at x
    Fv F1;
    field_eval<LOSSY, RAW>(F, p, x, y, F1);
    float px, py, dpx, dpy, dxx = 0.f, dxy = 0.f, T = 0.f, Tc = 0.f;
    float B = 0.f, Bc = 0.f;   // lossy media: B = int alpha ds by the rule of T; a gains exp(-B)
    // compensation terms of the position and of the paraxial ray's closed-form steps (T has
    // Tc). In the Heun steps the momentum, renormalised to n(x) at every step, and the
    // paraxial ray, which only sets the amplitude, take plain sums: compensated too, the
    // tables met the same parity bars against the FP64 oracle (T 1e-9 s, a 1e-5) and the
    // trace took 1.6 % longer.
    float cx = 0.f, cy = 0.f, cdx = 0.f, cdy = 0.f;

    // Uniform water near the ring (exact up to rounding). Beyond radius rho every cell that a
    // sample or an auxiliary point can touch holds the same medium with zero derivatives (rho
    // exceeds the largest radius of a non-uniform node by a cell diagonal and a step), so there
    // a ray is a straight line with constant n and a linearly growing paraxial deviation; rho
    // also stays two cells outside the mask, so a quad with all vertices beyond rho holds no
    // mask node. Up to its entry step kin (its last sample beyond rho on the way in) a ray
    // takes the closed form of the step; kin depends on the ray alone, so the ray shared by two
    // warps has identical samples in both. The warp rasterises nothing before its smallest kin.
    const float ru = __uint_as_float((unsigned)counters[7]);
    const float rho = fmaxf(ru + 1.5f * p.dx + ds, p.rmask + 2.f * p.dx), rho2 = rho * rho;
    int kin = 0;
    {
        float s0, c0;
        sincosf(gam0, &s0, &c0);
        px = F1.n * c0; py = F1.n * s0;
        dpx = -F1.n * s0; dpy = F1.n * c0;
        if (has_ray && R2 > rho2) {
            const float b = x * c0 + y * s0, disc = b * b - (fmaf(x, x, y * y) - rho2);
            const float s_in = disc >= 0.f ? -b - sqrtf(disc) : -b;   // entry, or closest approach
            kin = max(0, (int)floorf(s_in / ds) - 1);
        }
    }
    if (has_ray) atomicMin(&sh.i0, kin);
    __syncthreads();
    const int i0 = sh.i0;
    const float rm = p.rmask + 2.f * p.dx, rm2 = rm * rm;
    float sc1 = 0.f, Jlast = 0.f;   // sc1 = sqrt(n_1 |J_1| / ds): a_i = sc1 / sqrt(n_i |J_i|)
    int K = 0;
    bool alive = has_ray;
    Vtx prev{}, nprev{};

    for (int i = 0; i < p.maxs; i++) {
        Vtx cur{};
        bool have = false;
        if (alive && i < kin) {
            // the step below in a uniform medium: straight, p constant, dx += ds dp / n
            const float n = F1.n, in = rcp_nr(n);
            const float rp = rsqrtf(px * px + py * py), tx = px * rp, ty = py * rp;
            kadd(x, cx, ds * tx); kadd(y, cy, ds * ty);
            kadd(dxx, cdx, ds * (dpx * in)); kadd(dxy, cdy, ds * (dpy * in));
            kadd(T, Tc, hds * (F1.nr + F1.nr));
            if (LOSSY) kadd(B, Bc, hds * (F1.al + F1.al));
            const float J = dxx * ty - dxy * tx;
            if (i == 0) { sc1 = sqrtf(F1.nr * fabsf(J) / ds); Jlast = J; }
            else if (J * Jlast < 0.f) K++;
            if (J != 0.f) Jlast = J;
            cur.x = x; cur.y = y; cur.T = T; cur.kx = tx; cur.ky = ty; cur.K = K;
            cur.a = sc1 * rsqrtf(F1.nr * fabsf(J));
            if (LOSSY) cur.a *= expf(-B);
            have = true;
        } else if (alive) {
            // stage 1 at x: normalise p to n(x), q_x = p/n, q_p = grad n
            const float n = F1.n, in = rcp_ap(n);
            const float sc = n * rsqrtf(px * px + py * py);
            px *= sc; py *= sc;
            const float qx = px * in, qy = py * in;
            // stage 2 at the auxiliary point x + ds q_x
            Fv F2;
            // The new sample lies within ds times half the step's bend of the auxiliary point
            // (about 1e-4 cells), so the nodes of one cell serve both but where a grid line runs
            // between them: half the loads and their address arithmetic (16.4 -> 15.6 ms at 1024
            // transducers on 512 x 512).
            Cell<LOSSY, RAW> cell;
            {
                const float ax = x + ds * qx, ay = y + ds * qy;
                const float u = (ax - p.x0) * p.inv_dx, v = (ay - p.y0) * p.inv_dx;
                cell_load<LOSSY, RAW>(F, p, u, v, cell);
                cell_eval<LOSSY, RAW>(cell, u - cell.i, v - cell.j, F2);
            }
            const float na = F2.n, ina = rcp_ap(na);
            float pax = px + ds * F1.gx, pay = py + ds * F1.gy;
            const float sca = na * rsqrtf(pax * pax + pay * pay);
            pax *= sca; pay *= sca;
            const float qax = pax * ina, qay = pay * ina;
            const float sx = qx + qax, sy = qy + qay, rs = rsqrtf(sx * sx + sy * sy);
            const float dirx = sx * rs, diry = sy * rs;
            const float ddpx = hds * (F1.gx + F2.gx), ddpy = hds * (F1.gy + F2.gy);
            // paraxial system, both stages at the reference ray's stage values:
            // q_dx = (dp - p (g.dx)/n)/n, q_dp = H dx + g ((p.dp)/n - g.dx)/n
            const float gd = F1.gx * dxx + F1.gy * dxy, pd = px * dpx + py * dpy;
            const float qdxx = in * (dpx - px * gd * in), qdxy = in * (dpy - py * gd * in);
            const float w1 = in * (pd * in - gd);
            const float qdpx = F1.hxx * dxx + F1.hxy * dxy + F1.gx * w1;
            const float qdpy = F1.hxy * dxx + F1.hyy * dxy + F1.gy * w1;
            const float dpax = dpx + ds * qdpx, dpay = dpy + ds * qdpy;
            const float dxax = dxx + ds * qdxx, dxay = dxy + ds * qdxy;
            const float gda = F2.gx * dxax + F2.gy * dxay, pda = pax * dpax + pay * dpay;
            const float qdxax = ina * (dpax - pax * gda * ina), qdxay = ina * (dpay - pay * gda * ina);
            const float w2 = ina * (pda * ina - gda);
            const float qdpax = F2.hxx * dxax + F2.hxy * dxay + F2.gx * w2;
            const float qdpay = F2.hxy * dxax + F2.hyy * dxay + F2.gy * w2;
            const float ddxx = hds * (qdxx + qdxax), ddxy = hds * (qdxy + qdxay);
            const float ddpx2 = hds * (qdpx + qdpax), ddpy2 = hds * (qdpy + qdpay);
            const float xn = x + ds * dirx, yn = y + ds * diry;
            Fv Fn;
            {
                const float u = (xn - p.x0) * p.inv_dx, v = (yn - p.y0) * p.inv_dx;
                float tx = u - cell.i, ty = v - cell.j;
                if (!(tx >= 0.f && tx < 1.f && ty >= 0.f && ty < 1.f)) {
                    cell_load<LOSSY, RAW>(F, p, u, v, cell);
                    tx = u - cell.i; ty = v - cell.j;
                }
                cell_eval<LOSSY, RAW>(cell, tx, ty, Fn);
            }
            float inc = hds * (F1.nr + Fn.nr), incB = LOSSY ? hds * (F1.al + Fn.al) : 0.f;
            const bool last = xn * xn + yn * yn >= R2;
            if (last) {
                // final partial step: crossing of the step's chord with the ring; the other
                // quantities interpolated linearly along the chord. A first step starts at the
                // transducer, on the ring: |x|^2 - R^2 is 0 there, and its FP32 rounding residue
                // (~R ulp(R)) would swamp b^2 for the near-tangent rays that end within a step
                float b = x * dirx + y * diry, cc = i == 0 ? 0.f : x * x + y * y - R2;
                float disc = b * b - cc;
                float t = -b + sqrtf(disc > 0.f ? disc : 0.f);
                t = fminf(fmaxf(t, 0.f), ds);
                float fr = t / ds;
                x = x + t * dirx; y = y + t * diry;
                inc *= fr;
                incB *= fr;
                dxx += fr * ddxx; dxy += fr * ddxy;
                dpx += fr * ddpx2; dpy += fr * ddpy2;
                px += fr * ddpx; py += fr * ddpy;
                field_eval<LOSSY, RAW>(F, p, x, y, Fn);
            } else {
                kadd(x, cx, ds * dirx); kadd(y, cy, ds * diry);
                px += ddpx; py += ddpy;
                dxx += ddxx; dxy += ddxy;
                dpx += ddpx2; dpy += ddpy2;
            }
            kadd(T, Tc, inc);   // trapezoid of n along the samples
            if (LOSSY) kadd(B, Bc, incB);
            F1 = Fn;
            const float rp = rsqrtf(px * px + py * py), tx = px * rp, ty = py * rp;
            const float J = dxx * ty - dxy * tx;
            if (i == 0) { sc1 = sqrtf(F1.nr * fabsf(J) / ds); Jlast = J; }
            else if (J * Jlast < 0.f) K++;   // caustic: sign change of the ray Jacobian
            if (J != 0.f) Jlast = J;
            cur.x = x; cur.y = y; cur.T = T; cur.kx = tx; cur.ky = ty; cur.K = K;
            cur.a = sc1 * rsqrtf(F1.nr * fabsf(J));
            if (LOSSY) cur.a *= expf(-B);
            have = true;
            if (last) {
                alive = false;
                if (sub == 0 && (ray < 31 || j == N - 1))
                    exits[(size_t)e * (N - 1) + (j - 1)] = make_float4(atan2f(y, x), T, cur.a, (float)K);
            }
        }
        // the sample and what the neighbours need to know of the ray
        const bool ob = fmaf(cur.x, cur.x, cur.y * cur.y) > rm2 && fmaf(prev.x, prev.x, prev.y * prev.y) > rm2;
        const bool out = alive && i >= kin && fmaf(x, x, y * y) > rho2 && fmaf(x, px, y * py) > 0.f;
        const int par = i & 1;
        if (sub == 0) {
            // a ray that has ended leaves its last position, as its lanes hold it
            sh.a[par][ray] = make_float4(have ? cur.x : x, have ? cur.y : y, cur.T, cur.a);
            sh.b[par][ray] = make_float4(cur.kx, cur.ky, __int_as_float(cur.K),
                                         __int_as_float((have ? 1 : 0) | (ob ? 2 : 0) | (alive ? 4 : 0) | (out ? 8 : 0)));
        }
        if (!__syncthreads_or(have)) break;
        // neighbour ray j+1: its sample i+1
        const float4 na = sh.a[par][min(ray + 1, 31)], nb4 = sh.b[par][min(ray + 1, 31)];
        const int nflags = __float_as_int(nb4.w);
        Vtx ncur;
        ncur.x = na.x; ncur.y = na.y; ncur.T = na.z; ncur.a = na.w;
        ncur.kx = nb4.x; ncur.ky = nb4.y; ncur.K = __float_as_int(nb4.z);
        const bool valid = i >= 1 && i >= i0 && have && (nflags & 1) && ray < 31 && j + 1 <= N - 1;
        // skip where every quad lies beyond a line two cells outside the mask, as k_trace_raster
        bool skip = __all_sync(FULL, !valid || (ob && (nflags & 2)));
        if (skip) {
            bool hs = true;
            if (valid) {
                const float gx = (prev.x + cur.x) + (nprev.x + ncur.x), gy = (prev.y + cur.y) + (nprev.y + ncur.y);
                const float h = fminf(fminf(fmaf(gx, prev.x, gy * prev.y), fmaf(gx, cur.x, gy * cur.y)),
                                      fminf(fmaf(gx, nprev.x, gy * nprev.y), fmaf(gx, ncur.x, gy * ncur.y)));
                hs = h > 0.f && h * h > rm2 * fmaf(gx, gx, gy * gy);
            }
            skip = __all_sync(FULL, hs);
        }
        if (!skip)
            raster_quad_warp(valid, prev, cur, nprev, ncur, ((uint32_t)j << 11 | (uint32_t)i) << 1, p, inv_dx, sub, LPR,
                             rows, fan, hq, counters);
        prev = cur;
        nprev = ncur;
        // leaving through the uniform water, as k_trace_raster
        if (out) {
            const float4 la = sh.a[par][max(ray - 1, 0)];
            const int lflags = __float_as_int(sh.b[par][max(ray - 1, 0)].w);
            const bool aL = lflags & 4, aR = nflags & 4;
            bool okL = !aL || (lflags & 8), okR = !aR || (nflags & 8);
            const float xl = la.x, yl = la.y, xr = na.x, yr = na.y;
            const float gap = rho - p.rmask, gap2 = gap * gap;
            if (ray == 0) okL = true;
            else if (aL) okL = okL && (x - xl) * (x - xl) + (y - yl) * (y - yl) < gap2;
            if (ray == 31) okR = true;
            else if (aR) okR = okR && (x - xr) * (x - xr) + (y - yr) * (y - yr) < gap2;
            if (okL && okR) {
                const float n = F1.n, in = rcp_nr(n), inc = hds * (F1.nr + F1.nr);
                const float rp = rsqrtf(px * px + py * py), tx = px * rp, ty = py * rp;
                const float b = x * tx + y * ty, se = -b + sqrtf(fmaxf(b * b - over_ring(fmaf(x, x, y * y), p.R), 0.f));
                const int m = max(0, (int)floorf(se / ds));
                const float sm = (float)m * ds;
                const float xm = fmaf(sm, tx, x), ym = fmaf(sm, ty, y);
                const float b2 = xm * tx + ym * ty, disc = b2 * b2 - over_ring(fmaf(xm, xm, ym * ym), p.R);
                float t = -b2 + sqrtf(disc > 0.f ? disc : 0.f);
                t = fminf(fmaxf(t, 0.f), ds);
                x = fmaf(t, tx, xm); y = fmaf(t, ty, ym);
                kadd(T, Tc, (float)m * inc);
                kadd(T, Tc, (t / ds) * inc);
                if (LOSSY) {
                    const float incB = hds * (F1.al + F1.al);
                    kadd(B, Bc, (float)m * incB);
                    kadd(B, Bc, (t / ds) * incB);
                }
                dxx = fmaf(sm + t, dpx * in, dxx); dxy = fmaf(sm + t, dpy * in, dxy);
                field_eval<LOSSY, RAW>(F, p, x, y, F1);
                const float J = dxx * ty - dxy * tx;
                if (J * Jlast < 0.f) K++;
                const float a = sc1 * rsqrtf(F1.nr * fabsf(J)) * (LOSSY ? expf(-B) : 1.f);
                if (sub == 0 && (ray < 31 || j == N - 1))
                    exits[(size_t)e * (N - 1) + (j - 1)] = make_float4(atan2f(y, x), T, a, (float)K);
                alive = false;
            }
        }
        if (i == p.maxs - 1 && alive && sub == 0) atomicAdd(&counters[2], 1ull);   // ray never reached the ring
    }
    count_first(hq, lane < hq.n && drain_one(hq, lane, fan, counters));
    __syncwarp();
    if (lane == 0 && *hq.cov) atomicAdd(&counters[0], (unsigned long long)*hq.cov);
}

// Persistent form of the trace over several jobs (the batched form). Each block takes the
// next item from a device counter until the list is exhausted: items are numbered job by job
// in the order of g.j, and within a job as the blocks of the per-job grid (the fans of one rank
// of warps, then the next rank). An item is one block of the per-job kernel. The job list is a kernel parameter, so that the
// jobs' parameters stay in the constant bank (with them in shared memory the kernel spilled
// and ran 5.8 % slower per item; this form costs 1.1 %).
template <bool LOSSY, bool RAW>
__global__ __launch_bounds__(32 * kFansPerBlock, 20 / kFansPerBlock) void k_trace_grouped(const __grid_constant__ TraceGroup g,
                                                                                        int *next)
{
    extern __shared__ int4 rows[];   // [largest ny of the jobs]
    __shared__ BlockQueues bq;
    __shared__ int s_item, s_job;
    for (;;) {
        __syncthreads();   // the block's warps are done with the previous item
        if (threadIdx.x == 0) {
            const int it = atomicAdd(next, 1);
            int jb = 0;
            if (it < g.total)
                while (jb + 1 < g.njobs && g.j[jb + 1].item0 <= it) jb++;
            s_item = it;
            s_job = jb;
        }
        __syncthreads();
        const int it = s_item;
        if (it >= g.total) return;   // uniform over the block
        const TraceJob &J = g.j[s_job];
        for (int q = threadIdx.x; q < J.p.ny; q += blockDim.x) rows[q] = J.rows[q];
        if (threadIdx.x < kFansPerBlock) bq.cov[threadIdx.x] = 0u;
        __syncthreads();
        const int local = it - J.item0;
        const int nfb = (J.p.N + kFansPerBlock - 1) / kFansPerBlock;
        trace_block<LOSSY, RAW>(J.F, rows, J.tab, J.exits, J.p, J.counters, warp_of_rank(local / nfb, J.nwarps),
                                local % nfb, bq);
    }
}

// Largest radius of a node whose fields differ from the uniform medium of node (0, 0)
// (n, alpha and the integrated slowness there, all derivatives zero); +inf when node (0, 0)
// itself is not uniform.
__global__ void k_uniform_radius(const float4 *__restrict__ F, RayParams p, unsigned long long *ru)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned r = 0u;   // bits of a non-negative float: their order is the values' order
    if (k < p.nx * p.ny) {
        const size_t nxy = (size_t)p.nx * p.ny;
        const float2 *F2 = reinterpret_cast<const float2 *>(F + nxy), *F3 = F2 + nxy;
        const float4 u0 = F[0], a0 = F[k];
        const float2 v0 = F2[0], v1 = F3[0], b0 = F2[k], b1 = F3[k];
        const float4 u1 = make_float4(v0.x, v0.y, v1.x, v1.y), a1 = make_float4(b0.x, b0.y, b1.x, b1.y);
        if (k == 0 && !(u0.y == 0.f && u0.z == 0.f && u0.w == 0.f && u1.x == 0.f && u1.y == 0.f)) {
            r = 0x7f800000u;   // +inf
        } else {
            const bool uni = a0.x == u0.x && a0.y == 0.f && a0.z == 0.f && a0.w == 0.f && a1.x == 0.f &&
                             a1.y == 0.f && a1.z == u1.z && a1.w == u1.w;
            if (!uni) {
                const float px = p.x0 + (float)(k % p.nx) * p.dx, py = p.y0 + (float)(k / p.nx) * p.dx;
                r = __float_as_uint(sqrtf(px * px + py * py));
            }
        }
    }
    r = __reduce_max_sync(0xffffffffu, r);   // one atomic per warp
    if ((threadIdx.x & 31) == 0 && r) atomicMax(ru, (unsigned long long)r);
}

void launch_uniform_radius(const float *fields, const RayParams &p, unsigned long long *ru, cudaStream_t s)
{
    const int n = p.nx * p.ny;
    k_uniform_radius<<<(n + 255) / 256, 256, 0, s>>>(reinterpret_cast<const float4 *>(fields), p, ru);
}

// Lanes per ray: the most (up to 8) with which the traces running together (load: their warps with one
// lane per ray, this one's included) stay within a number of warps. Every lane of a ray integrates it, which
// costs nothing only while the GPU has issue slots to spare, and gives nothing where a ray's tube holds
// no node to share out. So the number is 3,040 for a trace alone, 1,216 (8 per SM) where the tubes are thin
// (2 R ds / (dx dx N), to a factor the nodes that a quad of the fan holds on average, below 1/2), and half of
// that beside other jobs, whose contractions take some of the slots. The GPU holds 2,432 warps of k_trace_wide (16 per SM) and
// 3,040 of k_trace_raster; that the line lies there is what was measured (rbx_trace_rays alone, ms, lanes 1 / 2 /
// 4 / 8, ds = dx / 2):
//   thick, N on nodes: 64 on 96 0.464 / 0.442 / 0.383 / 0.358, 128 on 160 0.865 / 0.842 / 0.789 / 1.088, 152 on 160
//     0.810 / 0.787 / 0.734 / 1.250, 215 on 224 1.299 / 1.290 / 1.829 / 3.094
//   thin: 64 on 48 0.173 / 0.171 / 0.165 / 0.169, 96 on 64 0.225 / 0.229 / 0.239 / 0.251, 128 on 80 0.284 / 0.306 /
//     0.335 / 0.502, 215 on 80 0.263 / 0.370 / 0.585 / 1.048 (the two lanes of 3,040 warps took longer than the
//     0.327 of the kernel before the present one)
//   together: four of 64 on 96 0.497 / 0.494 / 0.487 / 0.648, eight 0.561 / 0.604 / 0.735 / 1.229; 24 of 128 on 160 4.0
//     with one lane, 11.2 with the four of a ring alone; a batch of three updates each, eight of 64: 1.98 with one
//     lane, 2.53 with two
// The block keeps its queues and `rows_bytes` of mask rows in the 48 KB of shared memory that a launch
// has without asking for more (eight lanes to 2,173 grid rows, four to 2,558). One lane, and
// k_trace_raster, from about 215 transducers on.
static int lanes_per_ray(const RayParams &p, size_t load, size_t rows_bytes)
{
    const bool thin = 2.f * p.R * p.ds < 0.5f * p.dx * p.dx * (float)p.N;
    const size_t most = (thin ? 1216 : 3040) / (load > trace_warps(p.N) ? 2 : 1);
    int l = 1;
    while (l < 8 && load * 2 * l <= most) l *= 2;
    auto fits = [&](int lanes) {
        const size_t queues = lanes == 8 ? sizeof(WideShared<8>) : lanes == 4 ? sizeof(WideShared<4>) : sizeof(WideShared<2>);
        return queues + rows_bytes <= 48 * 1024;
    };
    while (l > 1 && !fits(l)) l /= 2;
    return l;
}

void launch_trace_raster(const float *fields, const int4 *rows, TabEntry *tab, float4 *exits, const RayParams &p,
                         unsigned long long *counters, size_t load, bool lossy, bool raw, cudaStream_t s)
{
    // the longest warps of every fan first: the blocks that start last, and those that share
    // an SM when the grid is a single wave, then differ least (1024 transducers on 512 x 512:
    // 17.8 -> 16.5 ms; 512 on 256 x 256: 2.7 -> 2.25; 256 on 288 x 288, one wave: 2.84 -> 2.50)
    int nwarps = (p.N - 2 + 30) / 31;
    dim3 grd((p.N + kFansPerBlock - 1) / kFansPerBlock, nwarps);
    const size_t sm = (size_t)p.ny * sizeof(int4);
    const int lpr = lanes_per_ray(p, load, sm);
    if (lpr > 1) {
        auto wide = [&](auto lp) {
            constexpr int L = decltype(lp)::value;
            const dim3 g(p.N, nwarps);
            if (lossy && raw)
                k_trace_wide<true, true, L><<<g, 32 * L, sm, s>>>(fields, rows, tab, exits, p, counters);
            else if (lossy)
                k_trace_wide<true, false, L><<<g, 32 * L, sm, s>>>(fields, rows, tab, exits, p, counters);
            else if (raw)
                k_trace_wide<false, true, L><<<g, 32 * L, sm, s>>>(fields, rows, tab, exits, p, counters);
            else
                k_trace_wide<false, false, L><<<g, 32 * L, sm, s>>>(fields, rows, tab, exits, p, counters);
        };
        if (lpr == 8) wide(std::integral_constant<int, 8>{});
        else if (lpr == 4) wide(std::integral_constant<int, 4>{});
        else wide(std::integral_constant<int, 2>{});
        return;
    }
    auto go = [&](auto w) {
        constexpr int W = decltype(w)::value;
        if (lossy && raw)
            k_trace_raster<true, true, W><<<grd, 32 * kFansPerBlock, sm, s>>>(fields, rows, tab, exits, p, counters);
        else if (lossy)
            k_trace_raster<true, false, W><<<grd, 32 * kFansPerBlock, sm, s>>>(fields, rows, tab, exits, p, counters);
        else if (raw)
            k_trace_raster<false, true, W><<<grd, 32 * kFansPerBlock, sm, s>>>(fields, rows, tab, exits, p, counters);
        else
            k_trace_raster<false, false, W><<<grd, 32 * kFansPerBlock, sm, s>>>(fields, rows, tab, exits, p, counters);
    };
    // 16 warps per SM with 128 registers each while they hold the whole grid (to about 260
    // transducers: 256 on 288 x 288 1.86 -> 1.75 ms), else 20 with 96 and a few spills (1024 on 512 x 512
    // 15.6 ms against 16.4)
    if ((size_t)p.N * nwarps <= 152 * 16)
        go(std::integral_constant<int, 16>{});
    else
        go(std::integral_constant<int, 20>{});
}

size_t trace_warps(int N) { return (size_t)N * ((N - 2 + 30) / 31); }

int trace_items(int N, int *nwarps)
{
    const int nw = (N - 2 + 30) / 31;
    if (nwarps) *nwarps = nw;
    return nw * ((N + kFansPerBlock - 1) / kFansPerBlock);
}

template <bool LOSSY, bool RAW>
static int grouped_blocks_of(int max_ny)
{
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_trace_grouped<LOSSY, RAW>, 32 * kFansPerBlock,
                                                      (size_t)max_ny * sizeof(int4)) != cudaSuccess)
        return 0;
    return sms * per_sm;
}

int trace_grouped_blocks(bool lossy, bool raw, int max_ny)
{
    if (lossy && raw) return grouped_blocks_of<true, true>(max_ny);
    if (lossy) return grouped_blocks_of<true, false>(max_ny);
    if (raw) return grouped_blocks_of<false, true>(max_ny);
    return grouped_blocks_of<false, false>(max_ny);
}

void launch_trace_grouped(const TraceGroup &g, int max_ny, int blocks, int *next, bool lossy, bool raw, cudaStream_t s)
{
    const int grd = blocks < g.total ? blocks : g.total;
    const size_t sm = (size_t)max_ny * sizeof(int4);
    if (lossy && raw)
        k_trace_grouped<true, true><<<grd, 32 * kFansPerBlock, sm, s>>>(g, next);
    else if (lossy)
        k_trace_grouped<true, false><<<grd, 32 * kFansPerBlock, sm, s>>>(g, next);
    else if (raw)
        k_trace_grouped<false, true><<<grd, 32 * kFansPerBlock, sm, s>>>(g, next);
    else
        k_trace_grouped<false, false><<<grd, 32 * kFansPerBlock, sm, s>>>(g, next);
}

// rows[iy] = (compact index of the row's first mask node, first ix, last ix); empty rows
// get first ix > last ix. The mask is a disc, so each row's mask nodes are contiguous.
__global__ void k_mask_rows(const int *__restrict__ node2x, int nx, int ny, int4 *__restrict__ rows)
{
    int iy = blockIdx.x * blockDim.x + threadIdx.x;
    if (iy >= ny) return;
    int first = -1, last = -2, off = 0;
    for (int ix = 0; ix < nx; ix++) {
        int k = node2x[iy * nx + ix];
        if (k >= 0) {
            if (first < 0) { first = ix; off = k; }
            last = ix;
        }
    }
    rows[iy] = make_int4(off, first < 0 ? 1 : first, first < 0 ? 0 : last, 0);
}

void launch_mask_rows(const int *node2x, int nx, int ny, int4 *rows, cudaStream_t s)
{
    k_mask_rows<<<(ny + 127) / 128, 128, 0, s>>>(node2x, nx, ny, rows);
}

// ---------------------------------------------------------------- a4

// ---------------------------------------------------------------- a5

// Phase in cycles: f T - K/4 + 1/8, with f = fhi + flo and the product f T formed
// exactly enough (two-product) that omega T ~ 10^3 rad keeps ~1e-7 rad accuracy.
__device__ __forceinline__ float phase_cycles(float T, int K, float fhi, float flo)
{
    float p = fhi * T;
    float err = fmaf(fhi, T, -p) + flo * T;
    float r = (p - rintf(p)) + err;
    return r + 0.125f - 0.25f * (float)K;
}

__device__ __forceinline__ float wrap2pi(float t)
{
    const float TWO_PI = 6.28318530717959f;
    return t - TWO_PI * floorf(t / TWO_PI);
}

// An angle difference d in (-4 pi, 4 pi) taken to [0, 2 pi) by whole turns.
__device__ __forceinline__ double wrap_turn(double d)
{
    const double TWO_PI = 6.283185307179586476925;
    if (d < 0.0) d += TWO_PI;
    if (d < 0.0) d += TWO_PI;
    if (d >= TWO_PI) d -= TWO_PI;
    if (d >= TWO_PI) d -= TWO_PI;
    return d;
}

// Angle of the receiver m ring places after transducer e (r = (e + m) mod N) relative to it,
// in [0, 2 pi), increasing with m: m steps of step = 2 pi / N on the uniform ring (no FP64
// division or rounding to whole turns: FP64 is slow on this GPU), else the difference of the
// caller's position angles.
__device__ __forceinline__ double recv_rel_m(int m, int e, int N, double step, const double *beta, double be)
{
    return beta ? wrap_turn(beta[(e + m) % N] - be) : (double)m * step;
}

// Position angle of transducer e.
__device__ __forceinline__ double xducer_angle(int e, int N, double step, const double *beta)
{
    return beta ? beta[e] : (double)e * step;
}

// For every receiver r != e of fan e, the first pair of consecutive fan rays (j, j + 1),
// j = 1..N-2, whose exit angles th (relative to beta_e, in [0, 2 pi)) bracket beta_r, as
// first[r] = j, or INT_MAX when no pair does. relt[m] is the receiver angle relative to beta_e
// of ring place m (increasing in m). Each pair marks the receivers between its two exit
// angles (a binary search for the first, then the run up to the larger angle) and the
// smallest j wins, so a fan costs O(N log N) rather than a scan over the pairs per receiver.
// Called by the whole block.
__device__ void first_brackets(const float *th, const float *relt, int N, int e, int *first)
{
    for (int r = threadIdx.x; r < N; r += blockDim.x) first[r] = INT_MAX;
    __syncthreads();
    for (int j = 1 + threadIdx.x; j <= N - 2; j += blockDim.x) {
        const float tj = th[j - 1], tk = th[j];
        if (tj == tk) continue;
        const float lo = fminf(tj, tk), hi = fmaxf(tj, tk);
        int a = 1, b = N;   // first ring place m in [1, N - 1] with relt[m] >= lo (N: none)
        while (a < b) {
            const int c = (a + b) >> 1;
            if (relt[c] < lo) a = c + 1; else b = c;
        }
        for (int m = a; m <= N - 1 && relt[m] <= hi; m++) atomicMin(&first[(e + m) % N], j);
    }
    __syncthreads();
}

__global__ void k_direct_green(const float4 *__restrict__ exits, int N, const double *__restrict__ beta, float fhi,
                               float flo, float C, float2 *__restrict__ g, unsigned long long *counters)
{
    extern __shared__ float4 ex[];
    double *reld = reinterpret_cast<double *>(ex + (N - 1));   // receiver angle relative to beta_e by ring place
    double *thd = reld + N;                                    // exit angle relative to beta_e, in [0, 2 pi)
    float *th = reinterpret_cast<float *>(thd + (N - 1));      // thd rounded to float
    float *relt = th + (N - 1);                                // reld rounded to float
    int *first = reinterpret_cast<int *>(relt + N);            // first bracketing pair per receiver
    const int e = blockIdx.x;
    const double step = 6.283185307179586476925 / N, be = xducer_angle(e, N, step, beta);
    for (int q = threadIdx.x; q < N - 1; q += blockDim.x) {
        float4 v = exits[(size_t)e * (N - 1) + q];
        ex[q] = v;
        thd[q] = wrap_turn((double)v.x - be);
        th[q] = (float)thd[q];
    }
    for (int m = threadIdx.x; m < N; m += blockDim.x) {
        reld[m] = recv_rel_m(m, e, N, step, beta, be);
        relt[m] = (float)reld[m];
    }
    __syncthreads();
    first_brackets(th, relt, N, e, first);
    for (int r = threadIdx.x; r < N; r += blockDim.x) {
        if (r == e) { g[(size_t)e * N + r] = make_float2(0.f, 0.f); continue; }
        const double td = reld[(r - e + N) % N];
        const float t = (float)td;
        // first consecutive pair (j, j+1) whose exit angles bracket beta_r
        const int found = first[r] == INT_MAX ? -1 : first[r];
        float T, a;
        int K;
        if (found > 0) {
            float4 A = ex[found - 1], B = ex[found];
            // the bracket fraction from the exit angles in double precision
            const double ta = thd[found - 1], tb = thd[found];
            const double fr = (td - ta) / (tb - ta);
            T = (float)((double)A.y + fr * ((double)B.y - (double)A.y));
            a = (float)((double)A.z + fr * ((double)B.z - (double)A.z));
            K = (int)(fr < 0.5 ? A.w : B.w);
        } else {
            int best = 1;
            float bd = 1e30f;
            for (int j = 1; j <= N - 1; j++) {
                float d = fabsf(th[j - 1] - t);
                if (d < bd) { bd = d; best = j; }
            }
            float4 A = ex[best - 1];
            T = A.y; a = A.z; K = (int)A.w;
            atomicAdd(&counters[1], 1ull);
        }
        float sn, cs;
        sincospif(2.f * phase_cycles(T, K, fhi, flo), &sn, &cs);
        g[(size_t)e * N + r] = make_float2(C * a * cs, C * a * sn);
    }
}

void launch_direct_green(const float4 *exits, int N, const double *beta, double f, double c0, float2 *g,
                         unsigned long long *counters, cudaStream_t s)
{
    float fhi = (float)f, flo = (float)(f - (double)fhi);
    float C = (float)(1.0 / sqrt(8.0 * 3.14159265358979323846 * (2.0 * 3.14159265358979323846 * f) / c0));
    size_t smem = (size_t)(N - 1) * (sizeof(float4) + sizeof(double) + sizeof(float)) +
                  (size_t)N * (sizeof(double) + sizeof(float) + sizeof(int));   // <= 180 KB at N = 4095
    if (smem > 48 * 1024) cudaFuncSetAttribute(k_direct_green, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_direct_green<<<N, 512, smem, s>>>(exits, N, beta, fhi, flo, C, g, counters);
}

// ---------------------------------------------------------------- ray linking

// Linked rays of the direct term (Sec. 4.4, Sec. 6.3.2), in two kernels.
//
// Linking, step 1, one block per transducer: the first bracketing pair of fan rays of every
// receiver (as in k_direct_green), or the nearest fan ray where none brackets it, kept in the
// unused first slot of linked[e][r] as j (> 0) or -j; the diagonal is zeroed.
__global__ void k_link_brackets(const float4 *__restrict__ exits, int N, const double *__restrict__ beta,
                                float4 *__restrict__ linked)
{
    extern __shared__ float4 ex_s[];
    float *th = reinterpret_cast<float *>(ex_s);
    float *relt = th + (N - 1);
    int *first = reinterpret_cast<int *>(relt + N);
    const int e = blockIdx.x;
    const double step = 6.283185307179586476925 / N, be = xducer_angle(e, N, step, beta);
    for (int q = threadIdx.x; q < N - 1; q += blockDim.x)
        th[q] = (float)wrap_turn((double)exits[(size_t)e * (N - 1) + q].x - be);
    for (int m = threadIdx.x; m < N; m += blockDim.x) relt[m] = (float)recv_rel_m(m, e, N, step, beta, be);
    __syncthreads();
    first_brackets(th, relt, N, e, first);
    for (int r = threadIdx.x; r < N; r += blockDim.x) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r != e) {
            int code = first[r];
            if (code == INT_MAX) {
                const float t = relt[(r - e + N) % N];
                int best = 1;
                float bd = 1e30f;
                for (int j = 1; j <= N - 1; j++) {
                    float d = fabsf(th[j - 1] - t);
                    if (d < bd) { bd = d; best = j; }
                }
                code = -best;
            }
            v.x = __int_as_float(code);
        }
        linked[(size_t)e * N + r] = v;
    }
}

// Linking, step 2. A warp takes `chunk` consecutive receiver offsets m = r - e of one transducer, a
// block's four warps the same offsets of four neighbouring ones, so their rays, rotated by one
// ring step, share L1 lines. From the bracketing fan rays a secant on the initial
// angle, kept inside the bracket (regula falsi with the Illinois weighting), stops when the
// exit lies within tol radians of beta_r (at most maxit new rays); T and a are then
// interpolated in exit angle between the two bracketing rays to beta_r exactly, K taken from
// the nearer; linked[e][r] = (0, T, a, K) serves every frequency of the trace. Unbracketed
// receivers take the nearest fan ray; those and the pairs that stopped on maxit are counted
// in counters[1].
//
// A lane whose pair is linked takes the warp's next pair at once, and every lane's ray advances one
// step per turn of the loop, whatever ray of whatever pair it is: rays of a warp differ in
// length and pairs in their number of rays, and with one pair per lane half of the lanes waited
// (16.5 of 32 at work). What happens between rays is in FP64, which is slow here, so it waits until
// `wait` lanes need it; the secant's state lies in shared memory meanwhile. A warp with one pair
// per lane (small rings) waits for all.
// Linking alone, trace excluded: 256 transducers (288 x 288) 4.15 -> 2.19 ms, 512 (256 x 256, lossy)
// 3.8 -> 2.6, 1024 (192 x 192) 9.05 -> 7.27; eight steps between looks at the other lanes (3.0 ms at
// 512 with a look at every step).
// The step is k_trace_raster's; the initial direction is formed in double so that the secant is not
// limited by FP32 rounding of the angle.
template <bool LOSSY, bool RAW>
__global__ __launch_bounds__(128, 4) void k_link_rays(const float *__restrict__ F, RayParams p,
                                                   const float4 *__restrict__ exits, int maxit, double tol, int chunk,
                                                   float4 *__restrict__ linked, unsigned long long *counters)
{
    enum { GA, GB, FA, FB, WA, WB, TA, TB, AA, AB, ND };
    __shared__ double sd[ND][128];
    __shared__ int sk[3][128];   // Ka, Kb, side
    const unsigned FULL = 0xffffffffu;
    const int N = p.N, q = threadIdx.x, lane = q & 31;
    const int e = blockIdx.x * 4 + (q >> 5);
    if (e >= N) return;
    const double PI = 3.14159265358979323846, TWO_PI = 2.0 * PI;
    const double step = TWO_PI / N, be = xducer_angle(e, N, step, p.beta);
    const float4 *ex = exits + (size_t)e * (N - 1);
    auto rel = [&](double ang) { return wrap_turn(ang - be); };
    const float xe = (float)(p.R * cos(be)), ye = (float)(p.R * sin(be));
    int next = 1 + warp_of_rank(blockIdx.y, gridDim.y) * chunk;   // the warp's next pair
    const int end = min(N, next + chunk);

    // the pair, its rays so far, and the ray on its way
    bool has = false, busy = false, reached = false;
    int m = 0, it = 0, i = 0, K = 0;
    double td = 0.0, gc = 0.0;
    float an = 0.f;
    float x = 0.f, y = 0.f, px = 0.f, py = 0.f, dpx = 0.f, dpy = 0.f;
    float dxx = 0.f, dxy = 0.f, T = 0.f, Tc = 0.f, B = 0.f, Bc = 0.f, cx = 0.f, cy = 0.f, sc1 = 0.f, Jlast = 0.f;
    Fv F1{};
    const float ds = p.ds, hds = 0.5f * p.ds, R2 = p.R * p.R;

    // the next ray of the pair, or its result when it is linked or out of rays
    auto advance = [&]() {
        const double ga = sd[GA][q], gb = sd[GB][q], fa = sd[FA][q], fb = sd[FB][q], wa = sd[WA][q], wb = sd[WB][q];
        if (fabs(fa) > tol && fabs(fb) > tol && it < maxit && wb != wa) {
            gc = (ga * wb - gb * wa) / (wb - wa);
            x = xe;
            y = ye;
            field_eval<LOSSY, RAW>(F, p, x, y, F1);
            double sn, cd;
            sincos(gc, &sn, &cd);
            px = F1.n * (float)cd; py = F1.n * (float)sn; dpx = -F1.n * (float)sn; dpy = F1.n * (float)cd;
            dxx = 0.f; dxy = 0.f; T = 0.f; Tc = 0.f; B = 0.f; Bc = 0.f;
            cx = 0.f; cy = 0.f;
            sc1 = 0.f; Jlast = 0.f;
            K = 0;
            i = 0;
            busy = true;
            return;
        }
        if (fabs(fa) > tol && fabs(fb) > tol) atomicAdd(&counters[1], 1ull);
        const double fr = (fb == fa) ? 0.0 : -fa / (fb - fa);
        const double To = sd[TA][q] + fr * (sd[TB][q] - sd[TA][q]);
        const double ao = sd[AA][q] + fr * (sd[AB][q] - sd[AA][q]);
        const int Ko = fabs(fa) <= fabs(fb) ? sk[0][q] : sk[1][q];
        linked[(size_t)e * N + (e + m) % N] = make_float4(0.f, (float)To, (float)ao, (float)Ko);
        has = false;
    };
    // the bracket after a ray (a ray that does not reach the ring ends the pair as it stands)
    auto narrow = [&]() {
        if (!reached) {
            it = maxit;
            return;
        }
        const float thc = atan2f(y, x);
        double fc = rel(thc) - td;
        if (fc > PI) fc -= TWO_PI;
        if (fc < -PI) fc += TWO_PI;
        it++;
        if ((fc > 0) == (sd[FB][q] > 0)) {
            sd[GB][q] = gc; sd[FB][q] = fc; sd[WB][q] = fc; sd[TB][q] = T; sd[AB][q] = an; sk[1][q] = K;
            if (sk[2][q] == -1) sd[WA][q] *= 0.5;
            sk[2][q] = -1;
        } else {
            sd[GA][q] = gc; sd[FA][q] = fc; sd[WA][q] = fc; sd[TA][q] = T; sd[AA][q] = an; sk[0][q] = K;
            if (sk[2][q] == 1) sd[WB][q] *= 0.5;
            sk[2][q] = 1;
        }
    };

    const int wait = chunk > 32 ? 12 : 32;
    for (;;) {
        unsigned b = __ballot_sync(FULL, busy);
        if (__popc(b) <= 32 - wait && (next < end || __any_sync(FULL, has && !busy))) {
            if (has && !busy) narrow();
            for (;;) {
                // lanes without a pair take the next ones
                const unsigned idle = __ballot_sync(FULL, !has);
                const int mine = next + __popc(idle & ((1u << lane) - 1));
                next += __popc(idle);
                if (!has && mine < end) {
                    m = mine;
                    const int r = (e + m) % N, code = __float_as_int(linked[(size_t)e * N + r].x);
                    if (code > 0) {
                        const float4 A = ex[code - 1], Bq = ex[code];
                        td = recv_rel_m(m, e, N, step, p.beta, be);
                        // every new ray starts between the two bracketing rays, so it points inward
                        // like the fan's
                        sd[GA][q] = be + PI / 2 + PI * code / N;
                        sd[GB][q] = be + PI / 2 + PI * (code + 1) / N;
                        const double fa = rel(A.x) - td, fb = rel(Bq.x) - td;
                        sd[FA][q] = sd[WA][q] = fa;
                        sd[FB][q] = sd[WB][q] = fb;
                        sd[TA][q] = A.y; sd[TB][q] = Bq.y; sd[AA][q] = A.z; sd[AB][q] = Bq.z;
                        sk[0][q] = (int)A.w; sk[1][q] = (int)Bq.w; sk[2][q] = 0;
                        it = 0;
                        has = true;
                    } else {
                        const float4 A = ex[-code - 1];
                        atomicAdd(&counters[1], 1ull);
                        linked[(size_t)e * N + r] = make_float4(0.f, (float)(double)A.y, (float)(double)A.z, (float)(int)A.w);
                    }
                }
                __syncwarp();
                if (has && !busy) advance();
                __syncwarp();
                if (next >= end || !__any_sync(FULL, !has)) break;
            }
            b = __ballot_sync(FULL, busy);
        }
        if (!b) break;
        if (busy) {
            int k = 0;   // eight steps between looks at the other lanes (all, where the warp waits for all)
            do {
                const float n = F1.n, in = rcp_ap(n);
                const float sc = n * rsqrtf(px * px + py * py);
                px *= sc; py *= sc;
                const float qx = px * in, qy = py * in;
                Fv F2;
                Cell<LOSSY, RAW> cell;   // one cell for both points, as in k_trace_raster
                {
                    const float ax = x + ds * qx, ay = y + ds * qy;
                    const float u = (ax - p.x0) * p.inv_dx, v = (ay - p.y0) * p.inv_dx;
                    cell_load<LOSSY, RAW>(F, p, u, v, cell);
                    cell_eval<LOSSY, RAW>(cell, u - cell.i, v - cell.j, F2);
                }
                const float na = F2.n, ina = rcp_ap(na);
                float pax = px + ds * F1.gx, pay = py + ds * F1.gy;
                const float sca = na * rsqrtf(pax * pax + pay * pay);
                pax *= sca; pay *= sca;
                const float qax = pax * ina, qay = pay * ina;
                const float sx = qx + qax, sy = qy + qay, rs = rsqrtf(sx * sx + sy * sy);
                const float dirx = sx * rs, diry = sy * rs;
                const float ddpx = hds * (F1.gx + F2.gx), ddpy = hds * (F1.gy + F2.gy);
                const float gd = F1.gx * dxx + F1.gy * dxy, pd = px * dpx + py * dpy;
                const float qdxx = in * (dpx - px * gd * in), qdxy = in * (dpy - py * gd * in);
                const float w1 = in * (pd * in - gd);
                const float qdpx = F1.hxx * dxx + F1.hxy * dxy + F1.gx * w1;
                const float qdpy = F1.hxy * dxx + F1.hyy * dxy + F1.gy * w1;
                const float dpax = dpx + ds * qdpx, dpay = dpy + ds * qdpy;
                const float dxax = dxx + ds * qdxx, dxay = dxy + ds * qdxy;
                const float gda = F2.gx * dxax + F2.gy * dxay, pda = pax * dpax + pay * dpay;
                const float qdxax = ina * (dpax - pax * gda * ina), qdxay = ina * (dpay - pay * gda * ina);
                const float w2 = ina * (pda * ina - gda);
                const float qdpax = F2.hxx * dxax + F2.hxy * dxay + F2.gx * w2;
                const float qdpay = F2.hxy * dxax + F2.hyy * dxay + F2.gy * w2;
                const float ddxx = hds * (qdxx + qdxax), ddxy = hds * (qdxy + qdxay);
                const float ddpx2 = hds * (qdpx + qdpax), ddpy2 = hds * (qdpy + qdpay);
                const float xn = x + ds * dirx, yn = y + ds * diry;
                Fv Fn;
                {
                    const float u = (xn - p.x0) * p.inv_dx, v = (yn - p.y0) * p.inv_dx;
                    float tx = u - cell.i, ty = v - cell.j;
                    if (!(tx >= 0.f && tx < 1.f && ty >= 0.f && ty < 1.f)) {
                        cell_load<LOSSY, RAW>(F, p, u, v, cell);
                        tx = u - cell.i; ty = v - cell.j;
                    }
                    cell_eval<LOSSY, RAW>(cell, tx, ty, Fn);
                }
                float inc = hds * (F1.nr + Fn.nr), incB = LOSSY ? hds * (F1.al + Fn.al) : 0.f;
                const bool last = xn * xn + yn * yn >= R2;
                if (last) {
                    // as in k_trace_raster: a first step starts on the ring (|x|^2 - R^2 = 0)
                    float b = x * dirx + y * diry, cc = i == 0 ? 0.f : __fsub_rn(__fmaf_rn(y, y, __fmul_rn(x, x)), R2);
                    float disc = b * b - cc;
                    float t = -b + sqrtf(disc > 0.f ? disc : 0.f);
                    t = fminf(fmaxf(t, 0.f), ds);
                    float fr = t / ds;
                    x = x + t * dirx; y = y + t * diry;
                    inc *= fr;
                    incB *= fr;
                    dxx += fr * ddxx; dxy += fr * ddxy;
                    dpx += fr * ddpx2; dpy += fr * ddpy2;
                    px += fr * ddpx; py += fr * ddpy;
                    field_eval<LOSSY, RAW>(F, p, x, y, Fn);
                } else {
                    kadd(x, cx, ds * dirx); kadd(y, cy, ds * diry);
                    px += ddpx; py += ddpy;
                    dxx += ddxx; dxy += ddxy;
                    dpx += ddpx2; dpy += ddpy2;
                }
                kadd(T, Tc, inc);
                if (LOSSY) kadd(B, Bc, incB);
                F1 = Fn;
                const float rp = rsqrtf(px * px + py * py), tx = px * rp, ty = py * rp;
                const float J = dxx * ty - dxy * tx;
                if (i == 0) { sc1 = sqrtf(F1.nr * fabsf(J) / ds); Jlast = J; }
                else if (J * Jlast < 0.f) K++;
                if (J != 0.f) Jlast = J;
                if (last) {
                    an = sc1 * rsqrtf(F1.nr * fabsf(J)) * (LOSSY ? expf(-B) : 1.f);
                    reached = true;
                    busy = false;
                } else if (++i == p.maxs) {
                    reached = false;
                    busy = false;
                }
            } while (busy && (wait == 32 || ++k < 8));
        }
        __syncwarp();
    }
}

// g[e][r] = C a exp(i 2 pi (f T - K/4 + 1/8)) from the linked rays' (-, T, a, K); 0 on the diagonal
__global__ void k_green_linked(const float4 *__restrict__ linked, int N, float fhi, float flo, float C,
                               float2 *__restrict__ g)
{
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= (size_t)N * N) return;
    const float4 v = linked[i];
    if (i / N == i % N) { g[i] = make_float2(0.f, 0.f); return; }
    float sn, cs;
    sincospif(2.f * phase_cycles(v.y, (int)v.w, fhi, flo), &sn, &cs);
    g[i] = make_float2(C * v.z * cs, C * v.z * sn);
}

void launch_green_linked(const float4 *linked, int N, double f, double c0, float2 *g, cudaStream_t s)
{
    float fhi = (float)f, flo = (float)(f - (double)fhi);
    float C = (float)(1.0 / sqrt(8.0 * 3.14159265358979323846 * (2.0 * 3.14159265358979323846 * f) / c0));
    const size_t n = (size_t)N * N;
    k_green_linked<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(linked, N, fhi, flo, C, g);
}

void launch_link_rays(const float *fields, const RayParams &p, const float4 *exits, int maxit, float4 *linked,
                      unsigned long long *counters, bool lossy, bool raw, cudaStream_t s)
{
    const size_t smem = (size_t)(p.N - 1) * sizeof(float) + (size_t)p.N * (sizeof(float) + sizeof(int));   // <= 49 KB
    if (smem > 48 * 1024) cudaFuncSetAttribute(k_link_brackets, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_link_brackets<<<p.N, 256, smem, s>>>(exits, p.N, p.beta, linked);
    const double tol = 1e-6;
    // two sets of warps for the GPU (152 SMs x 16), at least a pair and at most eight pairs per lane
    int chunk = (int)((size_t)p.N * (p.N - 1) / (2 * 152 * 16) + 31) / 32 * 32;
    chunk = chunk < 32 ? 32 : (chunk > 256 ? 256 : chunk);
    const dim3 grd((p.N + 3) / 4, (p.N - 1 + chunk - 1) / chunk);
    if (lossy && raw)
        k_link_rays<true, true><<<grd, 128, 0, s>>>(fields, p, exits, maxit, tol, chunk, linked, counters);
    else if (lossy)
        k_link_rays<true, false><<<grd, 128, 0, s>>>(fields, p, exits, maxit, tol, chunk, linked, counters);
    else if (raw)
        k_link_rays<false, true><<<grd, 128, 0, s>>>(fields, p, exits, maxit, tol, chunk, linked, counters);
    else
        k_link_rays<false, false><<<grd, 128, 0, s>>>(fields, p, exits, maxit, tol, chunk, linked, counters);
}

}  // namespace rbx
