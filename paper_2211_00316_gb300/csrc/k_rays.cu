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
// lockstep; a block's four warps take the same rays of four neighbouring transducers. At
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

// The state of a reference ray (x, p) and its paraxial ray (dx, dp), T = int n ds and, lossy
// media, B = int alpha ds by the same rule; F: the fields at x.
// cx, cy, Tc, Bc are compensation terms: position and T are sums of ~10^3 small steps. In the Heun
// steps the momentum, renormalised to n(x) at every step, and the paraxial ray, which only sets
// the amplitude, take plain sums: compensated too, the tables met the same parity bars against
// the FP64 oracle (T 1e-9 s, a 1e-5) and the trace took 1.6 % longer.
struct RayState {
    float x, y, cx, cy, px, py, dxx, dxy, dpx, dpy, T, Tc, B, Bc;
    Fv F;
};

// One step of Heun's method (Alg. 1) with the paraxial system of Eq. ray-equation-paraxial;
// returns true when the step ended on the ring (the final partial step).
// Both stages' directions p / n are unit vectors, so the auxiliary point x + ds q and the new
// sample are known before any field is read there; they lie within ds times half the step's
// bend of each other (about 1e-4 cells), so one cell's nodes serve both but where a grid line runs
// between them, and then the new sample's own cell is read.
template <bool LOSSY, bool RAW>
__device__ __forceinline__ bool heun_step(const float *__restrict__ F, const RayParams &p, RayState &s, bool first)
{
    const float ds = p.ds, hds = 0.5f * p.ds, R2 = p.R * p.R;
    const float n = s.F.n, in = rcp_ap(n);
    // stage 1 at x: normalise p to n(x), q_x = p/n, q_p = grad n
    const float r1 = rsqrtf(s.px * s.px + s.py * s.py), qx = s.px * r1, qy = s.py * r1;
    s.px = qx * n;
    s.py = qy * n;
    // stage 2 at the auxiliary point x + ds q_x, the direction of p + ds grad n
    float qax = s.px + ds * s.F.gx, qay = s.py + ds * s.F.gy;
    const float ra = rsqrtf(qax * qax + qay * qay);
    qax *= ra;
    qay *= ra;
    const float sx = qx + qax, sy = qy + qay, rs = rsqrtf(sx * sx + sy * sy);
    const float dirx = sx * rs, diry = sy * rs;
    const float xn = s.x + ds * dirx, yn = s.y + ds * diry;
    const float ua = (s.x + ds * qx - p.x0) * p.inv_dx, va = (s.y + ds * qy - p.y0) * p.inv_dx;
    const float un = (xn - p.x0) * p.inv_dx, vn = (yn - p.y0) * p.inv_dx;
    Fv F2, Fn;   // fields at the auxiliary point and at the new sample
    {
        Cell<LOSSY, RAW> c;
        cell_load<LOSSY, RAW>(F, p, ua, va, c);
        cell_eval<LOSSY, RAW>(c, ua - c.i, va - c.j, F2);
        const float tx = un - c.i, ty = vn - c.j;
        cell_eval<LOSSY, RAW>(c, tx, ty, Fn);
        if (!(tx >= 0.f && tx < 1.f && ty >= 0.f && ty < 1.f)) {
            cell_load<LOSSY, RAW>(F, p, un, vn, c);
            cell_eval<LOSSY, RAW>(c, un - c.i, vn - c.j, Fn);
        }
    }
    const float ina = rcp_ap(F2.n);
    const float ddpx = hds * (s.F.gx + F2.gx), ddpy = hds * (s.F.gy + F2.gy);
    // paraxial system, both stages at the reference ray's stage values:
    // q_dx = (dp - p (g.dx)/n)/n, q_dp = H dx + g ((p.dp)/n - g.dx)/n
    const float gd = s.F.gx * s.dxx + s.F.gy * s.dxy, qd = qx * s.dpx + qy * s.dpy;
    const float qdxx = in * (s.dpx - qx * gd), qdxy = in * (s.dpy - qy * gd);
    const float w1 = in * (qd - gd);
    const float qdpx = s.F.hxx * s.dxx + s.F.hxy * s.dxy + s.F.gx * w1;
    const float qdpy = s.F.hxy * s.dxx + s.F.hyy * s.dxy + s.F.gy * w1;
    const float dpax = s.dpx + ds * qdpx, dpay = s.dpy + ds * qdpy;
    const float dxax = s.dxx + ds * qdxx, dxay = s.dxy + ds * qdxy;
    const float gda = F2.gx * dxax + F2.gy * dxay, qda = qax * dpax + qay * dpay;
    const float qdxax = ina * (dpax - qax * gda), qdxay = ina * (dpay - qay * gda);
    const float w2 = ina * (qda - gda);
    const float qdpax = F2.hxx * dxax + F2.hxy * dxay + F2.gx * w2;
    const float qdpay = F2.hxy * dxax + F2.hyy * dxay + F2.gy * w2;
    const float ddxx = hds * (qdxx + qdxax), ddxy = hds * (qdxy + qdxay);
    const float ddpx2 = hds * (qdpx + qdpax), ddpy2 = hds * (qdpy + qdpay);
    float inc = hds * (s.F.nr + Fn.nr), incB = LOSSY ? hds * (s.F.al + Fn.al) : 0.f;   // trapezoid rule
    const bool last = xn * xn + yn * yn >= R2;
    if (last) {
        // final partial step: crossing of the step's chord with the ring; the other
        // quantities interpolated linearly along the chord. A first step starts at the
        // transducer, on the ring: |x|^2 - R^2 is 0 there, and its FP32 rounding residue
        // (~R ulp(R)) would swamp b^2 for the near-tangent rays that end within a step
        const float b = s.x * dirx + s.y * diry, cc = first ? 0.f : s.x * s.x + s.y * s.y - R2;
        const float disc = b * b - cc;
        float t = -b + sqrtf(disc > 0.f ? disc : 0.f);
        t = fminf(fmaxf(t, 0.f), ds);
        const float fr = t / ds;
        s.x = s.x + t * dirx; s.y = s.y + t * diry;
        inc *= fr;
        incB *= fr;
        s.dxx += fr * ddxx; s.dxy += fr * ddxy;
        s.dpx += fr * ddpx2; s.dpy += fr * ddpy2;
        s.px += fr * ddpx; s.py += fr * ddpy;
        field_eval<LOSSY, RAW>(F, p, s.x, s.y, Fn);
    } else {
        kadd(s.x, s.cx, ds * dirx); kadd(s.y, s.cy, ds * diry);
        s.px += ddpx; s.py += ddpy;
        s.dxx += ddxx; s.dxy += ddxy;
        s.dpx += ddpx2; s.dpy += ddpy2;
    }
    kadd(s.T, s.Tc, inc);
    if (LOSSY) kadd(s.B, s.Bc, incB);
    s.F = Fn;
    return last;
}

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
// quad holds 0.3 to 1.1 nodes.
// Folded quads and slivers (near a caustic) take the two-triangle test, the smaller key winning.
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
            use1 = (e3 > 0.f) == (ar1 > 0.f) && e3 != 0.f;
            const float mx = use1 ? P01.x : P10.x, my = use1 ? P01.y : P10.y;
            x1 = __fmaf_rn(P11.x - mx, py - my, -__fmul_rn(P11.y - my, px - mx));
            x2 = __fmaf_rn(mx - P00.x, py - P00.y, -__fmul_rn(my - P00.y, px - P00.x));
            hit = use1 != (ar1 > 0.f) ? fminf(x1, x2) >= 0.f : fmaxf(x1, x2) <= 0.f;
            fx += (float)lpr;
            wrap();
            more = fy <= fy1;
        }
        __syncwarp();
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        float2 u = make_float2(0.f, 0.f);
        const float sum = (x1 - e3) + x2;
        hit = hit && sum != 0.f;
        if (hit) {
            const int4 ro = rows[(int)hy];
            const int ix = (int)hx;
            hit = ix >= ro.y && ix <= ro.z;
            // barycentric weights of M and P11; in both triangles -e3 / sum and x2 / sum
            const float inv = rcp_nr(sum), wm = -e3 * inv, wc = x2 * inv, wa = 1.f - wm - wc;
            const float mT = use1 ? P01.T : P10.T, ma = use1 ? P01.a : P10.a, mkx = use1 ? P01.kx : P10.kx,
                        mky = use1 ? P01.ky : P10.ky;
            const int K = max(P00.K, max(P11.K, use1 ? P01.K : P10.K));
            v.x = (tid0 + (use1 ? 1u : 0u)) << 8 | (uint32_t)min(K, 255);
            v.y = __float_as_uint(P00.T + wm * (mT - P00.T) + wc * (P11.T - P00.T));
            v.z = __float_as_uint(wa * P00.a + wm * ma + wc * P11.a);
            v.w = __float_as_uint(wa * P00.kx + wm * mkx + wc * P11.kx);
            u = make_float2(wa * P00.ky + wm * mky + wc * P11.ky, __int_as_float(ro.x + ix - ro.y));
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
                const float px = p.x0 + fx * p.dx, py = p.y0 + fy * p.dx;
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
                if (k0 != ~0ull || k1 != ~0ull) {
                    const bool use0 = k0 < k1;
                    const float lb = use0 ? lb0 : lb1, lc = use0 ? lc0 : lc1, la = 1.f - lb - lc;
                    const float Ba = use0 ? P10.a : P11.a, Ca = use0 ? P11.a : P01.a;
                    const float Bkx = use0 ? P10.kx : P11.kx, Ckx = use0 ? P11.kx : P01.kx;
                    const float Bky = use0 ? P10.ky : P11.ky, Cky = use0 ? P11.ky : P01.ky;
                    const unsigned long long key = use0 ? k0 : k1;
                    v = make_uint4((uint32_t)key, (uint32_t)(key >> 32), __float_as_uint(la * P00.a + lb * Ba + lc * Ca),
                                   __float_as_uint(la * P00.kx + lb * Bkx + lc * Ckx));
                    u = make_float2(la * P00.ky + lb * Bky + lc * Cky, __int_as_float(ro.x + ix - ro.y));
                    hit = true;
                }
            }
            fx += (float)lpr;
            wrap();
            more = fy <= fy1;
        }
        push_hits(hit, v, u, fan, hq, counters);
    }
}

// Warps per block, each tracing the same rays of a neighbouring transducer; 20 warps per SM.
constexpr int kFansPerBlock = 4;

// The per-warp hit queues of a block (shared memory).
struct BlockQueues {
    uint4 v[kFansPerBlock][64];
    float2 w[kFansPerBlock][64];
    unsigned cov[kFansPerBlock];
};

// Rays of a warp and warps of a fan: `lpr` lanes per ray (a power of two up to 16) carry the same
// ray and share the rasterisation of its tube; neighbouring warps of a fan share a ray.
__host__ __device__ __forceinline__ int warp_rays(int lpr) { return 32 / lpr; }
__host__ __device__ __forceinline__ int fan_warps(int N, int lpr) { return (N - 2 + 32 / lpr - 2) / (32 / lpr - 1); }

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
    // the warps of a block trace the same rays of neighbouring transducers: rotated by one
    // ring step, those rays stay within about a cell of one another, so their field gathers
    // share L1 lines
    const int e = eblk * kFansPerBlock + wib;
    const int N = p.N, lpr = p.lpr, nr = warp_rays(lpr);
    if (e >= N) return;                        // whole warp leaves together
    const int ray = lane / lpr, sub = lane - ray * lpr;
    const int j = 1 + (nr - 1) * warp + ray;   // this lane's ray
    const bool has_ray = j <= N - 1;
    const bool writes_exit = sub == 0 && (ray < nr - 1 || j == N - 1);   // one warp of the two that trace a shared ray
    TabEntry *fan = tab + (size_t)e * p.X;
    const float ds = p.ds, hds = 0.5f * p.ds, inv_dx = p.inv_dx, R2 = p.R * p.R;
    HitQueue hq{bq.v[wib], bq.w[wib], &bq.cov[wib], 0};

    const double be = p.beta ? p.beta[e] : 2.0 * 3.14159265358979323846 * e / N;
    const float gam0 = (float)(be + 3.14159265358979323846 / 2 + 3.14159265358979323846 * j / N);
    RayState s{};
    s.x = (float)(p.R * cos(be));
    s.y = (float)(p.R * sin(be));
    field_eval<LOSSY, RAW>(F, p, s.x, s.y, s.F);
    float cdx = 0.f, cdy = 0.f;   // compensation terms of the paraxial ray's closed-form steps

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
        s.px = s.F.n * c0; s.py = s.F.n * s0;
        s.dpx = -s.F.n * s0; s.dpy = s.F.n * c0;
        if (has_ray && R2 > rho2) {
            const float b = s.x * c0 + s.y * s0, disc = b * b - (fmaf(s.x, s.x, s.y * s.y) - rho2);
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
        const bool have = alive;
        if (alive) {
            bool last = false;
            if (i < kin) {
                // the step in a uniform medium: straight, p constant, dx += ds dp / n
                const float in = rcp_nr(s.F.n);
                const float rp = rsqrtf(s.px * s.px + s.py * s.py), tx = s.px * rp, ty = s.py * rp;
                kadd(s.x, s.cx, ds * tx); kadd(s.y, s.cy, ds * ty);
                kadd(s.dxx, cdx, ds * (s.dpx * in)); kadd(s.dxy, cdy, ds * (s.dpy * in));
                kadd(s.T, s.Tc, hds * (s.F.nr + s.F.nr));
                if (LOSSY) kadd(s.B, s.Bc, hds * (s.F.al + s.F.al));
            } else {
                last = heun_step<LOSSY, RAW>(F, p, s, i == 0);
            }
            const float rp = rsqrtf(s.px * s.px + s.py * s.py), tx = s.px * rp, ty = s.py * rp;
            const float J = s.dxx * ty - s.dxy * tx;
            if (i == 0) { sc1 = sqrtf(s.F.nr * fabsf(J) / ds); Jlast = J; }
            else if (J * Jlast < 0.f) K++;   // caustic: sign change of the ray Jacobian
            if (J != 0.f) Jlast = J;
            cur.x = s.x; cur.y = s.y; cur.T = s.T; cur.kx = tx; cur.ky = ty; cur.K = K;
            cur.a = sc1 * rsqrtf(s.F.nr * fabsf(J));
            if (LOSSY) cur.a *= expf(-s.B);
            if (last) {
                alive = false;
                if (writes_exit)
                    exits[(size_t)e * (N - 1) + (j - 1)] = make_float4(atan2f(s.y, s.x), s.T, cur.a, (float)K);
            }
        }
        // neighbour ray j+1 (lpr lanes on): its sample i+1
        Vtx ncur;
        ncur.x = __shfl_down_sync(FULL, cur.x, lpr);
        ncur.y = __shfl_down_sync(FULL, cur.y, lpr);
        ncur.T = __shfl_down_sync(FULL, cur.T, lpr);
        ncur.a = __shfl_down_sync(FULL, cur.a, lpr);
        ncur.kx = __shfl_down_sync(FULL, cur.kx, lpr);
        ncur.ky = __shfl_down_sync(FULL, cur.ky, lpr);
        ncur.K = __shfl_down_sync(FULL, cur.K, lpr);
        const bool nhave = __shfl_down_sync(FULL, (int)have, lpr) != 0;
        const bool valid = i >= 1 && i >= i0 && have && nhave && ray < nr - 1 && j + 1 <= N - 1;
        // A quad beyond a line two cells outside the mask holds no mask node, in any medium:
        // the edge functions accept only points of its two triangles, which lie in the convex
        // hull of its corners, so when every corner q has u.q > rm for u the direction of the
        // corners' sum, so does every accepted point, and |q| > rm. The warp skips the step's
        // rasterisation when that holds for all its quads. The corners' own radii beyond rm
        // are necessary for it and cheap, so the line test runs only when they hold for the
        // whole warp (radii alone would not do: the cross edge of a wide tube can be a chord
        // through the mask).
        const bool ob = fmaf(cur.x, cur.x, cur.y * cur.y) > rm2 && fmaf(prev.x, prev.x, prev.y * prev.y) > rm2;
        const bool nb = __shfl_down_sync(FULL, (int)ob, lpr) != 0;
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
            raster_quad_warp(valid, prev, cur, nprev, ncur, ((uint32_t)j << 11 | (uint32_t)i) << 1, p, inv_dx, sub, lpr,
                             rows, fan, hq, counters);
        prev = cur;
        nprev = ncur;
        // Leaving through the uniform water: once a ray is beyond rho, moving outward, and so
        // are (or have ended) the rays it forms quads with in this warp, no later quad of it
        // can hold a mask node, and it goes straight to the ring in closed form (the chord's
        // crossing as in the last step above; J is linear in s there, so at most one caustic).
        {
            const bool out = alive && i >= kin && fmaf(s.x, s.x, s.y * s.y) > rho2 && fmaf(s.x, s.px, s.y * s.py) > 0.f;
            if (__any_sync(FULL, out)) {
                const bool okself = !alive || out;
                bool okL = __shfl_up_sync(FULL, okself, lpr), okR = __shfl_down_sync(FULL, okself, lpr);
                const bool aL = __shfl_up_sync(FULL, alive, lpr), aR = __shfl_down_sync(FULL, alive, lpr);
                const float xl = __shfl_up_sync(FULL, s.x, lpr), yl = __shfl_up_sync(FULL, s.y, lpr);
                const float xr = __shfl_down_sync(FULL, s.x, lpr), yr = __shfl_down_sync(FULL, s.y, lpr);
                const float gap = rho - p.rmask, gap2 = gap * gap;
                if (ray == 0) okL = true;
                else if (aL) okL = okL && (s.x - xl) * (s.x - xl) + (s.y - yl) * (s.y - yl) < gap2;
                if (ray == nr - 1) okR = true;
                else if (aR) okR = okR && (s.x - xr) * (s.x - xr) + (s.y - yr) * (s.y - yr) < gap2;
                if (out && okL && okR) {
                    const float in = rcp_nr(s.F.n), inc = hds * (s.F.nr + s.F.nr);
                    const float rp = rsqrtf(s.px * s.px + s.py * s.py), tx = s.px * rp, ty = s.py * rp;
                    const float b = s.x * tx + s.y * ty, se = -b + sqrtf(fmaxf(b * b - (fmaf(s.x, s.x, s.y * s.y) - R2), 0.f));
                    const int m = max(0, (int)floorf(se / ds));
                    const float sm = (float)m * ds;
                    const float xm = fmaf(sm, tx, s.x), ym = fmaf(sm, ty, s.y);
                    const float b2 = xm * tx + ym * ty, disc = b2 * b2 - (fmaf(xm, xm, ym * ym) - R2);
                    float t = -b2 + sqrtf(disc > 0.f ? disc : 0.f);
                    t = fminf(fmaxf(t, 0.f), ds);
                    s.x = fmaf(t, tx, xm); s.y = fmaf(t, ty, ym);
                    kadd(s.T, s.Tc, (float)m * inc);
                    kadd(s.T, s.Tc, (t / ds) * inc);
                    if (LOSSY) {
                        const float incB = hds * (s.F.al + s.F.al);
                        kadd(s.B, s.Bc, (float)m * incB);
                        kadd(s.B, s.Bc, (t / ds) * incB);
                    }
                    s.dxx = fmaf(sm + t, s.dpx * in, s.dxx); s.dxy = fmaf(sm + t, s.dpy * in, s.dxy);
                    field_eval<LOSSY, RAW>(F, p, s.x, s.y, s.F);
                    const float J = s.dxx * ty - s.dxy * tx;
                    if (J * Jlast < 0.f) K++;
                    const float a = sc1 * rsqrtf(s.F.nr * fabsf(J)) * (LOSSY ? expf(-s.B) : 1.f);
                    if (writes_exit)
                        exits[(size_t)e * (N - 1) + (j - 1)] = make_float4(atan2f(s.y, s.x), s.T, a, (float)K);
                    alive = false;
                }
            }
        }
        if (!__any_sync(FULL, alive)) break;
        if (i == p.maxs - 1 && alive && sub == 0) atomicAdd(&counters[2], 1ull);   // ray never reached the ring
    }
    // drain the rest of the queue; the covered-entry count goes to counters[0]
    count_first(hq, lane < hq.n && drain_one(hq, lane, fan, counters));
    __syncwarp();
    if (lane == 0 && *hq.cov) atomicAdd(&counters[0], (unsigned long long)*hq.cov);
}

template <bool LOSSY, bool RAW>
__global__ __launch_bounds__(32 * kFansPerBlock, 20 / kFansPerBlock) void k_trace_raster(const float *__restrict__ F, const int4 *__restrict__ rows_g,
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

void launch_trace_raster(const float *fields, const int4 *rows, TabEntry *tab, float4 *exits, const RayParams &p,
                         unsigned long long *counters, bool lossy, bool raw, cudaStream_t s)
{
    // the longest warps of every fan first: the blocks that start last, and those that share
    // an SM when the grid is a single wave, then differ least (256 transducers, 576 blocks in
    // one wave: the busiest scheduler issued 2.3 times the mean before, 1.4 times now)
    dim3 grd((p.N + kFansPerBlock - 1) / kFansPerBlock, fan_warps(p.N, p.lpr));
    const size_t sm = (size_t)p.ny * sizeof(int4);
    if (lossy && raw)
        k_trace_raster<true, true><<<grd, 32 * kFansPerBlock, sm, s>>>(fields, rows, tab, exits, p, counters);
    else if (lossy)
        k_trace_raster<true, false><<<grd, 32 * kFansPerBlock, sm, s>>>(fields, rows, tab, exits, p, counters);
    else if (raw)
        k_trace_raster<false, true><<<grd, 32 * kFansPerBlock, sm, s>>>(fields, rows, tab, exits, p, counters);
    else
        k_trace_raster<false, false><<<grd, 32 * kFansPerBlock, sm, s>>>(fields, rows, tab, exits, p, counters);
}

int trace_lanes_per_ray(int N)
{
    int lpr = 1;
    while (lpr < 8 && (size_t)N * fan_warps(N, 2 * lpr) <= 3040) lpr *= 2;
    return lpr;
}

int trace_items(int N, int *nwarps)
{
    const int nw = fan_warps(N, 1);
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

// Angular density of every entry (the back-projection's tensor-core operand synthesis forms
// the same values itself, from the same expression, and does not need this array).
__global__ void k_dgamma(const TabEntry *__restrict__ tab, float *__restrict__ dg, int N, int X)
{
    size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= (size_t)N * X) return;
    int e = (int)(i / X), k = (int)(i % X);
    const TabEntry &tp = tab[(size_t)((e + 1) % N) * X + k];
    const TabEntry &tm = tab[(size_t)((e + N - 1) % N) * X + k];
    dg[i] = (tp.idk == kUncovered || tm.idk == kUncovered) ? 0.f : dgamma_of(tp.gam, tm.gam);
}

void launch_dgamma(const TabEntry *tab, float *dg, int N, int X, cudaStream_t s)
{
    size_t n = (size_t)N * X;
    k_dgamma<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(tab, dg, N, X);
}

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

// One ray from (x, y) to the ring by one thread: the step of k_trace_raster without its
// rasterisation and straight-line shortcuts. The initial direction is formed in double so that a secant
// iteration on it is not limited by FP32 rounding of the angle. Returns false when the ray
// does not reach the ring within p.maxs steps.
template <bool LOSSY, bool RAW>
__device__ bool trace_one(const float *__restrict__ F, const RayParams &p, float x, float y, double gam0,
                          float &theta, float &Tout, float &aout, int &Kout)
{
    RayState s{};
    s.x = x;
    s.y = y;
    field_eval<LOSSY, RAW>(F, p, x, y, s.F);
    double sd, cd;
    sincos(gam0, &sd, &cd);
    s.px = s.F.n * (float)cd; s.py = s.F.n * (float)sd;
    s.dpx = -s.F.n * (float)sd; s.dpy = s.F.n * (float)cd;
    float sc1 = 0.f, Jlast = 0.f;
    int K = 0;
    for (int i = 0; i < p.maxs; i++) {
        const bool last = heun_step<LOSSY, RAW>(F, p, s, i == 0);
        const float rp = rsqrtf(s.px * s.px + s.py * s.py), tx = s.px * rp, ty = s.py * rp;
        const float J = s.dxx * ty - s.dxy * tx;
        if (i == 0) { sc1 = sqrtf(s.F.nr * fabsf(J) / p.ds); Jlast = J; }
        else if (J * Jlast < 0.f) K++;
        if (J != 0.f) Jlast = J;
        if (last) {
            theta = atan2f(s.y, s.x);
            Tout = s.T;
            aout = sc1 * rsqrtf(s.F.nr * fabsf(J)) * (LOSSY ? expf(-s.B) : 1.f);
            Kout = K;
            return true;
        }
    }
    return false;
}

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

// Linking, step 2, one thread per (transducer, receiver) pair; a block's four warps take the
// same 32 receiver offsets m = r - e of four neighbouring transducers, so their rays, rotated
// by one ring step, share L1 lines. From the bracketing fan rays a secant on the initial
// angle, kept inside the bracket (regula falsi with the Illinois weighting), stops when the
// exit lies within tol radians of beta_r (at most maxit new rays); T and a are then
// interpolated in exit angle between the two bracketing rays to beta_r exactly, K taken from
// the nearer; linked[e][r] = (0, T, a, K) serves every frequency of the trace. Unbracketed
// receivers take the nearest fan ray; those and the pairs that stopped on maxit are counted
// in counters[1].
template <bool LOSSY, bool RAW>
__global__ __launch_bounds__(128, 4) void k_link_rays(const float *__restrict__ F, RayParams p,
                                                   const float4 *__restrict__ exits, int maxit, double tol,
                                                   float4 *__restrict__ linked, unsigned long long *counters)
{
    const int N = p.N;
    const int e = blockIdx.y * 4 + (threadIdx.x >> 5), m = blockIdx.x * 32 + (threadIdx.x & 31) + 1;
    if (e >= N || m > N - 1) return;
    const int r = (e + m) % N;
    const double PI = 3.14159265358979323846, TWO_PI = 2.0 * PI;
    const double step = TWO_PI / N, be = xducer_angle(e, N, step, p.beta);
    const double td = recv_rel_m(m, e, N, step, p.beta, be);
    float4 *slot = linked + (size_t)e * N + r;
    const int code = __float_as_int(slot->x);
    const float4 *ex = exits + (size_t)e * (N - 1);
    auto rel = [&](double ang) { return wrap_turn(ang - be); };
    double T, a;
    int K;
    if (code > 0) {
        const int found = code;
        const float xe = (float)(p.R * cos(be)), ye = (float)(p.R * sin(be));
        const float4 A = ex[found - 1], Bq = ex[found];
        // bracketing secant (regula falsi, Illinois weighting): every new ray starts between
        // the two bracketing rays, so it points inward like the fan's
        double ga = be + PI / 2 + PI * found / N, gb = be + PI / 2 + PI * (found + 1) / N;
        double fa = rel(A.x) - td, fb = rel(Bq.x) - td, wa = fa, wb = fb;
        double Ta = A.y, Tb = Bq.y, aa = A.z, ab = Bq.z;
        int Ka = (int)A.w, Kb = (int)Bq.w, it = 0, side = 0;
        while (fabs(fa) > tol && fabs(fb) > tol && it < maxit && wb != wa) {
            const double gc = (ga * wb - gb * wa) / (wb - wa);
            float thc, Tc, ac;
            int Kc;
            if (!trace_one<LOSSY, RAW>(F, p, xe, ye, gc, thc, Tc, ac, Kc)) break;
            double fc = rel(thc) - td;
            if (fc > PI) fc -= TWO_PI;
            if (fc < -PI) fc += TWO_PI;
            it++;
            if ((fc > 0) == (fb > 0)) {
                gb = gc; fb = fc; wb = fc; Tb = Tc; ab = ac; Kb = Kc;
                if (side == -1) wa *= 0.5;
                side = -1;
            } else {
                ga = gc; fa = fc; wa = fc; Ta = Tc; aa = ac; Ka = Kc;
                if (side == 1) wb *= 0.5;
                side = 1;
            }
        }
        if (fabs(fa) > tol && fabs(fb) > tol) atomicAdd(&counters[1], 1ull);
        const double fr = (fb == fa) ? 0.0 : -fa / (fb - fa);
        T = Ta + fr * (Tb - Ta);
        a = aa + fr * (ab - aa);
        K = fabs(fa) <= fabs(fb) ? Ka : Kb;
    } else {
        const float4 A = ex[-code - 1];
        T = A.y; a = A.z; K = (int)A.w;
        atomicAdd(&counters[1], 1ull);
    }
    *slot = make_float4(0.f, (float)T, (float)a, (float)K);
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
    const dim3 grd((p.N - 1 + 31) / 32, (p.N + 3) / 4);
    if (lossy && raw)
        k_link_rays<true, true><<<grd, 128, 0, s>>>(fields, p, exits, maxit, tol, linked, counters);
    else if (lossy)
        k_link_rays<true, false><<<grd, 128, 0, s>>>(fields, p, exits, maxit, tol, linked, counters);
    else if (raw)
        k_link_rays<false, true><<<grd, 128, 0, s>>>(fields, p, exits, maxit, tol, linked, counters);
    else
        k_link_rays<false, false><<<grd, 128, 0, s>>>(fields, p, exits, maxit, tol, linked, counters);
}

// ---------------------------------------------------------------- table I/O

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

__global__ void k_get_tables(const TabEntry *tab, float *T, float *a, float *gam, uint8_t *K, size_t n)
{
    size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    TabEntry t = tab[i];
    bool cov = t.idk != kUncovered;
    if (T) T[i] = cov ? t.T : 0.f;
    if (a) a[i] = cov ? t.a : 0.f;
    if (gam) gam[i] = cov ? t.gam : 0.f;
    if (K) K[i] = cov ? (uint8_t)(t.idk & 0xffu) : 0;
}

void launch_get_tables(const TabEntry *tab, float *T, float *a, float *gam, uint8_t *K, size_t n, cudaStream_t s)
{
    k_get_tables<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(tab, T, a, gam, K, n);
}

}  // namespace rbx
