// Particle functions psi_mu (Sec. 3.2, App. A): linear finite elements on the
// periodic Delaunay triangulation of the particles (2D), hat functions over
// the periodically ordered particles (1D); and particle volumes
// v_mu = int psi_mu (Sec. 2.1, Eq. part_v).
//
// 2D: the Delaunay star of a particle p comes from one of four passes.
//  * k_delaunay, one thread per particle: the star is the convex hull of the
//    particles around p after inversion about p (the manner of quickhull), found
//    with float arithmetic whose every decision is certain (see below).
//  * k_delaunay_wide, 8 lanes per particle, for what the first pass gives up:
//    the same hull with a wider search, undecided tests made exactly.
//  * k_delaunay_exact, one thread per particle, for many ties (lattices), and
//    k_delaunay_last, a warp per particle, for the rest (crowds inside a cell, jumps
//    of density, coincident particles, sets too sparse to certify, stars of more
//    than 24 neighbours, which are refused): p's Voronoi cell is clipped by the
//    bisectors of nearby particles, scanned ring by ring of mesh cells. The cell
//    is a cyclic list of
//    neighbours q_k; its vertex k is the circumcentre of (p, q_k, q_k+1). A
//    candidate s removes vertex k iff s lies strictly inside the circle
//    through (p, q_k, q_k+1): the in-circle predicate, equivalently
//    2 c_k . s > |s|^2 for the circumcentre c_k. It is decided in float from
//    c_k and a rigorous bound on its error, and exactly on the 32-bit torus
//    coordinates (128-bit integers) when the float value falls inside the error
//    margin. After ring r the cell is final once every vertex v satisfies
//    2|v| < (distance from p to the unscanned cells).
// Exact ties are broken by symbolic perturbation of the lifted coordinate
// |r|^2 + eps^rank, rank = caller index. Because every decision is exact and
// the perturbation is a property of the point set, the stars of all particles
// agree, whatever pass made them: every triangle (p, a, b) appears in the stars
// of p, a and b. Its order does not tell the pass either (start_key).
//
// Measured (16.8M clustered particles on 2048^2, all passes): 6.1 ms, against
// 17.2 ms with the clipping alone as the main pass, every lane at its own
// candidate and its own polygon. Smallest calls gain too, 262,144 particles from
// 518 to 170 us: no lane walks a long chain. Sets that the hull cannot take (clipping
// alone, a hull attempt and one thread each after it, now): 1M on a square lattice
// 427, 710, 487 us; 1M with x = u^2 2959, 4027, 2179 us; 80,000 with 20,000 inside
// a quarter of a cell 35.7, 44.9, 5.8 ms.
#include <algorithm>

#include "internal.cuh"

PM_DEBUG_DECL(delaunay)

namespace {

__device__ __forceinline__ int sgn_ll(ll v) { return (v > 0) - (v < 0); }
__device__ __forceinline__ int sgn_i128(i128 v) { return (v > 0) - (v < 0); }

// Exact "s strictly inside circle(p = 0, a, b)" for counter-clockwise (p,a,b),
// coordinates relative to p with |.| <= 2^30 (every term below 2^124).
__device__ __noinline__ bool incircle_exact(int ax, int ay, int bx, int by, int sx, int sy, int pp, int pa, int pb,
                                            int ps) {
    ll al = (ll)ax * ax + (ll)ay * ay;
    ll bl = (ll)bx * bx + (ll)by * by;
    ll sl = (ll)sx * sx + (ll)sy * sy;
    i128 t1 = (i128)by * sl - (i128)sy * bl;
    i128 t2 = (i128)bx * sl - (i128)sx * bl;
    i128 t3 = (i128)((ll)bx * sy - (ll)by * sx);
    i128 det = (i128)ax * t1 - (i128)ay * t2 + (i128)al * t3;
    if (det != 0) return det < 0;
    // Symbolic perturbation: d/d(eps_k) of the lifted 4x4 determinant is a
    // signed orientation of the other three points.
    int sg[4], pr[4] = {pp, pa, pb, ps};
    i128 oabs = (i128)((ll)bx - ax) * ((ll)sy - ay) - (i128)((ll)by - ay) * ((ll)sx - ax);
    sg[0] = sgn_i128(oabs);
    sg[1] = -sgn_ll((ll)bx * sy - (ll)by * sx);
    sg[2] = sgn_ll((ll)ax * sy - (ll)ay * sx);
    sg[3] = -sgn_ll((ll)ax * by - (ll)ay * bx);
    for (int it = 0; it < 4; ++it) {
        int best = -1;
        for (int k = 0; k < 4; ++k)
            if (pr[k] >= 0 && (best < 0 || pr[k] < pr[best])) best = k;
        if (best < 0) break;
        if (sg[best] != 0) return sg[best] > 0;
        pr[best] = -1;
    }
    return false;
}

// Star entries carry the sorted index in the low 28 bits and the image code
// in the high 4 (so real entries may be negative as ints); the four virtual
// points of the initial cell use the indices PM_VIRT..PM_VIRT+3 and rank last.
#define PM_VIRT 0x0ffffff0
__device__ __forceinline__ int prio(int enc, const int *__restrict__ perm) {
    const int id = enc & 0x0fffffff;
    return id >= PM_VIRT ? 0x7ffffff0 + (id - PM_VIRT) : __ldg(perm + id);
}

#define EBLK 64     // threads per block of the exact pass
#define EMINB 12    // resident blocks per SM (24 warps, what the polygons in shared memory leave)
#define ECAP 9      // polygon capacity of the exact pass
#define LBLK 128    // threads per block of the last pass, a warp per particle
#define LCAP 31     // polygon capacity of the last pass (vertex masks are 32 bits)
#define ST_OVERFLOW 0x40000000  // internal: the cell outgrew the exact pass's capacity

// Float circumcentre c of (0, a, b) and a bound e on the error of each of its
// components (infinite when the triangle is too flat to bound). Inputs are
// exact integers below 2^30 in magnitude; every rounding, including the
// conversion of the inputs to float, is covered by the 8u factors.
__device__ __forceinline__ void circumcentre(float ax, float ay, float bx, float by, float &cx, float &cy, float &e) {
    const float u8 = 4.8e-7f;  // 8 units of roundoff
    float al = ax * ax + ay * ay, bl = bx * bx + by * by;
    float D = 2.0f * (ax * by - ay * bx);
    float eD = 2.0f * u8 * (fabsf(ax * by) + fabsf(ay * bx));
    float Nx = by * al - ay * bl, Ny = ax * bl - bx * al;
    float eN = u8 * fmaxf(fabsf(by * al) + fabsf(ay * bl), fabsf(ax * bl) + fabsf(bx * al));
    float den = fabsf(D) - eD;
    const float iD = __frcp_rn(D);
    cx = Nx * iD;
    cy = Ny * iD;
    if (!(den > 0.0f)) {
        e = INFINITY;
        return;
    }
    float cm = fmaxf(fabsf(cx), fabsf(cy));
    // per-component bound (the reciprocal and product roundings are inside
    // the u8 term), doubled to cover the vector norm (sqrt 2) with slack
    e = 2.0f * ((eN + cm * eD) * __frcp_ru(den) + u8 * cm);
    if (!(e < INFINITY) || !(cm < INFINITY)) e = INFINITY;
}

// Polygon state of one thread, one column per thread in shared memory:
// neighbour k, q[k] = (x, y, entry) with entry = sorted index | image code <<
// 28, and vertex k, v[k] = (c_k, w_k, rr_k): the circumcentre c_k of
// (p, q_k, q_k+1), the margin w_k = e_k + 8u |c_k| (the float test
// 2 c_k . s > |s|^2 is certain outside w_k |s| + 4u |s|^2), and rr_k, an
// upper bound of (|c_k| + w_k)^2 without square roots:
// (|c| + w)^2 <= |c|^2 + 2 sqrt2 max(|cx|,|cy|) w + w^2 (infinite when the
// vertex is unbounded).
template <int NB>
struct PolyS {
    int4 (*q)[NB];
    float4 (*v)[NB];
    int t;
};

template <int NB>
__device__ __forceinline__ float set_vertex(PolyS<NB> P, int k, float ax, float ay, float bx, float by) {
    float cx, cy, e;
    circumcentre(ax, ay, bx, by, cx, cy, e);
    const float cm = fmaxf(fabsf(cx), fabsf(cy));
    float w = e + 4.8e-7f * cm * 1.5f;
    w = w < INFINITY ? w : INFINITY;
    float rr = (cx * cx + cy * cy) * 1.000001f + 2.8285f * cm * w + w * w;
    rr = rr < INFINITY ? rr : INFINITY;
    P.v[k][P.t] = make_float4(cx, cy, w, rr);
    return rr;
}

// Work of one thread, counted by the counting instantiation of the kernel:
// candidates examined, candidates passing the distance test, vertex tests,
// clips, and the sum of the cell sizes after each clip.
// Work of the cells a pass completes (a pass that gives a cell up to a larger
// capacity drops what it counted for it), and the cells given up.
struct WorkCount {
    unsigned cand = 0, tested = 0, vtests = 0, clips = 0, msum = 0, over = 0, exact = 0;
};

// Clip the cell of p by the bisector of candidate s (relative position
// (sx, sy), sorted index sidx, image code). R2 = max_k rr_k is kept up to
// date: the vertices that survive a clip are those the candidate does not
// remove, plus the two new ones. Returns an error bit or 0.
template <int CAP, int NB, bool COUNT>
__device__ __forceinline__ int clip_by(PolyS<NB> P, int &m, float &R2, int sx, int sy, int sidx, int code, int p,
                                       int &pp, const int *__restrict__ perm, WorkCount &wc) {
    const float fsx = (float)sx, fsy = (float)sy;
    const float d2 = fsx * fsx + fsy * fsy;
    if (COUNT) wc.cand++;
    if (d2 > 4.0001f * R2) return 0;  // |s| > 2 max|c|: no vertex can be cut
    if (COUNT) {
        wc.tested++;
        wc.vtests += m;
    }
    // |s| <= sqrt2 max(|sx|, |sy|) stands in for the norm in the margin
    const float hs = 0.5f * d2, ns = 1.41422f * fmaxf(fabsf(fsx), fabsf(fsy)), mr = 2.4e-7f * d2;
    // float pass: certain inside -> mask, certain outside -> nothing, else
    // undecided (exact pass below, rare)
    // rkeep: the largest radius bound among the vertices not certainly
    // removed (an upper bound of the kept ones: undecided vertices that the
    // exact pass removes only make it larger, which is safe)
    unsigned mask = 0, undecided = 0;
    float rkeep = 0.0f;
    const int t = P.t;
    if (CAP <= 12) {
        // CAP predicated iterations on every lane: no loop exit that depends
        // on the lane's own cell size (lanes of a warp hold cells of
        // different sizes). Entries past m are stale but in bounds, and are
        // masked out.
#pragma unroll
        for (int k = 0; k < CAP; ++k) {
            const bool live = k < m;
            const float4 c = P.v[k][t];
            const float hk = c.x * fsx + c.y * fsy - hs;
            const float mg = c.z * ns + mr;
            const bool in = live && hk > mg, out = hk < -mg;  // NaN: neither
            mask |= (in ? 1u : 0u) << k;
            undecided |= (live && !in && !out ? 1u : 0u) << k;
            rkeep = (in || !live) ? rkeep : fmaxf(rkeep, c.w);
        }
    } else {
#pragma unroll 4
        for (int k = 0; k < m; ++k) {
            const float4 c = P.v[k][t];
            const float hk = c.x * fsx + c.y * fsy - hs;
            const float mg = c.z * ns + mr;
            const bool in = hk > mg, out = hk < -mg;  // both false also when hk or mg is NaN
            mask |= (in ? 1u : 0u) << k;
            undecided |= (!in && !out ? 1u : 0u) << k;
            rkeep = in ? rkeep : fmaxf(rkeep, c.w);
        }
    }
    if (undecided) {
        if (COUNT) wc.exact += __popc(undecided);
        const int ps = perm[sidx];
        if (pp == -2) pp = perm[p];
        for (unsigned u = undecided; u; u &= u - 1) {
            const int k = __ffs(u) - 1;
            const int4 A = P.q[k][t], Bq = P.q[k + 1 == m ? 0 : k + 1][t];
            if (incircle_exact(A.x, A.y, Bq.x, Bq.y, sx, sy, pp, prio(A.z, perm), prio(Bq.z, perm), ps))
                mask |= 1u << k;
        }
    }
    if (mask == 0) return 0;
    const unsigned full = (1u << m) - 1u;
    const int cnt = __popc(mask);
    const unsigned prevm = ((mask << 1) | (mask >> (m - 1))) & full;
    const unsigned starts = mask & ~prevm;
    if (cnt >= m || __popc(starts) != 1) return ST_RANGE;
    const int i0 = __ffs(starts) - 1;  // first removed vertex; q_i0 is kept
    const int nd = cnt - 1;            // neighbours q_{i0+1..i0+nd} are removed
    if (m - nd + 1 > CAP) return CAP < LCAP ? ST_OVERFLOW : ST_DEGREE;
    PM_CHK(m - nd + 1 <= CAP, 204, return ST_DEGREE)
    const int4 S = make_int4(sx, sy, sidx | (code << 28), 0);
    int ipos;
    if (i0 + nd < m) {
        if (nd == 0) {
            for (int k = m; k > i0 + 1; --k) {
                P.q[k][t] = P.q[k - 1][t];
                P.v[k][t] = P.v[k - 1][t];
            }
            m += 1;
        } else if (nd > 1) {
            for (int k = i0 + 2; k + nd - 1 < m; ++k) {
                P.q[k][t] = P.q[k + nd - 1][t];
                P.v[k][t] = P.v[k + nd - 1][t];
            }
            m -= nd - 1;
        }
        P.q[i0 + 1][t] = S;
        ipos = i0 + 1;
    } else {
        const int dbeg = nd - (m - 1 - i0);
        for (int k = 0; k <= i0 - dbeg; ++k) {
            P.q[k][t] = P.q[k + dbeg][t];
            P.v[k][t] = P.v[k + dbeg][t];
        }
        m = i0 - dbeg + 1;
        P.q[m][t] = S;
        ipos = m;
        m += 1;
    }
    const int iprev = ipos == 0 ? m - 1 : ipos - 1, inext = ipos + 1 == m ? 0 : ipos + 1;
    const int4 Q = P.q[iprev][t], Nq = P.q[inext][t];
    const float r1 = set_vertex(P, iprev, (float)Q.x, (float)Q.y, fsx, fsy);
    const float r2 = set_vertex(P, ipos, fsx, fsy, (float)Nq.x, (float)Nq.y);
    R2 = fmaxf(rkeep, fmaxf(r1, r2));
    if (COUNT) {
        wc.clips++;
        wc.msum += m;
    }
    return 0;
}

// Cell (dx, dy) of the neighbourhood of cell (cx, cy): wrapped index, image offsets.
__device__ __forceinline__ int nb_cell(int cx, int cy, int dx, int dy, int n, int &ox, int &oy) {
    int ux = cx + dx, uy = cy + dy;
    ox = ux < 0 ? -1 : (ux >= n ? 1 : 0);
    oy = uy < 0 ? -1 : (uy >= n ? 1 : 0);
    return (uy - oy * n) * n + (ux - ox * n);
}

// Squared distance from p (offset (fx, fy) inside its cell, torus units) to
// the cell (dx, dy) of its neighbourhood, rounded down a little so that a cell
// is skipped only when every point in it is certainly farther.
__device__ __forceinline__ float box_dist2(int dx, int dy, float fx, float fy, float cw) {
    const float gx = dx > 0 ? (float)dx * cw - fx : (dx < 0 ? fx - (float)(dx + 1) * cw : 0.0f);
    const float gy = dy > 0 ? (float)dy * cw - fy : (dy < 0 ? fy - (float)(dy + 1) * cw : 0.0f);
    return (gx * gx + gy * gy) * 0.99999f;
}

__device__ __forceinline__ void cswap(unsigned &a, unsigned &b) {
    const unsigned lo = min(a, b), hi = max(a, b);
    a = lo;
    b = hi;
}

// Ring-1 slot i (0..7) -> cell offset (dx, dy).
__device__ __forceinline__ void ring1(int i, int &dx, int &dy) {
    dx = i < 3 ? i - 1 : (i < 5 ? (i == 3 ? -1 : 1) : i - 6);
    dy = i < 3 ? -1 : (i < 5 ? 0 : 1);
}

// Star entry of sorted neighbour s at Xs: index and image code of its minimal
// image; (rx, ry) its offset from p.
__device__ __forceinline__ int star_entry(int s, uint2 Xs, uint2 Xp, int &rx, int &ry) {
    rx = (int)(Xs.x - Xp.x);
    ry = (int)(Xs.y - Xp.y);
    const int ox = rx >= 0 ? (Xs.x < Xp.x ? 1 : 0) : (Xs.x > Xp.x ? -1 : 0);
    const int oy = ry >= 0 ? (Xs.y < Xp.y ? 1 : 0) : (Xs.y > Xp.y ? -1 : 0);
    return s | (((ox + 1) * 3 + (oy + 1)) << 28);
}

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Inversion about Xp, in units of 1 / cell (cw: torus units per cell); the
// origin for p itself. The same bits in every kernel (explicit roundings).
struct Inversion {
    uint2 Xp;
    float cw;
    __device__ __forceinline__ float of(int rx, int ry, float &ux, float &uy) const {
        const float sx = (float)rx, sy = (float)ry, d2 = __fmaf_rn(sx, sx, __fmul_rn(sy, sy));
        const float iv = d2 > 0.0f ? __fmul_rn(rcp_approx(d2), cw) : 0.0f;
        ux = __fmul_rn(sx, iv);
        uy = __fmul_rn(sy, iv);
        return d2;
    }
    __device__ __forceinline__ float operator()(uint2 X, float &ux, float &uy) const {
        return of((int)(X.x - Xp.x), (int)(X.y - Xp.y), ux, uy);
    }
};

// A star is stored counter-clockwise from the neighbour of largest start_key,
// where the main pass begins its hull: the inversion farthest in x, its low 6
// bits dropped, then the place in the main pass's list (row of cells, beyond the
// box edge in x or not, sorted index). So a star is the same array whatever pass
// made it.
__device__ __forceinline__ ull start_key(const Inversion &inv, int rx, int ry, int entry, int n, int cy) {
    float ux, uy;
    inv.of(rx, ry, ux, uy);
    const int code = (unsigned)entry >> 28, ox = code / 3 - 1, oy = code % 3 - 1;
    const int dy = cell_of(inv.Xp.y + (unsigned)ry, n) + oy * n - cy;
    return (ull)(ux > 0.0f ? __float_as_uint(ux) >> 6 : 0u) << 34 | (ull)(dy + 16) << 29 | (ull)(ox != 0) << 28 |
           (ull)(entry & 0x0fffffff);
}

// Up to four particles around p that a hull pass found before it gave p up, -1
// for none; kept in p's star slots until its star is written. The last pass
// clips by them first: the cell is then near its final size, and most other
// candidates fail the distance test.
#define NSEED 4
struct Seeds {
    int s[NSEED];
    __device__ __forceinline__ void load(const int *nbr, ll np, int p) {
        s[0] = nbr[p];
#pragma unroll
        for (int k = 1; k < NSEED; ++k) s[k] = s[0] < 0 ? -1 : nbr[(ll)k * np + p];
    }
    __device__ __forceinline__ bool has(int i) const {
        bool h = false;
#pragma unroll
        for (int k = 0; k < NSEED; ++k) h |= s[k] == i;
        return h;
    }
    // seed k, if it is one and not an earlier one again
    __device__ __forceinline__ bool take(int k, int p) const {
        bool ok = s[k] >= 0 && s[k] != p;
        for (int j = 0; j < k; ++j) ok = ok && s[j] != s[k];
        return ok;
    }
};

// The initial cell: the square cut out by four virtual points at distance
// B = 2^30, the largest coordinate the exact predicates take. A vertex
// involving a virtual point is at least 2^29 from p, which the scan
// (< 2^30) can never certify, so a certified cell is bounded by real
// particles only; a cell still touching a virtual point after the last
// ring is reported as ST_SPARSE. Returns the bound R2 of its vertices.
template <int NB>
__device__ __forceinline__ float initial_cell(PolyS<NB> P) {
    const int t = P.t, B = 1 << 30;
    const float hb = 0.5f * (float)B;
    const float rb = 2.0f * hb * hb * 1.0001f;
    P.q[0][t] = make_int4(B, 0, PM_VIRT + 0, 0);
    P.q[1][t] = make_int4(0, B, PM_VIRT + 1, 0);
    P.q[2][t] = make_int4(-B, 0, PM_VIRT + 2, 0);
    P.q[3][t] = make_int4(0, -B, PM_VIRT + 3, 0);
    P.v[0][t] = make_float4(hb, hb, 0.0f, rb);
    P.v[1][t] = make_float4(-hb, hb, 0.0f, rb);
    P.v[2][t] = make_float4(-hb, -hb, 0.0f, rb);
    P.v[3][t] = make_float4(hb, -hb, 0.0f, rb);
    return rb;
}

// Clip the initial cell by the seeds.
template <int CAP, int NB, bool COUNT>
__device__ __forceinline__ int clip_by_seeds(PolyS<NB> P, int &m, float &R2, const Seeds &seeds, int p, uint2 Xp,
                                             const uint2 *__restrict__ pos, int &pp, const int *__restrict__ perm,
                                             WorkCount &wc) {
    for (int k = 0; k < NSEED; ++k) {
        if (!seeds.take(k, p)) continue;
        int rx, ry;
        const int e = star_entry(seeds.s[k], __ldg(pos + seeds.s[k]), Xp, rx, ry);
        if ((rx | ry) == 0) return ST_DUP;
        const int err = clip_by<CAP, NB, COUNT>(P, m, R2, rx, ry, seeds.s[k], (unsigned)e >> 28, p, pp, perm, wc);
        if (err) return err;
    }
    return 0;
}

// The Voronoi cell (star) of one particle p. Candidates are taken ring by
// ring of cells around p until the cell is certified. A neighbouring cell is
// skipped when its box is farther than 2 max|c_k| (none of its points can cut
// the cell: the same test as for a single candidate), and the eight cells of
// the first ring are visited nearest first, so that the cell shrinks early and
// later candidates fail the distance test. The visiting order does not change
// the result: the Voronoi cell is unique and every decision is exact.
// Returns 0, an error bit, or ST_OVERFLOW when the cell outgrew CAP.
template <int CAP, int NB, bool COUNT>
__device__ __forceinline__ int star_of(PolyS<NB> P, int p, const Geo &g, ll np, const uint2 *__restrict__ pos,
                                       const int *__restrict__ cell_start, const int *__restrict__ perm,
                                       int *__restrict__ nbr, unsigned char *__restrict__ deg,
                                       float *__restrict__ vol, float vol_scale, WorkCount &wc) {
    const int t = P.t;
    const int n = g.n;
    int m = 4;
    float R2 = initial_cell(P);
    const uint2 Xp = pos[p];
    const int cx = cell_of(Xp.x, n), cy = cell_of(Xp.y, n);
    const float cw = 4294967296.0f / (float)n;
    const float fxl = (float)cell_frac(Xp.x, n) / (float)n, fyl = (float)cell_frac(Xp.y, n) / (float)n;
    const float edge = fminf(fminf(fxl, cw - fxl), fminf(fyl, cw - fyl));
    int pp = -2;  // priority of p, loaded on first exact test
    int rmax = min(PM_RCAP, n / 4 - 1);
    if (rmax < 0) rmax = 0;
    int err = 0;
    bool done = false;
    // Candidates of one neighbouring cell. Differences of torus coordinates
    // in 32-bit arithmetic are the minimal-image offsets (all |.| < 2^31).
    auto scan_cell = [&](int dx, int dy) {
        if (dx != 0 || dy != 0) {
            if (box_dist2(dx, dy, fxl, fyl, cw) > 4.0001f * R2) return;
        }
        int ox, oy, c = nb_cell(cx, cy, dx, dy, n, ox, oy);
        const int code = (ox + 1) * 3 + (oy + 1);
        PM_CHK(c >= 0 && c < g.ncell, 201, return)
        const int s0 = __ldg(cell_start + c), s1 = __ldg(cell_start + c + 1);
        PM_CHK(s0 >= 0 && s1 <= np && s0 <= s1, 202, return)
        for (int s = s0; s < s1; ++s) {
            if (s == p) continue;
            const uint2 Xs = __ldg(pos + s);
            const int rx = (int)(Xs.x - Xp.x), ry = (int)(Xs.y - Xp.y);
            if ((rx | ry) == 0) { err |= ST_DUP; break; }
            if (rx > (1 << 30) || rx < -(1 << 30) || ry > (1 << 30) || ry < -(1 << 30)) continue;
            err |= clip_by<CAP, NB, COUNT>(P, m, R2, rx, ry, s, code, p, pp, perm, wc);
            if (err) break;
        }
    };
    for (int r = 0; r <= rmax && !done && !err; ++r) {
        if (r == 0) {
            scan_cell(0, 0);
        } else if (r == 1) {
            // the eight cells of ring 1 ordered by box distance: keys hold the
            // distance's float bits with the cell's slot in the low 3 bits
            unsigned k[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                int dx, dy;
                ring1(i, dx, dy);
                k[i] = (__float_as_uint(box_dist2(dx, dy, fxl, fyl, cw)) & ~7u) | (unsigned)i;
            }
            // Batcher's odd-even merge sort network for 8 keys (19 exchanges)
            cswap(k[0], k[1]); cswap(k[2], k[3]); cswap(k[4], k[5]); cswap(k[6], k[7]);
            cswap(k[0], k[2]); cswap(k[1], k[3]); cswap(k[4], k[6]); cswap(k[5], k[7]);
            cswap(k[1], k[2]); cswap(k[5], k[6]);
            cswap(k[0], k[4]); cswap(k[1], k[5]); cswap(k[2], k[6]); cswap(k[3], k[7]);
            cswap(k[2], k[4]); cswap(k[3], k[5]);
            cswap(k[1], k[2]); cswap(k[3], k[4]); cswap(k[5], k[6]);
            unsigned order = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) order |= (k[i] & 7u) << (3 * i);
            for (int i = 0; i < 8 && !err; ++i) {
                int dx, dy;
                ring1((order >> (3 * i)) & 7, dx, dy);
                scan_cell(dx, dy);
            }
        } else {
            const int ncells = 8 * r;
            for (int ci = 0; ci < ncells && !err; ++ci) {
                int dx, dy;
                if (ci < 2 * r + 1) { dx = ci - r; dy = -r; }
                else if (ci < 4 * r + 2) { dx = ci - (3 * r + 1); dy = r; }
                else if (ci < 6 * r + 1) { dx = -r; dy = ci - (5 * r + 1); }
                else { dx = r; dy = ci - (7 * r); }
                scan_cell(dx, dy);
            }
        }
        const float dmin = edge + (float)r * cw;
        if (4.0001f * R2 < dmin * dmin) done = true;
    }
    if (err) return err;
    if (!done) return ST_SPARSE;
    for (int k = 0; k < m; ++k)
        if ((P.q[k][t].z & 0x0fffffff) >= PM_VIRT) return ST_SPARSE;
    if (m > PM_MAXDEG) return ST_DEGREE;
    PM_CHK(m >= 3 && m <= PM_MAXDEG, 203, return ST_DEGREE)
    const Inversion inv{Xp, cw};
    int k0 = 0;
    ull best = 0;
    for (int k = 0; k < m; ++k) {
        const int4 q = P.q[k][t];
        const ull key = start_key(inv, q.x, q.y, q.z, n, cy);
        if (key > best) {
            best = key;
            k0 = k;
        }
    }
    ll area2 = 0;
    int4 A = P.q[k0][t];
    for (int k = 0; k < m; ++k) {
        k0 = k0 + 1 == m ? 0 : k0 + 1;
        int4 Bq = P.q[k0][t];
        area2 += (ll)A.x * Bq.y - (ll)A.y * Bq.x;
        nbr[(ll)k * np + p] = A.z;
        A = Bq;
    }
    deg[p] = (unsigned char)m;
    vol[p] = (float)area2 * vol_scale;
    return 0;
}

// Work counters 0..4 into wsum[0..4], the give-ups into wsum[over_slot], the
// vertex tests the float filter left to the exact predicate into wsum[7].
template <bool COUNT>
__device__ __forceinline__ void add_counts(const WorkCount &wc, ull *__restrict__ wsum, int over_slot) {
    if (!COUNT) return;
    // warp sums, one atomic per warp and counter
    unsigned v[7] = {wc.cand, wc.tested, wc.vtests, wc.clips, wc.msum, wc.over, wc.exact};
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        unsigned x = v[i];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) == 0 && x) atomicAdd(wsum + (i < 5 ? i : (i == 5 ? over_slot : 7)), (ull)x);
    }
}

// ---------------------------------------------------------------------------
// Main pass: the star as a convex hull.
//
// Inversion about p (u_s = (s - p) / |s - p|^2) takes the circles through p to
// lines, and the neighbours of p's Voronoi cell to the vertices of the convex
// hull of the inverted points: a circle through p, a, b is empty exactly when
// every other u_s lies on the origin's side of the line through u_a and u_b.
// So one thread per particle collects the candidates within a radius r_c and
// finds the hull of their inversions by repeated queries "the point farthest
// beyond the directed edge (a, b)": a point beyond the edge is inserted
// between a and b, and an edge with nothing beyond it is a star triangle. All
// lanes of a warp run the same straight-line query over the same number of
// list slots; only the number of queries differs (2 m - 1 for m neighbours).
//
// Every decision is certain or left to another pass. With E = 5.4e-7 bounding the
// relative error of each component of u (nine roundings of 2^-24: conversion, |s|^2,
// reciprocal, products) and U = max |u| (the nearest particle), the float value of
// n . (u_s - u_a), n the float normal of (a, b), is off by less than 1.1 mg,
//   mg = 2.7e-6 U (|u_a| + |u_b|)
// (2 E |n| U for the points, 2 E U (|u_a| + |u_b|) for the normal, 10 units of
// roundoff times |n| U for the evaluation, |n| <= |u_a| + |u_b|). Queries run on
// w = (n . (u_s - u_a)) / mg + 1.25, itself good to 0.1: a maximum above 2.5 is
// certainly beyond the edge; points with w < 0 are certainly not. When all slots
// but a and b have w < 0 (their sign bits are counted) nothing is beyond;
// otherwise the lane is undecided, and its particle goes to the wide pass, or to
// the exact pass where many lanes of the warp are undecided. The
// points that were not collected are at least r_c away, so their inversions lie
// in the disc of radius 1 / r_c, which a final edge must clear too (this is the
// test that the cell is certified: 2 |circumcentre| < r_c). A hull that meets
// the disc, a full list, more than HDEG neighbours, or an edge whose side of p
// is not certain sends the particle to the wide pass; coincident particles go
// to the exact pass. On the 1024^2 mixture 242 warp instructions a particle with
// 24.9 of 32 lanes active, issue active 67 %, 48.5 bytes of DRAM a particle (the wide
// pass, for 4 % of them: 38 more).
// ---------------------------------------------------------------------------
// HN and HL are a balance: fewer candidates make the queries shorter and the
// wide list longer (HN 24, 26, 28, 30 with HL 40: 6.57, 6.35, 6.43, 6.87 ms on
// the set above before the 5 x 5 density, 28 best with it; HL 32: 8.2 ms, HL 48:
// 8.3 ms). The lists take 80 registers, so 8 blocks of 64 threads are resident.
#define HBLK 64        // threads per block
#define HMINB 8        // resident blocks per SM
#define HL 40          // list slots per particle
#define HN 28.0f       // expected number of candidates within r_c
#define HRMAX 6        // largest r_c, in cells
#define HDEG 10        // largest star of this pass (6-bit indices packed into 64 bits)

__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The bits of w with the low 6 replaced by the slot (0..63); positive values
// order as integers.
__device__ __forceinline__ int tag6(float w, unsigned keep, unsigned slot) {
    unsigned r;  // (w & keep) | slot
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(__float_as_uint(w)), "r"(keep), "r"(slot));
    return (int)r;
}

// Search disc of a particle: radius in cells (at most lim) that holds about
// `want` particles at the density of the 3 x 3 cells around (cx, cy), or, where
// those hold fewer than 20, of the 5 x 5 (cut at the box edge in x).
__device__ __forceinline__ float search_radius(const Geo &g, const int *__restrict__ cell_start, int cx, int cy,
                                               float want, int lim) {
    const int n = g.n;
    int cnt = 0, cells = 0;
    for (int h = 1; h <= 2; ++h) {
        const int xa = max(cx - h, 0), xb = min(cx + h, n - 1);
        cnt = 0;
        cells = (2 * h + 1) * (xb - xa + 1);
        for (int dy = -h; dy <= h; ++dy) {
            int y = cy + dy;
            y = y < 0 ? y + n : (y >= n ? y - n : y);
            cnt += __ldg(cell_start + (ll)y * n + xb + 1) - __ldg(cell_start + (ll)y * n + xa);
        }
        if (cnt >= 20 || n < 8) break;
    }
    const float r2 = want * (1.0f / 3.14159265f) * (float)cells * rcp_approx((float)max(cnt, 1));
    return fminf(sqrt_approx(r2), (float)min(lim, n / 4 - 1));
}

// Sorted slots of the cells of row cy + dy that the disc of radius rs around p
// (offset (fx, fy) in its cell, cell units) meets: [s0, s1) and, where the row
// crosses the box edge, [t0, t1). rs carries the slack against the roundings.
__device__ __forceinline__ void row_range(const int *__restrict__ cell_start, int n, int cx, int cy, int dy, float fx,
                                          float fy, float rs, int &s0, int &s1, int &t0, int &t1) {
    const float gy = dy > 0 ? (float)dy - fy : (dy < 0 ? fy - (float)(dy + 1) : 0.0f);
    const float hw = sqrt_approx(fmaxf(rs * rs - gy * gy, 0.0f)) * 1.0001f;
    const int ux0 = cx + (int)floorf(fx - hw), ux1 = cx + (int)floorf(fx + hw);
    int y = cy + dy;
    y = y < 0 ? y + n : (y >= n ? y - n : y);
    const int *cs = cell_start + (ll)y * n;
    s0 = __ldg(cs + max(ux0, 0));
    s1 = __ldg(cs + min(ux1, n - 1) + 1);
    t0 = t1 = 0;
    if (ux0 < 0) {
        t0 = __ldg(cs + ux0 + n);
        t1 = __ldg(cs + n);
    } else if (ux1 >= n) {
        t0 = __ldg(cs);
        t1 = __ldg(cs + ux1 - n + 1);
    }
}

// Star written; needs a wider search; needs exact tests; undecided tests.
enum { HULL_DONE = 1, HULL_WIDER = 2, HULL_EXACT = 3, HULL_UNSURE = 4 };

// All lanes of the warp call this together (live: the lane has a particle).
// ids: the block's list columns, HL + 4 rows (the last rows take the candidates
// of a full list); stk: the stack of hull vertices (u, slot).
template <bool COUNT>
__device__ __forceinline__ int star_hull(int (*ids)[HBLK], float4 (*stk)[HBLK], bool live, int p, uint2 Xp, int ties, const Geo &g, ll np,
                                         const uint2 *__restrict__ pos, const int *__restrict__ cell_start,
                                         int *__restrict__ nbr, unsigned char *__restrict__ deg,
                                         float *__restrict__ vol, float vol_scale, WorkCount &wc) {
    const int t = (int)threadIdx.x, n = g.n;
    const Inversion inv{Xp, 4294967296.0f / (float)n};
    int *const col = &ids[0][0];
    int q = t;
    float ri2 = 0.0f;
    const bool mostly_ties = 3LL * ties > (ll)blockIdx.x * HBLK;  // of the blocks before this one (see on_lattice)
    if (live) {
        const int cx = cell_of(Xp.x, n), cy = cell_of(Xp.y, n);
        const float fx = frac_f(Xp.x, n), fy = frac_f(Xp.y, n);
        const float r = search_radius(g, cell_start, cx, cy, HN, HRMAX), rs = r * 1.0001f + 1e-6f;
        const float r2 = (r * inv.cw) * (r * inv.cw);
        ri2 = rcp_approx(r * r) * 1.0002f;
        const int y1 = mostly_ties ? -100 : (int)floorf(fy + rs);
        for (int dy = (int)floorf(fy - rs); dy <= y1; ++dy) {
            int s0, s1, t0, t1;
            row_range(cell_start, n, cx, cy, dy, fx, fy, rs, s0, s1, t0, t1);
            for (;;) {
                PM_CHK(s0 >= 0 && s1 <= np, 209, break)
                if (COUNT) wc.cand += s1 - s0;
                // four candidates at a time, the next four on their way, without
                // branches: every slot is stored, the column advances past the
                // ones in the disc. Loads past s1 stay within the array's
                // padding and are masked.
                uint2 Xn[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) Xn[k] = __ldg(pos + s0 + k);
                for (int s = s0; s < s1; s += 4) {
                    uint2 Xs[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) Xs[k] = Xn[k];
#pragma unroll
                    for (int k = 0; k < 4; ++k) Xn[k] = __ldg(pos + s + 4 + k);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float sx = (float)(int)(Xs[k].x - Xp.x), sy = (float)(int)(Xs[k].y - Xp.y);
                        col[q] = s + k;
                        q += (s + k < s1 && sx * sx + sy * sy < r2) ? HBLK : 0;
                    }
                    q = min(q, HL * HBLK + t);
                }
                if (t0 >= t1) break;
                s0 = t0;
                s1 = t1;
                t0 = t1;
            }
        }
    }
    const int cnt = (q - t) / HBLK;  // p itself included; HL: the list is full
    if (COUNT) wc.tested += cnt;
    int state = !live || cnt < 4 || cnt >= HL ? HULL_WIDER : 0;  // 0: running
    const int used = __reduce_max_sync(0xffffffffu, state == 0 ? cnt : 0);
    if (used == 0) {
        if (live) nbr[p] = -1;
        return mostly_ties ? HULL_EXACT : state;
    }
    // The inverted candidates, in registers; slots past the lane's own list
    // hold the origin, which is never beyond an edge. The extremes in x and y
    // start the hull: the largest bit pattern as a signed integer is the
    // largest positive value, as an unsigned one the most negative.
    f32x2 xx[HL / 2], yy[HL / 2];
    unsigned keep = 0xffffffc0u;
    asm("" : "+r"(keep));  // one register: (w & keep) | slot is a single LOP3
    int xmax = 0, ymax = 0, zeros = 0;
    unsigned xmin = 0u, ymin = 0u;
#pragma unroll
    for (int c = 0; c < HL / 8; ++c) {
        if (c * 8 < used) {
            uint2 Xs[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) Xs[k] = c * 8 + k < cnt ? __ldg(pos + ids[c * 8 + k][t]) : Xp;
#pragma unroll
            for (int k = 0; k < 8; k += 2) {
                const int j = c * 8 + k;
                float ux[2], uy[2];
                zeros += inv(Xs[k], ux[0], uy[0]) > 0.0f ? 0 : 1;
                zeros += inv(Xs[k + 1], ux[1], uy[1]) > 0.0f ? 0 : 1;
                const int x0 = tag6(ux[0], keep, j), x1 = tag6(ux[1], keep, j + 1);
                const int y0 = tag6(uy[0], keep, j), y1 = tag6(uy[1], keep, j + 1);
                xmax = __vimax3_s32(xmax, x0, x1);
                ymax = __vimax3_s32(ymax, y0, y1);
                xmin = __vimax3_u32(xmin, (unsigned)x0, (unsigned)x1);
                ymin = __vimax3_u32(ymin, (unsigned)y0, (unsigned)y1);
                xx[c * 4 + k / 2] = pk2(ux[0], ux[1]);
                yy[c * 4 + k / 2] = pk2(uy[0], uy[1]);
            }
        }
    }
    const int fill = (used + 7) & ~7;
    if (state == 0 && zeros != fill - cnt + 1) state = HULL_EXACT;  // coincident particles
    // no point on one side of p in x or y: p is not inside the hull
    if (state == 0 && (xmax < 64 || ymax < 64 || (int)xmin > -64 || (int)ymin > -64)) state = HULL_WIDER;
    // U >= |u| of every candidate (the tags take at most 2^-17 off a component)
    const float ex = fmaxf(__int_as_float(xmax), -__uint_as_float(xmin)), ey = fmaxf(__int_as_float(ymax), -__uint_as_float(ymin));
    const float U27 = 2.7e-6f * 1.00003f * sqrt_approx(ex * ex + ey * ey);
    const unsigned ext = (unsigned)(xmax & 63) | (ymin & 63u) << 8 | (xmin & 63u) << 16 | (unsigned)(ymax & 63) << 24;
    const bool seeded = state == 0;
    int a = 0, b = 0, m = 0, depth = 0;  // edge (a, b); the stack's top, b, is row depth; row 0 closes the cycle
    ull out = 0;
    float ax = 0.0f, ay = 0.0f, bx = 0.0f, by = 0.0f;
    if (state == 0) {
        // ccw from the largest x: the vertices still ahead, the last one first
        a = xmax & 63;
        inv(__ldg(pos + ids[a][t]), ax, ay);
        stk[0][t] = make_float4(ax, ay, __int_as_float(a), 0.0f);
        b = a;
        bx = ax;
        by = ay;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int v = (int)(ext >> (8 * (k + 1))) & 63;
            if (v != b && v != a) {
                b = v;
                inv(__ldg(pos + ids[b][t]), bx, by);
                stk[++depth][t] = make_float4(bx, by, __int_as_float(b), 0.0f);
            }
        }
        if (depth == 0) state = HULL_WIDER;
    }
    while (__any_sync(0xffffffffu, state == 0)) {
        // what lies beyond the edge (a, b)?
        const float nx = by - ay, ny = ax - bx, mg = U27 * ((fabsf(ax) + fabsf(ay)) + (fabsf(bx) + fabsf(by)));
        const float im = rcp_approx(mg), sx = nx * im, sy = ny * im, c0 = 1.25f - fmaf(sx, ax, sy * ay);
        const f32x2 sx2 = pk2(sx, sx), sy2 = pk2(sy, sy), c2 = pk2(c0, c0);
        int M = 0;       // largest w as an ordered integer, tagged with its slot
        unsigned S = 0;  // number of w < 0
#pragma unroll
        for (int c = 0; c < HL / 8; ++c) {
            if (c * 8 < used) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int j = c * 4 + k;
                    const f32x2 w = fma2(sy2, yy[j], fma2(sx2, xx[j], c2));
                    float w0, w1;
                    up2(w, w0, w1);
                    S += __float_as_uint(w0) >> 31;
                    S += __float_as_uint(w1) >> 31;
                    M = __vimax3_s32(M, tag6(w0, keep, 2 * j), tag6(w1, keep, 2 * j + 1));
                }
            }
        }
        if (state == 0) {
            const float T = fmaf(nx, ax, ny * ay);
            if (COUNT) wc.vtests += cnt;
            if (M >= 0x40200000 + 64) {  // w > 2.5: insert the vertex
                ++depth;
                b = M & 63;
                if (COUNT) {
                    wc.clips++;
                    wc.msum += m + depth + 1;
                }
                if (depth >= HDEG || b >= cnt) {
                    state = HULL_WIDER;
                } else {
                    inv(__ldg(pos + ids[b][t]), bx, by);
                    stk[depth][t] = make_float4(bx, by, __int_as_float(b), 0.0f);
                }
            } else if (!(T > mg && (T - mg) * (T - mg) > (nx * nx + ny * ny) * ri2) || m >= HDEG) {
                state = HULL_WIDER;
            } else if (S != (unsigned)(fill - 2)) {
                state = HULL_UNSURE;
            } else {  // a final edge
                out = (out << 6) | (ull)a;
                ++m;
                a = b;
                ax = bx;
                ay = by;
                if (--depth < 0) {
                    state = HULL_DONE;
                } else {
                    const float4 q4 = stk[depth][t];
                    bx = q4.x;
                    by = q4.y;
                    b = __float_as_int(q4.z);
                }
            }
        }
    }
    // A few undecided lanes go to the wide pass, which decides exactly; where
    // they are many (a regular lattice) the exact passes are the faster way.
    if (__popc(__ballot_sync(0xffffffffu, state == HULL_UNSURE)) > 4 && state == HULL_UNSURE) state = HULL_EXACT;
    if (state != HULL_DONE || m < 3) {
        if (live) {
            const bool keep = seeded && state != HULL_EXACT;
            nbr[p] = keep ? ids[ext & 63][t] : -1;
            if (keep)
                for (int k = 1; k < NSEED; ++k) nbr[(ll)k * np + p] = ids[(ext >> (8 * k)) & 63][t];
        }
        return state == HULL_EXACT ? HULL_EXACT : HULL_WIDER;
    }
    // the star, counter-clockwise from the largest x of the inversions
    ll area2 = 0;
    int fx0 = 0, fy0 = 0, px = 0, py = 0;
    for (int k = 0; k < m; ++k) {
        const int s = ids[(int)((out >> (6 * (m - 1 - k))) & 63)][t];
        PM_CHK(s >= 0 && s < np, 210, return HULL_EXACT)
        int rx, ry;
        nbr[(ll)k * np + p] = star_entry(s, __ldg(pos + s), Xp, rx, ry);
        if (k == 0) {
            fx0 = rx;
            fy0 = ry;
        } else {
            area2 += (ll)px * ry - (ll)py * rx;
        }
        px = rx;
        py = ry;
    }
    area2 += (ll)px * fy0 - (ll)py * fx0;
    deg[p] = (unsigned char)m;
    vol[p] = (float)area2 * vol_scale;
    return HULL_DONE;
}

// Append this lane's particle to a list (one atomic per warp).
__device__ __forceinline__ void push_list(bool add, int p, ll np, int *__restrict__ list, int *__restrict__ count) {
    const unsigned ball = __ballot_sync(0xffffffffu, add);
    if (!ball) return;
    const int lane = threadIdx.x & 31;
    int base = 0;
    if (lane == 0) base = atomicAdd(count, __popc(ball));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (add) {
        const int k = base + __popc(ball & ((1u << lane) - 1u));
        PM_CHK(k >= 0 && k < np, 205, return)
        list[k] = p;
    }
}

// The particles that a pass gives up: to the wide pass (counts[0]), to the exact
// pass (counts[1]: ties, from the main pass), to the last pass (counts[2], from both);
// counts[3]: the exact pass's next entry.
struct Lists {
    int *wide, *exact, *last, *counts;
};

// A warp goes to the exact pass without an attempt (the attempt costs a third to
// all of the hull, and the exact pass then starts over) in two cases:
//  - (here) its particles stand on a rectangular lattice along the axes: nearly all
//    share a coordinate with the one before or after them, and the next row above
//    has a particle straight above them, so every four are a tie;
//  - (in star_hull) of the particles of the blocks before it more than a third were
//    ties: hull and exact pass take about 270 + 450 f us for 1M particles with a
//    fraction f of ties, the exact pass alone 420. A block reads the count as it
//    stands, so its route may differ from run to run; its stars do not.
__device__ __forceinline__ bool on_lattice(bool live, uint2 X, const Geo &g, const uint2 *__restrict__ pos,
                                           const int *__restrict__ cell_start) {
    const unsigned FULL = 0xffffffffu;
    const uint2 N = make_uint2(__shfl_down_sync(FULL, X.x, 1), __shfl_down_sync(FULL, X.y, 1));
    const bool row = (threadIdx.x & 31) < 31 && (X.x == N.x || X.y == N.y);
    const unsigned rows = __ballot_sync(FULL, live && row);
    if (__popc(rows | rows << 1) < 28) return false;
    bool above = false;
    if (live) {
        const int n = g.n, cx = cell_of(X.x, n), cy = cell_of(X.y, n);
        unsigned dmin = 0xffffffffu;
        for (int h = 0; h < 2; ++h) {
            const int *cs = cell_start + (ll)(cy + h == n ? 0 : cy + h) * n + cx;
            const int s0 = __ldg(cs), s1 = min(__ldg(cs + 1), s0 + 16);
            for (int s = s0; s < s1; ++s) {
                const uint2 Y = __ldg(pos + s);
                const unsigned d = Y.y - X.y;  // up, modulo the box
                if (d == 0 || d > 0x7fffffffu) continue;
                if (d < dmin) above = false;
                if (d <= dmin) above |= Y.x == X.x;
                dmin = min(dmin, d);
            }
        }
    }
    return __popc(__ballot_sync(FULL, above)) >= 24;
}

// Counters: wsum[0..4] the work of completed cells, wsum[5] the cells given
// up by the main pass, wsum[6] large stars of the later passes.
template <bool COUNT>
__global__ void __launch_bounds__(HBLK, HMINB) k_delaunay(Geo g, ll np, const uint2 *__restrict__ pos,
                                                   const int *__restrict__ cell_start, int *__restrict__ nbr,
                                                   unsigned char *__restrict__ deg, float *__restrict__ vol,
                                                   float vol_scale, Lists L, ull *__restrict__ wsum) {
    __shared__ int ids[HL + 4][HBLK];
    __shared__ float4 stk[HDEG][HBLK];
    const ll pl = (ll)blockIdx.x * HBLK + threadIdx.x;
    const bool live = pl < np;
    const int ties = L.counts[1];
    const uint2 Xp = live ? pos[pl] : make_uint2(0u, 0u);
    WorkCount wc;
    int e = HULL_EXACT;
    if (!on_lattice(live, Xp, g, pos, cell_start))
        e = star_hull<COUNT>(ids, stk, live, (int)pl, Xp, ties, g, np, pos, cell_start, nbr, deg, vol, vol_scale, wc);
    else if (live)
        nbr[pl] = -1;
    if (COUNT && live && e != HULL_DONE) {
        wc = WorkCount{};
        wc.over = 1;
    }
    push_list(live && e == HULL_WIDER, (int)pl, np, L.wide, L.counts);
    push_list(live && e == HULL_EXACT, (int)pl, np, L.exact, L.counts + 1);
    add_counts<COUNT>(wc, wsum, 5);
}

// ---------------------------------------------------------------------------
// Wide pass: the hull of a particle of the wide list by a group of 8 lanes,
// over up to 96 candidates (12 registers per lane). A query is 12 candidates
// per lane and a 3-step reduction, so a star takes microseconds, where one lane
// with a long list would hold up a warp. The same tests and margins as in the
// main pass, with undecided candidates decided exactly on the spot. The first
// search takes a disc that should hold 48 candidates; where the hull of what it
// finds is complete but not certified, its largest circle gives the radius of
// the next. Up to PM_MAXDEG neighbours.
// ---------------------------------------------------------------------------
#define WBLK 128
#define WG (WBLK / 8)  // groups per block
#define WL 96          // list slots per group
#define WN 48.0f       // expected candidates of the first search
#define WTRIES 4       // searches per particle

struct WideS {
    float x[WL], y[WL];
    int id[WL];
    float ex[PM_MAXDEG], ey[PM_MAXDEG], et[PM_MAXDEG];  // edges of the last complete hull
    unsigned char st[PM_MAXDEG + 2], out[PM_MAXDEG + 2];
};

// All lanes of the warp call this together, the 8 lanes of a group with the
// same particle. HULL_DONE, or HULL_EXACT where the exact passes are needed.
template <bool COUNT>
__device__ __forceinline__ int star_wide(WideS &G, bool live, int p, const Geo &g, ll np, const uint2 *__restrict__ pos,
                                         const int *__restrict__ cell_start, const int *__restrict__ perm,
                                         int *__restrict__ nbr, unsigned char *__restrict__ deg,
                                         float *__restrict__ vol, float vol_scale, WorkCount &wc) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, sub = lane & 7, sh = lane & 24;
    const int n = g.n;
    const uint2 Xp = live ? pos[p] : make_uint2(0u, 0u);
    const Inversion inv{Xp, 4294967296.0f / (float)n};
    const int cx = cell_of(Xp.x, n), cy = cell_of(Xp.y, n);
    const float fx = frac_f(Xp.x, n), fy = frac_f(Xp.y, n);
    const float rlim = (float)min(PM_RCAP, n / 4 - 1);
    float r = live ? search_radius(g, cell_start, cx, cy, WN, PM_RCAP) : 0.0f;
    int result = live ? 0 : HULL_EXACT, cnt = 0, m = 0, edges = 0;  // result 0: not finished
    for (int tries = 0; tries < WTRIES && __any_sync(FULL, result == 0); ++tries) {
        const bool act = result == 0;
        const float rs = r * 1.0001f + 1e-6f, r2 = (r * inv.cw) * (r * inv.cw), ri2 = rcp_approx(r * r) * 1.0002f;
        bool dup = false;
        if (act) cnt = 0;
        const int y0 = (int)floorf(fy - rs), y1 = act ? (int)floorf(fy + rs) : y0 - 1;
        for (int dy = y0; __any_sync(FULL, dy <= y1); ++dy) {
            int s0 = 0, s1 = 0, t0 = 0, t1 = 0;
            if (dy <= y1) row_range(cell_start, n, cx, cy, dy, fx, fy, rs, s0, s1, t0, t1);
            for (;;) {
                PM_CHK(s0 >= 0 && s1 <= np, 211, s1 = s0)
                if (COUNT && sub == 0) wc.cand += s1 - s0;
                for (int s = s0 + sub; __any_sync(FULL, s - sub < s1); s += 8) {
                    bool hit = false;
                    if (s < s1) {
                        const uint2 Xs = __ldg(pos + s);
                        const int rx = (int)(Xs.x - Xp.x), ry = (int)(Xs.y - Xp.y);
                        const float sx = (float)rx, sy = (float)ry;
                        hit = sx * sx + sy * sy < r2 && s != p;
                        dup |= hit && (rx | ry) == 0;
                        if (hit && edges) {  // strictly inside the last hull: cannot matter
                            float ux, uy;
                            inv(Xs, ux, uy);
                            hit = false;
                            for (int k = 0; k < edges; ++k) hit |= fmaf(G.ex[k], ux, G.ey[k] * uy) > G.et[k];
                        }
                    }
                    const unsigned ball = (__ballot_sync(FULL, hit) >> sh) & 0xffu;
                    const int k = cnt + __popc(ball & ((1u << sub) - 1u));
                    if (hit && k < WL) G.id[k] = s;
                    cnt += __popc(ball);
                }
                if (!__any_sync(FULL, t0 < t1)) break;
                s0 = t0;
                s1 = t1;
                t0 = t1;
            }
        }
        __syncwarp();
        if (((__ballot_sync(FULL, dup) >> sh) & 0xffu) != 0 && act) result = HULL_EXACT;
        if (COUNT && sub == 0 && act) wc.tested += cnt;
        // 0: querying, 1: hull complete, 2: no use
        int state = act && result == 0 && cnt >= 3 && cnt <= WL ? 0 : 2;
        float X[WL / 8], Y[WL / 8];
        unsigned near = 0xffffffffu;
#pragma unroll
        for (int k = 0; k < WL / 8; ++k) {
            const int j = k * 8 + sub;
            X[k] = Y[k] = __int_as_float(0x7fc00000);  // no slot: never beyond an edge
            if (state == 0 && j < cnt) {
                const float d2 = inv(__ldg(pos + G.id[j]), X[k], Y[k]);
                G.x[j] = X[k];
                G.y[j] = Y[k];
                near = min(near, (__float_as_uint(d2) & ~127u) | (unsigned)j);
            }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) near = min(near, __shfl_xor_sync(FULL, near, o));
        __syncwarp();
        int a = (int)(near & 127u), depth = 1;
        // U >= |u| of the nearest (the tag takes at most 2^-16 off |s|^2)
        const float U = sqrt_approx(rcp_approx(__uint_as_float(near & ~127u)) * 1.00005f) * inv.cw;
        float ax = 0.0f, ay = 0.0f, bx = 0.0f, by = 0.0f, need2 = 0.0f;
        int b = 0;
        if (state == 0) {
            m = 0;
            ax = G.x[a];
            ay = G.y[a];
            if (sub == 0) G.st[0] = (unsigned char)a;
        }
        bool first = true;
        while (__any_sync(FULL, state == 0)) {
            float nx = by - ay, ny = ax - bx, mg = 2.7e-6f * U * ((fabsf(ax) + fabsf(ay)) + (fabsf(bx) + fabsf(by)));
            if (first) {
                nx = -ax;
                ny = -ay;
                mg = U * U;
            }
            const float im = rcp_approx(mg), sx = nx * im, sy = ny * im, c0 = 1.25f - fmaf(sx, ax, sy * ay);
            // largest w (as an ordered integer, tagged with its slot), number of w > 0
            unsigned M = 0u;
            int S = 0;
#pragma unroll
            for (int k = 0; k < WL / 8; ++k) {
                const float w = fmaf(sy, Y[k], fmaf(sx, X[k], c0));
                if (w > 0.0f) {
                    M = max(M, (__float_as_uint(w) & ~127u) | (unsigned)(k * 8 + sub));
                    ++S;
                }
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                M = max(M, __shfl_xor_sync(FULL, M, o));
                S += __shfl_xor_sync(FULL, S, o);
            }
            if (COUNT && state == 0 && sub == 0) wc.vtests += cnt;
            int v = first || M >= 0x40200000u + 128u ? (int)(M & 127u) : -1;  // w > 2.5: the vertex to insert
            if (__any_sync(FULL, state == 0 && v < 0 && S != 2)) {
                // undecided candidates, exactly
                int e = 255;
                if (state == 0 && v < 0 && S != 2 && fmaf(nx, ax, ny * ay) > mg) {
                    const uint2 A = __ldg(pos + G.id[a]), B = __ldg(pos + G.id[b]);
                    for (int j = sub; j < cnt && e == 255; j += 8) {
                        if (j == a || j == b || !(fmaf(sy, G.y[j], fmaf(sx, G.x[j], c0)) > 0.0f)) continue;
                        const uint2 Q = __ldg(pos + G.id[j]);
                        if (incircle_exact((int)(A.x - Xp.x), (int)(A.y - Xp.y), (int)(B.x - Xp.x), (int)(B.y - Xp.y),
                                           (int)(Q.x - Xp.x), (int)(Q.y - Xp.y), perm[p], perm[G.id[a]],
                                           perm[G.id[b]], perm[G.id[j]]))
                            e = j;
                    }
                    if (COUNT) wc.exact++;
                }
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) e = min(e, __shfl_xor_sync(FULL, e, o));
                if (v < 0 && e < 255) v = e;
            }
            if (state == 0) {
                const float T = fmaf(nx, ax, ny * ay);
                if (v >= 0) {
                    if (depth >= PM_MAXDEG || v >= cnt) {
                        state = 2;
                    } else {
                        b = v;
                        if (sub == 0) G.st[depth] = (unsigned char)b;
                        ++depth;
                        bx = G.x[b];
                        by = G.y[b];
                        if (COUNT && sub == 0) {
                            wc.clips++;
                            wc.msum += m + depth;
                        }
                    }
                } else if ((!(T > mg) && S != 2) || m >= PM_MAXDEG) {
                    state = 2;
                } else {
                    // a final edge of this hull; need2: the squared radius that certifies it
                    need2 = fmaxf(need2, T > mg ? (nx * nx + ny * ny) * rcp_approx((T - mg) * (T - mg)) : 1e30f);
                    if (sub == 0) G.out[m] = (unsigned char)a;
                    ++m;
                    a = b;
                    ax = bx;
                    ay = by;
                    if (--depth == 0) {
                        state = 1;
                    } else {
                        b = G.st[depth - 1];
                        bx = G.x[b];
                        by = G.y[b];
                    }
                }
            }
            first = false;
            __syncwarp();
        }
        if (act && result == 0) {
            if (state == 1 && need2 * ri2 * 1.0001f < 1.0f)
                result = m >= 3 ? HULL_DONE : HULL_EXACT;
            else if (cnt > WL)
                r *= sqrt_approx(0.7f * (float)WL * rcp_approx((float)cnt));
            else if (r >= rlim)
                result = HULL_EXACT;
            else
                r = fminf(state == 1 && need2 < 1e30f ? sqrt_approx(need2) * 1.001f : 1.6f * r, rlim);
            if (state == 1 && result != HULL_DONE && sub < NSEED) nbr[(ll)sub * np + p] = G.id[G.out[sub * m / NSEED]];
            if (result == 0 && state == 1) {  // the next search drops what lies inside this hull
                edges = m;
                for (int k = sub; k < m; k += 8) {
                    const int i0 = G.out[k], i1 = G.out[k + 1 == m ? 0 : k + 1];
                    const float x0 = G.x[i0], y0 = G.y[i0], x1 = G.x[i1], y1 = G.y[i1];
                    G.ex[k] = y1 - y0;
                    G.ey[k] = x0 - x1;
                    G.et[k] = fmaf(G.ex[k], x0, G.ey[k] * y0) -
                              1e-5f * U * ((fabsf(x0) + fabsf(y0)) + (fabsf(x1) + fabsf(y1)));
                }
            }
        }
        __syncwarp();
    }
    const bool done = result == HULL_DONE;
    ull key = 0;
    int first_k = 0;
    for (int k = sub; done && k < m; k += 8) {
        const int s = G.id[G.out[k]];
        int rx, ry;
        const int e = star_entry(s, __ldg(pos + s), Xp, rx, ry);
        const ull q = start_key(inv, rx, ry, e, n, cy);
        if (q > key) {
            key = q;
            first_k = k;
        }
    }
    ull best = key;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) best = max(best, (ull)__shfl_xor_sync(FULL, best, o));
    first_k = __shfl_sync(FULL, first_k, sh + __ffs((__ballot_sync(FULL, key == best) >> sh) & 0xffu) - 1);
    ll area2 = 0;
    for (int k = sub; done && k < m; k += 8) {
        const int s = G.id[G.out[k]], s2 = G.id[G.out[k + 1 == m ? 0 : k + 1]];
        const int slot = k >= first_k ? k - first_k : k + m - first_k;
        int rx, ry, qx, qy;
        nbr[(ll)slot * np + p] = star_entry(s, __ldg(pos + s), Xp, rx, ry);
        star_entry(s2, __ldg(pos + s2), Xp, qx, qy);
        area2 += (ll)rx * qy - (ll)ry * qx;
    }
    __syncwarp();
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) area2 += __shfl_xor_sync(FULL, area2, o);
    if (done && sub == 0) {
        deg[p] = (unsigned char)m;
        vol[p] = (float)area2 * vol_scale;
        if (COUNT && m > 12) wc.over++;
    }
    return done ? HULL_DONE : HULL_EXACT;
}

template <bool COUNT>
__global__ void __launch_bounds__(WBLK) k_delaunay_wide(Geo g, ll np, const uint2 *__restrict__ pos,
                                                        const int *__restrict__ cell_start,
                                                        const int *__restrict__ perm, int *__restrict__ nbr,
                                                        unsigned char *__restrict__ deg, float *__restrict__ vol,
                                                        float vol_scale, Lists L, ull *__restrict__ wsum) {
    __shared__ WideS G[WG];
    const int cnt = L.counts[0], gid = threadIdx.x >> 3;
    WorkCount wc;
    for (ll j0 = (ll)blockIdx.x * WG; j0 < cnt; j0 += (ll)gridDim.x * WG) {
        const ll j = j0 + gid;
        const bool live = j < cnt;
        const int p = live ? L.wide[j] : 0;
        const WorkCount before = wc;
        const int e = star_wide<COUNT>(G[gid], live, p, g, np, pos, cell_start, perm, nbr, deg, vol, vol_scale, wc);
        const bool over = live && e != HULL_DONE && (threadIdx.x & 7) == 0;
        if (COUNT && over) wc = before;
        push_list(over, p, np, L.last, L.counts + 2);
    }
    add_counts<COUNT>(wc, wsum, 6);
}

// The mesh of a particle: one mesh, or the particle's instance of a batch (from
// the packed offsets; stars hold packed sorted indices, < 2^28 in total).
struct OneMesh {
    Geo g;
    ll np;
    const int *cell_start;
    float vol_scale;
    __device__ __forceinline__ Geo geo(int) const { return g; }
    __device__ __forceinline__ const int *cells(int) const { return cell_start; }
    __device__ __forceinline__ float scale(int) const { return vol_scale; }
    __device__ __forceinline__ int instance(int) const { return 0; }
};
struct BatchMesh {
    BTab t;
    ll np;
    const int *cell_start;
    __device__ __forceinline__ Geo geo(int k) const { return batch_geo(t, k); }
    __device__ __forceinline__ const int *cells(int k) const { return cell_start + __ldg(t.coff + k); }
    __device__ __forceinline__ float scale(int k) const { return t.inst[k].vol_scale; }
    __device__ __forceinline__ int instance(int p) const { return find_slot(t.poff, t.ninst, (ll)p); }
};

// From this many particles on the exact pass takes its list, one thread each, and
// leaves those whose cell outgrows ECAP to the last pass; a shorter list goes to
// the last pass as it is.
#define EXACT_MIN 4096

__device__ __forceinline__ void fail_star(int err, int p, unsigned char *deg, float *vol, int *status) {
    atomicOr(status, (err & ~ST_OVERFLOW) | (err & ST_OVERFLOW ? ST_DEGREE : 0));
    deg[p] = 0;
    vol[p] = 0.0f;
}

template <class Mesh, bool COUNT>
__global__ void __launch_bounds__(EBLK, EMINB) k_delaunay_exact(Mesh M, const uint2 *__restrict__ pos,
                                                                const int *__restrict__ perm, int *__restrict__ nbr,
                                                                unsigned char *__restrict__ deg,
                                                                float *__restrict__ vol, int *__restrict__ status,
                                                                Lists L, ull *__restrict__ wsum) {
    __shared__ int4 sq[ECAP][EBLK];
    __shared__ float4 sv[ECAP][EBLK];
    const int cnt = L.counts[1];
    if (cnt < EXACT_MIN) return;
    WorkCount wc;
    PolyS<EBLK> P{sq, sv, (int)threadIdx.x};
    const int lane = threadIdx.x & 31;
    for (;;) {  // a warp takes the next 32
        int j = 0;
        if (lane == 0) j = atomicAdd(L.counts + 3, 32);
        j = __shfl_sync(0xffffffffu, j, 0);
        if (j >= cnt) break;
        j += lane;
        bool over = false;
        int p = 0;
        if (j < cnt) {
            p = L.exact[j];
            PM_CHK(p >= 0 && p < M.np, 206, p = 0)
            const WorkCount before = wc;
            const int k = M.instance(p);
            const int err = star_of<ECAP, EBLK, COUNT>(P, p, M.geo(k), M.np, pos, M.cells(k), perm, nbr, deg, vol,
                                                       M.scale(k), wc);
            over = err == ST_OVERFLOW;
            if (COUNT && over) wc = before;
            if (err && !over) fail_star(err, p, deg, vol, status);
        }
        push_list(over, p, M.np, L.last, L.counts + 2);
    }
    add_counts<COUNT>(wc, wsum, 6);
}

// ---------------------------------------------------------------------------
// Last pass: the cell of a particle by a warp. The lanes read a cell's particles
// 32 at a time and drop those that certainly cut nothing; what is left is clipped
// by lane 0, one after another. It takes the few particles whose neighbourhood is
// unlike the mean density (a blob inside a cell, a jump of density), where one
// thread walks over thousands of candidates with a load latency each: 80,000
// particles with 20,000 in a blob of a quarter of a cell, 33.5 + 7.3 ms by one
// thread each.
// ---------------------------------------------------------------------------
template <bool COUNT>
__device__ __forceinline__ int star_warp(PolyS<LBLK / 32> P, int p, const Geo &g, ll np, const uint2 *__restrict__ pos,
                                         const int *__restrict__ cell_start, const int *__restrict__ perm,
                                         int *__restrict__ nbr, unsigned char *__restrict__ deg,
                                         float *__restrict__ vol, float vol_scale, WorkCount &wc) {
    constexpr int NB = LBLK / 32;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, t = P.t, n = g.n;
    const uint2 Xp = pos[p];
    const int cx = cell_of(Xp.x, n), cy = cell_of(Xp.y, n);
    const float cw = 4294967296.0f / (float)n;
    const float fxl = (float)cell_frac(Xp.x, n) / (float)n, fyl = (float)cell_frac(Xp.y, n) / (float)n;
    const float edge = fminf(fminf(fxl, cw - fxl), fminf(fyl, cw - fyl));
    const int rmax = max(0, min(PM_RCAP, n / 4 - 1));
    Seeds seeds;
    seeds.load(nbr, np, p);
    int m = 4, pp = -2, err = 0;
    float R2 = 0.0f;
    if (lane == 0) {
        R2 = initial_cell(P);
        err = clip_by_seeds<LCAP, NB, COUNT>(P, m, R2, seeds, p, Xp, pos, pp, perm, wc);
    }
    __syncwarp();
    m = __shfl_sync(FULL, m, 0);
    R2 = __shfl_sync(FULL, R2, 0);
    err = __shfl_sync(FULL, err, 0);
    bool done = false;
    for (int r = 0; r <= rmax && !done && !err; ++r) {
        const int ncells = r == 0 ? 1 : 8 * r;
        for (int c0 = 0; c0 < ncells && !err; c0 += 32) {
            // the ring's cells, one a lane; those that can matter are visited
            const int ci = c0 + lane;
            int dx = 0, dy = 0;
            if (r > 0) {
                if (ci < 2 * r + 1) { dx = ci - r; dy = -r; }
                else if (ci < 4 * r + 2) { dx = ci - (3 * r + 1); dy = r; }
                else if (ci < 6 * r + 1) { dx = -r; dy = ci - (5 * r + 1); }
                else { dx = r; dy = ci - (7 * r); }
            }
            int s0 = 0, s1 = 0, ox = 0, oy = 0;
            const float bd = r == 0 ? 0.0f : box_dist2(dx, dy, fxl, fyl, cw);
            if (ci < ncells && bd <= 4.0001f * R2) {
                const int c = nb_cell(cx, cy, dx, dy, n, ox, oy);
                PM_CHK(c >= 0 && c < g.ncell, 201, s0 = s1)
                s0 = __ldg(cell_start + c);
                s1 = __ldg(cell_start + c + 1);
                PM_CHK(s0 >= 0 && s1 <= np && s0 <= s1, 202, s0 = s1 = 0)
            }
            for (unsigned cells = __ballot_sync(FULL, s0 < s1); cells && !err; cells &= cells - 1) {
                const int src = __ffs(cells) - 1;
                const int a = __shfl_sync(FULL, s0, src), b = __shfl_sync(FULL, s1, src);
                const int code = (__shfl_sync(FULL, ox, src) + 1) * 3 + (__shfl_sync(FULL, oy, src) + 1);
                if (__shfl_sync(FULL, bd, src) > 4.0001f * R2) continue;
                for (int k = a; k < b && !err; k += 32) {
                    const int s = k + lane;
                    bool hit = false, dup = false;
                    int rx = 0, ry = 0;
                    if (s < b && s != p) {
                        const uint2 Xs = __ldg(pos + s);
                        rx = (int)(Xs.x - Xp.x);
                        ry = (int)(Xs.y - Xp.y);
                        dup = (rx | ry) == 0;
                        hit = rx <= (1 << 30) && rx >= -(1 << 30) && ry <= (1 << 30) && ry >= -(1 << 30) && !seeds.has(s);
                        const float fx = (float)rx, fy = (float)ry, d2 = fx * fx + fy * fy;
                        hit = hit && d2 <= 4.0001f * R2;
                        if (hit) {  // certainly outside every vertex's circle: no cut (as in clip_by)
                            const float hs = 0.5f * d2, ns = 1.41422f * fmaxf(fabsf(fx), fabsf(fy)), mr = 2.4e-7f * d2;
                            bool cut = false;
                            for (int i = 0; i < m; ++i) {
                                const float4 v = P.v[i][t];
                                cut |= !(v.x * fx + v.y * fy - hs < -(v.z * ns + mr));
                            }
                            hit = cut;
                        }
                    }
                    if (COUNT && lane == 0) wc.cand += min(32, b - k);
                    if (__any_sync(FULL, dup)) err = ST_DUP;
                    for (unsigned hits = __ballot_sync(FULL, hit); hits && !err; hits &= hits - 1) {
                        const int h = __ffs(hits) - 1, hx = __shfl_sync(FULL, rx, h), hy = __shfl_sync(FULL, ry, h);
                        if (lane == 0) {
                            err = clip_by<LCAP, NB, COUNT>(P, m, R2, hx, hy, k + h, code, p, pp, perm, wc);
                            if (COUNT) wc.cand--;  // counted above
                        }
                        err = __shfl_sync(FULL, err, 0);
                    }
                    __syncwarp();
                    m = __shfl_sync(FULL, m, 0);
                    R2 = __shfl_sync(FULL, R2, 0);
                }
            }
        }
        const float dmin = edge + (float)r * cw;
        if (4.0001f * R2 < dmin * dmin) done = true;
    }
    if (err) return err;
    if (!done) return ST_SPARSE;
    const int4 q = P.q[lane < m ? lane : 0][t], q2 = P.q[lane + 1 < m ? lane + 1 : 0][t];
    if (__any_sync(FULL, lane < m && (q.z & 0x0fffffff) >= PM_VIRT)) return ST_SPARSE;
    if (m > PM_MAXDEG) return ST_DEGREE;
    ll area2 = lane < m ? (ll)q.x * q2.y - (ll)q.y * q2.x : 0;
    for (int o = 16; o > 0; o >>= 1) area2 += __shfl_xor_sync(FULL, area2, o);
    const ull key = lane < m ? start_key(Inversion{Xp, cw}, q.x, q.y, q.z, n, cy) : 0;
    ull best = key;
    for (int o = 16; o > 0; o >>= 1) best = max(best, (ull)__shfl_xor_sync(FULL, best, o));
    const int k0 = __ffs(__ballot_sync(FULL, key == best)) - 1;
    if (lane < m) nbr[(ll)(lane >= k0 ? lane - k0 : lane + m - k0) * np + p] = q.z;
    if (lane == 0) {
        deg[p] = (unsigned char)m;
        vol[p] = (float)area2 * vol_scale;
        if (COUNT && m > 12) wc.over++;
    }
    return 0;
}

template <class Mesh, bool COUNT>
__global__ void __launch_bounds__(LBLK) k_delaunay_last(Mesh M, const uint2 *__restrict__ pos,
                                                        const int *__restrict__ perm, int *__restrict__ nbr,
                                                        unsigned char *__restrict__ deg, float *__restrict__ vol,
                                                        int *__restrict__ status, Lists L, ull *__restrict__ wsum) {
    constexpr int NB = LBLK / 32;
    __shared__ int4 sq[LCAP][NB];
    __shared__ float4 sv[LCAP][NB];
    const int hard = L.counts[2], ties = L.counts[1] < EXACT_MIN ? L.counts[1] : 0;
    WorkCount wc;
    const int w = threadIdx.x >> 5;
    PolyS<NB> P{sq, sv, w};
    for (ll j = (ll)blockIdx.x * NB + w; j < (ll)hard + ties; j += (ll)gridDim.x * NB) {
        const int p = j < hard ? L.last[j] : L.exact[j - hard];
        PM_CHK(p >= 0 && p < M.np, 207, continue)
        const int k = M.instance(p);
        const int err = star_warp<COUNT>(P, p, M.geo(k), M.np, pos, M.cells(k), perm, nbr, deg, vol, M.scale(k), wc);
        if (err && (threadIdx.x & 31) == 0) fail_star(err, p, deg, vol, status);
        __syncwarp();
    }
    add_counts<COUNT>(wc, wsum, 6);
}

// Batched passes: the particle's instance comes from the packed offsets; its
// mesh, cell ranges and volume scale from the instance table. Stars hold
// packed sorted indices (< 2^28 in total).
__global__ void __launch_bounds__(HBLK, HMINB) k_delaunay_b(BTab t, const uint2 *__restrict__ pos,
                                                     const int *__restrict__ cell_start, int *__restrict__ nbr,
                                                     unsigned char *__restrict__ deg, float *__restrict__ vol, Lists L) {
    __shared__ int ids[HL + 4][HBLK];
    __shared__ float4 stk[HDEG][HBLK];
    const ll pl = (ll)blockIdx.x * HBLK + threadIdx.x;
    const bool live = pl < t.NP;
    const int ties = L.counts[1];
    const uint2 Xp = live ? pos[pl] : make_uint2(0u, 0u);
    WorkCount wc;
    int e = HULL_EXACT;
    const int k = find_slot(t.poff, t.ninst, live ? pl : t.NP - 1);
    const Geo g = batch_geo(t, k);
    const int *cs = cell_start + __ldg(t.coff + k);
    if (!on_lattice(live, Xp, g, pos, cs))
        e = star_hull<false>(ids, stk, live, (int)pl, Xp, ties, g, t.NP, pos, cs, nbr, deg, vol, t.inst[k].vol_scale, wc);
    else if (live)
        nbr[pl] = -1;
    push_list(live && e == HULL_WIDER, (int)pl, t.NP, L.wide, L.counts);
    push_list(live && e == HULL_EXACT, (int)pl, t.NP, L.exact, L.counts + 1);
}

__global__ void __launch_bounds__(WBLK) k_delaunay_wide_b(BTab t, const uint2 *__restrict__ pos,
                                                          const int *__restrict__ cell_start,
                                                        const int *__restrict__ perm, int *__restrict__ nbr,
                                                          unsigned char *__restrict__ deg, float *__restrict__ vol,
                                                          Lists L) {
    __shared__ WideS G[WG];
    const int cnt = L.counts[0], gid = threadIdx.x >> 3;
    WorkCount wc;
    for (ll j0 = (ll)blockIdx.x * WG; j0 < cnt; j0 += (ll)gridDim.x * WG) {
        const ll j = j0 + gid;
        const bool live = j < cnt;
        const int p = live ? L.wide[j] : 0;
        const int k = find_slot(t.poff, t.ninst, (ll)p);
        const Geo g = batch_geo(t, k);
        const int e = star_wide<false>(G[gid], live, p, g, t.NP, pos, cell_start + __ldg(t.coff + k), perm, nbr, deg,
                                       vol, t.inst[k].vol_scale, wc);
        push_list(live && e != HULL_DONE && (threadIdx.x & 7) == 0, p, t.NP, L.last, L.counts + 2);
    }
}

// 1D: v_mu = half the distance between the two neighbours on the circle.
__global__ void k_vol1d(ll np, const uint2 *__restrict__ pos, float *__restrict__ vol, float scale) {
    ll s = (ll)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= np) return;
    uint32_t x = pos[s].x;
    ull gn = s + 1 < np ? (ull)(pos[s + 1].x - x) : 4294967296ull - (ull)(x - pos[0].x);
    ull gp = s > 0 ? (ull)(x - pos[s - 1].x) : 4294967296ull - (ull)(pos[np - 1].x - x);
    vol[s] = (float)(gn + gp) * scale;
}

__global__ void k_export(ll np, const uint2 *__restrict__ pos, const int *__restrict__ nbr,
                         const unsigned char *__restrict__ deg, const int *__restrict__ perm, int *__restrict__ tri,
                         int *__restrict__ off, ll max_tri, ll *__restrict__ counter) {
    ll pl = (ll)blockIdx.x * blockDim.x + threadIdx.x;
    if (pl >= np) return;
    int p = (int)pl, m = deg[p];
    for (int k = 0; k < m; ++k) {
        int ea = nbr[(ll)k * np + p], eb = nbr[(ll)(k + 1 == m ? 0 : k + 1) * np + p];
        int a = ea & 0x0fffffff, b = eb & 0x0fffffff;
        if (a <= p || b <= p) continue;
        ll t = atomicAdd((ull *)counter, 1ull);
        if (t >= max_tri) continue;
        tri[3 * t] = perm[p];
        tri[3 * t + 1] = perm[a];
        tri[3 * t + 2] = perm[b];
        int ca = (unsigned)ea >> 28, cb = (unsigned)eb >> 28;
        off[4 * t] = ca / 3 - 1;
        off[4 * t + 1] = ca % 3 - 1;
        off[4 * t + 2] = cb / 3 - 1;
        off[4 * t + 3] = cb % 3 - 1;
    }
}

}  // namespace

namespace {
// The passes' lists: the sort's scratch is free once the particles are sorted.
Lists pass_lists(const Work &w) { return Lists{w.tmp, w.key, w.slot, w.nretry}; }

// Grids of the list passes (grid-stride): resident blocks per SM.
constexpr int kWideGrid = 8 * 152, kExactGrid = EMINB * 152, kLastGrid = 12 * 152;

template <class Mesh, bool COUNT>
void exact_passes(const Mesh &M, Work &w, const Lists &L, ull *wsum, cudaStream_t st) {
    k_delaunay_exact<Mesh, COUNT><<<min(kExactGrid, div_up(M.np, EBLK)), EBLK, 0, st>>>(M, w.pos, w.perm, w.nbr, w.deg,
                                                                                    w.vol, w.status, L, wsum);
    k_delaunay_last<Mesh, COUNT><<<min(kLastGrid, div_up(M.np, LBLK / 32)), LBLK, 0, st>>>(M, w.pos, w.perm, w.nbr, w.deg,
                                                                                       w.vol, w.status, L, wsum);
}

template <bool COUNT>
void triangulate_passes(const Geo &g, Work &w, ll np, float scale, ull *wsum, cudaStream_t st) {
    const Lists L = pass_lists(w);
    k_delaunay<COUNT><<<div_up(np, HBLK), HBLK, 0, st>>>(g, np, w.pos, w.cell_start, w.nbr, w.deg, w.vol, scale, L, wsum);
    k_delaunay_wide<COUNT><<<min(kWideGrid, div_up(np, WG)), WBLK, 0, st>>>(g, np, w.pos, w.cell_start, w.perm, w.nbr,
                                                                            w.deg, w.vol, scale, L, wsum);
    exact_passes<OneMesh, COUNT>(OneMesh{g, np, w.cell_start, scale}, w, L, wsum, st);
}
}  // namespace

void launch_triangulate(const Geo &g, Work &w, ll np, cudaStream_t st, bool count_work) {
    if (np <= 0) return;
    double u = g.L / 4294967296.0;
    float scale = (float)(u * u / 6.0);
    cudaMemsetAsync(w.nretry, 0, 4 * sizeof(int), st);
    if (count_work)
        triangulate_passes<true>(g, w, np, scale, w.wsum, st);
    else
        triangulate_passes<false>(g, w, np, scale, nullptr, st);
    count_launches(4);
}

void launch_triangulate_batched(const BTab &t, Work &w, cudaStream_t st) {
    if (t.NP <= 0) return;
    cudaMemsetAsync(w.nretry, 0, 4 * sizeof(int), st);
    const Lists L = pass_lists(w);
    k_delaunay_b<<<div_up(t.NP, HBLK), HBLK, 0, st>>>(t, w.pos, w.cell_start, w.nbr, w.deg, w.vol, L);
    k_delaunay_wide_b<<<min(kWideGrid, div_up(t.NP, WG)), WBLK, 0, st>>>(t, w.pos, w.cell_start, w.perm, w.nbr, w.deg,
                                                                         w.vol, L);
    exact_passes<BatchMesh, false>(BatchMesh{t, t.NP, w.cell_start}, w, L, nullptr, st);
    count_launches(4);
}

void launch_volumes_1d(const Geo &g, Work &w, ll np, cudaStream_t st) {
    if (np <= 0) return;
    float scale = (float)(0.5 * g.L / 4294967296.0);
    k_vol1d<<<div_up(np, 256), 256, 0, st>>>(np, w.pos, w.vol, scale);
    count_launches(1);
}

void launch_export_tris(const Geo &g, Work &w, ll np, int *tri, int *off, ll max_tri, cudaStream_t st) {
    cudaMemsetAsync(w.ntri, 0, sizeof(ll), st);
    if (np > 0) {
        k_export<<<div_up(np, 256), 256, 0, st>>>(np, w.pos, w.nbr, w.deg, w.perm, tri, off, max_tri, w.ntri);
        count_launches(1);
    }
}
