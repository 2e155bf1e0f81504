// Mesh mass matrix m_ij = int psi_i psi_j (Sec. 2.4) and the solve M Ab = b
// (Eq. phi_def).
//
// M is applied matrix-free: 1D (h/6)(x_{i-1} + 4 x_i + x_{i+1}); 2D bilinear
// elements give the tensor product (h^2/36) [1 4 1; 4 16 4; 1 4 1]; 2D P1
// elements on cells split by the (0,0)-(1,1) diagonal give (h^2/12) times 6 at
// the node and 1 at its six edge neighbours (row sums h^2 in every case). Stencil
// sums are compensated (error-free transformations), so M x is accurate to
// about one rounding whatever the cancellation.
//
// The mesh solves are ONE persistent cooperative kernel each (k_cg, k_cheb):
// every block owns a strided share of the nodes of all F fields, and the
// reductions go through the blocks' totals, which every block then sums in the
// same fixed order (deterministic and identical on all blocks, so all
// blocks take the same branch). Per-node products are accumulated per thread
// in compensated FP32, and the threads' sums lose nothing against FP64 (Sum3).
// Before iterating, the mean mode of x is set exactly from sum_j b_j (1 is an
// eigenvector of the circulant M with eigenvalue h^dim, and the iterations keep
// the mean of the start vector), which makes the result conservative (Eq. cons)
// to rounding at any iteration count.
//
// What bounds them is the grid barrier with its reduction on small meshes
// (FP64 runs at 1/64 of FP32 here, so one thread per field computes the step
// lengths) and the passes over the vectors on large ones.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "internal.cuh"

PM_DEBUG_DECL(solve)

namespace {

struct CG {
    Geo g;
    int F;
    const float *bsrc;      // float right-hand side (or null)
    const ll *bfix;         // fixed-point right-hand side (or null)
    const unsigned *maxabs; // fixed-point scale source
    float *x;               // [F][ncell] start and result (caller's)
    float *b, *xw, *p;      // float right-hand side, iterate, search direction
    float *r[2], *s[2], *w[2];  // CG: residual, M p, M r, alternating between passes
                                // Chebyshev: r and d (in s)
    double *red;            // [6 * PM_MAXF][grid]
    float4 *red4;           // [4 * PM_MAXF][grid]
    double *scal;           // [F][16]
    unsigned *bar;          // [2] barrier count
    int *status;
    double rtol;
    int max_iter;
    int has_start;
    const double *psum;     // particle sums per block (or null)
    int nblk_psum;
};

enum { S_ITERS = 0, S_INIT = 1, S_RESID = 2, S_SUMMESH = 3, S_SUMPART = 4, S_SUMABS = 5 };

// Grid-wide barrier with a bounded wait (about a second); on timeout the
// status word gets ST_TIMEOUT and false is returned. The count only grows:
// barrier k of a launch opens at k times the number of blocks. `passed` counts
// the barriers of this launch.
__device__ bool grid_sync(unsigned *bar, int *status, unsigned &passed) {
    ++passed;
    if (gridDim.x == 1) {
        __syncthreads();
        return true;
    }
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        const unsigned target = passed * gridDim.x;
        unsigned seen;
        asm volatile("atom.add.release.gpu.global.u32 %0, [%1], 1;" : "=r"(seen) : "l"(bar) : "memory");
        int spins = 0;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
            if ((int)(seen - target) >= 0) break;
            if (++spins > 64) __nanosleep(64);
            if (spins > (1 << 22)) {
                atomicOr(status, ST_TIMEOUT);
                ok = 0;
                break;
            }
        }
    }
    __syncthreads();
    return ok != 0;
}

// A sum over the grid: every thread puts its accumulator (the warp's total goes
// to shared memory), the block flushes its total, and after a grid barrier every
// block sums the blocks' totals in the same order. Sum3 throughout or FP64, so
// nothing is held in fewer bits than FP64 holds:
//  put_sum, flush_sums, grid_sum: any range; FP64 totals of the blocks in
//    red[(slot + kind) * F + f][block]. The start, the closing residual.
//  put_scaled, flush_scaled, grid_scaled: the inner products of an iteration,
//    brought to order one by powers of two, so that no exponents are carried;
//    Sum3 in red4[(slot + kind) * F + f][block]. A single block keeps its totals
//    in shared memory.
// An FP64 addition takes 62 cycles here, a sum over a warp 680 in FP64 and 228 in
// Sum3 (180 in FP32 pairs, which this replaces: whole solves by CG take the
// same time to 5 %, 256^2 122.5 -> 125.7 us, 255^2 166 -> 147 us).
struct BlockSums {
    Sum3 v[3][PM_MAXF][8];
    Sum3 one[2 * PM_MAXF];  // totals of a single block's inner products
};
__device__ __forceinline__ void put_sum(BlockSums &B, int kind, int f, const Dot2 &a) {
    const Sum3 t = fold_warp(warp_parts(a));
    if ((threadIdx.x & 31) == 0) B.v[kind][f][threadIdx.x >> 5] = t;
}
// Kinds 0 and 1 at once.
__device__ __forceinline__ void put_sums(BlockSums &B, int f, const Dot2 &a0, const Dot2 &a1) {
    const Sum3 t = fold_warp(warp_parts(a0), warp_parts(a1));
    if ((threadIdx.x & 15) == 0) B.v[threadIdx.x >> 4 & 1][f][threadIdx.x >> 5] = t;
}
__device__ __forceinline__ void flush_sums(const BlockSums &B, int kinds, int F, double *red, int slot) {
    __syncthreads();
    const int t = threadIdx.x;
    if (t < kinds * F) {
        const Sum3 *v = B.v[t / F][t % F];
        Sum3 a = v[0], b = v[4];
#pragma unroll
        for (int w = 1; w < 4; ++w) {
            join(a, v[w]);
            join(b, v[w + 4]);
        }
        join(a, b);
        red[(ll)(slot * F + t) * gridDim.x + blockIdx.x] = total(a);
    }
}
// Total of (slot, f) over all blocks, by one warp.
__device__ __forceinline__ double grid_sum(const double *red, int F, int slot, int f) {
    const int lane = threadIdx.x & 31;
    const double *src = red + (ll)(slot * F + f) * gridDim.x;
    double s = 0;
#pragma unroll 4
    for (unsigned i = lane; i < gridDim.x; i += 32) s += __ldcg(src + i);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}
__device__ __forceinline__ void put_scaled(BlockSums &B, int kind, int f, const Dot2 &a, float scale) {
    const Sum3 t = fold_warp(scaled_parts(a, scale, 0));
    if ((threadIdx.x & 31) == 0) B.v[kind][f][threadIdx.x >> 5] = t;
}
// Kinds 0 and 1 at once.
__device__ __forceinline__ void put_scaled(BlockSums &B, int f, const Dot2 &a0, float s0, const Dot2 &a1, float s1) {
    const Sum3 t = fold_warp(scaled_parts(a0, s0, 0), scaled_parts(a1, s1, 0));
    if ((threadIdx.x & 15) == 0) B.v[threadIdx.x >> 4 & 1][f][threadIdx.x >> 5] = t;
}
__device__ __forceinline__ void flush_scaled(BlockSums &B, int kinds, int F, float4 *red4, int slot) {
    __syncthreads();
    const int t = threadIdx.x;
    if (t < kinds * F) {
        const Sum3 *v = B.v[t / F][t % F];
        Sum3 a = v[0], b = v[4];
#pragma unroll
        for (int w = 1; w < 4; ++w) {
            add_parts(a, v[w].a, v[w].b, v[w].c);
            add_parts(b, v[w + 4].a, v[w + 4].b, v[w + 4].c);
        }
        add_parts(a, b.a, b.b, b.c);
        if (gridDim.x == 1) {
            B.one[t] = a;
            return;
        }
        red4[(ll)(slot * F + t) * gridDim.x + blockIdx.x] = make_float4(a.a, a.b, a.c, 0.0f);
    }
}
// Totals of field f in K consecutive slots (1 or 2) over all blocks, by one
// warp, half of it for each of two slots; lane 0 has them.
template <int K>
__device__ __forceinline__ void grid_scaled(const BlockSums &B, const float4 *red4, int F, int slot, int f,
                                            double (&out)[K]) {
    constexpr int W = 32 / K;
    const unsigned lane = threadIdx.x & 31;
    Sum3 s{0.0f, 0.0f, 0.0f, 0};
    if (gridDim.x == 1) {
        s = B.one[(int)(lane / W) * F + f];
    } else {
        const float4 *src = red4 + (ll)((slot + (int)(lane / W)) * F + f) * gridDim.x;
        // eight loads in flight, also at the end: a load is an L2 latency
        for (unsigned i = lane % W; i < gridDim.x; i += 8 * W) {
            float4 t[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) t[j] = i + j * W < gridDim.x ? __ldcg(src + i + j * W) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
            for (int j = 0; j < 8; ++j) add_parts(s, t[j].x, t[j].y, t[j].z);
        }
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) fold_down(s, o);
    }
    out[0] = ((double)s.a + (double)s.b) + (double)s.c;
    if (K == 2) out[K - 1] = __shfl_down_sync(0xffffffffu, out[0], W);
}

// Totals of the per-block particle sums of one row (sum v A or sum v |A|) by
// the whole block, the same order on every run; thread 0 has it.
__device__ __forceinline__ double particle_sum(const double *psum, int nblk, int row) {
    __shared__ double sh[8];
    const double *src = psum + (ll)row * nblk;
    double s = 0;
#pragma unroll 4
    for (int i = threadIdx.x; i < nblk; i += 256) s += src[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    s = ((sh[0] + sh[1]) + (sh[2] + sh[3])) + ((sh[4] + sh[5]) + (sh[6] + sh[7]));
    __syncthreads();
    return s;
}

struct Q4 {
    float v[4];
};
__device__ __forceinline__ Q4 ld4(const float *p) {
    const float4 t = *(const float4 *)p;
    return Q4{{t.x, t.y, t.z, t.w}};
}

// VEC consecutive nodes of a row (VEC = 4: 16-byte accesses, n % 4 == 0).
template <int VEC>
__device__ __forceinline__ void ldn(const float *p, float (&v)[VEC]) {
    if (VEC == 4) {
        const Q4 q = ld4(p);
#pragma unroll
        for (int j = 0; j < VEC; ++j) v[j] = q.v[j & 3];
    } else {
        v[0] = *p;
    }
}
template <int VEC>
__device__ __forceinline__ void stn(float *p, const float (&v)[VEC]) {
    if (VEC == 4) *(float4 *)p = make_float4(v[0], v[1 % VEC], v[2 % VEC], v[3 % VEC]);
    else *p = v[0];
}

// Compensated stencil sums (hi, lo) of the VEC nodes starting at flat index i0
// (unscaled: the caller multiplies by h/6, h^2/36 or h^2/12) of the vector that
// val gives, val.get(index, out) for VEC nodes from an aligned index and
// val.one(index) for one; ctr: its values there. The additions are those of
// stencil<>, in the same order.
template <int DIM, int P1, int VEC, class Val>
__device__ __forceinline__ void stencil_of(const Val &val, int n, int i0, float (&hi)[VEC], float (&lo)[VEC],
                                           float (&ctr)[VEC]) {
    if (DIM == 1) {
        val.get(i0, ctr);
        const float l = val.one(i0 == 0 ? n - 1 : i0 - 1), r = val.one(i0 + VEC == n ? 0 : i0 + VEC);
#pragma unroll
        for (int j = 0; j < VEC; ++j) {
            Dot2 acc;
            acc.add(4.0f * ctr[j]);
            acc.add(j == 0 ? l : ctr[j == 0 ? 0 : j - 1]);
            acc.add(j == VEC - 1 ? r : ctr[j == VEC - 1 ? 0 : j + 1]);
            hi[j] = acc.hi;
            lo[j] = acc.lo;
        }
        return;
    }
    const int iy = (int)((unsigned)i0 / (unsigned)n), ix = i0 - iy * n;
    const int r0 = (iy == 0 ? n - 1 : iy - 1) * n, r1 = iy * n, r2 = (iy + 1 == n ? 0 : iy + 1) * n;
    const int xl = ix == 0 ? n - 1 : ix - 1, xr = ix + VEC == n ? 0 : ix + VEC;
    float a[VEC], c[VEC];
    val.get(r0 + ix, a);
    val.get(r1 + ix, ctr);
    val.get(r2 + ix, c);
    const float a_l = val.one(r0 + xl), a_r = P1 ? 0.0f : val.one(r0 + xr), b_l = val.one(r1 + xl),
                b_r = val.one(r1 + xr), c_l = P1 ? 0.0f : val.one(r2 + xl), c_r = val.one(r2 + xr);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
        const int jm = j == 0 ? 0 : j - 1, jp = j == VEC - 1 ? 0 : j + 1;
        const float am = j == 0 ? a_l : a[jm], ap = j == VEC - 1 ? a_r : a[jp];
        const float bm = j == 0 ? b_l : ctr[jm], bp = j == VEC - 1 ? b_r : ctr[jp];
        const float cm = j == 0 ? c_l : c[jm], cp = j == VEC - 1 ? c_r : c[jp];
        Dot2 acc;
        if (P1) {
            acc.add(6.0f * ctr[j]);
            acc.add(bm);
            acc.add(bp);
            acc.add(a[j]);
            acc.add(c[j]);
            acc.add(am);
            acc.add(cp);
        } else {
            acc.add(16.0f * ctr[j]);
            acc.add(4.0f * bm);
            acc.add(4.0f * bp);
            acc.add(4.0f * a[j]);
            acc.add(4.0f * c[j]);
            acc.add(am);
            acc.add(ap);
            acc.add(cm);
            acc.add(cp);
        }
        hi[j] = acc.hi;
        lo[j] = acc.lo;
    }
}

// A stored vector.
template <int VEC>
struct Plain {
    const float *v;
    __device__ __forceinline__ void get(int o, float (&q)[VEC]) const { ldn<VEC>(v + o, q); }
    __device__ __forceinline__ float one(int o) const { return v[o]; }
};
// The scaled start with its exact mean, S x + sh (sh alone without a start).
template <int VEC>
struct Start {
    const float *x;
    float S, sh;
    __device__ __forceinline__ void get(int o, float (&q)[VEC]) const {
#pragma unroll
        for (int j = 0; j < VEC; ++j) q[j] = 0.0f;
        if (x) ldn<VEC>(x + o, q);
#pragma unroll
        for (int j = 0; j < VEC; ++j) q[j] = fmaf(q[j], S, sh);
    }
    __device__ __forceinline__ float one(int o) const { return fmaf(x ? x[o] : 0.0f, S, sh); }
};
// The next residual of a CG pass, r - alpha (w + beta s).
template <int VEC>
struct NextR {
    const float *r, *w, *s;
    float al, be;
    bool first;  // no s yet: it is w
    __device__ __forceinline__ void get(int o, float (&q)[VEC]) const {
        float t[VEC], u[VEC];
        ldn<VEC>(r + o, q);
        ldn<VEC>(w + o, t);
        if (!first) {
            ldn<VEC>(s + o, u);
#pragma unroll
            for (int j = 0; j < VEC; ++j) t[j] = fmaf(be, u[j], t[j]);
        }
#pragma unroll
        for (int j = 0; j < VEC; ++j) q[j] = fmaf(-al, t[j], q[j]);
    }
    __device__ __forceinline__ float one(int o) const {
        float t = w[o];
        if (!first) t = fmaf(be, s[o], t);
        return fmaf(-al, t, r[o]);
    }
};

// Per-field state of a mesh solve, the same on every block.
struct SolveState {
    double bb[PM_MAXF], rr[PM_MAXF], rr0[PM_MAXF], pMp[PM_MAXF], sumb[PM_MAXF], tr[PM_MAXF], sx[PM_MAXF];
    double thr[PM_MAXF];  // the iteration's tolerance for rr
    float S[PM_MAXF], sh[PM_MAXF], al[PM_MAXF], be[PM_MAXF], ka[PM_MAXF];
    float kr[PM_MAXF], kw[PM_MAXF];  // powers of two that bring (r, r) and (w, r) to order one; rr and pMp hold them
    int act[PM_MAXF], first[PM_MAXF], its[PM_MAXF], steps[PM_MAXF];
};

// Right-hand side as float, its sum and sum of |b|, sum of the start; the field
// scale S (a power of two that brings the mean |b| to order one: exact scaling,
// FP32 inner products of any field stay in range) and the shift that sets the
// mean of S x + sh to the exact one. Ends with a block barrier.
template <int DIM, int VEC>
__device__ __forceinline__ bool solve_begin(const CG &a, SolveState &V, BlockSums &B, unsigned &passed) {
    const Geo &g = a.g;
    const int F = a.F;
    const unsigned nv = (unsigned)(g.ncell / VEC);
    const ll nn = g.ncell;
    const unsigned tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    const float hd32 = DIM == 1 ? g.h : g.h * g.h;
    const double hd = DIM == 1 ? (double)g.h : (double)g.h * g.h;
    for (int f = 0; f < F; ++f) {
        const ll fo = (ll)f * nn;
        // the fixed-point scale 2^-E in two factors, so that neither overflows (E is
        // at most 120 + 149) and only the second product can round, as in ldexpf
        const int E = a.bfix ? fixed_point_exp(__uint_as_float(a.maxabs[f]), hd32) : 0;
        const float s1 = ldexpf(1.0f, -(E / 2)), s2 = ldexpf(1.0f, E / 2 - E);
        Dot2 sb, sa, sx;
        for (unsigned i = tid; i < nv; i += nth) {
            const ll o = fo + (ll)i * VEC;
            float bv[VEC], xv[VEC];
            if (a.bfix) {
                ll q[VEC];
                if (VEC == 4) {
                    const longlong2 u = *(const longlong2 *)(a.bfix + o), v = *(const longlong2 *)(a.bfix + o + 2);
                    q[0] = u.x, q[1 % VEC] = u.y, q[2 % VEC] = v.x, q[3 % VEC] = v.y;
                } else {
                    q[0] = a.bfix[o];
                }
#pragma unroll
                for (int j = 0; j < VEC; ++j) bv[j] = (float)q[j] * s1 * s2;
            } else {
                ldn<VEC>(a.bsrc + o, bv);
            }
            stn<VEC>(a.b + o, bv);
            if (a.has_start) ldn<VEC>(a.x + o, xv);
#pragma unroll
            for (int j = 0; j < VEC; ++j) {
                // times 2^-10: a thread's sums stay in range where the nodes do
                sb.add(bv[j] * 0x1p-10f);
                sa.add(fabsf(bv[j]) * 0x1p-10f);
                if (a.has_start) sx.add(xv[j] * 0x1p-10f);
            }
        }
        put_sums(B, f, sb, sa);
        put_sum(B, 2, f, sx);
    }
    flush_sums(B, 3, F, a.red, 0);
    if (!grid_sync(a.bar, a.status, passed)) return false;
    const int f = threadIdx.x >> 5;
    if (f < F) {
        const double sumb = 1024.0 * grid_sum(a.red, F, 0, f), suma = 1024.0 * grid_sum(a.red, F, 1, f),
                     sumx = 1024.0 * grid_sum(a.red, F, 2, f);
        if ((threadIdx.x & 31) == 0) {
            const float S = solve_scale(suma / (double)nn);
            V.S[f] = S;
            V.sumb[f] = sumb;
            V.sh[f] = (float)((double)S * (sumb / ((double)nn * hd) - (a.has_start ? sumx / (double)nn : 0.0)));
            V.its[f] = 0;
        }
    }
    __syncthreads();
    return true;
}

// True residual r = S b - M xw into r (and, if out, the unscaled result into
// out), sums of r^2 and xw; with START, xw = S x + sh is formed and stored and
// the second sum is that of (S b)^2. Ends before the reduction's barrier.
template <int DIM, int P1, int VEC, bool START>
__device__ __forceinline__ void residual_pass(const CG &a, SolveState &V, BlockSums &B, float *r, float *out, int slot) {
    const Geo &g = a.g;
    const int F = a.F, n = g.n;
    const unsigned nv = (unsigned)(g.ncell / VEC);
    const ll nn = g.ncell;
    const unsigned tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    const float c = DIM == 1 ? g.h / 6.0f : (P1 ? g.h * g.h / 12.0f : g.h * g.h / 36.0f);
    for (int f = 0; f < F; ++f) {
        const ll fo = (ll)f * nn;
        const float S = V.S[f], inv = 1.0f / S;  // powers of two: exact
        const Start<VEC> st{a.has_start ? a.x + fo : nullptr, S, V.sh[f]};
        const Plain<VEC> xw{a.xw + fo};
        Dot2 s, t;
        for (unsigned i = tid; i < nv; i += nth) {
            const int i0 = (int)(i * VEC);
            float hi[VEC], lo[VEC], ct[VEC], bv[VEC], rv[VEC];
            if (START) stencil_of<DIM, P1, VEC>(st, n, i0, hi, lo, ct);
            else stencil_of<DIM, P1, VEC>(xw, n, i0, hi, lo, ct);
            ldn<VEC>(a.b + fo + i0, bv);
#pragma unroll
            for (int j = 0; j < VEC; ++j) {
                bv[j] *= S;
                rv[j] = fmaf(-c, hi[j], bv[j]) - c * lo[j];
                s.fma_acc(rv[j], rv[j]);
                if (START) t.fma_acc(bv[j], bv[j]);
                else t.add(ct[j]);
            }
            stn<VEC>(r + fo + i0, rv);
            if (START) stn<VEC>(a.xw + fo + i0, ct);
            if (out) {
#pragma unroll
                for (int j = 0; j < VEC; ++j) ct[j] *= inv;
                stn<VEC>(out + fo + i0, ct);
            }
        }
        put_sums(B, f, s, t);
    }
    flush_sums(B, 2, F, a.red, slot);
}

// The report of a solve whose closing residual pass is summed (V.tr, V.sx).
__device__ __forceinline__ void solve_report(const CG &a, const SolveState &V, double hd) {
    // the particle sums, a row to a block from the last block down
    if (a.psum)
        for (int row = gridDim.x - 1 - blockIdx.x; row < 2 * a.F; row += gridDim.x) {
            const double ps = particle_sum(a.psum, a.nblk_psum, row);
            if (threadIdx.x == 0) a.scal[(row >> 1) * 16 + (row & 1 ? S_SUMABS : S_SUMPART)] = ps;
        }
    if (blockIdx.x != 0) return;
    const int f = threadIdx.x >> 1, k = threadIdx.x & 1;  // k: residual at exit, at the start
    if (f >= a.F) return;
    const double res = V.bb[f] > 0.0 ? sqrt((k ? V.rr0[f] : V.tr[f]) / V.bb[f]) : 0.0;
    if (k) {
        a.scal[f * 16 + S_INIT] = res;
        return;
    }
    a.scal[f * 16 + S_ITERS] = V.its[f];
    a.scal[f * 16 + S_RESID] = res;
    a.scal[f * 16 + S_SUMMESH] = V.sx[f] * hd / (double)V.S[f];
    if (!a.psum) {
        a.scal[f * 16 + S_SUMPART] = V.sumb[f];
        a.scal[f * 16 + S_SUMABS] = 0.0;
    }
    if (res > a.rtol) atomicOr(a.status, ST_NOTCONV);
}

// Field f (re)starts from a residual of squared norm rr.
__device__ __forceinline__ void restart_state(SolveState &V, int f, double rr, double tol2, ll nn, double hd) {
    const float kr = solve_scale(rr / (double)nn), kw = solve_scale(rr / (double)nn * hd);
    V.rr[f] = rr * (double)kr;
    V.thr[f] = tol2 * V.bb[f] * (double)kr;
    V.kr[f] = kr;
    V.kw[f] = kw;
    V.ka[f] = kw / kr;
}

// Conjugate gradients with one pass and one grid barrier per iteration. With
// w = M r at hand, (r, r) and (w, r) give both step lengths (Chronopoulos and
// Gear): beta = rr / rr_old, alpha = rr / pMp, pMp = (w, r) - beta^2 pMp_old, and
//   s = w + beta s (= M p),  p = r + beta p,  x += alpha p,  r -= alpha s,  w = M r
// is one pass: each node forms the next r at its stencil's nodes from the old r,
// w and s (the same FMAs everywhere, so every copy has the same bits), and r, s
// and w alternate between two buffers. The separate passes for M p, x and r,
// and p took three barriers. Whole solves from zero, before and now: 128 nodes in
// 1D (one block) 168 -> 46 us; 256^2 327 -> 126 us; 512^2, 3 fields 684 -> 285 us; 2048^2, 4
// fields (19 iterations) 4165 -> 2859 us: 40 bytes per node and iteration, and 44 in
// the other passes, 4.7 TB/s.
// Consecutive reductions never share slots, so that a block that runs ahead never
// overwrites partials another block is summing: {0, 1, 2} and {3, 4} of red, {0}
// and then alternately {2, 3} and {0, 1} of red4, and {0, 1} of red at the end.
template <int DIM, int P1, int VEC>
__global__ void __launch_bounds__(256, VEC == 4 ? 3 : 4) k_cg(CG a) {
    __shared__ SolveState V;
    __shared__ BlockSums B;
    unsigned passed = 0;
    const Geo &g = a.g;
    const int F = a.F, n = g.n;
    const unsigned nv = (unsigned)(g.ncell / VEC);
    const ll nn = g.ncell;
    const unsigned tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    const float c = DIM == 1 ? g.h / 6.0f : (P1 ? g.h * g.h / 12.0f : g.h * g.h / 36.0f);
    const double hd = DIM == 1 ? (double)g.h : (double)g.h * g.h;
    const double tol2 = a.rtol * a.rtol;
    const int wf = threadIdx.x >> 5;  // warp f sums field f's partials, its lane 0 keeps the state
    const bool lane0 = (threadIdx.x & 31) == 0;
    if (!solve_begin<DIM, VEC>(a, V, B, passed)) return;
    residual_pass<DIM, P1, VEC, true>(a, V, B, a.r[0], nullptr, 3);
    if (!grid_sync(a.bar, a.status, passed)) return;
    if (wf < F) {
        const double rr = grid_sum(a.red, F, 3, wf), bb = grid_sum(a.red, F, 4, wf);
        if (lane0) {
            V.rr0[wf] = rr;
            V.bb[wf] = bb;
            restart_state(V, wf, rr, tol2, nn, hd);
            V.act[wf] = V.first[wf] = bb > 0.0 && rr > tol2 * bb;
        }
    }
    __syncthreads();
    int cur = 0, it = 0;
    for (int restarts = 0;; ++restarts) {
        bool any = false;
        for (int f = 0; f < F; ++f) any |= V.act[f] != 0;
        if (any && it < a.max_iter) {
            // w = M r, (w, r) of the fields that (re)start
            for (int f = 0; f < F; ++f) {
                if (!V.act[f]) continue;
                const ll fo = (ll)f * nn;
                const Plain<VEC> rp{a.r[cur] + fo};
                Dot2 d;
                for (unsigned i = tid; i < nv; i += nth) {
                    float hi[VEC], lo[VEC], ct[VEC];
                    stencil_of<DIM, P1, VEC>(rp, n, (int)(i * VEC), hi, lo, ct);
#pragma unroll
                    for (int j = 0; j < VEC; ++j) {
                        hi[j] = fmaf(c, hi[j], c * lo[j]);
                        d.fma_acc(hi[j], ct[j]);
                    }
                    stn<VEC>(a.w[cur] + fo + i * VEC, hi);
                }
                put_scaled(B, 0, f, d, V.kw[f]);
            }
            flush_scaled(B, 1, F, a.red4, 0);
            if (!grid_sync(a.bar, a.status, passed)) return;
            if (wf < F && V.act[wf]) {
                double t[1];
                grid_scaled<1>(B, a.red4, F, 0, wf, t);
                if (lane0) {
                    const double wr = t[0];
                    V.pMp[wf] = wr;
                    V.al[wf] = (float)(V.rr[wf] / wr) * V.ka[wf];
                    V.be[wf] = 0.0f;
                    V.first[wf] = 1;
                    if (!(wr > 0.0)) V.act[wf] = 0;  // r below the range of its products
                }
            }
            __syncthreads();
            int slot = 2;
            while (any && it < a.max_iter) {
                const int nxt = cur ^ 1;
                for (int f = 0; f < F; ++f) {
                    if (!V.act[f]) continue;
                    const ll fo = (ll)f * nn;
                    const float al = V.al[f], be = V.be[f];
                    const bool first = V.first[f] != 0;
                    const NextR<VEC> rn{a.r[cur] + fo, a.w[cur] + fo, a.s[cur] + fo, al, be, first};
                    Dot2 sr, sw;
                    for (unsigned i = tid; i < nv; i += nth) {
                        const int i0 = (int)(i * VEC);
                        const ll o = fo + i0;
                        float hi[VEC], lo[VEC], ct[VEC], sv[VEC], pv[VEC], xv[VEC];
                        stencil_of<DIM, P1, VEC>(rn, n, i0, hi, lo, ct);
                        ldn<VEC>(a.w[cur] + o, sv);
                        ldn<VEC>(a.r[cur] + o, pv);
                        ldn<VEC>(a.xw + o, xv);
                        if (!first) {
                            float t[VEC], u[VEC];
                            ldn<VEC>(a.s[cur] + o, t);
                            ldn<VEC>(a.p + o, u);
#pragma unroll
                            for (int j = 0; j < VEC; ++j) {
                                sv[j] = fmaf(be, t[j], sv[j]);
                                pv[j] = fmaf(be, u[j], pv[j]);
                            }
                        }
#pragma unroll
                        for (int j = 0; j < VEC; ++j) {
                            xv[j] = fmaf(al, pv[j], xv[j]);
                            hi[j] = fmaf(c, hi[j], c * lo[j]);
                            sr.fma_acc(ct[j], ct[j]);
                            sw.fma_acc(hi[j], ct[j]);
                        }
                        stn<VEC>(a.r[nxt] + o, ct);
                        stn<VEC>(a.s[nxt] + o, sv);
                        stn<VEC>(a.w[nxt] + o, hi);
                        stn<VEC>(a.p + o, pv);
                        stn<VEC>(a.xw + o, xv);
                    }
                    put_scaled(B, f, sr, V.kr[f], sw, V.kw[f]);
                }
                flush_scaled(B, 2, F, a.red4, slot);
                if (!grid_sync(a.bar, a.status, passed)) return;
                if (wf < F && V.act[wf]) {
                    double t[2];
                    grid_scaled<2>(B, a.red4, F, slot, wf, t);
                    if (lane0) {
                        const double rr = t[0], wr = t[1];
                        const double beta = rr / V.rr[wf], pMp = wr - beta * (beta * V.pMp[wf]);
                        V.pMp[wf] = pMp;
                        V.al[wf] = (float)(rr / pMp) * V.ka[wf];
                        V.be[wf] = (float)beta;
                        V.rr[wf] = rr;
                        V.first[wf] = 0;
                        ++V.its[wf];
                        if (rr <= V.thr[wf] || !(pMp > 0.0)) V.act[wf] = 0;
                    }
                }
                __syncthreads();
                slot ^= 2;
                cur = nxt;
                ++it;
                any = false;
                for (int f = 0; f < F; ++f) any |= V.act[f] != 0;
            }
        }
        // the true residual of every field, and the result
        residual_pass<DIM, P1, VEC, false>(a, V, B, a.r[cur], a.x, 0);
        if (!grid_sync(a.bar, a.status, passed)) return;
        if (wf < F) {
            const double tr = grid_sum(a.red, F, 0, wf), sx = grid_sum(a.red, F, 1, wf);
            if (lane0) {
                V.tr[wf] = tr;
                V.sx[wf] = sx;
                V.act[wf] = V.bb[wf] > 0.0 && tr > tol2 * V.bb[wf];
                if (V.act[wf]) restart_state(V, wf, tr, tol2, nn, hd);
            }
        }
        __syncthreads();
        bool again = false;
        for (int f = 0; f < F; ++f) again |= V.act[f] != 0;
        // drifted fields restart from their true residual
        if (!again || restarts >= 3 || it >= a.max_iter) break;
    }
    solve_report(a, V, hd);
}

// ---------------------------------------------------------------------------
// Chebyshev iteration for M x = b. The spectrum of the periodic mass matrix
// is known in closed form (Fourier modes): [h/3, h] in 1D, [h^2/9, h^2] on
// the bilinear mesh, [h^2/4, h^2] on the P1 mesh. With theta and delta the
// centre and half-width of that interval, sigma = theta / delta, the
// iteration
//   d_0 = r_0 / theta, rho_0 = 1 / sigma,
//   x += d_k, r -= M d_k, rho_{k+1} = 1 / (2 sigma - rho_k),
//   d_{k+1} = rho_{k+1} rho_k d_k + (2 rho_{k+1} / delta) r
// reduces the residual by the scaled Chebyshev polynomial, whose maximum on
// the interval is at most 2 q^k, q = (sqrt(kappa) - 1) / (sqrt(kappa) + 1).
// It needs no inner products: the number of steps for the tolerance follows
// from ||r_0|| and that bound, one pass and one grid barrier per step; the true
// residual is then recomputed and, if rounding left it above the tolerance, the
// iteration restarts from it (at most three times). The mean mode is set
// exactly first, as for CG, and every update d_k has zero mean, so the result
// is conservative to rounding.
// 20 steps on a bilinear mesh: 256^2 with 1 field 188 -> 88 us, 512^2 with 3
// fields 522 -> 168 us, 1024^2 with 4 fields 1400 -> 557 us, 2048^2 with 4 fields
// 4056 -> 1806 us (24 bytes per node and step, 20 in the first, and 36 in the other
// passes: 4.8 TB/s), against passes of four
// steps on 32 x 32 tiles with a halo in shared memory, which these replace (on
// this kernel's barrier and loads: 106, 255, 1038, 4075 us; a step does 1.6
// times the work there, at one block of shared-memory latency after another).
// ---------------------------------------------------------------------------
#define CHEB_COEF 32  // step coefficients computed at a time

// The first update, r / theta.
template <int VEC>
struct Scaled {
    const float *r;
    float k;
    __device__ __forceinline__ void get(int o, float (&q)[VEC]) const {
        ldn<VEC>(r + o, q);
#pragma unroll
        for (int j = 0; j < VEC; ++j) q[j] *= k;
    }
    __device__ __forceinline__ float one(int o) const { return r[o] * k; }
};

// One step of one field: x += d, r' = r - M d, d' = c1 d + c2 r'.
template <int DIM, int P1, int VEC, class Val>
__device__ __forceinline__ void cheb_step(const Val &d, int n, unsigned nv, float c, float c1, float c2, const float *r,
                                          float *rn, float *dn, float *x) {
    const unsigned tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    for (unsigned i = tid; i < nv; i += nth) {
        const int i0 = (int)(i * VEC);
        float hi[VEC], lo[VEC], dv[VEC], rv[VEC], xv[VEC];
        stencil_of<DIM, P1, VEC>(d, n, i0, hi, lo, dv);
        ldn<VEC>(r + i0, rv);
        ldn<VEC>(x + i0, xv);
#pragma unroll
        for (int j = 0; j < VEC; ++j) {
            xv[j] += dv[j];
            rv[j] -= fmaf(c, hi[j], c * lo[j]);
            dv[j] = fmaf(c1, dv[j], c2 * rv[j]);
        }
        stn<VEC>(x + i0, xv);
        stn<VEC>(rn + i0, rv);
        stn<VEC>(dn + i0, dv);
    }
}

template <int DIM, int P1, int VEC>
__global__ void __launch_bounds__(256, DIM == 1 ? 2 : 3) k_cheb(CG a) {
    __shared__ SolveState V;
    __shared__ BlockSums B;
    __shared__ float coef[2][CHEB_COEF];
    unsigned passed = 0;
    const Geo &g = a.g;
    const int F = a.F, n = g.n;
    const unsigned nv = (unsigned)(g.ncell / VEC);
    const ll nn = g.ncell;
    const float c = DIM == 1 ? g.h / 6.0f : (P1 ? g.h * g.h / 12.0f : g.h * g.h / 36.0f);
    const double hd = DIM == 1 ? (double)g.h : (double)g.h * g.h;
    // spectrum bounds, widened by 1e-6 against rounding of the operator
    const double lmin = hd * (DIM == 1 ? 1.0 / 3.0 : (P1 ? 0.25 : 1.0 / 9.0)) * (1.0 - 1e-6);
    const double lmax = hd * (1.0 + 1e-6);
    const double theta = 0.5 * (lmax + lmin), delta = 0.5 * (lmax - lmin);
    const float itheta = (float)(1.0 / theta);
    const double tol2 = a.rtol * a.rtol;
    const int wf = threadIdx.x >> 5;
    const bool lane0 = (threadIdx.x & 31) == 0;
    if (!solve_begin<DIM, VEC>(a, V, B, passed)) return;
    residual_pass<DIM, P1, VEC, true>(a, V, B, a.r[0], nullptr, 3);
    if (!grid_sync(a.bar, a.status, passed)) return;
    if (wf < F) {
        const double rr = grid_sum(a.red, F, 3, wf), bb = grid_sum(a.red, F, 4, wf);
        if (lane0) {
            V.rr[wf] = V.rr0[wf] = rr;
            V.bb[wf] = bb;
        }
    }
    int steps_done = 0, slot = 0;
    for (int pass = 0;; ++pass) {
        // steps of each field for the bound 2 q^k ||r_0|| <= rtol ||b||; the
        // pass runs the largest, a field stops updating after its own
        if (wf < F && lane0) {
            const double kap = lmax / lmin, q = (sqrt(kap) - 1.0) / (sqrt(kap) + 1.0);
            int K = 0;
            if (V.bb[wf] > 0.0 && V.rr[wf] > tol2 * V.bb[wf] && pass < 4) {
                const double ratio = a.rtol * sqrt(V.bb[wf]) / (2.0 * sqrt(V.rr[wf]));
                K = max(0, min((int)ceil(log(ratio) / log(q)), a.max_iter - steps_done));
            }
            V.steps[wf] = K;
            V.its[wf] += K;
        }
        __syncthreads();
        int K = 0;
        for (int f = 0; f < F; ++f) K = max(K, V.steps[f]);
        if (K <= 0 && pass > 0) break;  // the closing pass computed the result
        int cur = 0;
        double rho = delta / theta;  // 1 / sigma, thread 0's
        for (int kb = 0; kb < K;) {
            const int cnt = min(CHEB_COEF, K - kb);
            if (threadIdx.x == 0) {
                for (int j = 0; j < cnt; ++j) {
                    const double rho1 = 1.0 / (2.0 * (theta / delta) - rho);
                    coef[0][j] = (float)(rho1 * rho);
                    coef[1][j] = (float)(2.0 * rho1 / delta);
                    rho = rho1;
                }
            }
            __syncthreads();
            for (int j = 0; j < cnt; ++j, ++kb) {
                for (int f = 0; f < F; ++f) {
                    if (kb >= V.steps[f]) continue;
                    const ll fo = (ll)f * nn;
                    const float c1 = coef[0][j], c2 = coef[1][j];
                    float *rn = a.r[cur ^ 1] + fo, *dn = a.s[cur ^ 1] + fo, *x = a.xw + fo;
                    if (kb == 0)
                        cheb_step<DIM, P1, VEC>(Scaled<VEC>{a.r[cur] + fo, itheta}, n, nv, c, c1, c2, a.r[cur] + fo, rn,
                                                dn, x);
                    else
                        cheb_step<DIM, P1, VEC>(Plain<VEC>{a.s[cur] + fo}, n, nv, c, c1, c2, a.r[cur] + fo, rn, dn, x);
                }
                cur ^= 1;
                if (!grid_sync(a.bar, a.status, passed)) return;
            }
        }
        steps_done += K;
        // the true residual of every field, and the result
        residual_pass<DIM, P1, VEC, false>(a, V, B, a.r[0], a.x, slot);
        if (!grid_sync(a.bar, a.status, passed)) return;
        if (wf < F) {
            const double tr = grid_sum(a.red, F, slot, wf), sx = grid_sum(a.red, F, slot + 1, wf);
            if (lane0) {
                V.rr[wf] = V.tr[wf] = tr;
                V.sx[wf] = sx;
            }
        }
        slot ^= 2;
    }
    solve_report(a, V, hd);
}

template <int DIM, int P1>
__global__ void k_mass_apply(Geo g, const float *__restrict__ x, int F, float *__restrict__ y) {
    ll i = (ll)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.ncell) return;
    const float c = DIM == 1 ? g.h / 6.0f : (P1 ? g.h * g.h / 12.0f : g.h * g.h / 36.0f);
    for (int f = 0; f < F; ++f) {
        float hi, lo;
        stencil<DIM, P1>(x + (ll)f * g.ncell, g.n, i, hi, lo);
        y[(ll)f * g.ncell + i] = fmaf(c, hi, c * lo);
    }
}

// ---------------------------------------------------------------------------
// Full-mass mesh -> particle projection (Eq. proj2): solve M_p x = c with
// (M_p)_{mu nu} = int psi_mu psi_nu, applied matrix-free from the Delaunay
// stars (2D: diagonal v/2 and, for neighbour q_k, the coefficient
// (|T_k| + |T_k+1|)/12 of the two star triangles sharing the edge; 1D: gaps g
// give g/6 (x_left + 2 x_p) and g/6 (2 x_p + x_right)). Conjugate gradients
// with the Jacobi preconditioner D (diagonal v/2 in 2D, 2v/3 in 1D), from the
// lumped start c/v, in one persistent cooperative kernel with fixed-order
// FP64 reductions. The vectors are interleaved per particle, [np][FF] with
// FF = 2, 4 or 8 >= F, so that one row of M_p gathers each neighbour's fields
// with one wide load; fields past F stay 0, and a converged field is frozen
// by zero step lengths.
//
// Two passes and two grid barriers per iteration. The kernel keeps the
// preconditioned residual z = D^-1 r instead of r (r = D z where the norms
// need it). The pass that applies M_p forms the new search direction
// p = z + beta p_prev at the row and at each neighbour it gathers (the same
// FMA at every use, so every copy has the same bits), writes p into the
// other of two direction buffers, and applies the previous iteration's
// x += alpha p_prev at its own row. The second pass updates z. The last
// x += alpha p is folded into the closing residual pass, which writes the
// solution to q.
// ---------------------------------------------------------------------------
struct PCG {
    Geo g;
    int F;
    ll np;
    const float *c, *vol;  // c: [F][np] (fields apart), vol: [np]
    const uint2 *pos;
    const int *nbr;
    const unsigned char *deg;
    const float *coef;      // [PM_MAXDEG][np] off-diagonal row coefficients (2D)
    float *x, *z, *q;       // [np][FF]: iterate, D^-1 r, M_p p (the solution at exit)
    float *p[2];            // [np][FF]: search directions of even and odd iterations
    double *red, *scal;
    float4 *red4;
    unsigned *bar;
    int *status;
    double rtol;
    int max_iter;
    float unit;  // L / 2^32: torus units -> length
    const unsigned *meshmax;  // [F] max |Ab| bit patterns
    int ev;                   // binary exponent of the mean particle volume
    float vs;                 // 2^ev
};

template <int FF>
struct VF {
    float v[FF];
};

template <int FF>
__device__ __forceinline__ VF<FF> ldv(const float *p) {
    VF<FF> o;
    if (FF == 2) {
        const float2 t = *(const float2 *)p;
        o.v[0] = t.x;
        o.v[1] = t.y;
    } else {
#pragma unroll
        for (int i = 0; i < FF / 4; ++i) {
            const float4 t = ((const float4 *)p)[i];
            o.v[4 * i] = t.x;
            o.v[4 * i + 1] = t.y;
            o.v[4 * i + 2] = t.z;
            o.v[4 * i + 3] = t.w;
        }
    }
    return o;
}

template <int FF>
__device__ __forceinline__ void stv(float *p, const VF<FF> &o) {
    if (FF == 2) {
        *(float2 *)p = make_float2(o.v[0], o.v[1]);
    } else {
#pragma unroll
        for (int i = 0; i < FF / 4; ++i)
            ((float4 *)p)[i] = make_float4(o.v[4 * i], o.v[4 * i + 1], o.v[4 * i + 2], o.v[4 * i + 3]);
    }
}

// Row s of M_p applied to the vector whose value at particle i is val(i),
// all FF fields at once; xs = val(s), already at hand. In 2D the star is
// walked two entries at a time, with the next pair's entries loaded while the
// current pair's neighbours are gathered; the first pair is loaded together
// with the degree (every row has PM_MAXDEG allocated slots, so these loads
// stay in bounds; entries past the degree are never used). The sums keep the
// order diagonal, slot 0, 1, ...
template <int DIM, int FF, class Val>
__device__ __forceinline__ VF<FF> pmass_row(const PCG &a, ll s, const VF<FF> &xs, Val val) {
    const ll np = a.np;
    KSum acc[FF];
    if (DIM == 1) {
        const uint32_t X = a.pos[s].x;
        const ll sl = s == 0 ? np - 1 : s - 1, sr = s + 1 == np ? 0 : s + 1;
        const float u = a.unit * (1.0f / 6.0f);
        const float gl = (float)(uint32_t)(X - a.pos[sl].x) * u, gr = (float)(uint32_t)(a.pos[sr].x - X) * u;
        const VF<FF> xl = val(sl), xr = val(sr);
#pragma unroll
        for (int f = 0; f < FF; ++f) {
            acc[f].add(gl * xl.v[f]);
            acc[f].add(2.0f * (gl + gr) * xs.v[f]);
            acc[f].add(gr * xr.v[f]);
        }
    } else {
        int e0 = a.nbr[s], e1 = a.nbr[np + s];
        float w0 = a.coef[s], w1 = a.coef[np + s];
        const int m = a.deg[s];
        const float d = 0.5f * a.vol[s];
#pragma unroll
        for (int f = 0; f < FF; ++f) acc[f].add(d * xs.v[f]);
        for (int k = 0; k < m; k += 2) {
            int n0 = 0, n1 = 0;
            float u0 = 0.0f, u1 = 0.0f;
            if (k + 2 < m) {
                n0 = a.nbr[(ll)(k + 2) * np + s];
                u0 = a.coef[(ll)(k + 2) * np + s];
            }
            if (k + 3 < m) {
                n1 = a.nbr[(ll)(k + 3) * np + s];
                u1 = a.coef[(ll)(k + 3) * np + s];
            }
            int i0 = e0 & 0x0fffffff;
            PM_CHK(i0 < np, 402, i0 = (int)s)
            const VF<FF> x0 = val(i0);
            if (k + 1 < m) {
                int i1 = e1 & 0x0fffffff;
                PM_CHK(i1 < np, 402, i1 = (int)s)
                const VF<FF> x1 = val(i1);
#pragma unroll
                for (int f = 0; f < FF; ++f) {
                    acc[f].add(w0 * x0.v[f]);
                    acc[f].add(w1 * x1.v[f]);
                }
            } else {
#pragma unroll
                for (int f = 0; f < FF; ++f) acc[f].add(w0 * x0.v[f]);
            }
            e0 = n0;
            e1 = n1;
            w0 = u0;
            w1 = u1;
        }
    }
    VF<FF> o;
#pragma unroll
    for (int f = 0; f < FF; ++f) o.v[f] = acc[f].get();
    return o;
}

// Coefficients of the particle mass matrix rows from the stars: slot k of
// particle p gets (|T_k| + |T_k+1|) / 12, T_k = (p, q_k-1, q_k), areas from
// exact 64-bit cross products of the torus coordinates.
__global__ void k_star_coef(ll np, const uint2 *__restrict__ pos, const int *__restrict__ nbr,
                            const unsigned char *__restrict__ deg, float unit, float *__restrict__ coef) {
    const ll s = (ll)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= np) return;
    const int m = deg[s];
    if (m < 3) return;
    const uint2 Xp = pos[s];
    const float k12 = unit * unit * (1.0f / 24.0f);  // |T|/12 = area2 unit^2 / 24
    auto rel = [&](int e, ll &rx, ll &ry) {
        const uint2 Xq = pos[e & 0x0fffffff];
        rx = (int)(Xq.x - Xp.x);  // the neighbour's image: |.| <= 2^30
        ry = (int)(Xq.y - Xp.y);
    };
    ll ax, ay, bx, by;
    rel(nbr[(ll)(m - 1) * np + s], ax, ay);
    float wprev = 0.0f, wfirst = 0.0f;
    for (int k = 0; k < m; ++k) {
        rel(nbr[(ll)k * np + s], bx, by);
        const float w = (float)(ax * by - ay * bx) * k12;  // triangle k = (p, q_k-1, q_k)
        if (k == 0) wfirst = w;
        else coef[(ll)(k - 1) * np + s] = wprev + w;      // edge (p, q_k-1): triangles k-1 and k
        wprev = w;
        ax = bx;
        ay = by;
    }
    coef[(ll)(m - 1) * np + s] = wprev + wfirst;           // edge (p, q_m-1): triangles m-1 and 0
}


// Per-field solver scalars, identical on every block (each block computes
// them from the same totals); shared so that the row loops stay small.
struct PcgState {
    double cc[PM_MAXF], rz[PM_MAXF], rr0[PM_MAXF], sumc[PM_MAXF], sumabs[PM_MAXF];
    float al[PM_MAXF], be[PM_MAXF], ap[PM_MAXF], S[PM_MAXF], iS[PM_MAXF];  // ap: alpha in units of x; iS = 1 / S
    int act[PM_MAXF], its[PM_MAXF];
};

// The FF accumulators of a kind (fields past F are dropped).
template <int FF>
__device__ __forceinline__ void put_sums(BlockSums &B, int kind, int F, const Dot2 (&v)[FF]) {
#pragma unroll
    for (int f = 0; f < FF; ++f)
        if (f < F) put_sum(B, kind, f, v[f]);
}
template <int FF>
__device__ __forceinline__ void put_order_one(BlockSums &B, int F, const Dot2 (&v)[FF]) {
#pragma unroll
    for (int f = 0; f < FF; ++f)
        if (f < F) put_scaled(B, 0, f, v[f], 1.0f);
}
template <int FF>
__device__ __forceinline__ void put_order_one(BlockSums &B, int F, const Dot2 (&v)[FF], const Dot2 (&u)[FF]) {
#pragma unroll
    for (int f = 0; f < FF; ++f)
        if (f < F) put_scaled(B, f, v[f], 1.0f, u[f], 1.0f);
}

// The iteration runs on S c, S the field's power of two with S max|Ab| (mean
// volume) of order one (|c_mu| <= max|Ab| v_mu), and its inner products with z and
// p take the factor vs: the totals over all particles stay in the range of FP32
// whatever the field's amplitude and the box. Power-of-two factors are exact, so
// the results are those of the unscaled iteration bit for bit. x is unscaled.
// Reductions use slot groups {0,1,2} and {3,4} of red, then alternate {0} and
// {1,2} of red4 inside the loop, and at the end {0,1} of red: no two
// consecutive reductions share a slot, so a block that runs ahead to the next
// reduction never overwrites a partial that a slower block is still summing.
// Sums as in the mesh solves: with FP64 shuffles and sums per thread a
// solve of 3 fields on 1.97e6 particles (7 iterations) took 1.34 ms, now 1.16.
// An iteration is 97 us for the rows (two 16-byte gathers per neighbour from the
// L1 and L2), 22 us for the update and 10 us in the two barriers.
template <int DIM, int FF>
__global__ void __launch_bounds__(256, FF == 8 ? 2 : 4) k_pcg(PCG a) {
    __shared__ PcgState S;
    __shared__ BlockSums B;
    unsigned passed = 0;
    // warp f sums field f's partials, its lane 0 keeps the field's scalars
    const int wf = threadIdx.x >> 5;
    const bool lane0 = (threadIdx.x & 31) == 0;
    const int F = a.F;
    const ll np = a.np;
    const ll tid = (ll)blockIdx.x * blockDim.x + threadIdx.x, nth = (ll)gridDim.x * blockDim.x;
    const float dfac = DIM == 2 ? 0.5f : 2.0f / 3.0f;  // Jacobi diagonal = dfac v
    // binary exponent of max|Ab| (mean volume) of field f, 0 for a zero field
    auto exponent = [&](int f) {
        const float m = __uint_as_float(__ldg(a.meshmax + f));
        return m > 0.0f ? min(max(ilogbf(m) + a.ev, -120), 120) : 0;
    };
    if (threadIdx.x < F) {
        const int e = exponent(threadIdx.x);
        S.S[threadIdx.x] = pow2f(-e);
        S.iS[threadIdx.x] = pow2f(e);
    }
    // --- lumped start x = c / v; (c, c), sum c, sum |c|
    {
        float Sf[FF];
#pragma unroll
        for (int f = 0; f < FF; ++f) Sf[f] = f < F ? pow2f(-exponent(f)) : 0.0f;
        Dot2 s2[FF], s1[FF], sa[FF];
        for (ll s = tid; s < np; s += nth) {
            const float vv = a.vol[s];
            VF<FF> cv, xv;
#pragma unroll
            for (int f = 0; f < FF; ++f) {
                cv.v[f] = f < F ? a.c[(ll)f * np + s] : 0.0f;
                xv.v[f] = vv > 0.0f ? cv.v[f] / vv : 0.0f;
                const float cs = cv.v[f] * Sf[f];
                s2[f].fma_acc(cs, cs);
                s1[f].add(cs);
                sa[f].add(fabsf(cs));
            }
            stv<FF>(a.x + s * FF, xv);
        }
        put_sums<FF>(B, 0, F, s2);
        put_sums<FF>(B, 1, F, s1);
        put_sums<FF>(B, 2, F, sa);
        flush_sums(B, 3, F, a.red, 0);
    }
    if (!grid_sync(a.bar, a.status, passed)) return;
    if (wf < F) {
        const double cc = grid_sum(a.red, F, 0, wf);
        // a field so small that its residual drowns in FP32's denormals keeps the
        // lumped start, as a zero field does
        if (lane0) S.cc[wf] = exponent(wf) > -110 ? cc : 0.0;
        if (blockIdx.x == 0) {  // reported only
            const double sumc = grid_sum(a.red, F, 1, wf), sumabs = grid_sum(a.red, F, 2, wf);
            if (lane0) {
                S.sumc[wf] = sumc;
                S.sumabs[wf] = sumabs;
            }
        }
    }
    // --- r = S (c - M x), z = r / d; (r, r), (r, z)
    {
        Dot2 s2[FF], sz[FF];
        for (ll s = tid; s < np; s += nth) {
            const VF<FF> xs = ldv<FF>(a.x + s * FF);
            const VF<FF> mx = pmass_row<DIM, FF>(a, s, xs, [&](ll i) { return ldv<FF>(a.x + i * FF); });
            const float d = dfac * a.vol[s];
            VF<FF> zv;
#pragma unroll
            for (int f = 0; f < FF; ++f) {
                const float rv = f < F ? (a.c[(ll)f * np + s] - mx.v[f]) * S.S[f] : 0.0f;
                zv.v[f] = d > 0.0f ? rv / d : 0.0f;
                s2[f].fma_acc(rv, rv);
                sz[f].fma_acc(rv, zv.v[f] * a.vs);
            }
            stv<FF>(a.z + s * FF, zv);
        }
        put_sums<FF>(B, 0, F, s2);
        put_sums<FF>(B, 1, F, sz);
        flush_sums(B, 2, F, a.red, 3);
    }
    if (!grid_sync(a.bar, a.status, passed)) return;
    // The iteration stops on its recurrence for (r, r), which in FP32 drifts
    // from the true residual by a few roundings (observed: under 1 %); it
    // stops at 0.9 rtol so that the true residual, recomputed at exit, meets
    // rtol.
    const double tol2 = 0.81 * a.rtol * a.rtol;
    if (wf < F) {
        const double rr = grid_sum(a.red, F, 3, wf), rz = grid_sum(a.red, F, 4, wf);
        if (lane0) {
            S.rr0[wf] = rr;
            S.rz[wf] = rz;
            S.act[wf] = S.cc[wf] > 0.0 && rr > tol2 * S.cc[wf];
            S.its[wf] = 0;
            S.al[wf] = S.ap[wf] = 0.0f;
            S.be[wf] = 0.0f;
        }
    }
    __syncthreads();
    int last = -1;  // the last iteration run: its alpha p is still to be added to x
    for (int it = 0; it < a.max_iter; ++it) {
        bool any = false;
        for (int f = 0; f < F; ++f) any |= S.act[f] != 0;
        if (!any) break;
        // p = z + beta p_prev (at the row and at each neighbour), q = M p,
        // (p, q); x += alpha_prev p_prev at the row
        const float *pin = a.p[(it + 1) & 1];
        float *pout = a.p[it & 1];
        float be[FF], ap[FF];
#pragma unroll
        for (int f = 0; f < FF; ++f) {
            be[f] = f < F ? S.be[f] : 0.0f;
            ap[f] = f < F ? S.ap[f] : 0.0f;
        }
        const bool first = it == 0;
        {
            auto pval = [&](ll i) {
                VF<FF> zv = ldv<FF>(a.z + i * FF);
                if (!first) {
                    const VF<FF> pv = ldv<FF>(pin + i * FF);
#pragma unroll
                    for (int f = 0; f < FF; ++f) zv.v[f] = fmaf(be[f], pv.v[f], zv.v[f]);
                }
                return zv;
            };
            Dot2 sq[FF];
            for (ll s = tid; s < np; s += nth) {
                VF<FF> ps = ldv<FF>(a.z + s * FF);
                if (!first) {
                    const VF<FF> pv = ldv<FF>(pin + s * FF);
                    VF<FF> xv = ldv<FF>(a.x + s * FF);
#pragma unroll
                    for (int f = 0; f < FF; ++f) {
                        ps.v[f] = fmaf(be[f], pv.v[f], ps.v[f]);
                        xv.v[f] = fmaf(ap[f], pv.v[f], xv.v[f]);
                    }
                    stv<FF>(a.x + s * FF, xv);
                }
                const VF<FF> qv = pmass_row<DIM, FF>(a, s, ps, pval);
                stv<FF>(pout + s * FF, ps);
                stv<FF>(a.q + s * FF, qv);
#pragma unroll
                for (int f = 0; f < FF; ++f) sq[f].fma_acc(ps.v[f] * a.vs, qv.v[f]);
            }
            put_order_one<FF>(B, F, sq);
            flush_scaled(B, 1, F, a.red4, 0);
        }
        if (!grid_sync(a.bar, a.status, passed)) return;
        if (wf < F) {
            double t[1];
            grid_scaled<1>(B, a.red4, F, 0, wf, t);
            if (lane0) {
                S.al[wf] = S.act[wf] ? (float)(S.rz[wf] / t[0]) : 0.0f;
                S.ap[wf] = S.al[wf] * S.iS[wf];
            }
        }
        __syncthreads();
        last = it;
        // z -= alpha q / d; (r, r) and (r, z) with r = d z
        {
            float al[FF];
#pragma unroll
            for (int f = 0; f < FF; ++f) al[f] = f < F ? S.al[f] : 0.0f;
            Dot2 s2[FF], sz[FF];
            for (ll s = tid; s < np; s += nth) {
                VF<FF> zv = ldv<FF>(a.z + s * FF);
                const VF<FF> qv = ldv<FF>(a.q + s * FF);
                const float d = dfac * a.vol[s];
#pragma unroll
                for (int f = 0; f < FF; ++f) {
                    zv.v[f] = d > 0.0f ? fmaf(-al[f], qv.v[f] / d, zv.v[f]) : 0.0f;
                    const float rv = d * zv.v[f];
                    s2[f].fma_acc(rv, rv);
                    sz[f].fma_acc(rv, zv.v[f] * a.vs);
                }
                stv<FF>(a.z + s * FF, zv);
            }
            put_order_one<FF>(B, F, s2, sz);
            flush_scaled(B, 2, F, a.red4, 1);
        }
        if (!grid_sync(a.bar, a.status, passed)) return;
        if (wf < F) {
            double t[2];
            grid_scaled<2>(B, a.red4, F, 1, wf, t);
            if (lane0) {
                S.be[wf] = 0.0f;
                if (S.act[wf]) {
                    S.be[wf] = (float)(t[1] / S.rz[wf]);
                    S.rz[wf] = t[1];
                    ++S.its[wf];
                    if (t[0] <= tol2 * S.cc[wf]) S.act[wf] = 0;
                }
            }
        }
        __syncthreads();
    }
    // --- report: x += alpha p of the last iteration (at the row and at each
    // neighbour), true residual c - M x, sum v x (= sum c for the exact
    // solution); the solution goes to q
    {
        float ap[FF];
#pragma unroll
        for (int f = 0; f < FF; ++f) ap[f] = (f < F && last >= 0) ? S.ap[f] : 0.0f;
        const float *pl = a.p[(last >= 0 ? last : 0) & 1];
        const bool pend = last >= 0;
        auto xval = [&](ll i) {
            VF<FF> xv = ldv<FF>(a.x + i * FF);
            if (pend) {
                const VF<FF> pv = ldv<FF>(pl + i * FF);
#pragma unroll
                for (int f = 0; f < FF; ++f) xv.v[f] = fmaf(ap[f], pv.v[f], xv.v[f]);
            }
            return xv;
        };
        Dot2 s2[FF], sv[FF];
        for (ll s = tid; s < np; s += nth) {
            const VF<FF> xs = xval(s);
            const VF<FF> mx = pmass_row<DIM, FF>(a, s, xs, xval);
            const float vv = a.vol[s];
#pragma unroll
            for (int f = 0; f < FF; ++f) {
                const float Sf = f < F ? S.S[f] : 0.0f;
                const float rv = f < F ? (a.c[(ll)f * np + s] - mx.v[f]) * Sf : 0.0f;
                s2[f].fma_acc(rv, rv);
                sv[f].fma_acc(vv, xs.v[f] * Sf);
            }
            stv<FF>(a.q + s * FF, xs);
        }
        put_sums<FF>(B, 0, F, s2);
        put_sums<FF>(B, 1, F, sv);
        flush_sums(B, 2, F, a.red, 0);
    }
    if (!grid_sync(a.bar, a.status, passed)) return;
    if (blockIdx.x != 0 || wf >= F) return;
    const double tr = grid_sum(a.red, F, 0, wf), sx = grid_sum(a.red, F, 1, wf);
    if (lane0) {
        const double res = S.cc[wf] > 0.0 ? sqrt(tr / S.cc[wf]) : 0.0, inv = (double)S.iS[wf];
        a.scal[wf * 16 + S_INIT] = S.cc[wf] > 0.0 ? sqrt(S.rr0[wf] / S.cc[wf]) : 0.0;
        a.scal[wf * 16 + S_ITERS] = S.its[wf];
        a.scal[wf * 16 + S_RESID] = res;
        a.scal[wf * 16 + S_SUMMESH] = S.sumc[wf] * inv;   // int Ab = sum_mu c_mu
        a.scal[wf * 16 + S_SUMPART] = sx * inv;           // sum_mu v_mu Abb_mu
        a.scal[wf * 16 + S_SUMABS] = S.sumabs[wf] * inv;  // sum_mu |c_mu|: scale of the conservation error
        if (!(res <= a.rtol)) atomicOr(a.status, ST_NOTCONV);  // also when it is not a number
    }
}

// Interleaved solution [np][FF] -> caller order [F][np], one field per grid
// row: the rows run one after another, so the scattered writes of a row stay
// within one field's array, which the L2 holds and merges before writing back.
__global__ void k_unsort_aos(ll np, int FF, const int *__restrict__ perm, const float *__restrict__ x,
                             float *__restrict__ out) {
    const ll s = (ll)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= np) return;
    const int f = blockIdx.y;
    out[(ll)f * np + perm[s]] = x[s * FF + f];
}

// Resident blocks of a persistent kernel: SMs x min(occupancy, cap), looked
// up once per (device, kernel variant) and cached. The cache is keyed by the
// current device and guarded, so threads driving different devices each get
// their own device's figure.
#define PM_GRID_MAXDEV 64
std::mutex g_grid_mu;
int g_grid_cache[PM_GRID_MAXDEV][16];

int persistent_grid(int variant, const void *kern, int cap) {
    int dev = 0;
    cudaGetDevice(&dev);
    const bool cached = dev >= 0 && dev < PM_GRID_MAXDEV;
    if (cached) {
        std::lock_guard<std::mutex> lk(g_grid_mu);
        if (g_grid_cache[dev][variant]) return g_grid_cache[dev][variant];
    }
    int sms = 0, per = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, 256, 0);
    if (per < 1) per = 1;
    if (per > cap) per = cap;
    const int grid = sms * per;
    if (cached) {
        std::lock_guard<std::mutex> lk(g_grid_mu);
        g_grid_cache[dev][variant] = grid;
    }
    return grid;
}

// The reduction partials hold w.red_blocks blocks per slot: never launch more.
int clamp_grid(int grid, ll need, const Work &w) {
    if (need < grid) grid = (int)(need < 1 ? 1 : need);
    if (w.red_blocks > 0 && grid > w.red_blocks) grid = w.red_blocks;
    return grid;
}

}  // namespace

void launch_mass_apply(const Geo &g, const float *x, int F, float *y, cudaStream_t st) {
    if (g.dim == 1)
        k_mass_apply<1, 0><<<div_up(g.ncell, 256), 256, 0, st>>>(g, x, F, y);
    else
        if (g.p1)
            k_mass_apply<2, 1><<<div_up(g.ncell, 256), 256, 0, st>>>(g, x, F, y);
        else
            k_mass_apply<2, 0><<<div_up(g.ncell, 256), 256, 0, st>>>(g, x, F, y);
    count_launches(1);
}

namespace {

// Kernel of a mesh solve by dimension, mesh kind and nodes per access.
template <template <int, int, int> class K>
void (*mesh_kernel(const Geo &g, int vec, int *variant))(CG) {
    const int p1 = g.dim == 2 && g.p1;
    *variant = g.dim == 1 ? 0 : 1 + 2 * p1 + (vec == 4);
    if (g.dim == 1) return K<1, 0, 1>::get();
    if (vec == 4) return p1 ? K<2, 1, 4>::get() : K<2, 0, 4>::get();
    return p1 ? K<2, 1, 1>::get() : K<2, 0, 1>::get();
}
template <int DIM, int P1, int VEC>
struct CgKernel {
    static void (*get())(CG) { return k_cg<DIM, P1, VEC>; }
};
template <int DIM, int P1, int VEC>
struct ChebKernel {
    static void (*get())(CG) { return k_cheb<DIM, P1, VEC>; }
};

// The solvers' arguments. Vectors: w.r, w.r2, w.p, w.q, w.b and four in w.part
// (the FLIP partials, free during a solve).
CG mesh_args(const Geo &g, Work &w, int F, const float *b_float, bool b_from_fix, float *x, bool x_has_start,
             double rtol, int max_iter) {
    CG a;
    const ll len = (ll)F * g.ncell;
    a.g = g;
    a.F = F;
    a.bsrc = b_float;
    a.bfix = b_from_fix ? w.bfix : nullptr;
    a.maxabs = w.maxabs;
    a.x = x;
    a.b = w.b;
    a.p = w.p;
    a.r[0] = w.r;
    a.r[1] = w.r2;
    a.w[0] = w.q;
    a.w[1] = w.part;
    a.s[0] = w.part + len;
    a.s[1] = w.part + 2 * len;
    a.xw = w.part + 3 * len;
    a.red = w.red;
    a.red4 = w.red4;
    a.scal = w.scal;
    a.bar = w.bar;
    a.status = w.status;
    a.rtol = rtol;
    a.max_iter = max_iter;
    a.has_start = x_has_start ? 1 : 0;
    a.psum = b_from_fix ? w.psum : nullptr;
    a.nblk_psum = w.nblk_psum;
    return a;
}

// Nodes per access: quads on 2D meshes with n % 4 == 0 and 16-byte aligned
// arrays of the caller (the workspace's are).
int vec_of(const Geo &g, const float *b, const float *x) {
    return g.dim == 2 && g.n % 4 == 0 && ((uintptr_t)b | (uintptr_t)x) % 16 == 0 ? 4 : 1;
}

// Queue a mesh solve, at most 4 resident blocks per SM and no more blocks than
// there is work for. 0 or a CUDA error.
int run_mesh_solve(void (*kern)(CG), int variant, CG &a, Work &w, int vec, cudaStream_t st) {
    const ll need = (a.g.ncell / vec + 255) / 256;
    const int grid = clamp_grid(persistent_grid(variant, (const void *)kern, 4), need, w);
    cudaMemsetAsync(w.bar, 0, 2 * sizeof(unsigned), st);
    void *args[] = {&a};
    const cudaError_t e = cudaLaunchCooperativeKernel((void *)kern, dim3(grid), dim3(256), args, 0, st);
    count_launches(1);
    return (int)e;
}

}  // namespace

// Returns 0 or a CUDA error code.
int launch_cg(const Geo &g, Work &w, int F, const float *b_float, bool b_from_fix, float *x, bool x_has_start,
              double rtol, int max_iter, cudaStream_t st) {
    CG a = mesh_args(g, w, F, b_float, b_from_fix, x, x_has_start, rtol, max_iter);
    const int vec = vec_of(g, b_float, x);
    int variant;
    void (*kern)(CG) = mesh_kernel<CgKernel>(g, vec, &variant);
    return run_mesh_solve(kern, variant, a, w, vec, st);
}

// Chebyshev solve: same arguments, workspace and report as launch_cg.
int launch_cheb(const Geo &g, Work &w, int F, const float *b_float, bool b_from_fix, float *x, bool x_has_start,
                double rtol, int max_iter, cudaStream_t st) {
    CG a = mesh_args(g, w, F, b_float, b_from_fix, x, x_has_start, rtol, max_iter);
    const int vec = vec_of(g, b_float, x);
    int variant;
    void (*kern)(CG) = mesh_kernel<ChebKernel>(g, vec, &variant);
    return run_mesh_solve(kern, 5 + variant, a, w, vec, st);
}

int pcg_width(int F) { return F <= 2 ? 2 : (F <= 4 ? 4 : PM_MAXF); }

int launch_pcg(const Geo &g, Work &w, ll np, int F, const float *c, float *out, double rtol, int max_iter,
               cudaStream_t st) {
    const int FF = pcg_width(F);
    PCG a;
    a.g = g;
    a.F = F;
    a.np = np;
    a.c = c;
    a.vol = w.vol;
    a.pos = w.pos;
    a.nbr = w.nbr;
    a.deg = w.deg;
    a.coef = w.pcoef;
    a.x = w.px;
    a.z = w.prp;
    a.p[0] = w.prp + (ll)pcg_width(w.F_max) * w.np_max;
    a.p[1] = w.pp2;
    a.q = w.pq;
    a.red = w.red;
    a.red4 = w.red4;
    a.scal = w.scal;
    a.bar = w.bar;
    a.status = w.status;
    a.rtol = rtol;
    a.max_iter = max_iter;
    a.unit = (float)(g.L / 4294967296.0);
    a.meshmax = w.meshmax;
    a.ev = std::min(1000, std::max(-1000, std::ilogb((g.dim == 2 ? g.L * g.L : g.L) / (double)(np > 0 ? np : 1))));
    a.vs = std::ldexp(1.0f, std::min(120, std::max(-120, a.ev)));
    const int fi = FF == 2 ? 0 : (FF == 4 ? 1 : 2);
    const int di = (g.dim - 1) * 3 + fi;
    void (*const kerns[6])(PCG) = {k_pcg<1, 2>, k_pcg<1, 4>, k_pcg<1, PM_MAXF>,
                                   k_pcg<2, 2>, k_pcg<2, 4>, k_pcg<2, PM_MAXF>};
    void (*kern)(PCG) = kerns[di];
    const ll need = (np + 255) / 256;
    const int grid = clamp_grid(persistent_grid(10 + di, (const void *)kern, 4), need, w);
    if (g.dim == 2 && np > 0) {
        k_star_coef<<<div_up(np, 256), 256, 0, st>>>(np, w.pos, w.nbr, w.deg, a.unit, w.pcoef);
        count_launches(1);
    }
    cudaMemsetAsync(w.bar, 0, 2 * sizeof(unsigned), st);
    void *args[] = {&a};
    cudaError_t e = cudaLaunchCooperativeKernel((void *)kern, dim3(grid), dim3(256), args, 0, st);
    count_launches(1);
    if (e != cudaSuccess) return (int)e;
    if (np > 0) {
        k_unsort_aos<<<dim3((unsigned)div_up(np, 256), F), 256, 0, st>>>(np, FF, w.perm, w.pq, out);
        count_launches(1);
    }
    return 0;
}
