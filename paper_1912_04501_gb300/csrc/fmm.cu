// The near image sum by a fast multipole method: O(N) instead of the direct
// 9 N^2 (or 4 N^2) pair evaluations.
//
// In complex notation (z the target, n its normal, zeta a source, q = sigma w
// its strength, r = z - zeta) the traction kernel of Eq. Gt is
//   c r = -(1/4pi) [ 2 n Re(q / r) + conj(n) conj( conj(q) / r + q conj(r) / r^2 ) ],
// so the sum over a set of sources needs two analytic functions of z,
//   A(z) = sum q / r,   F(z) = sum conj(q) / r + q conj(r) / r^2 = E(z) - conj(w) A'(z),
// w = z - c about a box centre c.  About the centre of the sources' box
//   A = sum_k a_k / w^{k+1},  a_k = sum q eta^k,  eta = zeta - c,
//   E = sum_k e_k / w^{k+1},  e_k = sum conj(q) eta^k - k q conj(eta) eta^{k-1};
// about the centre of the targets' box A and E are power series.  Moving the
// centre by d adds -conj(d) A' to E; a shifted series is then diagonal powers
// around a constant matrix of binomials, because
//   1 / (z0 + w)^{k+1} = sum_l C(k+l, l) (-w)^l / z0^{k+l+1}.
// Lengths are in units of the box side of the level throughout.
//
// Boxes: a uniform grid of squares of side h over the rectangle that holds the
// cell's nodes, and coarser levels of twice the side each.  Lattice images are
// the same boxes shifted, so a (target box, source box, image) triple is near
// when the centres differ by less than two sides in both coordinates.  Far
// triples whose parents are near (every far triple at the top) pass by
// expansions; near triples of the finest level are evaluated pair by pair.
// Truncation: 0.547^P for two box corners that face each other, P = 24 in single
// precision, P = 48 in double; of a corner's whole far sum 2e-16 in double.
//
// Three arithmetics: float, double, and double-float (df, bie_internal.cuh) for
// the double-float application, all of it on the FP32 pipe.
//
// What bounds it.  Single precision: latency up to some 10^4 nodes, then the
// pair sum (about 20 instructions per pair, a few hundred pairs per target);
// double: the FP64 pipe in the translations (a warp DFMA per 19 cycles and SM).
// Whole applications on GB300, direct sum before and this now: single precision
// 32.8 -> 0.185 ms on the 400-ellipse cell (102400 nodes), 0.94 -> 0.095 ms at
// 16000 nodes, 0.21 -> 0.077 ms at 6400; double-float 340 -> 1.10 ms at 102400;
// FP64 12.2 -> 0.85 ms at 6400.  The single-precision application's error
// against 64 bits falls (5.0e-7 -> 1.9e-7 in the 2-norm at 6400 nodes): near pairs are
// differenced exactly.  So does the double-float application's against FP64
// (4.1e-13 -> 8.5e-14; 1 to 400 bodies, shear to 0.45), whose walls and proxies were
// summed in FP64 before.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "bie_internal.cuh"

namespace bie {

template <typename R>
struct __align__(8) C2 {
    R x, y;
};
template <>
struct __align__(16) C2<double> {
    double x, y;
};
// coefficient pair of one order: (a, e)
template <typename R>
struct __align__(16) V4 {
    R x, y, z, w;
};

template <typename R>
__device__ __forceinline__ C2<R> cmul(C2<R> a, C2<R> b) {
    return {renorm(fma_(a.x, b.x, -(a.y * b.y))), renorm(fma_(a.x, b.y, a.y * b.x))};
}
template <typename R>
__device__ __forceinline__ C2<R> czero() {
    return {R(0), R(0)};
}
template <typename R>
__device__ __forceinline__ V4<R> vzero() {
    return {R(0), R(0), R(0), R(0)};
}
// s += c v
template <typename R>
__device__ __forceinline__ void axpy(V4<R>& s, R c, const V4<R>& v) {
    s.x = fma_(c, v.x, s.x);
    s.y = fma_(c, v.y, s.y);
    s.z = fma_(c, v.z, s.z);
    s.w = fma_(c, v.w, s.w);
}
// acc += p s (both series by one complex power)
template <typename R>
__device__ __forceinline__ void add_scaled(V4<R>& acc, C2<R> p, const V4<R>& s) {
    const R sx = renorm(s.x), sy = renorm(s.y), sz = renorm(s.z), sw = renorm(s.w);
    acc.x = fma_(p.x, sx, fma_(-p.y, sy, acc.x));
    acc.y = fma_(p.x, sy, fma_(p.y, sx, acc.y));
    acc.z = fma_(p.x, sz, fma_(-p.y, sw, acc.z));
    acc.w = fma_(p.x, sw, fma_(p.y, sz, acc.w));
}
template <typename R>
__device__ __forceinline__ V4<R> scaled(C2<R> p, C2<R> a, C2<R> e) {
    const C2<R> va = cmul(p, a), ve = cmul(p, e);
    return {va.x, va.y, ve.x, ve.y};
}
template <typename R>
__device__ __forceinline__ V4<R> vadd(const V4<R>& a, const V4<R>& b) {
    return {a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w};
}

// Powers z^k, 0 <= k < 64, from three small tables (radix 4, 4, 4): entries
// 0..2 z, z^2, z^3; 3..5 z^4, z^8, z^12; 6..8 z^16, z^32, z^48.
constexpr int kPowTab = 9;
template <typename R>
__device__ __forceinline__ void pow_table(C2<R> z, C2<R>* t) {
    t[0] = z;
    t[1] = cmul(z, z);
    t[2] = cmul(t[1], z);
    t[3] = cmul(t[1], t[1]);
    t[4] = cmul(t[3], t[3]);
    t[5] = cmul(t[4], t[3]);
    t[6] = cmul(t[4], t[4]);
    t[7] = cmul(t[6], t[6]);
    t[8] = cmul(t[7], t[6]);
}
template <typename R>
__device__ __forceinline__ C2<R> pow_at(const C2<R>* t, int k) {
    const int a = k & 3, b = (k >> 2) & 3, c = k >> 4;
    C2<R> r{R(1), R(0)};
    if (a) r = t[a - 1];
    if (b) r = cmul(r, t[2 + b]);
    if (c) r = cmul(r, t[5 + c]);
    return r;
}

// storage type <-> arithmetic: strengths (double in memory for double)
template <typename R>
struct FmmTypes {
    static constexpr int P = kFmmP64;
};
template <>
struct FmmTypes<float> {
    static constexpr int P = kFmmP32;
};
constexpr int kFmmItems = 96;  // orders x groups of sources or entries per warp: three per lane
static_assert(kFmmItems % kFmmP32 == 0 && kFmmItems % kFmmP64 == 0, "items");

__host__ __device__ inline int fmm_ix(int4 b) { return b.z & 0xffff; }
__host__ __device__ inline int fmm_iy(int4 b) { return (b.z >> 16) & 0xffff; }

// ---------------------------------------------------------------------------
// per geometry: sort the sources (and, with the doubled cell, the targets) by box
// ---------------------------------------------------------------------------
// Position of source record r (relative to the cell centre): a node, or with
// the doubled cell one of its four images.
__device__ __forceinline__ double2 fmm_source(const FmmGeom& g, const Cell& cl, int r, int mul) {
    if (mul == 1) return make_double2(g.x[r] - cl.C[0], g.y[r] - cl.C[1]);
    const int i = r >> 2, sh = img_shift(g.imc[i], r & 3);
    return make_double2((g.x[i] + cl.sx[sh]) - cl.C[0], (g.y[i] + cl.sy[sh]) - cl.C[1]);
}

__device__ __forceinline__ int fmm_leaf(const FmmCell& f, double2 p) {
    int ix = (int)floor((p.x - f.ox) * f.inv_h), iy = (int)floor((p.y - f.oy) * f.inv_h);
    ix = max(0, min(f.gx[0] - 1, ix));
    iy = max(0, min(f.gy[0] - 1, iy));
    return f.off[0] + iy * f.gx[0] + ix;
}

// Leaf of every record, and the record counts of its box and the box's ancestors.
// set 0: sources, set 1: targets (doubled cell only).  With `owned` also the counts of the
// nodes n0 <= i < n1 and of the cell's first: a target partition's own targets.
// Bound by the atomics of the
// coarse boxes, which every record adds to: a warp's records of one box (neighbours on
// a curve, mostly) go as one, 102400 records in 9 us against 148.
__global__ void k_fmm_bin(FmmGeom g, const Cell* __restrict__ cells, const FmmCell* __restrict__ fc,
                          const int4* __restrict__ box, int n, int mul, int targets, int* __restrict__ leaf,
                          int* __restrict__ count, int n0, int n1, int* __restrict__ owned) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    int b = -1;
    bool own = false;
    if (r < n) {
        const int c = g.node_cell[mul == 1 ? r : r >> 2];
        const Cell& cl = cells[c];
        const double2 p = targets ? make_double2(g.xw[r] - cl.C[0], g.yw[r] - cl.C[1]) : fmm_source(g, cl, r, mul);
        b = fmm_leaf(fc[c], p);
        leaf[r] = b;
        own = owned && ((r >= n0 && r < n1) || r == cl.node_off);
    }
    const unsigned mine = __ballot_sync(0xffffffffu, own);
    while (__any_sync(0xffffffffu, b >= 0)) {
        const unsigned same = __match_any_sync(0xffffffffu, b);
        if (b >= 0) {
            if ((threadIdx.x & 31) == __ffs(same) - 1) {
                atomicAdd(count + b, __popc(same));
                if (same & mine) atomicAdd(owned + b, __popc(same & mine));
            }
            b = box[b].w;
        }
    }
}

// Exclusive scan of the leaf counts (one CTA); cursor starts as a copy.
__global__ void __launch_bounds__(1024)
k_fmm_scan(const int* __restrict__ count, int n, int* __restrict__ start, int* __restrict__ cursor) {
    __shared__ int s[32];
    __shared__ int carry;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (t == 0) carry = 0;
    __syncthreads();
    for (int b = 0; b < n; b += 1024) {
        const int v = b + t < n ? count[b + t] : 0;
        int x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s[w] = x;
        __syncthreads();
        if (w == 0) {
            int y = s[lane];
            for (int o = 1; o < 32; o <<= 1) {
                const int z = __shfl_up_sync(0xffffffffu, y, o);
                if (lane >= o) y += z;
            }
            s[lane] = y;
        }
        __syncthreads();
        const int e = carry + x - v + (w ? s[w - 1] : 0);
        if (b + t < n) start[b + t] = cursor[b + t] = e;
        __syncthreads();
        if (t == 1023) carry = e + v;
        __syncthreads();
    }
    if (t == 0) start[n] = carry;
}

__global__ void k_fmm_fill(const int* __restrict__ leaf, int n, int* __restrict__ cursor, int* __restrict__ raw) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n) raw[atomicAdd(cursor + leaf[r], 1)] = r;
}

// Orders every box's records by index (the order of the atomics is not
// reproducible, the sums must be) and stores the sorted positions: double-float
// relative to the cell centre, and double.  One CTA per leaf.
__global__ void __launch_bounds__(64)
k_fmm_sort(FmmGeom g, const Cell* __restrict__ cells, const int4* __restrict__ box, const int* __restrict__ start,
           const int* __restrict__ raw, int mul, int targets, int* __restrict__ perm, float4* __restrict__ pos,
           double2* __restrict__ pos64) {
    const int s0 = start[blockIdx.x], s1 = start[blockIdx.x + 1];
    if (s0 == s1) return;
    const Cell& cl = cells[box[blockIdx.x].x];
    for (int k = s0 + threadIdx.x; k < s1; k += blockDim.x) {
        const int r = raw[k];
        int rank = 0;
        for (int j = s0; j < s1; ++j) rank += raw[j] < r;
        const double2 p = targets ? make_double2(g.xw[r] - cl.C[0], g.yw[r] - cl.C[1]) : fmm_source(g, cl, r, mul);
        perm[s0 + rank] = r;
        if (pos) {
            float4 v;
            split_df(p.x, v.x, v.y);
            split_df(p.y, v.z, v.w);
            pos[s0 + rank] = v;
        }
        if (pos64) pos64[s0 + rank] = p;
    }
}

// ---------------------------------------------------------------------------
// upward: moments of every box
// ---------------------------------------------------------------------------
// (p - c) / h for double-float positions: the high parts' difference is exact,
// or rounded relative to itself
__device__ __forceinline__ C2<float> fmm_local(float4 p, float4 c, float inv_h) {
    return {((p.x - c.x) + (p.y - c.y)) * inv_h, ((p.z - c.z) + (p.w - c.w)) * inv_h};
}

__host__ __device__ inline double2 fmm_centre(const FmmCell& f, int level, int ix, int iy) {
    const double H = f.h * (1 << level);
    return make_double2(f.ox + (ix + 0.5) * H, f.oy + (iy + 0.5) * H);
}

// Constant tables of one precision (host: fmm_tables): the matrix C(k + l, l)
// [k][l], the binomials C(m, k) [k][m], and for a child at (+-1/4, +-1/4) of its
// parent delta^m and (1 / (2 delta))^k.
template <typename R>
struct FmmTab {
    const R *hankel, *binom, *binomt;  // binomt: [k][m] = C(k, m)
    const C2<R>*dpow, *gpow;  // [quadrant][order]
};

template <typename R>
__device__ __forceinline__ C2<R> fmm_offset(const FmmTree& t, int s, double2 c, float4 cf, double inv_h);
template <>
__device__ __forceinline__ C2<float> fmm_offset<float>(const FmmTree& t, int s, double2 c, float4 cf, double inv_h) {
    return fmm_local(t.spos[s], cf, (float)inv_h);
}
template <>
__device__ __forceinline__ C2<double> fmm_offset<double>(const FmmTree& t, int s, double2 c, float4 cf, double inv_h) {
    const double2 p = t.spos64[s];
    return {(p.x - c.x) * inv_h, (p.y - c.y) * inv_h};
}
template <>
__device__ __forceinline__ C2<df> fmm_offset<df>(const FmmTree& t, int s, double2 c, float4 cf, double inv_h) {
    const double2 p = t.spos64[s];
    return {df((p.x - c.x) * inv_h), df((p.y - c.y) * inv_h)};
}

// One CTA per box.  Boxes of at most kFmmDirect sources (every leaf) sum their
// moments from the sources, rows of leaves at a time; a leaf's CTA also gathers
// the strengths q = sigma w in sorted order.  A warp takes 32 sources at a time; a
// lane sums three (order, group of sources) items, eta^k = eta^(k % 4)
// (eta^4)^(k / 4) from two small tables per source.  Larger boxes' moments come
// from their children's, a warp per child, in the CTA of the last child to finish,
// and so on up: each such level waits for the one below (some 3 us), which is why
// only boxes too large to sum in that time do it (single precision; the double
// sums cost more, so their line is lower).
// The CTAs past the boxes form the bodies' moments (F_b, tau_b), one body each,
// with the per-node records that velocities and the direct walls read.
struct FmmBodies {
    const double *x, *y, *body;
    const int* body_cell;
    float4* src32;   // cell-centred, or null
    Src64* src64;    // or null
    double* bodyF;
};

__device__ void fmm_body(const FmmBodies& p, int b, const Cell* cells, const double2* sigma, const double* w) {
    __shared__ double red[33];
    const double* bd = p.body + 8 * b;
    const double xc = bd[2], yc = bd[3];
    const int n = (int)bd[5], off = (int)bd[6];
    const Cell& cl = cells[p.body_cell[b]];
    double fx = 0, fy = 0, tq = 0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int i = off + k;
        const double2 sg = sigma[i];
        const double wi = w[i], X = p.x[i], Y = p.y[i];
        const double qx = sg.x * wi, qy = sg.y * wi;
        fx += qx;
        fy += qy;
        tq += -(Y - yc) * qx + (X - xc) * qy;
        if (p.src32) p.src32[i] = make_float4((float)(X - cl.C[0]), (float)(Y - cl.C[1]), (float)qx, (float)qy);
        if (p.src64) p.src64[i] = Src64{X, Y, qx, qy};
    }
    fx = block_sum_d(fx, red);
    fy = block_sum_d(fy, red);
    tq = block_sum_d(tq, red);
    if (threadIdx.x == 0) {
        p.bodyF[3 * b] = fx;
        p.bodyF[3 * b + 1] = fy;
        p.bodyF[3 * b + 2] = tq;
    }
}

// Measured (whole application, us, on a stream of the context's own): single precision
// at 6400 / 102400 nodes 64.4 / 167 with 128, 67.1 / 170 with 512, 80.9 / 188 with 2048;
// double-float 270 / 1119 with 64, 262 / 1132 with 256, 278 / 1178 with 512.
template <typename R>
constexpr int kFmmDirect = sizeof(R) == 4 ? 128 : 256;

template <typename R>
__global__ void __launch_bounds__(128)
k_fmm_up(FmmTree t, const Cell* __restrict__ cells, const double2* sigma, const double* __restrict__ w,
         int shift, C2<R>* __restrict__ sq, V4<R>* __restrict__ mp, unsigned* __restrict__ ticket, FmmTab<R> tab,
         FmmBodies bodies) {
    constexpr int P = FmmTypes<R>::P, G = kFmmItems / P, PER = 32 / G, HI = P / 4;
    struct Tables {
        C2<R> lo[4][4][33], hi[4][HI][33], q[4][32], s[4][32];
    };
    __shared__ __align__(16) Tables sh;
    __shared__ bool s_last;
    auto& s_lo = sh.lo;
    auto& s_hi = sh.hi;
    auto& s_q = sh.q;
    auto& s_s = sh.s;
    // the tables' space holds the warps' sums (6 numbers per item), then the
    // children's translated series
    R* s_sum = reinterpret_cast<R*>(&sh);
    static_assert(4 * kFmmItems * 6 * sizeof(R) <= sizeof(Tables), "sums");
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x >= t.nbox) {
        fmm_body(bodies, blockIdx.x - t.nbox, cells, sigma, w);
        return;
    }
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    constexpr int kDirect = kFmmDirect<R>;
    const int b = blockIdx.x;
    int4 bx = t.box[b];
    const int total = t.scount[b];
    if (bx.y > 0 && total > kDirect) return;  // from its children
    const FmmCell& f = t.cells[bx.x];
    if (!cells[bx.x].active) return;
    const int lv0 = bx.y;
    if (total > 0) {
        const double2 c = sizeof(R) == 4 ? make_double2(0.0, 0.0) : fmm_centre(f, lv0, fmm_ix(bx), fmm_iy(bx));
        const float4 cf = sizeof(R) == 4 ? t.centre[b] : make_float4(0.f, 0.f, 0.f, 0.f);
        const double inv_h = f.inv_h / (1 << lv0);
        // per item the moments of q_x and q_y and of s = q conj(eta)
        C2<R> X[3], Y[3], D[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) X[r] = Y[r] = D[r] = czero<R>();
        // the rows of leaves in turn, chunks of 32 sources dealt to the warps
        const int gx0 = f.gx[0], x0 = fmm_ix(bx) << lv0, x1 = min(gx0, x0 + (1 << lv0)), y0 = fmm_iy(bx) << lv0,
                  y1 = min(f.gy[0], y0 + (1 << lv0)), off0 = f.off[0];
        int turn = 0;
        for (int y = y0; y < y1; ++y) {
        const int s0 = t.sstart[off0 + y * gx0 + x0], s1 = t.sstart[off0 + y * gx0 + x1];
        const int first = (wid - turn) & 3;
        turn += (s1 - s0 + 31) >> 5;
        for (int k0 = s0 + 32 * first; k0 < s1; k0 += 128) {
            const int s = k0 + lane, cnt = min(32, s1 - k0);
            C2<R> eta = czero<R>(), q = czero<R>();
            if (lane < cnt) {
                eta = fmm_offset<R>(t, s, c, cf, inv_h);
                const int i = t.sperm[s] >> shift;
                const double2 sg = sigma[i];
                const double wi = w[i];
                q = {R(sg.x * wi), R(sg.y * wi)};
                if (lv0 == 0) sq[s] = q;
            }
            const C2<R> e2 = cmul(eta, eta), e4 = cmul(e2, e2);
            __syncwarp();
            s_lo[wid][0][lane] = {R(1), R(0)};
            s_lo[wid][1][lane] = eta;
            s_lo[wid][2][lane] = e2;
            s_lo[wid][3][lane] = cmul(e2, eta);
            C2<R> h{R(1), R(0)};
#pragma unroll
            for (int a = 0; a < HI; ++a) {
                s_hi[wid][a][lane] = h;
                h = cmul(h, e4);
            }
            s_q[wid][lane] = q;
            s_s[wid][lane] = {fma_(q.x, eta.x, q.y * eta.y), fma_(q.y, eta.x, -(q.x * eta.y))};
            __syncwarp();
            for (int j = 0; j < PER; ++j) {
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    const int it = lane + 32 * r, k = it % P, js = (it / P) * PER + j;
                    if (js < cnt) {
                        const C2<R> qj = s_q[wid][js], sj = s_s[wid][js];
                        const C2<R> pw = cmul(s_lo[wid][k & 3][js], s_hi[wid][k >> 2][js]);
                        X[r].x = fma_(qj.x, pw.x, X[r].x);
                        X[r].y = fma_(qj.x, pw.y, X[r].y);
                        Y[r].x = fma_(qj.y, pw.x, Y[r].x);
                        Y[r].y = fma_(qj.y, pw.y, Y[r].y);
                        D[r].x = fma_(sj.x, pw.x, fma_(-sj.y, pw.y, D[r].x));
                        D[r].y = fma_(sj.x, pw.y, fma_(sj.y, pw.x, D[r].y));
                    }
                }
            }
            __syncwarp();
        }
        }
        __syncthreads();
        // the sums of 4 warps x G groups, in order; number n of order k at n P + k
        R* mine = s_sum + (size_t)wid * kFmmItems * 6;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int it = lane + 32 * r;
            const R v[6] = {X[r].x, X[r].y, Y[r].x, Y[r].y, D[r].x, D[r].y};
#pragma unroll
            for (int n = 0; n < 6; ++n) mine[n * kFmmItems + it] = renorm(v[n]);
        }
        __syncthreads();
        for (int e = tid; e < 6 * P; e += 128) {
            const int n = e / P, k = e % P;
            R v = s_sum[n * kFmmItems + k];
            for (int g = 1; g < 4 * G; ++g)
                v = v + s_sum[(size_t)(g / G) * kFmmItems * 6 + n * kFmmItems + (g % G) * P + k];
            // only this thread reads (n, k) of warp 0's group 0 below this line's write
            s_sum[n * kFmmItems + k] = v;
        }
        __syncthreads();
        // a = X + i Y, b = X - i Y, e_k = b_k - k d_{k-1}
        if (tid < P) {
            const int k = tid;
            const R xx = s_sum[k], xy = s_sum[kFmmItems + k], yx = s_sum[2 * kFmmItems + k],
                    yy = s_sum[3 * kFmmItems + k];
            R dx(0), dy(0);
            if (k) {
                dx = s_sum[4 * kFmmItems + k - 1];
                dy = s_sum[5 * kFmmItems + k - 1];
            }
            mp[(size_t)b * P + k] = {xx - yy, xy + yx, (xx + yy) - R(k) * dx, (xy - yx) - R(k) * dy};
        }
    }
    // parents: the series translated from the four children, a warp each
    V4<R>* s_v = reinterpret_cast<V4<R>*>(&sh);  // [4][P] scaled, then [4][P] translated
    static_assert(8 * P * sizeof(V4<R>) <= sizeof(Tables), "series");
    for (int level = lv0; bx.w >= 0; ++level) {
        const int parent = bx.w;
        if (t.scount[parent] <= kDirect) return;  // summed by its own CTA
        const int px = fmm_ix(t.box[parent]), py = fmm_iy(t.box[parent]);
        const int nx = min(2, f.gx[level] - 2 * px), ny = min(2, f.gy[level] - 2 * py);
        __threadfence();
        __syncthreads();
        if (tid == 0) s_last = atomicAdd(ticket + parent, 1u) == (unsigned)(nx * ny) - 1;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        if (tid == 0) ticket[parent] = 0u;
        bx = t.box[parent];
        const int jx = wid & 1, jy = wid >> 1;
        const int child = f.off[level] + (2 * py + jy) * f.gx[level] + 2 * px + jx;
        const bool have = jx < nx && jy < ny && t.scount[child] > 0;
        V4<R>* v = s_v + wid * P;
        V4<R>* o = s_v + (4 + wid) * P;
        if (have) {
            // child's unit is half the parent's: v_k = a_k (1 / (2 delta))^k; with
            // delta = (+-1/2, +-1/2) in the child's unit, e_k - conj(delta) k a_{k-1}
            const R hx(jx ? 0.5 : -0.5), hy(jy ? 0.5 : -0.5);
            for (int k = lane; k < P; k += 32) {
                const R* src = reinterpret_cast<const R*>(mp + (size_t)child * P + k);
                const C2<R> a{ldcg(src), ldcg(src + 1)};
                C2<R> e{ldcg(src + 2), ldcg(src + 3)};
                if (k) {
                    const R pax = ldcg(src - 4), pay = ldcg(src - 3);
                    e.x = e.x - R(k) * fma_(hx, pax, hy * pay);
                    e.y = e.y - R(k) * fma_(hx, pay, -(hy * pax));
                }
                v[k] = scaled(tab.gpow[wid * P + k], a, e);
            }
            __syncwarp();
            for (int m = lane; m < P; m += 32) {
                V4<R> s = vzero<R>();
                // C(m, k), 0 for k > m: whole rows keep the loads in flight
                const int rows = m < 32 ? min(P, 32) : P;
#pragma unroll 8
                for (int k = 0; k < rows; ++k) axpy(s, tab.binom[(size_t)k * P + m], v[k]);
                V4<R> r = vzero<R>();
                add_scaled(r, tab.dpow[wid * P + m], s);
                o[m] = r;
            }
        }
        if (!have)
            for (int m = lane; m < P; m += 32) o[m] = vzero<R>();
        __syncthreads();
        if (tid < P) {
            const V4<R>* q = s_v + 4 * P + tid;
            mp[(size_t)parent * P + tid] = vadd(vadd(q[0], q[P]), vadd(q[2 * P], q[3 * P]));
        }
    }
}

// ---------------------------------------------------------------------------
// beside the translations: wall discrepancy and close pairs
// ---------------------------------------------------------------------------
// The wall discrepancy (Sec. 6.2 step 2, the far-image form of k_disc) from the
// moments of the boxes of one level, which the six far images of a wall point are well
// away from (fmm_wall_side).
// With u = 1 / W, W = (p - c) / H, per box
//   velocity   4 pi mu u = -a_0 log|w| + (sum_{k>0} a_k u^k / k + conj(sum_{k>0} e_k u^k / k)
//                          + conj(conj(W) A) + a_0) / 2,
//   traction  -4 pi H T = 2 n Re A + conj(n (E - conj(W) A')).
// The single-layer sum took 12 N (4 m) kernel evaluations with a logarithm
// each: 3.5 ms of the FP64 pipe at 102400 nodes, 0.23 ms at 6400.
// the sums' type: float, or double (double-float too)
template <typename R>
struct WallReal {
    typedef double T;
};
template <>
struct WallReal<float> {
    typedef float T;
};
template <typename S, typename R>
__device__ __forceinline__ S to_real(R a) {
    return (S)to_double(a);
}
template <>
__device__ __forceinline__ float to_real<float, float>(float a) {
    return a;
}

template <typename R>
__device__ __forceinline__ void wall_box(const V4<R>* mp, C2<R> W, typename WallReal<R>::T ln_w, R n0, R n1,
                                         const R* inv_k, typename WallReal<R>::T* v) {
    typedef typename WallReal<R>::T S;
    constexpr int P = FmmTypes<R>::P;
    const R s = rcp(fma_(W.x, W.x, W.y * W.y));
    const C2<R> u{renorm(W.x * s), renorm(-(W.y * s))};
    C2<R> A = czero<R>(), B = czero<R>(), E = czero<R>(), L = czero<R>(), M = czero<R>();
    auto step = [&](C2<R>& a, R vx, R vy) {
        a = {renorm(fma_(a.x, u.x, fma_(-a.y, u.y, vx))), renorm(fma_(a.x, u.y, fma_(a.y, u.x, vy)))};
    };
    for (int k = P - 1; k > 0; --k) {
        const V4<R> m = mp[k];
        const R k1(k + 1), ik = inv_k[k];
        step(A, m.x, m.y);
        step(B, k1 * m.x, k1 * m.y);
        step(E, m.z, m.w);
        step(L, ik * m.x, ik * m.y);
        step(M, ik * m.z, ik * m.w);
    }
    const V4<R> m = mp[0];
    step(A, m.x, m.y);
    step(B, m.x, m.y);
    step(E, m.z, m.w);
    L = cmul(L, u);
    M = cmul(M, u);
    A = cmul(A, u);
    E = cmul(E, u);
    B = cmul(cmul(B, u), u);  // -A'
    // F = E - conj(W) A'
    const C2<R> F{E.x + fma_(W.x, B.x, W.y * B.y), E.y + fma_(W.x, B.y, -(W.y * B.x))};
    // conj(conj(W) A) = W conj(A)
    const R wx = fma_(W.x, A.x, W.y * A.y), wy = fma_(W.y, A.x, -(W.x * A.y));
    v[0] = S(0.5) * to_real<S>(L.x + M.x + wx + m.x) - ln_w * to_real<S>(m.x);
    v[1] = S(0.5) * to_real<S>(L.y - M.y + wy + m.y) - ln_w * to_real<S>(m.y);
    v[2] = -to_real<S>(R(2) * n0 * A.x + (n0 * F.x - n1 * F.y));
    v[3] = -to_real<S>(R(2) * n1 * A.x - (n0 * F.y + n1 * F.x));
}
constexpr int kWallImages = 6;

// One warp per task: first (cell, wall point, far image), writing
// gpart[((cell 7) + image) 8m + 4 wp + component]; then one per cell for its
// total force (slot 6); then the close pairs (Sec. 6.3), C_p sigma into psum[p].
struct SideArgs {
    int ncell, m, walls, ctas;  // ctas: four tasks each
    const int* npairs;          // on the device (a replayed capture meets later geometries), or null: none
    const double *wall, *bodyF;
    const double *x, *y;
    double* gpart;
    const int4* pairs;
    const int* node_cell;
    const long long* blk_off;
    const void* blocks;  // float (single precision: on q = sigma w), or double
    const double* body;
    const double2* sigma;
    const double* w;
    void* psum;
};

// B: the blocks' type
template <typename B>
__device__ __forceinline__ void close_pair(const SideArgs& a, const Cell* cells, int p, int lane) {
    const int4 pr = a.pairs[p];
    if (!cells[a.node_cell[pr.x]].active) return;
    const int n = (int)a.body[8 * pr.y + 5], off = (int)a.body[8 * pr.y + 6];
    const B* C = reinterpret_cast<const B*>(a.blocks) + a.blk_off[p];
    B bx = 0, by = 0;
#pragma unroll 4
    for (int j = lane; j < n; j += 32) {
        const double2 sg = a.sigma[off + j];
        B sx = (B)sg.x, sy = (B)sg.y;
        if constexpr (sizeof(B) == 4) {
            const float wj = (float)a.w[off + j];
            sx *= wj;
            sy *= wj;
        }
        const B c0 = C[3 * j], c1 = C[3 * j + 1], c2 = C[3 * j + 2];
        bx = fma(c0, sx, fma(c1, sy, bx));
        by = fma(c1, sx, fma(c2, sy, by));
    }
    for (int o = 16; o > 0; o >>= 1) {
        bx += __shfl_xor_sync(0xffffffffu, bx, o);
        by += __shfl_xor_sync(0xffffffffu, by, o);
    }
    if (lane) return;
    if constexpr (sizeof(B) == 4) reinterpret_cast<float2*>(a.psum)[p] = make_float2(bx, by);
    else reinterpret_cast<double2*>(a.psum)[p] = make_double2(bx, by);
}

template <typename B>
__global__ void __launch_bounds__(128) k_close_pairs(SideArgs a, const Cell* __restrict__ cells) {
    for (int p = blockIdx.x * 4 + (threadIdx.x >> 5); p < *a.npairs; p += 4 * a.ctas)
        close_pair<B>(a, cells, p, threadIdx.x & 31);
}

// The same for one far image node by node, for a cell whose bodies reach so near to the
// walls' images that no box is well away from them (FmmCell::wall -1: centres set far
// outside the cell): velocity times 4 pi mu and traction times -pi, by k_disc's formulas,
// in single precision (cell-centred) or double.
template <typename S>
__device__ __forceinline__ void wall_nodes(const SideArgs& a, const Cell& cl, S px, S py, S n0, S n1, int lane, S* v) {
    constexpr bool F32 = sizeof(S) == 4;
    for (int j = cl.node_off + lane; j < cl.node_off + cl.n_nodes; j += 32) {
        const double2 sg = a.sigma[j];
        const double w = a.w[j];
        const S qx = (S)(sg.x * w), qy = (S)(sg.y * w);
        const S rx = px - (F32 ? (S)(a.x[j] - cl.C[0]) : (S)a.x[j]), ry = py - (F32 ? (S)(a.y[j] - cl.C[1]) : (S)a.y[j]);
        const S r2 = rx * rx + ry * ry, inv = S(1) / r2, rq = (rx * qx + ry * qy) * inv, l = S(-0.5) * log(r2);
        const S cc = (rx * n0 + ry * n1) * rq * inv;
        v[0] += l * qx + rx * rq;
        v[1] += l * qy + ry * rq;
        v[2] += cc * rx;
        v[3] += cc * ry;
    }
}

template <typename R>
__device__ void side_tasks(const SideArgs& a, const FmmTree& t, const Cell* cells, const V4<R>* mp, int cta) {
    constexpr int P = FmmTypes<R>::P;
    typedef typename WallReal<R>::T S;
    __shared__ R s_inv[P];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int task = cta * 4 + wid, step = 4 * a.ctas;
    if (a.walls) {
        for (int k = threadIdx.x; k < P; k += 128) s_inv[k] = R(k ? 1.0 / k : 0.0);
        __syncthreads();
        const int per = 2 * a.m * kWallImages + 1;
        if (task < a.ncell * per) {
            const int ci = task / per, q = task % per;
            const Cell& cl = cells[ci];
            if (!cl.active) return;
            double* gp = a.gpart + (size_t)ci * 7 * 8 * a.m;
            if (q == per - 1) {
                double fx = 0, fy = 0;
                for (int b = cl.body_off + lane; b < cl.body_off + cl.n_bodies; b += 32) {
                    fx += a.bodyF[3 * b];
                    fy += a.bodyF[3 * b + 1];
                }
                fx = warp_sum_d(fx);
                fy = warp_sum_d(fy);
                if (lane < 2) gp[6 * 8 * (size_t)a.m + lane] = lane ? fy : fx;
                return;
            }
            const int wp = q / kWallImages, im = q % kWallImages;
            const FmmCell& f = t.cells[ci];
            const int lv = f.wall, gx = f.gx[max(lv, 0)], n = gx * f.gy[max(lv, 0)];
            const double* wt = a.wall + ((size_t)ci * 2 * a.m + wp) * kWallStride;
            S v[4] = {0, 0, 0, 0};
            if (lv < 0) {
                if constexpr (sizeof(R) == 4) {
                    const float* wf = reinterpret_cast<const float*>(wt + 16);
                    wall_nodes<float>(a, cl, wf[2 * im], wf[2 * im + 1], wf[12], wf[13], lane, v);
                } else {
                    wall_nodes<double>(a, cl, wt[2 * im], wt[2 * im + 1], wt[12], wt[13], lane, v);
                }
            } else if constexpr (sizeof(R) == 4) {  // cell-centred single precision
                const float* wf = reinterpret_cast<const float*>(wt + 16);
                const float H = (float)f.h * (1 << lv), iH = 1.f / H;
                const float px = wf[2 * im] - (float)f.ox, py = wf[2 * im + 1] - (float)f.oy, n0 = wf[12], n1 = wf[13];
                const float lh = logf(H);
                for (int e = lane; e < n; e += 32) {
                    const int b = f.off[lv] + e;
                    if (t.scount[b] == 0) continue;
                    const C2<R> W{fmaf(px, iH, -(e % gx + 0.5f)), fmaf(py, iH, -(e / gx + 0.5f))};
                    float o[4];
                    wall_box<R>(mp + (size_t)b * P, W, 0.5f * logf(W.x * W.x + W.y * W.y) + lh, n0, n1, s_inv, o);
#pragma unroll
                    for (int k = 0; k < 4; ++k) v[k] += o[k];
                }
            } else {
                const double H = f.h * (1 << lv), iH = f.inv_h / (1 << lv);
                const double px = wt[2 * im] - cl.C[0] - f.ox, py = wt[2 * im + 1] - cl.C[1] - f.oy;
                const double lh = log(H);
                const R n0(wt[12]), n1(wt[13]);
                for (int e = lane; e < n; e += 32) {
                    const int b = f.off[lv] + e;
                    if (t.scount[b] == 0) continue;
                    const double wx = fma(px, iH, -(e % gx + 0.5)), wy = fma(py, iH, -(e / gx + 0.5));
                    double o[4];
                    wall_box<R>(mp + (size_t)b * P, C2<R>{R(wx), R(wy)}, 0.5 * log(wx * wx + wy * wy) + lh, n0, n1,
                                s_inv, o);
#pragma unroll
                    for (int k = 0; k < 4; ++k) v[k] += o[k];
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
            if (lane < 4) {
                const double sg = im < 3 ? 1.0 : -1.0;
                const double g = lane < 2 ? sg / (4.0 * kPi * cl.mu)
                                          : (lv < 0 ? -sg / kPi : sg * f.inv_h / (4.0 * kPi * (1 << lv)));
                gp[(size_t)im * 8 * a.m + 4 * wp + lane] =
                    g * (double)(lane == 0 ? v[0] : (lane == 1 ? v[1] : (lane == 2 ? v[2] : v[3])));
            }
            return;
        }
        task -= a.ncell * per;
        step -= a.ncell * per;
    }
    if (!a.npairs) return;
    for (const int n = *a.npairs; task < n; task += step) {
        if constexpr (sizeof(R) == 4) close_pair<float>(a, cells, task, lane);
        else close_pair<double>(a, cells, task, lane);
    }
}

// ---------------------------------------------------------------------------
// across: local expansion of every target box from the far boxes whose
// parents are near
// ---------------------------------------------------------------------------
// Which boxes are near is decided in whole numbers: an image shift is rounded
// to 2^-16 of a leaf side (kFmmBits), and boxes ix and jx of a level (unit
// 2^(kFmmBits + level)) are near in one coordinate when their centres under the
// shift are less than two units apart.  The same numbers at every level make a
// level's far list, its children's and the pair sum's rows partition the pairs
// exactly; the FP64 pipe, which took 6000 cycles per box to list its far boxes,
// is left to the sums.
constexpr int kFmmBits = 16;
__device__ __forceinline__ bool fmm_close(int ix, int jx, int s, int level) {
    return abs(((ix - jx) << (kFmmBits + level)) - s) < (2 << (kFmmBits + level));
}
// the first of the (at most four) boxes near ix
__device__ __forceinline__ int fmm_first(int ix, int s, int level) { return ix - 1 + ((-s) >> (kFmmBits + level)); }
__device__ __forceinline__ int fmm_shift(double s, double inv_h) { return __double2int_rn(s * inv_h * (1 << kFmmBits)); }
constexpr int kFmmShares = 4;            // most CTAs a box's list is split over

// Near rows of a leaf's targets, compacted in (image, row) order by one warp.
__device__ __forceinline__ int fmm_ranges(const FmmTree& t, const FmmCell& f, const int2* shift, int4 bx, int nimg,
                                          FmmRange* out, int lane) {
    int n = 0;
    for (int q0 = 0; q0 < 4 * nimg; q0 += 32) {
        const int q = q0 + lane;
        FmmRange r{0, 0, 0};
        if (q < 4 * nimg) {
            r.im = nimg == 1 ? 4 : q >> 2;
            const int sx = shift[r.im].x, sy = shift[r.im].y;
            const int ix = fmm_ix(bx), iy = fmm_iy(bx);
            const int jy = fmm_first(iy, sy, 0) + (q & 3);
            if (fmm_close(iy, jy, sy, 0) && jy >= 0 && jy < f.gy[0]) {
                int x0 = fmm_first(ix, sx, 0), x1 = x0 + 3;
                if (!fmm_close(ix, x0, sx, 0)) ++x0;
                if (!fmm_close(ix, x1, sx, 0)) --x1;
                x0 = max(x0, 0);
                x1 = min(x1, f.gx[0] - 1);
                if (x0 <= x1) {
                    const int row = f.off[0] + jy * f.gx[0];
                    r.s0 = t.sstart[row + x0];
                    r.s1 = t.sstart[row + x1 + 1];
                }
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, r.s1 > r.s0);
        if (r.s1 > r.s0) out[n + __popc(m & ((1u << lane) - 1))] = r;
        n += __popc(m);
    }
    return n;
}

// Per geometry and box: the far boxes to translate from (box | image << 28, in a
// fixed order; at most 9 images x 64 children of near parents, and 9 x 16 at the
// top) and, for a leaf, its near rows (ranges of sorted records); per cell the
// image shifts in leaf sides as float pairs.
__global__ void __launch_bounds__(128)
k_fmm_lists(FmmTree t, const Cell* __restrict__ cells, int nimg) {
    __shared__ int2 s_shift[9];
    __shared__ int s_n[4];
    const int b = blockIdx.x, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int4 bx = t.box[b];
    const FmmCell& f = t.cells[bx.x];
    const Cell& cl = cells[bx.x];
    const int level = bx.y, ix = fmm_ix(bx), iy = fmm_iy(bx);
    const bool top = level == f.nlev - 1;
    const int gx = f.gx[level], gy = f.gy[level], off = f.off[level];
    if (threadIdx.x < 9) {
        const double sx = cl.sx[threadIdx.x], sy = cl.sy[threadIdx.x];
        s_shift[threadIdx.x] = make_int2(fmm_shift(sx, f.inv_h), fmm_shift(sy, f.inv_h));
        if (top && ix == 0 && iy == 0) {
            float4 v;
            split_df(sx * f.inv_h, v.x, v.y);
            split_df(sy * f.inv_h, v.z, v.w);
            t.shift[9 * bx.x + threadIdx.x] = v;
        }
    }
    __syncthreads();
    if (t.wanted[b] == 0) {
        if (threadIdx.x == 0) t.nfar[b] = 0;
        if (threadIdx.x == 0 && level == 0) t.nnear[b] = 0;
        return;
    }
    if (level == 0 && wid == 0) {
        const int n = fmm_ranges(t, f, s_shift, bx, nimg, t.near + (size_t)b * kFmmRanges, lane);
        if (lane == 0) t.nnear[b] = n;
    }
    const int per = top ? gx * gy : 64, ncand = per * nimg;
    int listed = 0;
    for (int q0 = 0; q0 < ncand; q0 += 128) {
        const int q = q0 + threadIdx.x;
        bool far = false;
        int entry = 0;
        if (q < ncand) {
            const int im = nimg == 1 ? 4 : q / per, e = nimg == 1 ? q : q % per;
            const int2 sh = s_shift[im];
            int jx, jy;
            bool ok = true;
            if (top) {
                jx = e % gx;
                jy = e / gx;
            } else {
                // children of the (up to 4 x 4) near parents
                const int kx = ix >> 1, ky = iy >> 1;
                const int px = fmm_first(kx, sh.x, level + 1) + (e & 7) / 2;
                const int py = fmm_first(ky, sh.y, level + 1) + (e >> 3) / 2;
                ok = fmm_close(kx, px, sh.x, level + 1) && fmm_close(ky, py, sh.y, level + 1);
                jx = 2 * px + (e & 1);
                jy = 2 * py + ((e >> 3) & 1);
            }
            if (ok && jx >= 0 && jx < gx && jy >= 0 && jy < gy) {
                const int src = off + jy * gx + jx;
                far = !(fmm_close(ix, jx, sh.x, level) && fmm_close(iy, jy, sh.y, level)) && t.scount[src] > 0;
                entry = src | (im << 28);
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, far);
        if (lane == 0) s_n[wid] = __popc(m);
        __syncthreads();
        int at = listed;
        for (int k = 0; k < 4; ++k) {
            if (k < wid) at += s_n[k];
            listed += s_n[k];
        }
        if (far) t.far[(size_t)b * kFmmFar + at + __popc(m & ((1u << lane) - 1))] = entry;
        __syncthreads();
    }
    if (threadIdx.x == 0) t.nfar[b] = listed;
}

// The first CTAs take the side tasks above.  Then one CTA per (target box of any
// level, share of its list): its warps translate the listed boxes in turn.
// Single precision: an entry per warp and step, lane l holding order l and its
// row of the matrix.  Double: two entries per warp and step, three (entry, order)
// items per lane.  The shares' sums are separate (one slot of loc each): without
// shares the longest lists (90 boxes, at the coarse levels) held up the launch.
template <typename R>
__global__ void __launch_bounds__(128)
k_fmm_m2l(FmmTree t, const Cell* cells, const V4<R>* mp, V4<R>* loc, FmmTab<R> tab, int shares,
          SideArgs side) {
    constexpr int P = FmmTypes<R>::P;
    constexpr bool F32 = sizeof(R) == 4;
    constexpr int ENT = F32 ? 1 : 2, ITEMS = F32 ? 1 : 3;
    __shared__ C2<R> s_tab[4][F32 ? 32 : 16][kPowTab], s_z[4][F32 ? 32 : 16];
    __shared__ V4<R> s_v[4][ENT][P + (F32 ? 0 : 1)];
    __shared__ int s_src[4][F32 ? 32 : 16];
    if ((int)blockIdx.x < side.ctas) {
        pdl_wait();
        pdl_trigger();
        side_tasks<R>(side, t, cells, mp, blockIdx.x);
        return;
    }
    const int id = blockIdx.x - side.ctas, b = id / shares, share = id % shares;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int4 bx = t.box[b];
    const Cell& cl = cells[bx.x];
    if (t.wanted[b] == 0 || !cl.active) {
        pdl_wait();
        return;
    }
    const int4 grid = t.grid[b];  // (first box of the level, its width, ...)
    const int* far = t.far + (size_t)b * kFmmFar;
    const int mine = (t.nfar[b] - share + shares - 1) / shares;  // this share's entries
    const int level = bx.y, ix = fmm_ix(bx), iy = fmm_iy(bx), off = grid.x, gx = grid.y;
    V4<R> acc[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) acc[r] = vzero<R>();
    R row[F32 ? P : 1];  // single precision: lane l's row of the matrix in registers
    if constexpr (F32) {
#pragma unroll
        for (int k = 0; k < P; ++k) row[k] = lane < P ? tab.hankel[(size_t)k * P + lane] : R(0);
    }
    if (mine <= 0) pdl_wait();
    {
        constexpr int GRP = F32 ? 32 : 16;  // entries whose power tables a warp holds
        for (int g0 = 0; g0 * 4 < mine; g0 += GRP) {
            // the warp's entries of this group: e = (g0 + n) 4 + wid (single), or
            // consecutive pairs (double)
            const int stepn = ENT == 1 ? 1 : 2;
            auto entry = [&](int n) { return ENT == 1 ? (g0 + n) * 4 + wid : ((g0 + n) / 2 * 4 + wid) * 2 + (n & 1); };
            __syncwarp();
            if (lane < GRP && entry(lane) < mine) {
                // target centre minus source centre in sides, its inverse's powers
                const int v = far[entry(lane) * shares + share], src = v & 0xfffffff, im = (unsigned)v >> 28;
                const int jy = (src - off) / gx, jx = src - off - jy * gx;
                s_src[wid][lane] = src;
                const float4 sh = t.shift[9 * bx.x + im];  // leaf sides
                R x, y;
                if constexpr (F32) {
                    const float iu = 1.f / (1 << level);
                    x = (((float)((ix - jx) << level) - sh.x) - sh.y) * iu;
                    y = (((float)((iy - jy) << level) - sh.z) - sh.w) * iu;
                } else {
                    const double inv = t.cells[bx.x].inv_h / (1 << level);
                    x = R((ix - jx) - cl.sx[im] * inv);
                    y = R((iy - jy) - cl.sy[im] * inv);
                }
                s_z[wid][lane] = {x, y};
                C2<R> u;
                if constexpr (F32) {
                    const float sc = 1.f / (x * x + y * y);
                    u = {x * sc, -y * sc};
                } else {
                    const double dx = to_double(x), dy = to_double(y), sc = rcp64(dx * dx + dy * dy);
                    u = {R(dx * sc), R(-dy * sc)};
                }
                pow_table(u, s_tab[wid][lane]);
            }
            __syncwarp();
            pdl_wait();
            pdl_trigger();
            if constexpr (F32) {
                V4<R> nxt = vzero<R>();
                if (entry(0) < mine && lane < P) nxt = mp[(size_t)s_src[wid][0] * P + lane];
                for (int n = 0; n < GRP && entry(n) < mine; ++n) {
                    const C2<R> z = s_z[wid][n];
                    const V4<R> m4 = nxt;
                    const int en = entry(n + 1);
                    if (n + 1 < GRP && en < mine && lane < P) nxt = mp[(size_t)s_src[wid][n + 1] * P + lane];
                    const C2<R> u = s_tab[wid][n][0];
                    C2<R> pw = pow_at(s_tab[wid][n], lane);
                    C2<R> pa{__shfl_up_sync(0xffffffffu, m4.x, 1), __shfl_up_sync(0xffffffffu, m4.y, 1)};
                    if (lane == 0) pa = czero<R>();
                    // e_k + conj(z0) k a_{k-1}
                    const C2<R> ev{m4.z + R(lane) * (z.x * pa.x + z.y * pa.y),
                                   m4.w + R(lane) * (z.x * pa.y - z.y * pa.x)};
                    if (lane < P) s_v[wid][0][lane] = scaled(pw, C2<R>{m4.x, m4.y}, ev);
                    __syncwarp();
                    V4<R> s = vzero<R>();
#pragma unroll
                    for (int k = 0; k < P; ++k) axpy(s, row[k], s_v[wid][0][k]);
                    __syncwarp();
                    pw = cmul(pw, u);
                    if (lane & 1) pw = {-pw.x, -pw.y};
                    add_scaled(acc[0], pw, s);
                }
            } else {
                for (int n = 0; n < GRP && entry(n) < mine; n += stepn) {
                    C2<R> pw[ITEMS];
#pragma unroll
                    for (int r = 0; r < ITEMS; ++r) {
                        const int it = lane + 32 * r, en = it / P, k = it % P, e = entry(n + en);
                        V4<R> v = vzero<R>();
                        pw[r] = czero<R>();
                        if (e < mine) {
                            const V4<R>* src4 = mp + (size_t)s_src[wid][n + en] * P + k;
                            const V4<R> m4 = *src4;
                            C2<R> ev{m4.z, m4.w};
                            if (k) {
                                const C2<R> z = s_z[wid][n + en];
                                const R pax = src4[-1].x, pay = src4[-1].y;
                                ev.x = ev.x + R(k) * fma_(z.x, pax, z.y * pay);
                                ev.y = ev.y + R(k) * fma_(z.x, pay, -(z.y * pax));
                            }
                            pw[r] = pow_at(s_tab[wid][n + en], k);
                            v = scaled(pw[r], C2<R>{m4.x, m4.y}, ev);
                            pw[r] = cmul(pw[r], s_tab[wid][n + en][0]);
                            if (k & 1) pw[r] = {-pw[r].x, -pw[r].y};
                        }
                        s_v[wid][en][k] = v;
                    }
                    __syncwarp();
                    V4<R> s[ITEMS];
#pragma unroll
                    for (int r = 0; r < ITEMS; ++r) s[r] = vzero<R>();
#pragma unroll 2
                    for (int k = 0; k < P; ++k) {
#pragma unroll
                        for (int r = 0; r < ITEMS; ++r) {
                            const int it = lane + 32 * r;
                            axpy(s[r], tab.hankel[(size_t)k * P + it % P], s_v[wid][it / P][k]);
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int r = 0; r < ITEMS; ++r) add_scaled(acc[r], pw[r], s[r]);
                }
            }
        }
    }
    // the warps' sums, in order
    V4<R>* flat = &s_v[wid][0][0];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int it = lane + 32 * r;
        if (it < ENT * P) flat[it] = V4<R>{renorm(acc[r].x), renorm(acc[r].y), renorm(acc[r].z), renorm(acc[r].w)};
    }
    __syncthreads();
    for (int k = threadIdx.x; k < P; k += 128) {
        V4<R> s = vzero<R>();
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int en = 0; en < ENT; ++en) s = vadd(s, (&s_v[q][0][0])[en * P + k]);
        loc[((size_t)share * t.nbox + b) * P + k] = s;
    }
}

// ---------------------------------------------------------------------------
// down: at every target, the ancestors' expansions moved to its leaf and the
// near boxes pair by pair
// ---------------------------------------------------------------------------
// The local expansion of a leaf with its ancestors' moved to its centre, in
// s_l[0] (the shares of k_fmm_m2l added on the way): warp w moves levels w,
// w + 4, ... (level 0 is the leaf's own); every thread of the 128 takes part.
template <typename R>
__device__ __forceinline__ void fmm_local_to_leaf(const FmmTree& t, const FmmCell& f, int4 bx, const V4<R>* loc,
                                                  int shares, const FmmTab<R>& tab, V4<R> (*s_l)[FmmTypes<R>::P],
                                                  C2<R> (*s_pw)[2][kPowTab], int wid, int lane) {
    constexpr int P = FmmTypes<R>::P, ROWS = (P + 31) / 32;
    V4<R>* s_v = s_l[wid];
    V4<R> acc[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) acc[r] = vzero<R>();
    for (int level = wid; level < f.nlev; level += 4) {
        const int jx = fmm_ix(bx) >> level, jy = fmm_iy(bx) >> level;
        const V4<R>* src = loc + (size_t)(f.off[level] + jy * f.gx[level] + jx) * P;
        auto get = [&](int l) {
            V4<R> m = src[l];
            for (int q = 1; q < shares; ++q) m = vadd(m, src[(size_t)q * t.nbox * P + l]);
            return m;
        };
        if (level == 0) {
#pragma unroll
            for (int r = 0; r < ROWS; ++r)
                if (lane + 32 * r < P) acc[r] = get(lane + 32 * r);
            continue;
        }
        // leaf centre minus ancestor centre, in the ancestor's unit (exact)
        const float u = 1.f / (1 << level);
        const float dx = (fmm_ix(bx) + 0.5f) * u - (jx + 0.5f), dy = (fmm_iy(bx) + 0.5f) * u - (jy + 0.5f);
        const C2<R>*pd = s_pw[wid][0], *pg = s_pw[wid][1];  // powers of delta and of 2^-level / delta
        __syncwarp();
        if (lane < 2) {
            const R i2 = lane ? R(double(u) / ((double)dx * dx + (double)dy * dy)) : R(1);
            pow_table(C2<R>{R(dx) * i2, R(lane ? -dy : dy) * i2}, s_pw[wid][lane]);
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int l = lane + 32 * r;
            if (l < P) {
                const V4<R> m = get(l);
                C2<R> e{m.z, m.w};
                if (l + 1 < P) {  // e_l - conj(d) (l + 1) a_{l+1}
                    const V4<R> n = get(l + 1);
                    e.x = e.x - R(l + 1) * fma_(R(dx), n.x, R(dy) * n.y);
                    e.y = e.y - R(l + 1) * fma_(R(dx), n.y, -(R(dy) * n.x));
                }
                s_v[l] = scaled(pow_at(pd, l), C2<R>{m.x, m.y}, e);
            }
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int m = lane + 32 * r;
            if (m < P) {
                V4<R> s = vzero<R>();
                // C(l, m), 0 for l < m: whole rows keep the loads in flight
#pragma unroll 8
                for (int l = r ? 32 : 0; l < P; ++l) axpy(s, tab.binomt[(size_t)l * P + m], s_v[l]);
                // to the leaf's unit: 2^-level per order and one more for the field's own scale
                C2<R> p = pow_at(pg, m);
                p = {p.x * R(u), p.y * R(u)};
                add_scaled(acc[r], p, s);
            }
        }
        __syncwarp();
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
        if (lane + 32 * r < P)
            s_v[lane + 32 * r] = V4<R>{renorm(acc[r].x), renorm(acc[r].y), renorm(acc[r].z), renorm(acc[r].w)};
    __syncthreads();
    for (int k = threadIdx.x; k < P; k += 128) s_l[0][k] = vadd(vadd(s_l[0][k], s_l[1][k]), vadd(s_l[2][k], s_l[3][k]));
    __syncthreads();
}

// Traction, times 4 pi h, of the local expansion's orders r, r + STEP, ... at W
// (leaf units) with normal n; the STEP residues add up to the whole.
template <typename R, int STEP>
__device__ __forceinline__ C2<R> fmm_local_at(const V4<R>* c, C2<R> W, int r, R nx, R ny) {
    constexpr int P = FmmTypes<R>::P;
    static_assert(P % STEP == 0, "residues");
    C2<R> S = W;  // W^STEP
#pragma unroll
    for (int k = 1; k < STEP; k <<= 1) S = cmul(S, S);
    // sums over l = r + STEP j of a_l, l a_l and e_l: A and E times W^r, and A'
    // times W^(r - 1) (r = 0: its j = 0 term is nil, the rest times W^(STEP - 1))
    C2<R> A = czero<R>(), B = czero<R>(), E = czero<R>();
    auto step = [&](C2<R>& a, R vx, R vy) {
        a = {renorm(fma_(a.x, S.x, fma_(-a.y, S.y, vx))), renorm(fma_(a.x, S.y, fma_(a.y, S.x, vy)))};
    };
#pragma unroll 2
    for (int l = P - STEP + r; l >= 0; l -= STEP) {
        const V4<R> v = c[l];
        const R fl(l);
        step(A, v.x, v.y);
        if (l) step(B, fl * v.x, fl * v.y);
        step(E, v.z, v.w);
    }
    if constexpr (STEP > 1) {
        C2<R> p{R(1), R(0)}, pb{R(1), R(0)};
        for (int k = 0; k < r; ++k) p = cmul(p, W);
        for (int k = 1; k < (r ? r : STEP); ++k) pb = cmul(pb, W);
        A = cmul(A, p);
        E = cmul(E, p);
        B = cmul(B, pb);
    }
    // F = E - conj(W) A';  -(2 n Re A + conj(n F))
    const C2<R> F{E.x - fma_(W.x, B.x, W.y * B.y), E.y - fma_(W.x, B.y, -(W.y * B.x))};
    return {-(R(2) * nx * A.x + nx * F.x - ny * F.y), -(R(2) * ny * A.x - (nx * F.y + ny * F.x))};
}

// xi = P g~ (Sec. 6.2 step 3) by the CTAs in front of the leaves', four rows of P
// each: the CTA gathers g~ = g0 - g from the far images' parts (side_tasks), a
// warp takes a row by compensated products and sums (Ogita, Rump & Oishi's
// Dot2, as k_xi, which says why).
struct XiArgs {
    int m, M, ctas, per_cell;  // ctas in all, per cell
    const double *gpart, *P;
    double* xi;
    float* xif;
};
__device__ void xi_rows(const XiArgs& a, const Cell* cells, int cta) {
    __shared__ double d[8 * kMaxColl];
    const int ci = cta / a.per_cell, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = (cta % a.per_cell) * 4 + wid, nv = 8 * a.m;
    const Cell& cl = cells[ci];
    if (!cl.active) return;
    const double* gp = a.gpart + (size_t)ci * 7 * nv;
    for (int cc = threadIdx.x; cc < nv; cc += 128) {
        const bool L = cc < 4 * a.m;
        const int k = (cc % (4 * a.m)) / a.m, wp = (L ? 0 : a.m) + cc % a.m;
        double g = 0;
#pragma unroll
        for (int im = 0; im < kWallImages; ++im) g += gp[(size_t)im * nv + 4 * wp + k];
        d[cc] = (k < 2 ? 0.0 : gp[kWallImages * (size_t)nv + k - 2] / (2.0 * (L ? cl.l2 : cl.l1))) - g;
    }
    __syncthreads();
    if (r >= 2 * a.M) return;
    const double* P = a.P + ((size_t)ci * 2 * a.M + r) * nv;
    double s = 0, e = 0;
    for (int cc = lane; cc < nv; cc += 32) {
        const double x = P[cc], y = d[cc], p = x * y, pe = fma(x, y, -p), u = s + p, z = u - s;
        e += pe + ((s - (u - z)) + (p - z));
        s = u;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double s2 = __shfl_xor_sync(0xffffffffu, s, o), e2 = __shfl_xor_sync(0xffffffffu, e, o);
        const double u = s + s2, z = u - s;
        e = e + e2 + ((s - (u - z)) + (s2 - z));
        s = u;
    }
    if (lane == 0) {
        a.xi[(size_t)ci * 2 * a.M + r] = s + e;
        a.xif[(size_t)ci * 2 * a.M + r] = (float)(s + e);
    }
}

// Lanes per target of a tile of n <= 32 targets: a short tile's spare lanes take
// every g-th source (leaves hold some 10 to 60 targets, so half the lanes would
// otherwise idle).
__device__ __forceinline__ int fmm_split(int n) { return n > 16 ? 1 : (n > 8 ? 2 : (n > 4 ? 4 : 8)); }

// Single precision.  One CTA per (leaf, tile share): four warps share a tile of 64
// targets, two per lane (a source read from shared memory then serves two pairs:
// 72 us against 83 with one target per lane at 102400 nodes), and split the near
// sources; a tile of at most 32 splits them over its spare lanes too.  The
// double-float positions make every difference exact to single precision, so no
// later pass has to redo near pairs.
__global__ void __launch_bounds__(128, 6)
k_fmm_down32(FmmTree t, const Cell* cells, const C2<float>* sq, const V4<float>* loc, int shares, FmmTab<float> tab,
             const float4* __restrict__ tgt32, int n0, int n1, float2* __restrict__ part, XiArgs xi, int tiles) {
    constexpr int P = kFmmP32;
    __shared__ V4<float> s_l[4][P];
    __shared__ C2<float> s_pw[4][2][kPowTab];
    __shared__ float4 s_p[4][32];
    __shared__ float2 s_q[4][32];
    __shared__ float2 s_acc[4][64];
    if ((int)blockIdx.x < xi.ctas) {
        pdl_wait();
        pdl_trigger();
        xi_rows(xi, cells, blockIdx.x);
        return;
    }
    const int id = blockIdx.x - xi.ctas, b = id / tiles, tile = id % tiles;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = t.tstart[b], t1 = t.tstart[b + 1];
    const int4 bx = t.box[b];
    const FmmCell& f = t.cells[bx.x];
    const Cell& cl = cells[bx.x];
    if (t0 + 64 * tile >= t1 || t.wanted[b] == 0 || !cl.active) {
        pdl_wait();
        return;
    }
    const FmmRange* near = t.near + (size_t)b * kFmmRanges;
    const int nr = t.nnear[b];
    const float4 cf = t.centre[b];
    const float inv_h = (float)f.inv_h;
    pdl_wait();
    pdl_trigger();
    fmm_local_to_leaf<float>(t, f, bx, loc, shares, tab, s_l, s_pw, wid, lane);
    for (int k0 = t0 + 64 * tile; k0 < t1; k0 += 64 * tiles) {
        const int n = min(64, t1 - k0);
        const bool two = n > 32;
        const int g = two ? 1 : fmm_split(n), per = 32 / g, sub = lane / per;
        float4 p[2];
        float nx[2], ny[2], ax[2] = {0.f, 0.f}, ay[2] = {0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int k = k0 + lane % per + 32 * q;
            int node = k < t1 && (q == 0 || two) ? t.tperm[k] : -1;
            if (node >= 0 && (node < n0 || node >= n1) && node != cl.node_off) node = -1;
            p[q] = make_float4(1e4f, 0.f, 1e4f, 0.f);
            nx[q] = ny[q] = 0.f;
            if (node >= 0) {
                p[q] = t.tpos[k];
                const float4 tv = tgt32[node];
                nx[q] = tv.z;
                ny[q] = tv.w;
            }
        }
        int turn = 0;
        for (int r = 0; r < nr; ++r) {
            const FmmRange rg = near[r];
            const int chunks = (rg.s1 - rg.s0 + 31) >> 5;
            const int first = (wid - turn) & 3;
            turn += chunks;
            if (first >= chunks) continue;
            float px[2], pxl[2], py[2], pyl[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                df_diff(p[q].x, p[q].y, cl.sxf[rg.im], cl.sxl[rg.im], px[q], pxl[q]);
                df_diff(p[q].z, p[q].w, cl.syf[rg.im], cl.syl[rg.im], py[q], pyl[q]);
            }
            for (int ch = first; ch < chunks; ch += 4) {
                const int s = rg.s0 + 32 * ch + lane, cnt = min(32, rg.s1 - rg.s0 - 32 * ch);
                __syncwarp();
                if (lane < cnt) {
                    s_p[wid][lane] = t.spos[s];
                    s_q[wid][lane] = make_float2(sq[s].x, sq[s].y);
                }
                __syncwarp();
                auto pair = [&](int q, const float4& sp, const float2& ss) {
                    const float dx = (px[q] - sp.x) + (pxl[q] - sp.y);
                    const float dy = (py[q] - sp.z) + (pyl[q] - sp.w);
                    const float cc = pair32(dx, dy, nx[q], ny[q], ss.x, ss.y);
                    ax[q] = fmaf(cc, dx, ax[q]);
                    ay[q] = fmaf(cc, dy, ay[q]);
                };
                if (two) {
#pragma unroll 4
                    for (int j = 0; j < cnt; ++j) {
                        const float4 sp = s_p[wid][j];
                        const float2 ss = s_q[wid][j];
                        pair(0, sp, ss);
                        pair(1, sp, ss);
                    }
                } else {
#pragma unroll 4
                    for (int j = sub; j < cnt; j += g) pair(0, s_p[wid][j], s_q[wid][j]);
                }
            }
        }
        for (int o = per; o < 32; o <<= 1) {
            ax[0] += __shfl_xor_sync(0xffffffffu, ax[0], o);
            ay[0] += __shfl_xor_sync(0xffffffffu, ay[0], o);
        }
        __syncthreads();  // the previous tile's sums have been read
        s_acc[wid][lane] = make_float2(ax[0], ay[0]);
        s_acc[wid][lane + 32] = make_float2(ax[1], ay[1]);
        __syncthreads();
        // two lanes per target split the local expansion and the warps' sums
        const int q = threadIdx.x >> 1, res = threadIdx.x & 1, kq = k0 + q;
        int nd = q < n ? t.tperm[kq] : -1;
        if (nd >= 0 && (nd < n0 || nd >= n1) && nd != cl.node_off) nd = -1;
        float fx = 0.f, fy = 0.f;
        if (nd >= 0) {
            const float4 tv = tgt32[nd];
            const C2<float> F = fmm_local_at<float, 2>(s_l[0], fmm_local(t.tpos[kq], cf, inv_h), res, tv.z, tv.w);
            const float gl = (float)(1.0 / (4.0 * kPi)) * inv_h, cp = (float)(-1.0 / kPi);
            fx = fmaf(cp, s_acc[res][q].x + s_acc[res + 2][q].x, gl * F.x);
            fy = fmaf(cp, s_acc[res][q].y + s_acc[res + 2][q].y, gl * F.y);
        }
        fx += __shfl_xor_sync(0xffffffffu, fx, 1);
        fy += __shfl_xor_sync(0xffffffffu, fy, 1);
        if (nd >= 0 && res == 0) part[cl.part_off[0] + (nd - cl.node_off)] = make_float2(fx, fy);
    }
}

// Double precision, native or double-float (everything but the last sums).  One
// CTA per (leaf, tile share): four warps share a tile of 32 targets and split
// the near sources, then four lanes per target split the local expansion.
template <typename R>
__global__ void __launch_bounds__(128, 4)
k_fmm_down64(FmmTree t, const Cell* cells, const C2<R>* sq, const V4<R>* loc, int shares, FmmTab<R> tab,
             const double* __restrict__ nxv, const double* __restrict__ nyv, int prec, int n0, int n1, double2* __restrict__ part,
             XiArgs xi, int tiles) {
    constexpr int P = FmmTypes<R>::P;
    constexpr bool DF = std::is_same<R, df>::value;
    __shared__ V4<R> s_l[4][P];
    __shared__ C2<R> s_pw[4][2][kPowTab];
    __shared__ double2 s_p[4][32], s_q[4][32];  // double-float: a float4 each
    __shared__ double2 s_acc[4][32], s_t[32], s_n[32];
    __shared__ int s_node[32];
    if ((int)blockIdx.x < xi.ctas) {
        pdl_wait();
        pdl_trigger();
        xi_rows(xi, cells, blockIdx.x);
        return;
    }
    const int id = blockIdx.x - xi.ctas, b = id / tiles, tile = id % tiles;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = t.tstart[b], t1 = t.tstart[b + 1];
    const int4 bx = t.box[b];
    const FmmCell& f = t.cells[bx.x];
    const Cell& cl = cells[bx.x];
    if (t0 + 32 * tile >= t1 || t.wanted[b] == 0 || !cl.active) {
        pdl_wait();
        return;
    }
    const FmmRange* near = t.near + (size_t)b * kFmmRanges;
    const int nr = t.nnear[b];
    pdl_wait();
    pdl_trigger();
    fmm_local_to_leaf<R>(t, f, bx, loc, shares, tab, s_l, s_pw, wid, lane);
    const double2 c = fmm_centre(f, 0, fmm_ix(bx), fmm_iy(bx));
    for (int k0 = t0 + 32 * tile; k0 < t1; k0 += 32 * tiles) {
        const int n = min(32, t1 - k0), g = fmm_split(n), per = 32 / g, sub = lane / per, k = k0 + lane % per;
        int node = k < t1 ? t.tperm[k] : -1;
        if (node >= 0 && (node < n0 || node >= n1) && node != cl.node_off) node = -1;
        double2 p = make_double2(1e4, 1e4);
        double nx = 0, ny = 0;
        if (node >= 0) {
            p = t.tpos64[k];
            nx = nxv[node];
            ny = nyv[node];
        }
        float nxh, nxl, nyh, nyl;
        if constexpr (DF) {
            split_df(nx, nxh, nxl);
            split_df(ny, nyh, nyl);
        }
        double ax = 0, ay = 0;
        int turn = 0;
        for (int r = 0; r < nr; ++r) {
            const FmmRange rg = near[r];
            const int chunks = (rg.s1 - rg.s0 + 31) >> 5;
            const int first = (wid - turn) & 3;
            turn += chunks;
            if (first >= chunks) continue;
            const double px = p.x - cl.sx[rg.im], py = p.y - cl.sy[rg.im];
            float pxh, pxl, pyh, pyl;
            if constexpr (DF) {
                split_df(px, pxh, pxl);
                split_df(py, pyh, pyl);
            }
            for (int ch = first; ch < chunks; ch += 4) {
                const int s = rg.s0 + 32 * ch + lane, cnt = min(32, rg.s1 - rg.s0 - 32 * ch);
                __syncwarp();
                if (lane < cnt) {
                    if constexpr (DF) {
                        *reinterpret_cast<float4*>(&s_p[wid][lane]) = t.spos[s];
                        *reinterpret_cast<float4*>(&s_q[wid][lane]) = reinterpret_cast<const float4*>(sq)[s];
                    } else {
                        s_p[wid][lane] = t.spos64[s];
                        s_q[wid][lane] = reinterpret_cast<const double2*>(sq)[s];
                    }
                }
                __syncwarp();
                if constexpr (DF) {
                    // chunk sums as (TwoSum high part, float error), folded into
                    // double after every chunk
                    float axh = 0, axe = 0, ayh = 0, aye = 0;
#pragma unroll 2
                    for (int j = sub; j < cnt; j += g) {
                        const float4 sp = *reinterpret_cast<const float4*>(&s_p[wid][j]);
                        const float4 ss = *reinterpret_cast<const float4*>(&s_q[wid][j]);
                        pair_df(pxh, pxl, pyh, pyl, nxh, nxl, nyh, nyl,
                                SrcDF{sp.x, sp.y, sp.z, sp.w, ss.x, ss.y, ss.z, ss.w}, axh, axe, ayh, aye);
                    }
                    ax += (double)axh + (double)axe;
                    ay += (double)ayh + (double)aye;
                } else {
#pragma unroll 2
                    for (int j = sub; j < cnt; j += g) {
                        const double2 sp = s_p[wid][j], ss = s_q[wid][j];
                        const double dx = px - sp.x, dy = py - sp.y;
                        const double inv = rcp64(fma(dx, dx, fma(dy, dy, 1e-300)));
                        const double rn = fma(dy, ny, dx * nx), rq = fma(dy, ss.y, dx * ss.x);
                        const double cc = (rn * inv) * (rq * inv);
                        ax = fma(cc, dx, ax);
                        ay = fma(cc, dy, ay);
                    }
                }
            }
        }
        for (int o = per; o < 32; o <<= 1) {
            ax += __shfl_xor_sync(0xffffffffu, ax, o);
            ay += __shfl_xor_sync(0xffffffffu, ay, o);
        }
        __syncthreads();  // also: the previous tile's targets have been read
        s_acc[wid][lane] = make_double2(ax, ay);
        if (wid == 0) {
            s_t[lane] = make_double2((p.x - c.x) * f.inv_h, (p.y - c.y) * f.inv_h);
            s_n[lane] = make_double2(nx, ny);
            s_node[lane] = lane < per ? node : -1;
        }
        __syncthreads();
        const int q = threadIdx.x >> 2, res = threadIdx.x & 3, nd = s_node[q];
        double fx = 0, fy = 0;
        if (nd >= 0) {
            const C2<R> F = fmm_local_at<R, 4>(s_l[0], C2<R>{R(s_t[q].x), R(s_t[q].y)}, res, R(s_n[q].x),
                                               R(s_n[q].y));
            const double g = f.inv_h / (4.0 * kPi), cp = -1.0 / kPi;
            fx = fma(cp, s_acc[res][q].x, g * to_double(F.x));
            fy = fma(cp, s_acc[res][q].y, g * to_double(F.y));
        }
        fx += __shfl_xor_sync(0xffffffffu, fx, 1);
        fy += __shfl_xor_sync(0xffffffffu, fy, 1);
        fx += __shfl_xor_sync(0xffffffffu, fx, 2);
        fy += __shfl_xor_sync(0xffffffffu, fy, 2);
        if (nd >= 0 && res == 0) part[cl.part_off[prec] + (nd - cl.node_off)] = make_double2(fx, fy);
    }
}

// ---------------------------------------------------------------------------
// host: choice of the boxes, storage, launches
// ---------------------------------------------------------------------------
// Compile-time switches for measurements: BIE_FMM 0 keeps the direct sums,
// BIE_FMM_HSCALE scales the chosen box side.
#ifndef BIE_FMM
#define BIE_FMM 1
#endif
#ifndef BIE_FMM_HSCALE
#define BIE_FMM_HSCALE 1.0
#endif

// Modelled time (seconds, GB300) of a near sum over a cell, direct or with
// leaves of side h.  Rates per precision (0 single, 1 double, 2 double-float):
// a direct pair, a pair of the fast sum's leaves, a translation.
static constexpr double kDirectPair[3] = {0.345e-12, 31.7e-12, 3.57e-12};
static constexpr double kLeafPair[3] = {1.2e-12, 25e-12, 5e-12};
static constexpr double kTranslate[3] = {0.7e-9, 26e-9, 7e-9};
static constexpr double kFmmFixed[3] = {5e-6, 20e-6, 20e-6};
// What sums of few long items cost a direct application of a cell alone in its
// context.  Measured (us, direct / fast): double-float 480 nodes 88 / 119, 1024 130 / 142,
// 1536 192 / 153; double 480 163 / 303, 1024 470 / 383.  (Single precision: 128 nodes
// 42 / 46, 1024 49 / 51, 1536 56 / 54, 2560 73 / 64, as the model has it.)
static constexpr double kDirectFixed[3] = {0, 220e-6, 85e-6};
// Boxes that any cell may have, in a batch and alone: with 64, cells below 500 nodes
// had no leaf small enough for the walls.
static constexpr double kFmmBoxes[2] = {64, 256};

struct FmmPlanCell {
    double ox, oy, w, ht;  // rectangle (relative to the cell centre)
    double area;
};

static double body_perimeter(const bie_ctx* c, int b) {
    const double* sh = &c->bshape_host[4 * (size_t)b];
    if (sh[0] == 1.0) {
        const int n = 512;
        double s = 0;
        for (int k = 0; k < n; ++k) {
            const double t = 2 * kPi * k / n, r = sh[1] * (1 + sh[2] * std::cos(sh[3] * t)),
                         d = -sh[1] * sh[2] * sh[3] * std::sin(sh[3] * t);
            s += std::sqrt(r * r + d * d);
        }
        return s * 2 * kPi / n;
    }
    const double a = sh[1], q = sh[2];
    return kPi * (3 * (a + q) - std::sqrt((3 * a + q) * (a + 3 * q)));
}

static double fmm_cost(const bie_ctx* c, const Cell& cl, const std::vector<double>& per, double area, double h,
                       int prec) {
    // (idle: leaves too few to fill the chip)
    double pairs = 0, occ = 0;
    for (int b = cl.body_off; b < cl.body_off + cl.n_bodies; ++b) {
        const double n = c->n_nodes[b], hb = per[b] / n;
        pairs += n * (std::min(n, 3.3 * h / hb + 1) + 9 * h * h / area * (cl.n_nodes - n));
        occ += std::min(n, 1.3 * per[b] / h + 1);
    }
    occ = std::max(1.0, std::min(occ, area / (h * h) * 1.1 + 4));
    const double idle = std::max(1.0, 2.0 * c->sms / (occ * c->ncell));
    return (pairs * kLeafPair[prec] + occ * 45 * kTranslate[prec]) * idle;
}

// The rectangle that holds every node of a cell whatever its lattice does in
// time stepping (|e2_x| <= |e1_x| / 2 there) and wherever its bodies are now.
static FmmPlanCell fmm_rect(const bie_ctx* c, int k) {
    const Cell& cl = c->cells_h[k];
    double R = 0;
    for (int b = cl.body_off; b < cl.body_off + cl.n_bodies; ++b)
        R = std::max(R, std::max(c->body_host[8 * (size_t)b], c->body_host[8 * (size_t)b + 1]));
    double e2x = std::fabs(cl.e2[0]);
    if (cl.e1[1] == 0.0) e2x = std::max(e2x, 0.5 * std::fabs(cl.e1[0]));
    const double m = c->utilde ? 1.0 : 0.5;
    double x1 = m * (std::fabs(cl.e1[0]) + e2x) + R, y1 = m * (std::fabs(cl.e1[1]) + std::fabs(cl.e2[1])) + R;
    double x0 = -x1, y0 = -y1;
    for (int b = cl.body_off; b < cl.body_off + cl.n_bodies; ++b) {
        const double px = c->body_host[8 * (size_t)b + 2] - cl.C[0], py = c->body_host[8 * (size_t)b + 3] - cl.C[1];
        x0 = std::min(x0, px - R);
        x1 = std::max(x1, px + R);
        y0 = std::min(y0, py - R);
        y1 = std::max(y1, py + R);
    }
    const double pad = 1e-6 * ((x1 - x0) + (y1 - y0));
    FmmPlanCell p;
    p.ox = x0 - pad;
    p.oy = y0 - pad;
    p.w = x1 - x0 + 2 * pad;
    p.ht = y1 - y0 + 2 * pad;
    p.area = std::fabs(cl.e1[0] * cl.e2[1] - cl.e1[1] * cl.e2[0]);
    return p;
}

int fmm_work(bie_ctx* c, int prec, int64_t* pairs, int64_t* translations, int32_t* order) {
    *pairs = *translations = 0;
    *order = prec == 0 ? kFmmP32 : kFmmP64;
    const Fmm& f = c->fmm[prec];
    if (!f.on) {
        for (const Cell& cl : c->cells_h) {
            const int own = c->shard.on ? c->shard.n1 - c->shard.n0 + (c->shard.n0 > 0) : cl.n_nodes;
            *pairs += (int64_t)own * cl.n_nodes * (c->utilde ? 4 : 9);
        }
        return BIE_OK;
    }
    if (int rc = fmm_build(c, prec)) return rc;
    std::vector<int> count(f.t.nleaf), nnear(f.t.nleaf), nfar(f.t.nbox);
    std::vector<FmmRange> near((size_t)f.t.nleaf * kFmmRanges);
    BIE_CUDA(c, cudaStreamSynchronize(c->stream));
    BIE_CUDA(c, cudaMemcpy(count.data(), f.t.wanted, count.size() * sizeof(int), cudaMemcpyDeviceToHost));
    BIE_CUDA(c, cudaMemcpy(nnear.data(), f.t.nnear, nnear.size() * sizeof(int), cudaMemcpyDeviceToHost));
    BIE_CUDA(c, cudaMemcpy(nfar.data(), f.t.nfar, nfar.size() * sizeof(int), cudaMemcpyDeviceToHost));
    BIE_CUDA(c, cudaMemcpy(near.data(), f.t.near, near.size() * sizeof(FmmRange), cudaMemcpyDeviceToHost));
    for (int b = 0; b < f.t.nleaf; ++b) {
        if (!count[b]) continue;
        for (int r = 0; r < nnear[b]; ++r) {
            const FmmRange& g = near[(size_t)b * kFmmRanges + r];
            *pairs += (int64_t)count[b] * (g.s1 - g.s0);
        }
    }
    for (int n : nfar) *translations += n;
    return BIE_OK;
}

void free_fmm(bie_ctx* c) {
    for (Fmm& f : c->fmm) {
        if (f.arena) cudaFree(f.arena);
        f = Fmm{};
    }
    if (c->fmm_ws) cudaFree(c->fmm_ws);
    c->fmm_ws = nullptr;
    c->ws.fsq = c->ws.fmp = c->ws.floc = nullptr;
    c->ws.ftick = nullptr;
    c->fmm_static = Workspace{};
}

// Table sizes in numbers of R: hankel, binom, then the child powers.
template <typename R>
static FmmTab<R> fmm_tab(const bie_ctx* c, int prec) {
    constexpr int P = FmmTypes<R>::P;
    const R* h = (const R*)c->fmm[prec].tables;
    const C2<R>* pw = (const C2<R>*)(h + 3 * P * P);
    return FmmTab<R>{h, h + P * P, h + 2 * P * P, pw, pw + 4 * P};
}

static df to_df(long double v) { return df((float)v, (float)(v - (long double)(float)v)); }

template <typename R>
static constexpr size_t kTableSize = (3 * (size_t)FmmTypes<R>::P * FmmTypes<R>::P + 16 * FmmTypes<R>::P) * sizeof(R);

template <typename R>
static void fmm_tables(void* out) {
    constexpr int P = FmmTypes<R>::P;
    R* t = (R*)out;
    auto put = [&](size_t k, long double v) {
        if constexpr (std::is_same<R, df>::value) t[k] = to_df(v);
        else t[k] = (R)v;
    };
    std::vector<std::vector<long double>> b(2 * P, std::vector<long double>(2 * P, 0.0L));
    for (int n = 0; n < 2 * P; ++n) {
        b[n][0] = 1;
        for (int k = 1; k <= n; ++k) b[n][k] = b[n - 1][k - 1] + (k <= n - 1 ? b[n - 1][k] : 0.0L);
    }
    for (int k = 0; k < P; ++k)
        for (int l = 0; l < P; ++l) {
            put((size_t)k * P + l, b[k + l][l]);
            put((size_t)(P + k) * P + l, b[l][k]);
            put((size_t)(2 * P + l) * P + k, b[l][k]);
        }
    for (int q = 0; q < 4; ++q) {
        // delta = (+-1/4, +-1/4); 1 / (2 delta) = (+-1, -+1)
        const long double dx = q & 1 ? 0.25L : -0.25L, dy = q >> 1 ? 0.25L : -0.25L;
        long double d[2] = {1, 0}, g[2] = {1, 0};
        for (int k = 0; k < P; ++k) {
            const size_t o = 3 * (size_t)P * P + 2 * ((size_t)q * P + k);
            put(o, d[0]);
            put(o + 1, d[1]);
            put(o + 8 * P, g[0]);
            put(o + 8 * P + 1, g[1]);
            const long double nd[2] = {d[0] * dx - d[1] * dy, d[0] * dy + d[1] * dx};
            const long double ex = 4 * dx, ey = -4 * dy;
            const long double ng[2] = {g[0] * ex - g[1] * ey, g[0] * ey + g[1] * ex};
            d[0] = nd[0];
            d[1] = nd[1];
            g[0] = ng[0];
            g[1] = ng[1];
        }
    }
}

// The largest box side that the walls' far images are well away from; <= 0: none.  The
// images of L and R lie on the lines lattice coordinate s = +-3/2, those of D and U on
// t = +-3/2; nodes lie within a bounding radius of their centres, so at least d from any
// image.  A source at a box's corner is e = side / sqrt 2 from its centre, and an image may
// be as near as d - e to that, so the moments converge by e / (d - e) per order at worst:
// 3/7 in single precision (e = 0.3 d; 24 orders reach 1.5e-9) and 1/2 in double (e = d / 3;
// 48 orders reach 3.6e-15, and sources elsewhere far less).  With e = 0.45 d, 0.45 per order
// as the source sees it but 9/11 from the centre, the first terms left out added up to
// 8e-12 on 25 bodies in a cell sheared by half.
static double fmm_wall_side(const bie_ctx* c, int k, int prec) {
    const Cell& cl = c->cells_h[k];
    const double det = cl.e1[0] * cl.e2[1] - cl.e1[1] * cl.e2[0];
    double R = 0, far = 0.5;  // bounding radius; largest |s|, |t| of a centre
    for (int b = cl.body_off; b < cl.body_off + cl.n_bodies; ++b) {
        const double* h = &c->body_host[8 * (size_t)b];
        R = std::max(R, std::max(h[0], h[1]));
        const double px = h[2] - cl.C[0], py = h[3] - cl.C[1];
        far = std::max(far, std::max(std::fabs(px * cl.e2[1] - py * cl.e2[0]), std::fabs(cl.e1[0] * py - cl.e1[1] * px)) /
                                std::fabs(det));
    }
    // perpendicular spacing of the lattice lines; a sheared cell's e2 lengthens
    // to (e1 / 2, e2_y) at most
    double e2x = std::fabs(cl.e2[0]);
    if (cl.e1[1] == 0.0) e2x = std::max(e2x, 0.5 * std::fabs(cl.e1[0]));
    const double l2 = std::hypot(e2x, cl.e2[1]), l1 = std::hypot(cl.e1[0], cl.e1[1]);
    const double d = (1.5 - far) * std::fabs(det) / std::max(l1, l2) - R;
    return (prec == 0 ? 0.3 : 1.0 / 3.0) * d * std::sqrt(2.0);
}

// The boxes of one cell for where its bodies are now: the grid as planned while it
// covers their rectangle, and else moved and its side stretched until it does; then the
// coarsest level that the walls' far images are well away from, which depends on the
// lattice and the centres too.
static FmmCell fmm_place(const bie_ctx* c, int k, int prec) {
    FmmCell f = c->fmm[prec].plan[k];
    const FmmPlanCell r = fmm_rect(c, k);
    const double x1 = std::max(f.ox + f.gx[0] * f.h, r.ox + r.w), y1 = std::max(f.oy + f.gy[0] * f.h, r.oy + r.ht);
    if (r.ox < f.ox || r.oy < f.oy || r.ox + r.w > f.ox + f.gx[0] * f.h || r.oy + r.ht > f.oy + f.gy[0] * f.h) {
        f.ox = std::min(f.ox, r.ox);
        f.oy = std::min(f.oy, r.oy);
        f.h = std::max(std::max((x1 - f.ox) / f.gx[0], (y1 - f.oy) / f.gy[0]), f.h * (1 + 1e-15));
        f.inv_h = 1.0 / f.h;
    }
    const double wall = fmm_wall_side(c, k, prec);
    f.wall = -1;
    for (int l = 0; l < f.nlev; ++l)
        if (f.h * (1 << l) <= wall) f.wall = l;
    return f;
}

static void fmm_centres(const std::vector<FmmCell>& cells, float4* centre) {
    for (const FmmCell& f : cells)
        for (int l = 0; l < f.nlev; ++l)
            for (int y = 0; y < f.gy[l]; ++y)
                for (int x = 0; x < f.gx[l]; ++x) {
                    const double2 p = fmm_centre(f, l, x, y);
                    float4& o = centre[f.off[l] + (size_t)y * f.gx[l] + x];
                    o.x = (float)p.x;
                    o.y = (float)(p.x - (double)o.x);
                    o.z = (float)p.y;
                    o.w = (float)(p.y - (double)o.z);
                }
}

// Called when a configuration is set (host mirrors of bodies and lattices).  A context
// that bie_apply_static takes keeps its counts of boxes, and with them every kernel's
// arguments, so that an application captured before stays right; stretched leaves cost
// it pairs (a side 1.6 times as long for bodies listed a lattice vector away).  Larger
// ones are planned anew when their bodies leave the grid: leaves of many more targets than
// planned would leave the chip to a few CTAs.  (The epoch then tells that the layout
// of the sums may have changed.)
int fmm_fit(bie_ctx* c) {
    std::vector<FmmCell> place[3];
    bool left = false;
    for (int prec = 0; prec < 3; ++prec)
        for (int k = 0; k < c->ncell && c->fmm[prec].on; ++k) {
            place[prec].push_back(fmm_place(c, k, prec));
            left = left || place[prec][k].h > c->fmm[prec].plan[k].h;
        }
    if (left && c->N > kStaticMaxNodes) {
        ++c->epoch;
        free_fmm(c);
        return fmm_plan(c);
    }
    for (int prec = 0; prec < 3; ++prec) {
        Fmm& f = c->fmm[prec];
        if (!f.on) continue;
        bool moved = false;
        for (int k = 0; k < c->ncell; ++k) {
            const FmmCell &q = place[prec][k], &o = f.now[k];
            moved = moved || q.ox != o.ox || q.oy != o.oy || q.h != o.h || q.wall != o.wall;
        }
        if (!moved) continue;
        f.now = place[prec];
        std::vector<float4> centre(f.t.nbox);
        fmm_centres(f.now, centre.data());
        BIE_CUDA(c, cudaMemcpyAsync(f.cells, f.now.data(), f.now.size() * sizeof(FmmCell), cudaMemcpyHostToDevice, c->stream));
        BIE_CUDA(c, cudaMemcpyAsync(f.t.centre, centre.data(), centre.size() * sizeof(float4), cudaMemcpyHostToDevice,
                                    c->stream));
        BIE_CUDA(c, cudaStreamSynchronize(c->stream));
    }
    return BIE_OK;
}

// Boxes of every precision whose near sums run faster this way.  Called when
// a context is made, after all else has its memory (and by fmm_fit): a precision whose boxes do not fit
// beside it keeps the direct sum (all of them, where the moments do not fit).  Nothing
// of the context refers to the boxes before they are complete.
int fmm_plan(bie_ctx* c) {
    std::vector<FmmPlanCell> rect(c->ncell);
    for (int k = 0; k < c->ncell; ++k) rect[k] = fmm_rect(c, k);
    if (!BIE_FMM) return BIE_OK;
    std::vector<double> per(c->nb);
    for (int b = 0; b < c->nb; ++b) per[b] = body_perimeter(c, b);
    const int N = c->N, nsrc = N * c->srcmul;
    size_t mp_bytes = 0, loc_bytes = 0, sq_bytes = 0;
    int max_box = 0;
    Fmm made[3];
    auto drop = [&](cudaError_t e, const char* what) {  // nothing kept; BIE_OK if memory was short
        for (Fmm& f : made)
            if (f.arena) cudaFree(f.arena);
        if (c->fmm_ws) cudaFree(c->fmm_ws);
        c->fmm_ws = nullptr;
        cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? BIE_OK : cuda_check(c, e, what);
    };
    for (int prec = 0; prec < 3; ++prec) {
        Fmm f;
        std::vector<FmmCell> cells(c->ncell);
        double t_fast = kFmmFixed[prec], t_direct = 0;
        long long nleaf = 0, nbox = 0;
        for (int k = 0; k < c->ncell; ++k) {
            const Cell& cl = c->cells_h[k];
            const FmmPlanCell& rc = rect[k];
            FmmCell& fc = cells[k];
            // leaf side: the modelled best of a geometric ladder, with at most
            // one box per 8 source records (kFmmBoxes at least)
            const double most = std::max(kFmmBoxes[c->ncell == 1], cl.n_nodes * (double)c->srcmul / 8);
            const double wall = fmm_wall_side(c, k, prec);
            double best = INFINITY, bh = 0;
            for (int j = 0; j < 48; ++j) {
                const double h = std::sqrt(rc.area) * std::pow(2.0, -0.25 * j);
                if (std::ceil(rc.w / h) * std::ceil(rc.ht / h) * 1.34 + 8 > most) break;
                if (wall > 0 && h > wall) continue;
                if (std::ceil(rc.w / h) > 4000 || std::ceil(rc.ht / h) > 4000) break;
                const double t = fmm_cost(c, cl, per, rc.area, h, prec);
                if (t < best) {
                    best = t;
                    bh = h;
                }
            }
            if (!(bh > 0)) {
                best = INFINITY;
                bh = std::max(rc.w, rc.ht);
            }
            bh *= BIE_FMM_HSCALE;
            t_fast += best;
            t_direct += (double)cl.n_nodes * cl.n_nodes * (c->utilde ? 4 : 9) * kDirectPair[prec];
            fc.ox = rc.ox;
            fc.oy = rc.oy;
            fc.h = bh;
            fc.inv_h = 1.0 / bh;
            fc.gx[0] = std::max(1, (int)std::ceil(rc.w / bh));
            fc.gy[0] = std::max(1, (int)std::ceil(rc.ht / bh));
            fc.nlev = 1;
            while (fc.nlev < kFmmLevels && (fc.gx[fc.nlev - 1] > 4 || fc.gy[fc.nlev - 1] > 4)) {
                fc.gx[fc.nlev] = (fc.gx[fc.nlev - 1] + 1) / 2;
                fc.gy[fc.nlev] = (fc.gy[fc.nlev - 1] + 1) / 2;
                ++fc.nlev;
            }
            fc.wall = -1;
            for (int l = 0; l < fc.nlev; ++l)
                if (bh * (1 << l) <= wall) fc.wall = l;
            fc.off[0] = (int)nleaf;
            nleaf += (long long)fc.gx[0] * fc.gy[0];
        }
        f.walls = !c->utilde;
        for (const FmmCell& fc : cells) f.walls = f.walls && fc.wall >= 0;
        if (f.walls && c->ncell == 1) t_direct += kDirectFixed[prec];
        f.on = (t_fast < t_direct || BIE_FMM == 2) && nleaf < (1 << 26);
        f.walls = f.walls && f.on;
        if (!f.on) continue;
        // leaves of all cells first, then the coarser levels cell by cell
        nbox = nleaf;
        for (FmmCell& fc : cells)
            for (int l = 1; l < fc.nlev; ++l) {
                fc.off[l] = (int)nbox;
                nbox += (long long)fc.gx[l] * fc.gy[l];
            }
        // one block: what the host writes first (cells, boxes, leaf centres, tables)
        const bool dbl = prec != 0;
        size_t total = 0;
        auto place = [&](size_t bytes) {
            const size_t at = total;
            total += (bytes + 255) & ~(size_t)255;
            return at;
        };
        const size_t tab_bytes = prec == 0 ? kTableSize<float> : (prec == 1 ? kTableSize<double> : kTableSize<df>);
        const size_t o_cells = place(cells.size() * sizeof(FmmCell)), o_box = place(nbox * sizeof(int4)),
                     o_centre = place(nbox * sizeof(float4)), o_grid = place(nbox * sizeof(int4)), o_tab = place(tab_bytes), written = total;
        const size_t o_scount = place(nbox * sizeof(int)), o_sstart = place((nleaf + 1) * sizeof(int)),
                     o_sperm = place(nsrc * sizeof(int)), o_cursor = place(nleaf * sizeof(int)),
                     o_leaf = place(nsrc * sizeof(int)), o_raw = place(nsrc * sizeof(int)),
                     o_spos = prec != 1 ? place(nsrc * sizeof(float4)) : 0,
                     o_spos64 = dbl ? place(nsrc * sizeof(double2)) : 0;
        const size_t o_far = place((size_t)nbox * kFmmFar * sizeof(int)), o_nfar = place(nbox * sizeof(int)),
                     o_near = place((size_t)nleaf * kFmmRanges * sizeof(FmmRange)), o_nnear = place(nleaf * sizeof(int)),
                     o_shift = place(9 * cells.size() * sizeof(float4));
        const bool ut = c->utilde;
        const size_t o_tcount = ut ? place(nbox * sizeof(int)) : 0, o_tstart = ut ? place((nleaf + 1) * sizeof(int)) : 0,
                     o_tperm = ut ? place(N * sizeof(int)) : 0,
                     o_tpos = ut ? place(N * (dbl ? sizeof(double2) : sizeof(float4))) : 0;
        const size_t o_owned = c->ncell == 1 ? place(nbox * sizeof(int)) : 0;
        if (const cudaError_t e = cudaMalloc(&f.arena, total)) {
            f.arena = nullptr;
            if (e != cudaErrorMemoryAllocation) return drop(e, "cudaMalloc");
            cudaGetLastError();
            continue;
        }
        std::vector<unsigned char> host(written);
        std::memcpy(&host[o_cells], cells.data(), cells.size() * sizeof(FmmCell));
        int4* box = (int4*)&host[o_box];
        for (int k = 0; k < c->ncell; ++k) {
            const FmmCell& fc = cells[k];
            for (int l = 0; l < fc.nlev; ++l)
                for (int y = 0; y < fc.gy[l]; ++y)
                    for (int x = 0; x < fc.gx[l]; ++x)
                        box[fc.off[l] + (size_t)y * fc.gx[l] + x] =
                            make_int4(k, l, x | (y << 16),
                                      l + 1 < fc.nlev ? fc.off[l + 1] + (y / 2) * fc.gx[l + 1] + x / 2 : -1);
        }
        fmm_centres(cells, (float4*)&host[o_centre]);
        int4* grid = (int4*)&host[o_grid];
        for (long long b = 0; b < nbox; ++b)
            grid[b] = make_int4(cells[box[b].x].off[box[b].y], cells[box[b].x].gx[box[b].y], 0, 0);
        if (prec == 0) fmm_tables<float>(&host[o_tab]);
        else if (prec == 1) fmm_tables<double>(&host[o_tab]);
        else fmm_tables<df>(&host[o_tab]);
        cudaError_t e = cudaMemcpyAsync(f.arena, host.data(), written, cudaMemcpyHostToDevice, c->stream);
        if (!e) e = cudaStreamSynchronize(c->stream);  // (the copy in host memory goes)
        if (e) {
            cudaFree(f.arena);
            return drop(e, "cudaMemcpyAsync");
        }
        f.plan = f.now = cells;
        unsigned char* a = (unsigned char*)f.arena;
        FmmTree& t = f.t;
        t.nleaf = (int)nleaf;
        t.nbox = (int)nbox;
        t.cells = f.cells = (FmmCell*)(a + o_cells);
        t.box = f.box = (int4*)(a + o_box);
        t.centre = (float4*)(a + o_centre);
        t.grid = (int4*)(a + o_grid);
        t.far = (int*)(a + o_far);
        t.nfar = (int*)(a + o_nfar);
        t.near = (FmmRange*)(a + o_near);
        t.nnear = (int*)(a + o_nnear);
        t.shift = (float4*)(a + o_shift);
        f.tables = a + o_tab;
        f.owned = c->ncell == 1 ? (int*)(a + o_owned) : nullptr;
        t.tcount = t.scount = (int*)(a + o_scount);
        t.tstart = t.sstart = (int*)(a + o_sstart);
        t.tperm = t.sperm = (int*)(a + o_sperm);
        f.cursor = (int*)(a + o_cursor);
        f.leaf = (int*)(a + o_leaf);
        f.raw = (int*)(a + o_raw);
        t.tpos = t.spos = prec != 1 ? (float4*)(a + o_spos) : nullptr;
        t.tpos64 = t.spos64 = dbl ? (double2*)(a + o_spos64) : nullptr;
        if (ut) {
            t.tcount = (int*)(a + o_tcount);
            t.tstart = (int*)(a + o_tstart);
            t.tperm = (int*)(a + o_tperm);
            t.tpos = dbl ? nullptr : (float4*)(a + o_tpos);
            t.tpos64 = dbl ? (double2*)(a + o_tpos) : nullptr;
        }
        t.wanted = t.tcount;
        f.built = 0;
        f.mp_bytes = (size_t)nbox * (dbl ? kFmmP64 * sizeof(V4<double>) : kFmmP32 * sizeof(V4<float>));
        // lists split into shares until the boxes (about half of them occupied)
        // fill the SMs four times over
        f.shares = std::max(1, std::min(kFmmShares, (int)(8LL * c->sms / std::max(1LL, nbox))));
        f.loc_bytes = f.mp_bytes * f.shares;
        f.sq_bytes = (size_t)nsrc * (dbl ? sizeof(double2) : sizeof(float2));
        mp_bytes = std::max(mp_bytes, f.mp_bytes);
        loc_bytes = std::max(loc_bytes, f.loc_bytes);
        sq_bytes = std::max(sq_bytes, f.sq_bytes);
        max_box = std::max(max_box, (int)nbox);
        made[prec] = f;
    }
    if (max_box) {
        auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
        // counters (a set for bie_apply_static's single-precision sum after the context's),
        // then sorted strengths and expansions, again for the context and for that call
        const size_t tick = up(max_box * sizeof(unsigned));
        const Fmm& s = made[0];
        const bool own = s.on && N <= kStaticMaxNodes;
        const size_t whole = up(sq_bytes) + up(mp_bytes) + up(loc_bytes),
                     second = own ? up(s.sq_bytes) + up(s.mp_bytes) + up(s.loc_bytes) : 0;
        if (const cudaError_t e = cudaMalloc(&c->fmm_ws, 2 * tick + whole + second)) {
            c->fmm_ws = nullptr;
            return drop(e, "cudaMalloc");
        }
        // (on the context's stream, which need not wait for the default one)
        if (const cudaError_t e = cudaMemsetAsync(c->fmm_ws, 0, 2 * tick, c->stream)) return drop(e, "cudaMemsetAsync");
        unsigned char* a = (unsigned char*)c->fmm_ws;
        auto lay = [&](Workspace& ws, unsigned char* ticks, unsigned char* at, size_t sq, size_t mp) {
            ws.ftick = (unsigned*)ticks;
            ws.fsq = at;
            ws.fmp = at + up(sq);
            ws.floc = at + up(sq) + up(mp);
        };
        lay(c->ws, a, a + 2 * tick, sq_bytes, mp_bytes);
        if (own) lay(c->fmm_static, a + tick, a + 2 * tick + whole, s.sq_bytes, s.mp_bytes);
    }
    for (int prec = 0; prec < 3; ++prec) c->fmm[prec] = made[prec];
    return BIE_OK;
}

// Sorts the current geometry's records into the boxes (once per geometry and
// precision, when an application first needs it; work that is only recorded by a stream
// capture has not sorted anything yet).
int fmm_build(bie_ctx* c, int prec) {
    Fmm& f = c->fmm[prec];
    if (!f.on || f.built == c->geometry) return BIE_OK;
    const FmmGeom g{c->x, c->y, c->xw, c->yw, c->imc, c->node_cell};
    FmmTree& t = f.t;
    t.wanted = t.tcount;
    if (c->shard.on) {
        // (the kernels pass over the boxes without a target of the partition's own; whole
        // leaves, so that an owned target's sums stay what they are without it, bit for bit)
        t.wanted = f.owned;
        BIE_CUDA(c, cudaMemsetAsync(f.owned, 0, t.nbox * sizeof(int), c->stream));
    }
    for (int set = 0; set < (c->utilde ? 2 : 1); ++set) {
        const int mul = set ? 1 : c->srcmul, n = c->N * mul;
        int* count = set ? t.tcount : t.scount;
        int* start = set ? t.tstart : t.sstart;
        BIE_CUDA(c, cudaMemsetAsync(count, 0, t.nbox * sizeof(int), c->stream));
        k_fmm_bin<<<(n + 255) / 256, 256, 0, c->stream>>>(g, c->cells, f.cells, f.box, n, mul, set, f.leaf, count,
                                                             c->shard.n0, c->shard.n1,
                                                             c->shard.on && (set || !c->utilde) ? f.owned : nullptr);
        BIE_LAUNCH(c, "k_fmm_bin");
        k_fmm_scan<<<1, 1024, 0, c->stream>>>(count, t.nleaf, start, f.cursor);
        BIE_LAUNCH(c, "k_fmm_scan");
        k_fmm_fill<<<(n + 255) / 256, 256, 0, c->stream>>>(f.leaf, n, f.cursor, f.raw);
        BIE_LAUNCH(c, "k_fmm_fill");
        k_fmm_sort<<<t.nleaf, 64, 0, c->stream>>>(g, c->cells, f.box, start, f.raw, mul, set, set ? t.tperm : t.sperm,
                                                  set ? t.tpos : t.spos, set ? t.tpos64 : t.spos64);
        BIE_LAUNCH(c, "k_fmm_sort");
    }
    k_fmm_lists<<<t.nbox, 128, 0, c->stream>>>(t, c->cells, c->utilde ? 1 : 9);
    BIE_LAUNCH(c, "k_fmm_lists");
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusActive;
    if (cudaStreamIsCapturing(c->stream, &capture) != cudaSuccess) cudaGetLastError();
    if (capture == cudaStreamCaptureStatusNone) f.built = c->geometry;
    return BIE_OK;
}

// bie_apply_static may be captured by the caller and replayed for later geometries: the
// contexts that it takes have their boxes sorted with every geometry, so that no capture
// holds the sorting and every replay finds the current one.  (All other applications end
// in a wait and cannot be captured.)
int fmm_build_static(bie_ctx* c) { return c->N <= kStaticMaxNodes ? fmm_build(c, 0) : BIE_OK; }

template <typename R>
static int up_launch(bie_ctx* c, const double* sigma, int prec, Workspace& ws) {
    const Fmm& f = c->fmm[prec];
    // the per-node records: the direct walls' (single precision, or double), and
    // for velocities_device after a double-precision application
    FmmBodies p{c->x, c->y, c->body, c->body_cell, nullptr, nullptr, ws.bodyF};
    if (!f.walls && prec == 0) p.src32 = c->utilde ? ws.src32n : ws.src32;
    if (!f.walls || prec != 0) p.src64 = ws.src64;
    BIE_CUDA(c, launch_after(fmm_chained(c, prec), k_fmm_up<R>, f.t.nbox + c->nb, 128, 0u, c->stream, f.t, c->cells, reinterpret_cast<const double2*>(sigma), c->w,
                                                          c->utilde ? 2 : 0, (C2<R>*)ws.fsq, (V4<R>*)ws.fmp, ws.ftick,
                                                          fmm_tab<R>(c, prec), p));
    ++c->launches;
    return BIE_OK;
}

int fmm_up(bie_ctx* c, const double* sigma, int prec, Workspace& ws) {
    return prec == 0 ? up_launch<float>(c, sigma, prec, ws)
                     : (prec == 1 ? up_launch<double>(c, sigma, prec, ws) : up_launch<df>(c, sigma, prec, ws));
}

static SideArgs side_args(bie_ctx* c, const double* sigma, int prec, bool walls, Workspace& ws) {
    SideArgs a;
    a.ncell = c->ncell;
    a.m = c->m;
    a.walls = walls ? 1 : 0;
    a.npairs = c->cl.npairs > 0 ? c->cl.pair_base + c->N : nullptr;
    const long long tasks = (walls ? (long long)c->ncell * (2 * c->m * kWallImages + 1) : 0) + c->cl.npairs;
    a.ctas = (int)((tasks + 3) / 4);
    a.wall = c->wall;
    a.bodyF = ws.bodyF;
    a.x = c->x;
    a.y = c->y;
    a.gpart = ws.gpart;
    a.pairs = c->cl.pairs;
    a.node_cell = c->node_cell;
    a.blk_off = c->cl.blk_off;
    a.blocks = prec == 0 ? (const void*)c->cl.blocks32 : (const void*)c->cl.blocks;
    a.body = c->body;
    a.sigma = reinterpret_cast<const double2*>(sigma);
    a.w = c->w;
    a.psum = ws.of_static ? (void*)c->cl.psum_static : (void*)c->cl.psum;
    return a;
}

int close_pairs(bie_ctx* c, const double* sigma, int prec, Workspace& ws, cudaStream_t st) {
    const SideArgs a = side_args(c, sigma, prec, false, ws);
    if (!a.npairs) return BIE_OK;
    if (prec == 0) k_close_pairs<float><<<a.ctas, 128, 0, st>>>(a, c->cells);
    else k_close_pairs<double><<<a.ctas, 128, 0, st>>>(a, c->cells);
    BIE_LAUNCH(c, "k_close_pairs");
    return BIE_OK;
}

template <typename R>
static int across_launch(bie_ctx* c, const double* sigma, int prec, Workspace& ws) {
    const Fmm& f = c->fmm[prec];
    const FmmTree& t = f.t;
    const FmmTab<R> tab = fmm_tab<R>(c, prec);
    const int tiles = 2;
    const int n0 = c->shard.on ? c->shard.n0 : 0, n1 = c->shard.on ? c->shard.n1 : c->N;
    const V4<R>* loc = (const V4<R>*)ws.floc;
    const SideArgs side = side_args(c, sigma, prec, f.walls, ws);
    const bool early = fmm_chained(c, prec);
    BIE_CUDA(c, launch_after(early, k_fmm_m2l<R>, side.ctas + t.nbox * f.shares, 128, 0u, c->stream, t, c->cells,
                             (const V4<R>*)ws.fmp, (V4<R>*)ws.floc, tab, f.shares, side));
    ++c->launches;
    XiArgs xi{c->m, c->M, 0, (2 * c->M + 3) / 4, ws.gpart, c->P, ws.xi, ws.xif};
    if (f.walls) xi.ctas = xi.per_cell * c->ncell;
    const unsigned down = xi.ctas + t.nleaf * tiles;
    if constexpr (sizeof(R) == 4)
        BIE_CUDA(c, launch_after(early, k_fmm_down32, down, 128, 0u, c->stream, t, c->cells, (const C2<float>*)ws.fsq, loc,
                                 f.shares, tab, c->tgt32, n0, n1, (float2*)ws.part, xi, tiles));
    else
        BIE_CUDA(c, launch_after(early, k_fmm_down64<R>, down, 128, 0u, c->stream, t, c->cells, (const C2<R>*)ws.fsq, loc,
                                 f.shares, tab, c->nx, c->ny, prec, n0, n1, (double2*)ws.part, xi, tiles));
    ++c->launches;
    return BIE_OK;
}

int fmm_across(bie_ctx* c, const double* sigma, int prec, Workspace& ws) {
    return prec == 0 ? across_launch<float>(c, sigma, prec, ws)
                     : (prec == 1 ? across_launch<double>(c, sigma, prec, ws)
                                  : across_launch<df>(c, sigma, prec, ws));
}

}  // namespace bie
