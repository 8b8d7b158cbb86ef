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
// Truncation: worst case (two box corners) 0.547^P, typically 1e-2 of that:
// P = 24 in single precision, P = 56 in double.
//
// What bounds it.  Single precision: the pair sum (about 20 instructions per
// pair, a few hundred pairs per target), then latency; double: the FP64 pipe in
// the translations (two DFMA per SM and cycle).  Whole applications on GB300,
// direct sum before and this now: single precision 32.8 -> 0.60 ms on the
// 400-ellipse cell (102400 nodes), 0.94 -> 0.20 ms at 16000 nodes, 0.21 ->
// 0.15 ms at 6400; double-float 338 -> 6.6 ms at 102400; FP64 12.2 -> 1.55 ms
// at 6400.  The single-precision application's error against 64 bits falls
// (8.6e-7 -> 2.0e-7 at 6400 nodes): near pairs are differenced exactly.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "bie_internal.cuh"

namespace bie {

template <typename R>
struct __align__(sizeof(R) * 2) C2 {
    R x, y;
};
// coefficient pair: (a, e) of one order
template <typename R>
struct __align__(16) V4 {
    R x, y, z, w;
};

template <typename R>
__device__ __forceinline__ C2<R> cmul(C2<R> a, C2<R> b) {
    return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename R>
__device__ __forceinline__ R fma_(R a, R b, R c) {
    return fma(a, b, c);
}
// z^n, 0 <= n < 64, by repeated squaring
template <typename R>
__device__ __forceinline__ C2<R> cpow(C2<R> z, int n) {
    C2<R> r{R(1), R(0)};
#pragma unroll
    for (int b = 0; b < 6; ++b) {
        if ((n >> b) & 1) r = cmul(r, z);
        z = cmul(z, z);
    }
    return r;
}
template <typename R>
__device__ __forceinline__ C2<R> cinv(C2<R> z) {
    const R s = R(1) / (z.x * z.x + z.y * z.y);
    return {z.x * s, -z.y * s};
}

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
// set 0: sources, set 1: targets (doubled cell only).
__global__ void k_fmm_bin(FmmGeom g, const Cell* __restrict__ cells, const FmmCell* __restrict__ fc,
                          const int4* __restrict__ box, int n, int mul, int targets, int* __restrict__ leaf,
                          int* __restrict__ count) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int c = g.node_cell[mul == 1 ? r : r >> 2];
    const Cell& cl = cells[c];
    const double2 p = targets ? make_double2(g.xw[r] - cl.C[0], g.yw[r] - cl.C[1]) : fmm_source(g, cl, r, mul);
    int b = fmm_leaf(fc[c], p);
    leaf[r] = b;
    for (; b >= 0; b = box[b].w) atomicAdd(count + b, 1);
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

__device__ __forceinline__ double2 fmm_centre(const FmmCell& f, int level, int ix, int iy) {
    const double H = f.h * (1 << level);
    return make_double2(f.ox + (ix + 0.5) * H, f.oy + (iy + 0.5) * H);
}

// One warp per leaf: gathers the strengths q = sigma w of the box's sources in
// sorted order (sq, or sqdf as double-float pairs) and sums their moments (lane
// k: orders k and k + 32; eta^k = eta^(k % 4) (eta^4)^(k / 4) from two small
// tables per source); the last child of a parent to finish forms the parent's
// moments, and so on up.
template <typename R, int P>
__global__ void __launch_bounds__(128)
k_fmm_up(FmmTree t, const Cell* __restrict__ cells, const double2* __restrict__ sigma, const double* __restrict__ w,
         int shift, C2<R>* __restrict__ sq, float4* __restrict__ sqdf, V4<R>* __restrict__ mp, unsigned* __restrict__ ticket,
         const R* __restrict__ binom) {
    constexpr int ROWS = (P + 31) / 32, HI = (P + 3) / 4;
    __shared__ __align__(16) C2<R> s_lo[4][4][33], s_hi[4][HI][33], s_q[4][32], s_s[4][32];
    static_assert(P * sizeof(V4<R>) <= HI * 33 * sizeof(C2<R>), "translation buffer");
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int b = blockIdx.x * 4 + wid;
    if (b >= t.nleaf) return;
    int4 bx = t.box[b];
    const FmmCell& f = t.cells[bx.x];
    if (!cells[bx.x].active) return;
    const int s0 = t.sstart[b], s1 = t.sstart[b + 1];
    if (s1 > s0) {
        const double2 c = fmm_centre(f, 0, fmm_ix(bx), fmm_iy(bx));
        float4 cf;
        split_df(c.x, cf.x, cf.y);
        split_df(c.y, cf.z, cf.w);
        // real moments of q_x and q_y (complex each) and of s = q conj(eta)
        C2<R> X[ROWS], Y[ROWS], D[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) X[r] = Y[r] = D[r] = {R(0), R(0)};
        for (int k0 = s0; k0 < s1; k0 += 32) {
            const int s = k0 + lane, cnt = min(32, s1 - k0);
            C2<R> eta{R(0), R(0)}, q{R(0), R(0)};
            if (lane < cnt) {
                if constexpr (sizeof(R) == 4) {
                    eta = fmm_local(t.spos[s], cf, (float)f.inv_h);
                } else {
                    const double2 p = t.spos64[s];
                    eta = {(p.x - c.x) * f.inv_h, (p.y - c.y) * f.inv_h};
                }
                const int i = t.sperm[s] >> shift;
                const double2 sg = sigma[i];
                const double wi = w[i];
                q = {(R)(sg.x * wi), (R)(sg.y * wi)};
                if (sqdf) {
                    float4 v;
                    split_df((double)q.x, v.x, v.y);
                    split_df((double)q.y, v.z, v.w);
                    sqdf[s] = v;
                } else {
                    sq[s] = q;
                }
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
            s_s[wid][lane] = {q.x * eta.x + q.y * eta.y, q.y * eta.x - q.x * eta.y};
            __syncwarp();
            for (int j = 0; j < cnt; ++j) {
                const C2<R> qj = s_q[wid][j], sj = s_s[wid][j], lo = s_lo[wid][lane & 3][j];
#pragma unroll
                for (int r = 0; r < ROWS; ++r) {
                    const int a = (lane >> 2) + 8 * r;
                    if (a < HI) {
                        const C2<R> pw = cmul(lo, s_hi[wid][a][j]);
                        X[r].x = fma_(qj.x, pw.x, X[r].x);
                        X[r].y = fma_(qj.x, pw.y, X[r].y);
                        Y[r].x = fma_(qj.y, pw.x, Y[r].x);
                        Y[r].y = fma_(qj.y, pw.y, Y[r].y);
                        D[r].x = fma_(sj.x, pw.x, fma_(-sj.y, pw.y, D[r].x));
                        D[r].y = fma_(sj.x, pw.y, fma_(sj.y, pw.x, D[r].y));
                    }
                }
            }
        }
        // a = X + i Y, b = X - i Y, e_k = b_k - k d_{k-1}
        C2<R> carry{R(0), R(0)};
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int k = lane + 32 * r;
            C2<R> d{__shfl_up_sync(0xffffffffu, D[r].x, 1), __shfl_up_sync(0xffffffffu, D[r].y, 1)};
            if (lane == 0) d = carry;
            carry = {__shfl_sync(0xffffffffu, D[r].x, 31), __shfl_sync(0xffffffffu, D[r].y, 31)};
            if (k < P)
                mp[(size_t)b * P + k] = {X[r].x - Y[r].y, X[r].y + Y[r].x, X[r].x + Y[r].y - R(k) * d.x,
                                         X[r].y - Y[r].x - R(k) * d.y};
        }
    }
    // parents (a warp's power table is free now: it holds the translated series)
    V4<R>* s_v = reinterpret_cast<V4<R>*>(&s_hi[wid][0][0]);
    for (int level = 0; bx.w >= 0; ++level) {
        const int parent = bx.w;
        const int px = fmm_ix(t.box[parent]), py = fmm_iy(t.box[parent]);
        const int nx = min(2, f.gx[level] - 2 * px), ny = min(2, f.gy[level] - 2 * py);
        __threadfence();
        __syncwarp();
        unsigned old = 0;
        if (lane == 0) old = atomicAdd(ticket + parent, 1u);
        old = __shfl_sync(0xffffffffu, old, 0);
        if (old != (unsigned)(nx * ny) - 1) return;
        __threadfence();
        if (lane == 0) ticket[parent] = 0u;
        V4<R> acc[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) acc[r] = {R(0), R(0), R(0), R(0)};
        for (int q = 0; q < nx * ny; ++q) {
            const int jx = q % nx, jy = q / nx;
            const int child = f.off[level] + (2 * py + jy) * f.gx[level] + 2 * px + jx;
            if (t.scount[child] == 0) continue;
            const C2<R> dl{jx ? R(0.25) : R(-0.25), jy ? R(0.25) : R(-0.25)};
            // child's unit is half the parent's: v_k = a_k (1/2)^k delta^-k = a_k (1 / (2 delta))^k
            const C2<R> g = cinv(C2<R>{2 * dl.x, 2 * dl.y});
            C2<R> carry{R(0), R(0)};
            __syncwarp();
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const int k = lane + 32 * r;
                V4<R> m{R(0), R(0), R(0), R(0)};
                if (k < P) {
                    const R* src = reinterpret_cast<const R*>(mp + (size_t)child * P + k);
                    m = {__ldcg(src), __ldcg(src + 1), __ldcg(src + 2), __ldcg(src + 3)};
                }
                C2<R> pa{__shfl_up_sync(0xffffffffu, m.x, 1), __shfl_up_sync(0xffffffffu, m.y, 1)};
                if (lane == 0) pa = carry;
                carry = {__shfl_sync(0xffffffffu, m.x, 31), __shfl_sync(0xffffffffu, m.y, 31)};
                // e_k - conj(delta) k a_{k-1}, delta in the child's unit: 2 dl
                m.z -= R(2 * k) * (dl.x * pa.x + dl.y * pa.y);
                m.w -= R(2 * k) * (dl.x * pa.y - dl.y * pa.x);
                const C2<R> pg = cpow(g, k);
                if (k < P) {
                    const C2<R> va = cmul(pg, C2<R>{m.x, m.y}), ve = cmul(pg, C2<R>{m.z, m.w});
                    s_v[k] = {va.x, va.y, ve.x, ve.y};
                }
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const int m = lane + 32 * r;
                if (m < P) {
                    V4<R> s{R(0), R(0), R(0), R(0)};
                    for (int k = 0; k <= m; ++k) {
                        const R cb = binom[(size_t)k * P + m];  // C(m, k)
                        const V4<R> v = s_v[k];
                        s.x = fma_(cb, v.x, s.x);
                        s.y = fma_(cb, v.y, s.y);
                        s.z = fma_(cb, v.z, s.z);
                        s.w = fma_(cb, v.w, s.w);
                    }
                    const C2<R> pd = cpow(dl, m);
                    const C2<R> ra = cmul(pd, C2<R>{s.x, s.y}), re = cmul(pd, C2<R>{s.z, s.w});
                    acc[r].x += ra.x;
                    acc[r].y += ra.y;
                    acc[r].z += re.x;
                    acc[r].w += re.y;
                }
            }
        }
        if (t.scount[parent] > 0)
#pragma unroll
            for (int r = 0; r < ROWS; ++r)
                if (lane + 32 * r < P) mp[(size_t)parent * P + lane + 32 * r] = acc[r];
        bx = t.box[parent];
    }
}

// ---------------------------------------------------------------------------
// across: local expansion of every target box from the far boxes whose
// parents are near
// ---------------------------------------------------------------------------
// Boxes ix and jx (under a shift of s sides) near in one coordinate: centres
// closer than two sides.  One expression everywhere, so that a level's far
// list, its children's and the pair sum's rows partition the pairs exactly.
__device__ __forceinline__ bool fmm_close(int ix, int jx, double s) { return fabs((double)(ix - jx) - s) < 2.0 - 1e-9; }
constexpr int kFmmList = 512;            // far boxes listed at a time

// One CTA per target box (all levels).  Its threads scan the candidate (box,
// image) pairs, compact the far ones into shared memory in a fixed order, and
// the warps translate them in turn (lane l: orders l and l + 32).
template <typename R, int P>
__global__ void __launch_bounds__(128)
k_fmm_m2l(FmmTree t, const Cell* __restrict__ cells, int nimg, const V4<R>* __restrict__ mp, V4<R>* __restrict__ loc,
          const R* __restrict__ hankel) {
    constexpr int ROWS = (P + 31) / 32;
    __shared__ int s_src[kFmmList];
    __shared__ C2<R> s_z[kFmmList];
    __shared__ V4<R> s_v[4][P];
    __shared__ int s_n[4];
    const int b = blockIdx.x, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (t.tcount[b] == 0) return;
    const int4 bx = t.box[b];
    const FmmCell& f = t.cells[bx.x];
    const Cell& cl = cells[bx.x];
    if (!cl.active) return;
    const int level = bx.y, ix = fmm_ix(bx), iy = fmm_iy(bx);
    const bool top = level == f.nlev - 1;
    const int gx = f.gx[level], gy = f.gy[level];
    const double H = f.h * (1 << level), inv = 1.0 / H;
    const int per = top ? gx * gy : 64;
    V4<R> acc[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) acc[r] = {R(0), R(0), R(0), R(0)};
    R row[sizeof(R) == 4 ? P : 1];  // single precision: lane l's row of the matrix in registers
    if constexpr (sizeof(R) == 4) {
#pragma unroll
        for (int k = 0; k < P; ++k) row[k] = lane < P ? hankel[(size_t)k * P + lane] : R(0);
    }
    int listed = 0;
    const int ncand = per * nimg;
    for (int q0 = 0; q0 < ncand; q0 += 128) {
        const int q = q0 + threadIdx.x;
        bool far = false;
        int src = 0;
        double zx = 0, zy = 0;
        if (q < ncand) {
            const int im = nimg == 1 ? 4 : q / per, e = nimg == 1 ? q : q % per;
            const double sx = cl.sx[im] * inv, sy = cl.sy[im] * inv;  // sides of this level
            int jx, jy;
            bool ok = true;
            if (top) {
                jx = e % gx;
                jy = e / gx;
            } else {
                // children of the (up to 4 x 4) near parents
                const int kx = ix >> 1, ky = iy >> 1;
                const int px = (int)floor(kx - 0.5 * sx - 2.0) + 1 + (e & 7) / 2;
                const int py = (int)floor(ky - 0.5 * sy - 2.0) + 1 + (e >> 3) / 2;
                ok = fmm_close(kx, px, 0.5 * sx) && fmm_close(ky, py, 0.5 * sy);
                jx = 2 * px + (e & 1);
                jy = 2 * py + ((e >> 3) & 1);
            }
            if (ok && jx >= 0 && jx < gx && jy >= 0 && jy < gy) {
                zx = (ix - jx) - sx;
                zy = (iy - jy) - sy;
                src = f.off[level] + jy * gx + jx;
                far = !(fmm_close(ix, jx, sx) && fmm_close(iy, jy, sy)) && t.scount[src] > 0;
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, far);
        if (lane == 0) s_n[wid] = __popc(m);
        __syncthreads();
        int at = listed, all = listed;
        for (int k = 0; k < 4; ++k) {
            if (k < wid) at += s_n[k];
            all += s_n[k];
        }
        if (far) {
            at += __popc(m & ((1u << lane) - 1));
            s_src[at] = src;
            s_z[at] = {(R)zx, (R)zy};
        }
        __syncthreads();
        listed = all;
        if (listed <= kFmmList - 128 && q0 + 128 < ncand) continue;
        V4<R> nxt[ROWS];
        auto fetch = [&](int e) {
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const int k = lane + 32 * r;
                nxt[r] = {R(0), R(0), R(0), R(0)};
                if (e < listed && k < P) nxt[r] = mp[(size_t)s_src[e] * P + k];
            }
        };
        fetch(wid);
        for (int e = wid; e < listed; e += 4) {
            const C2<R> z = s_z[e], u = cinv(z);
            C2<R> pw[ROWS], carry{R(0), R(0)};
            V4<R> m4[ROWS];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) m4[r] = nxt[r];
            fetch(e + 4);
            pw[0] = cpow(u, lane);
            if constexpr (ROWS > 1) {
                C2<R> u32 = u;
#pragma unroll
                for (int k = 0; k < 5; ++k) u32 = cmul(u32, u32);
                pw[1] = cmul(pw[0], u32);
            }
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const int k = lane + 32 * r;
                C2<R> pa{__shfl_up_sync(0xffffffffu, m4[r].x, 1), __shfl_up_sync(0xffffffffu, m4[r].y, 1)};
                if (lane == 0) pa = carry;
                carry = {__shfl_sync(0xffffffffu, m4[r].x, 31), __shfl_sync(0xffffffffu, m4[r].y, 31)};
                // e_k + conj(z0) k a_{k-1}
                const C2<R> ev{m4[r].z + R(k) * (z.x * pa.x + z.y * pa.y), m4[r].w + R(k) * (z.x * pa.y - z.y * pa.x)};
                const C2<R> pu = cmul(pw[r], u);
                const C2<R> va = cmul(pu, C2<R>{m4[r].x, m4[r].y}), ve = cmul(pu, ev);
                if (k < P) s_v[wid][k] = {va.x, va.y, ve.x, ve.y};
            }
            __syncwarp();
            V4<R> s[ROWS];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) s[r] = {R(0), R(0), R(0), R(0)};
            if constexpr (sizeof(R) == 4) {
#pragma unroll
                for (int k = 0; k < P; ++k) {
                    const V4<R> v = s_v[wid][k];
                    s[0].x = fma_(row[k], v.x, s[0].x);
                    s[0].y = fma_(row[k], v.y, s[0].y);
                    s[0].z = fma_(row[k], v.z, s[0].z);
                    s[0].w = fma_(row[k], v.w, s[0].w);
                }
            } else {
#pragma unroll 4
                for (int k = 0; k < P; ++k) {
                    const V4<R> v = s_v[wid][k];
#pragma unroll
                    for (int r = 0; r < ROWS; ++r) {
                        const int l = lane + 32 * r;
                        const R c = l < P ? __ldg(hankel + (size_t)k * P + l) : R(0);
                        s[r].x = fma_(c, v.x, s[r].x);
                        s[r].y = fma_(c, v.y, s[r].y);
                        s[r].z = fma_(c, v.z, s[r].z);
                        s[r].w = fma_(c, v.w, s[r].w);
                    }
                }
            }
            __syncwarp();
            const R sg = (lane & 1) ? R(-1) : R(1);  // (-1)^l, l = lane or lane + 32
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const C2<R> pl{sg * pw[r].x, sg * pw[r].y};
                const C2<R> ra = cmul(pl, C2<R>{s[r].x, s[r].y}), re = cmul(pl, C2<R>{s[r].z, s[r].w});
                acc[r].x += ra.x;
                acc[r].y += ra.y;
                acc[r].z += re.x;
                acc[r].w += re.y;
            }
        }
        listed = 0;
        __syncthreads();
    }
    // the warps' sums, in warp order
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
        if (lane + 32 * r < P) s_v[wid][lane + 32 * r] = acc[r];
    __syncthreads();
    for (int k = threadIdx.x; k < P; k += 128) {
        V4<R> s = s_v[0][k];
#pragma unroll
        for (int q = 1; q < 4; ++q) {
            s.x += s_v[q][k].x;
            s.y += s_v[q][k].y;
            s.z += s_v[q][k].z;
            s.w += s_v[q][k].w;
        }
        loc[(size_t)b * P + k] = s;
    }
}

// ---------------------------------------------------------------------------
// down: at every target, the ancestors' expansions moved to its leaf and the
// near boxes pair by pair
// ---------------------------------------------------------------------------
// The sources of a near row of boxes are contiguous: a range of sorted records
// under one image shift.
struct FmmRange {
    int s0, s1, im;
};
constexpr int kFmmRanges = 36;  // 9 images x 4 rows

// The local expansion of a leaf with its ancestors' moved to its centre, in
// s_l[0]: warp w moves levels w, w + 4, ... (level 0 is the leaf's own); every
// thread of the 128 takes part.
template <typename R, int P>
__device__ __forceinline__ void fmm_local_to_leaf(const FmmTree& t, const FmmCell& f, int4 bx, const V4<R>* loc,
                                                  const R* binom, V4<R> (*s_l)[P], int wid, int lane) {
    V4<R>* s_v = s_l[wid];
    constexpr int ROWS = (P + 31) / 32;
    V4<R> acc[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) acc[r] = {R(0), R(0), R(0), R(0)};
    for (int level = wid; level < f.nlev; level += 4) {
        const int jx = fmm_ix(bx) >> level, jy = fmm_iy(bx) >> level;
        const int b = f.off[level] + jy * f.gx[level] + jx;
        const V4<R>* src = loc + (size_t)b * P;
        if (level == 0) {
#pragma unroll
            for (int r = 0; r < ROWS; ++r)
                if (lane + 32 * r < P) acc[r] = src[lane + 32 * r];
            continue;
        }
        // leaf centre minus ancestor centre, in the ancestor's unit
        const R u = R(1) / R(1 << level);
        const C2<R> d{(R(fmm_ix(bx)) + R(0.5)) * u - (R(jx) + R(0.5)), (R(fmm_iy(bx)) + R(0.5)) * u - (R(jy) + R(0.5))};
        __syncwarp();
        C2<R> next_a{R(0), R(0)};
#pragma unroll
        for (int r = ROWS - 1; r >= 0; --r) {
            const int l = lane + 32 * r;
            V4<R> m{R(0), R(0), R(0), R(0)};
            if (l < P) m = src[l];
            C2<R> na{__shfl_down_sync(0xffffffffu, m.x, 1), __shfl_down_sync(0xffffffffu, m.y, 1)};
            if (lane == 31) na = next_a;
            next_a = {__shfl_sync(0xffffffffu, m.x, 0), __shfl_sync(0xffffffffu, m.y, 0)};
            // e_l - conj(d) (l + 1) a_{l+1}
            m.z -= R(l + 1) * (d.x * na.x + d.y * na.y);
            m.w -= R(l + 1) * (d.x * na.y - d.y * na.x);
            const C2<R> pd = cpow(d, l);
            if (l < P) {
                const C2<R> va = cmul(pd, C2<R>{m.x, m.y}), ve = cmul(pd, C2<R>{m.z, m.w});
                s_v[l] = {va.x, va.y, ve.x, ve.y};
            }
        }
        __syncwarp();
        const C2<R> g = cinv(d);
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int m = lane + 32 * r;
            V4<R> s{R(0), R(0), R(0), R(0)};
            if (m < P)
                for (int l = m; l < P; ++l) {
                    const R cb = binom[(size_t)m * P + l];  // C(l, m)
                    const V4<R> v = s_v[l];
                    s.x = fma_(cb, v.x, s.x);
                    s.y = fma_(cb, v.y, s.y);
                    s.z = fma_(cb, v.z, s.z);
                    s.w = fma_(cb, v.w, s.w);
                }
            // to the leaf's unit: 2^-level per order and one more for the field's own scale
            C2<R> pg = cpow(C2<R>{g.x * u, g.y * u}, m);
            pg = {pg.x * u, pg.y * u};
            const C2<R> ra = cmul(pg, C2<R>{s.x, s.y}), re = cmul(pg, C2<R>{s.z, s.w});
            acc[r].x += ra.x;
            acc[r].y += ra.y;
            acc[r].z += re.x;
            acc[r].w += re.y;
        }
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
        if (lane + 32 * r < P) s_v[lane + 32 * r] = acc[r];
    __syncthreads();
    for (int k = threadIdx.x; k < P; k += 128) {
        V4<R> s = s_l[0][k];
#pragma unroll
        for (int q = 1; q < 4; ++q) {
            s.x += s_l[q][k].x;
            s.y += s_l[q][k].y;
            s.z += s_l[q][k].z;
            s.w += s_l[q][k].w;
        }
        s_l[0][k] = s;
    }
    __syncthreads();
}

// Traction of the local expansion at W (leaf units) with normal n, times 4 pi h
template <typename R, int P>
__device__ __forceinline__ C2<R> fmm_local_at(const V4<R>* c, C2<R> W, R nx, R ny) {
    C2<R> A{R(0), R(0)}, dA{R(0), R(0)}, E{R(0), R(0)};
    for (int l = P - 1; l >= 0; --l) {
        const V4<R> v = c[l];
        dA = {fma_(dA.x, W.x, fma_(-dA.y, W.y, A.x)), fma_(dA.x, W.y, fma_(dA.y, W.x, A.y))};
        A = {fma_(A.x, W.x, fma_(-A.y, W.y, v.x)), fma_(A.x, W.y, fma_(A.y, W.x, v.y))};
        E = {fma_(E.x, W.x, fma_(-E.y, W.y, v.z)), fma_(E.x, W.y, fma_(E.y, W.x, v.w))};
    }
    // F = E - conj(W) A';  -(2 n Re A + conj(n F))
    const C2<R> F{E.x - (W.x * dA.x + W.y * dA.y), E.y - (W.x * dA.y - W.y * dA.x)};
    return {-(2 * nx * A.x + nx * F.x - ny * F.y), -(2 * ny * A.x - (nx * F.y + ny * F.x))};
}

// Near rows of a leaf's targets, compacted in (image, row) order by warp 0.
__device__ __forceinline__ int fmm_ranges(const FmmTree& t, const FmmCell& f, const Cell& cl, int4 bx, int nimg,
                                          FmmRange* out, int lane) {
    int n = 0;
    for (int q0 = 0; q0 < 4 * nimg; q0 += 32) {
        const int q = q0 + lane;
        FmmRange r{0, 0, 0};
        if (q < 4 * nimg) {
            r.im = nimg == 1 ? 4 : q >> 2;
            const double sx = cl.sx[r.im] * f.inv_h, sy = cl.sy[r.im] * f.inv_h;
            const int ix = fmm_ix(bx), iy = fmm_iy(bx);
            const int jy = (int)floor(iy - sy - 2.0) + 1 + (q & 3);
            if (fmm_close(iy, jy, sy) && jy >= 0 && jy < f.gy[0]) {
                int x0 = (int)floor(ix - sx - 2.0) + 1, x1 = x0 + 3;
                if (!fmm_close(ix, x0, sx)) ++x0;
                if (!fmm_close(ix, x1, sx)) --x1;
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

// Single precision.  One CTA per (leaf, tile share): four warps share the
// tile's 64 targets (two per lane) and split the near sources; the double-
// float positions make every difference exact to single precision, so no
// later pass has to redo near pairs.
__global__ void __launch_bounds__(128, 6)
k_fmm_down32(FmmTree t, const Cell* __restrict__ cells, int nimg, const C2<float>* __restrict__ sq,
             const V4<float>* __restrict__ loc, const float* __restrict__ binom, const float4* __restrict__ tgt32,
             int n0, int n1, float2* __restrict__ part) {
    constexpr int P = kFmmP32;
    __shared__ V4<float> s_l[4][P];
    __shared__ FmmRange s_r[kFmmRanges];
    __shared__ int s_nr;
    __shared__ float4 s_p[4][32];
    __shared__ float2 s_q[4][32];
    __shared__ float2 s_acc[4][64];
    const int b = blockIdx.x, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = t.tstart[b], t1 = t.tstart[b + 1];
    if (t0 + 64 * (int)blockIdx.y >= t1) return;
    const int4 bx = t.box[b];
    const FmmCell& f = t.cells[bx.x];
    const Cell& cl = cells[bx.x];
    if (!cl.active) return;
    if (wid == 0) {
        const int n = fmm_ranges(t, f, cl, bx, nimg, s_r, lane);
        if (lane == 0) s_nr = n;
    }
    fmm_local_to_leaf<float, P>(t, f, bx, loc, binom, s_l, wid, lane);
    const int nr = s_nr;
    const double2 c = fmm_centre(f, 0, fmm_ix(bx), fmm_iy(bx));
    float4 cf;
    split_df(c.x, cf.x, cf.y);
    split_df(c.y, cf.z, cf.w);
    const float inv_h = (float)f.inv_h;
    for (int k0 = t0 + 64 * blockIdx.y; k0 < t1; k0 += 64 * gridDim.y) {
        const bool two = t1 - k0 > 32;  // uniform: the second target of every lane
        float4 p[2];
        float nx[2], ny[2], ax[2] = {0.f, 0.f}, ay[2] = {0.f, 0.f};
        int node[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int k = k0 + lane + 32 * q;
            node[q] = k < t1 ? t.tperm[k] : -1;
            if (node[q] >= 0 && (node[q] < n0 || node[q] >= n1) && node[q] != cl.node_off) node[q] = -1;
            p[q] = make_float4(1e4f, 0.f, 1e4f, 0.f);
            nx[q] = ny[q] = 0.f;
            if (node[q] >= 0) {
                p[q] = t.tpos[k];
                const float4 tv = tgt32[node[q]];
                nx[q] = tv.z;
                ny[q] = tv.w;
            }
        }
        int turn = 0;
        for (int r = 0; r < nr; ++r) {
            const FmmRange rg = s_r[r];
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
                    for (int j = 0; j < cnt; ++j) pair(0, s_p[wid][j], s_q[wid][j]);
                }
            }
        }
        __syncthreads();
        s_acc[wid][lane] = make_float2(ax[0], ay[0]);
        s_acc[wid][lane + 32] = make_float2(ax[1], ay[1]);
        __syncthreads();
        if (wid < 2) {  // warp 0 finishes the first 32 targets, warp 1 the others
            const int nd = wid ? node[1] : node[0];
            const float4 pt = wid ? p[1] : p[0];
            if (nd >= 0) {
                float sx = 0.f, sy = 0.f;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    sx += s_acc[q][lane + 32 * wid].x;
                    sy += s_acc[q][lane + 32 * wid].y;
                }
                const C2<float> W = fmm_local(pt, cf, inv_h);
                const C2<float> F = fmm_local_at<float, P>(s_l[0], W, wid ? nx[1] : nx[0], wid ? ny[1] : ny[0]);
                const float g = (float)(1.0 / (4.0 * kPi)) * inv_h, cp = (float)(-1.0 / kPi);
                part[cl.part_off[0] + (nd - cl.node_off)] = make_float2(fmaf(cp, sx, g * F.x), fmaf(cp, sy, g * F.y));
            }
        }
    }
}

// 1 / x by the hardware's approximation (20 bits) and one step of the cubic
// iteration r <- r (1 + e + e^2), e = 1 - x r
__device__ __forceinline__ double rcp64(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// Double precision (DF: the pairs in double-float arithmetic on the FP32 pipe).
// One CTA per (leaf, tile share): four warps share a tile of 32 targets and
// split the near sources.
template <bool DF>
__global__ void __launch_bounds__(128, 4)
k_fmm_down64(FmmTree t, const Cell* __restrict__ cells, int nimg, const C2<double>* __restrict__ sq,
             const float4* __restrict__ sqdf, const V4<double>* __restrict__ loc, const double* __restrict__ binom,
             const double* __restrict__ nxv, const double* __restrict__ nyv, int prec, int n0, int n1,
             double2* __restrict__ part) {
    constexpr int P = kFmmP64;
    __shared__ V4<double> s_l[4][P];
    __shared__ FmmRange s_r[kFmmRanges];
    __shared__ int s_nr;
    __shared__ double2 s_p[4][32], s_q[4][32];  // double-float: a float4 each
    __shared__ double2 s_acc[4][32];
    const int b = blockIdx.x, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = t.tstart[b], t1 = t.tstart[b + 1];
    if (t0 + 32 * (int)blockIdx.y >= t1) return;
    const int4 bx = t.box[b];
    const FmmCell& f = t.cells[bx.x];
    const Cell& cl = cells[bx.x];
    if (!cl.active) return;
    if (wid == 0) {
        const int n = fmm_ranges(t, f, cl, bx, nimg, s_r, lane);
        if (lane == 0) s_nr = n;
    }
    fmm_local_to_leaf<double, P>(t, f, bx, loc, binom, s_l, wid, lane);
    const int nr = s_nr;
    const double2 c = fmm_centre(f, 0, fmm_ix(bx), fmm_iy(bx));
    for (int k0 = t0 + 32 * blockIdx.y; k0 < t1; k0 += 32 * gridDim.y) {
        const int k = k0 + lane;
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
            const FmmRange rg = s_r[r];
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
                        *reinterpret_cast<float4*>(&s_q[wid][lane]) = sqdf[s];
                    } else {
                        s_p[wid][lane] = t.spos64[s];
                        s_q[wid][lane] = make_double2(sq[s].x, sq[s].y);
                    }
                }
                __syncwarp();
                if constexpr (DF) {
                    // chunk sums as (TwoSum high part, float error), folded into
                    // double after every chunk
                    float axh = 0, axe = 0, ayh = 0, aye = 0;
                    for (int j = 0; j < cnt; ++j) {
                        const float4 sp = *reinterpret_cast<const float4*>(&s_p[wid][j]);
                        const float4 ss = *reinterpret_cast<const float4*>(&s_q[wid][j]);
                        pair_df(pxh, pxl, pyh, pyl, nxh, nxl, nyh, nyl,
                                SrcDF{sp.x, sp.y, sp.z, sp.w, ss.x, ss.y, ss.z, ss.w}, axh, axe, ayh, aye);
                    }
                    ax += (double)axh + (double)axe;
                    ay += (double)ayh + (double)aye;
                } else {
#pragma unroll 2
                    for (int j = 0; j < cnt; ++j) {
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
        __syncthreads();
        s_acc[wid][lane] = make_double2(ax, ay);
        __syncthreads();
        if (wid == 0 && node >= 0) {
            double sx = 0, sy = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                sx += s_acc[q][lane].x;
                sy += s_acc[q][lane].y;
            }
            const C2<double> W{(p.x - c.x) * f.inv_h, (p.y - c.y) * f.inv_h};
            const C2<double> F = fmm_local_at<double, P>(s_l[0], W, nx, ny);
            const double g = f.inv_h / (4.0 * kPi), cp = -1.0 / kPi;
            part[cl.part_off[prec] + (node - cl.node_off)] = make_double2(fma(cp, sx, g * F.x), fma(cp, sy, g * F.y));
        }
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
static constexpr double kLeafPair[3] = {1.0e-12, 25e-12, 4.5e-12};
static constexpr double kTranslate[3] = {0.5e-9, 26e-9, 26e-9};
static constexpr double kFmmFixed[3] = {12e-6, 20e-6, 20e-6};

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

void free_fmm(bie_ctx* c) {
    for (Fmm& f : c->fmm) {
        for (void* p : f.owned)
            if (p) cudaFree(p);
        f = Fmm{};
    }
    for (void*& p : c->fmm_tab) {
        if (p) cudaFree(p);
        p = nullptr;
    }
    for (void* p : {c->ws.fsq, c->ws.fmp, c->ws.floc, (void*)c->ws.ftick})
        if (p) cudaFree(p);
    c->ws.fsq = c->ws.fmp = c->ws.floc = nullptr;
    c->ws.ftick = nullptr;
}

template <typename R>
static int fmm_tables(bie_ctx* c, int P, void** out) {
    // [C(k + l, l)], [k][l]; then [C(m, k)], [k][m] (0 for k > m)
    std::vector<R> t(2 * (size_t)P * P);
    std::vector<std::vector<long double>> b(2 * P, std::vector<long double>(2 * P, 0.0L));
    for (int n = 0; n < 2 * P; ++n) {
        b[n][0] = 1;
        for (int k = 1; k <= n; ++k) b[n][k] = b[n - 1][k - 1] + (k <= n - 1 ? b[n - 1][k] : 0.0L);
    }
    for (int k = 0; k < P; ++k)
        for (int l = 0; l < P; ++l) {
            t[(size_t)k * P + l] = (R)b[k + l][l];
            t[(size_t)(P + k) * P + l] = (R)b[l][k];
        }
    BIE_CUDA(c, cudaMalloc(out, t.size() * sizeof(R)));
    BIE_CUDA(c, cudaMemcpy(*out, t.data(), t.size() * sizeof(R), cudaMemcpyHostToDevice));
    return BIE_OK;
}

// Boxes of every precision whose near sums run faster this way.  Called when
// a context is made and when a configuration is set; a plan whose rectangles
// still hold every body is kept.
int fmm_plan(bie_ctx* c) {
    std::vector<FmmPlanCell> rect(c->ncell);
    for (int k = 0; k < c->ncell; ++k) rect[k] = fmm_rect(c, k);
    if (!c->fmm_rects.empty()) {
        bool holds = true;
        for (int k = 0; k < c->ncell; ++k) {
            const double* o = &c->fmm_rects[4 * (size_t)k];
            holds = holds && rect[k].ox >= o[0] && rect[k].oy >= o[1] && rect[k].ox + rect[k].w <= o[0] + o[2] &&
                    rect[k].oy + rect[k].ht <= o[1] + o[3];
        }
        if (holds) return BIE_OK;
        ++c->epoch;
        free_fmm(c);
    }
    c->fmm_rects.resize(4 * (size_t)c->ncell);
    for (int k = 0; k < c->ncell; ++k) {
        double* o = &c->fmm_rects[4 * (size_t)k];
        o[0] = rect[k].ox;
        o[1] = rect[k].oy;
        o[2] = rect[k].w;
        o[3] = rect[k].ht;
    }
    if (!BIE_FMM) return BIE_OK;
    std::vector<double> per(c->nb);
    for (int b = 0; b < c->nb; ++b) per[b] = body_perimeter(c, b);
    const int N = c->N, nsrc = N * c->srcmul;
    size_t mp_bytes = 0, sq_bytes = 0;
    int max_box = 0;
    for (int prec = 0; prec < 3; ++prec) {
        Fmm& f = c->fmm[prec];
        std::vector<FmmCell> cells(c->ncell);
        double t_fast = kFmmFixed[prec], t_direct = 0;
        long long nleaf = 0, nbox = 0;
        for (int k = 0; k < c->ncell; ++k) {
            const Cell& cl = c->cells_h[k];
            const FmmPlanCell& rc = rect[k];
            FmmCell& fc = cells[k];
            // leaf side: the modelled best of a geometric ladder, with at most
            // one box per 8 source records (64 at least)
            const double most = std::max(64.0, cl.n_nodes * (double)c->srcmul / 8);
            double best = INFINITY, bh = 0;
            for (int j = 0; j < 48; ++j) {
                const double h = std::sqrt(rc.area) * std::pow(2.0, -0.25 * j);
                if (std::ceil(rc.w / h) * std::ceil(rc.ht / h) * 1.34 + 8 > most) break;
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
            fc.off[0] = (int)nleaf;
            nleaf += (long long)fc.gx[0] * fc.gy[0];
        }
        f.on = t_fast < t_direct && nleaf < (1 << 26);
        if (!f.on) continue;
        // leaves of all cells first, then the coarser levels cell by cell
        nbox = nleaf;
        for (FmmCell& fc : cells)
            for (int l = 1; l < fc.nlev; ++l) {
                fc.off[l] = (int)nbox;
                nbox += (long long)fc.gx[l] * fc.gy[l];
            }
        std::vector<int4> box(nbox);
        for (int k = 0; k < c->ncell; ++k) {
            const FmmCell& fc = cells[k];
            for (int l = 0; l < fc.nlev; ++l)
                for (int y = 0; y < fc.gy[l]; ++y)
                    for (int x = 0; x < fc.gx[l]; ++x)
                        box[fc.off[l] + (size_t)y * fc.gx[l] + x] =
                            make_int4(k, l, x | (y << 16),
                                      l + 1 < fc.nlev ? fc.off[l + 1] + (y / 2) * fc.gx[l + 1] + x / 2 : -1);
        }
        const bool dbl = prec != 0;
        auto get = [&](void* pp, size_t bytes) -> int {
            void* p = nullptr;
            BIE_CUDA(c, cudaMalloc(&p, bytes + 16));
            f.owned.push_back(p);
            std::memcpy(pp, &p, sizeof p);
            return BIE_OK;
        };
        FmmTree& t = f.t;
        t.nleaf = (int)nleaf;
        t.nbox = (int)nbox;
        int rc = get(&f.cells, cells.size() * sizeof(FmmCell));
        rc = rc ? rc : get(&f.box, box.size() * sizeof(int4));
        rc = rc ? rc : get(&t.scount, nbox * sizeof(int));
        rc = rc ? rc : get(&t.sstart, (nleaf + 1) * sizeof(int));
        rc = rc ? rc : get(&t.sperm, nsrc * sizeof(int));
        rc = rc ? rc : get(&f.cursor, nleaf * sizeof(int));
        rc = rc ? rc : get(&f.leaf, nsrc * sizeof(int));
        rc = rc ? rc : get(&f.raw, nsrc * sizeof(int));
        if (prec != 1) rc = rc ? rc : get(&t.spos, nsrc * sizeof(float4));
        if (dbl) rc = rc ? rc : get(&t.spos64, nsrc * sizeof(double2));
        t.tcount = t.scount;
        t.tstart = t.sstart;
        t.tperm = t.sperm;
        t.tpos = t.spos;
        t.tpos64 = t.spos64;
        if (c->utilde) {
            t.tpos = nullptr;
            t.tpos64 = nullptr;
            rc = rc ? rc : get(&t.tcount, nbox * sizeof(int));
            rc = rc ? rc : get(&t.tstart, (nleaf + 1) * sizeof(int));
            rc = rc ? rc : get(&t.tperm, N * sizeof(int));
            if (!dbl) rc = rc ? rc : get(&t.tpos, N * sizeof(float4));
            if (dbl) rc = rc ? rc : get(&t.tpos64, N * sizeof(double2));
        }
        if (rc) return rc;
        BIE_CUDA(c, cudaMemcpy(f.cells, cells.data(), cells.size() * sizeof(FmmCell), cudaMemcpyHostToDevice));
        BIE_CUDA(c, cudaMemcpy(f.box, box.data(), box.size() * sizeof(int4), cudaMemcpyHostToDevice));
        t.cells = f.cells;
        t.box = f.box;
        f.built = 0;
        if (!c->fmm_tab[dbl]) {
            rc = dbl ? fmm_tables<double>(c, kFmmP64, &c->fmm_tab[1]) : fmm_tables<float>(c, kFmmP32, &c->fmm_tab[0]);
            if (rc) return rc;
        }
        f.mp_bytes = (size_t)nbox * (dbl ? kFmmP64 * sizeof(V4<double>) : kFmmP32 * sizeof(V4<float>));
        f.sq_bytes = (size_t)nsrc * (dbl ? sizeof(double2) : sizeof(float2));
        mp_bytes = std::max(mp_bytes, f.mp_bytes);
        sq_bytes = std::max(sq_bytes, f.sq_bytes);
        max_box = std::max(max_box, (int)nbox);
    }
    if (max_box) {
        BIE_CUDA(c, cudaMalloc(&c->ws.fsq, sq_bytes + 16));
        BIE_CUDA(c, cudaMalloc(&c->ws.fmp, mp_bytes + 16));
        BIE_CUDA(c, cudaMalloc(&c->ws.floc, mp_bytes + 16));
        BIE_CUDA(c, cudaMalloc((void**)&c->ws.ftick, max_box * sizeof(unsigned)));
        BIE_CUDA(c, cudaMemset(c->ws.ftick, 0, max_box * sizeof(unsigned)));
    }
    return BIE_OK;
}

// Sorts the current geometry's records into the boxes (once per geometry and
// precision, when an application first needs it).
int fmm_build(bie_ctx* c, int prec) {
    Fmm& f = c->fmm[prec];
    if (!f.on || f.built == c->geometry) return BIE_OK;
    const FmmGeom g{c->x, c->y, c->xw, c->yw, c->imc, c->node_cell};
    FmmTree& t = f.t;
    for (int set = 0; set < (c->utilde ? 2 : 1); ++set) {
        const int mul = set ? 1 : c->srcmul, n = c->N * mul;
        int* count = set ? t.tcount : t.scount;
        int* start = set ? t.tstart : t.sstart;
        BIE_CUDA(c, cudaMemsetAsync(count, 0, t.nbox * sizeof(int), c->stream));
        k_fmm_bin<<<(n + 255) / 256, 256, 0, c->stream>>>(g, c->cells, f.cells, f.box, n, mul, set, f.leaf, count);
        BIE_LAUNCH(c, "k_fmm_bin");
        k_fmm_scan<<<1, 1024, 0, c->stream>>>(count, t.nleaf, start, f.cursor);
        BIE_LAUNCH(c, "k_fmm_scan");
        k_fmm_fill<<<(n + 255) / 256, 256, 0, c->stream>>>(f.leaf, n, f.cursor, f.raw);
        BIE_LAUNCH(c, "k_fmm_fill");
        k_fmm_sort<<<t.nleaf, 64, 0, c->stream>>>(g, c->cells, f.box, start, f.raw, mul, set, set ? t.tperm : t.sperm,
                                                  set ? t.tpos : t.spos, set ? t.tpos64 : t.spos64);
        BIE_LAUNCH(c, "k_fmm_sort");
    }
    f.built = c->geometry;
    return BIE_OK;
}

// The near sum's partials (one split per cell) of sigma in ws.part.
int fmm_near(bie_ctx* c, const double* sigma, int prec, Workspace& ws) {
    Fmm& f = c->fmm[prec];
    const FmmTree& t = f.t;
    const int nimg = c->utilde ? 1 : 9, shift = c->utilde ? 2 : 0;
    const double2* sg = reinterpret_cast<const double2*>(sigma);
    const int n0 = c->shard.on ? c->shard.n0 : 0, n1 = c->shard.on ? c->shard.n1 : c->N;
    const dim3 down(t.nleaf, 2);
    if (prec == 0) {
        const float* tab = (const float*)c->fmm_tab[0];
        const float* bin = tab + kFmmP32 * kFmmP32;
        k_fmm_up<float, kFmmP32><<<(t.nleaf + 3) / 4, 128, 0, c->stream>>>(
            t, c->cells, sg, c->w, shift, (C2<float>*)ws.fsq, nullptr, (V4<float>*)ws.fmp, ws.ftick, bin);
        BIE_LAUNCH(c, "k_fmm_up");
        k_fmm_m2l<float, kFmmP32><<<t.nbox, 128, 0, c->stream>>>(t, c->cells, nimg, (const V4<float>*)ws.fmp,
                                                               (V4<float>*)ws.floc, tab);
        BIE_LAUNCH(c, "k_fmm_m2l");
        k_fmm_down32<<<down, 128, 0, c->stream>>>(t, c->cells, nimg, (const C2<float>*)ws.fsq,
                                                  (const V4<float>*)ws.floc, bin, c->tgt32, n0, n1,
                                                  (float2*)ws.part);
        BIE_LAUNCH(c, "k_fmm_down32");
        return BIE_OK;
    }
    const double* tab = (const double*)c->fmm_tab[1];
    const double* bin = tab + kFmmP64 * kFmmP64;
    const bool df = prec == 2;
    k_fmm_up<double, kFmmP64><<<(t.nleaf + 3) / 4, 128, 0, c->stream>>>(
        t, c->cells, sg, c->w, shift, (C2<double>*)ws.fsq, df ? (float4*)ws.fsq : nullptr, (V4<double>*)ws.fmp,
        ws.ftick, bin);
    BIE_LAUNCH(c, "k_fmm_up");
    k_fmm_m2l<double, kFmmP64><<<t.nbox, 128, 0, c->stream>>>(t, c->cells, nimg, (const V4<double>*)ws.fmp,
                                                            (V4<double>*)ws.floc, tab);
    BIE_LAUNCH(c, "k_fmm_m2l");
    if (df)
        k_fmm_down64<true><<<down, 128, 0, c->stream>>>(t, c->cells, nimg, nullptr, (const float4*)ws.fsq,
                                                        (const V4<double>*)ws.floc, bin, c->nx, c->ny, prec, n0, n1,
                                                        (double2*)ws.part);
    else
        k_fmm_down64<false><<<down, 128, 0, c->stream>>>(t, c->cells, nimg, (const C2<double>*)ws.fsq, nullptr,
                                                         (const V4<double>*)ws.floc, bin, c->nx, c->ny, prec, n0, n1,
                                                         (double2*)ws.part);
    BIE_LAUNCH(c, "k_fmm_down64");
    return BIE_OK;
}

}  // namespace bie
