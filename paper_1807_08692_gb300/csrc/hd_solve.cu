// Online query path: spectral term + temporal term by multi-RHS CG (Eq. 17-20).
//
// Layout: every n x B block (R, P, Q, X) is row-major with a padded width Bp
// (B rounded up to a multiple of 4) so that one gathered row of P is Bp
// contiguous fp32 values: a group of Bp/4 lanes moves it with float4 loads.
// P alone may be kept in panels of a 128-byte line instead (Panels, panels_for).
//
// One CG iteration for B columns at once (per-column scalars in fp64):
//   Q = c1 P - c2 W P [+ U (c3 Lambda o (U^T P))]                 Eq. 20
//   sigma = P^T Q  (SpMM partials + c3 sum_k lambda_k C_k^2, C = U^T P)
//   a = rho / sigma; X += a P; R -= a Q; rr = ||R||^2               (CG, Sec. 4.4)
//   [PCG: C = U^T R, rho' = rr + sum_k D_k C_k^2, Z = R + U (D o C)]
//   beta = rho' / rho; P = Z + beta P
// Columns stop individually (||r|| <= tol ||b||, max_iter, breakdown); a
// stopped column keeps X and R bit-for-bit (its step length is 0).  When every
// column has stopped, the true residual b - A x is formed for the batch; a
// column whose recursive residual met tol but whose true residual did not is
// restarted from x with r := b - A x (residual replacement, at most
// MAX_CONFIRM times), and the true value is what the solve reports.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include <cuda_fp16.h>

#include "hd_solve.cuh"

// ------------------------------------------------------------------ helpers
__device__ __forceinline__ float4 ld4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 ld4v(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
// the same for a result that the next kernel reads as a stream: first to leave
// L2, so that it does not push out the rows being gathered
__device__ __forceinline__ void st4s(float* p, float4 v) { __stcs(reinterpret_cast<float4*>(p), v); }

// ------------------------------------------------------------------ kernels
// R[:, j] += y_j, one block per column.  Entries with one index are added in
// input order by the thread of the first of them; ascending indices (as
// hd_observe returns them) need no search for such entries, and a longer list
// in another order is left to one thread.
constexpr int SCATTER_SEARCH = 1024;
__global__ void __launch_bounds__(128) k_scatter_y(const int32_t* y_ptr, const int32_t* y_idx, const float* y_val,
                                                   int32_t nnz, int64_t n, int32_t ld, float* R, int* err) {
    const int j = blockIdx.x;
    const int32_t b = y_ptr[j], e = y_ptr[j + 1];
    if (b > e || b < 0 || e > nnz) {  // nnz = y_ptr[B], the entries there are
        if (threadIdx.x == 0) atomicExch(err, 1);
        return;
    }
    int unsorted = 0;
    for (int32_t t = b + (int)threadIdx.x; t + 1 < e; t += blockDim.x) unsorted |= y_idx[t] >= y_idx[t + 1];
    unsorted = __syncthreads_or(unsorted);
    const bool serial = unsorted && e - b > SCATTER_SEARCH;
    if (serial && threadIdx.x) return;
    for (int32_t t = b + (int)threadIdx.x; t < e; t += serial ? 1 : (int)blockDim.x) {
        const int32_t i = y_idx[t];
        const float v = y_val[t];
        if (i < 0 || i >= n || !isfinite(v)) {
            atomicExch(err, 1);
            continue;
        }
        float* a = R + (int64_t)i * ld + j;
        if (serial || !unsorted) {
            *a += v;
            continue;
        }
        bool first = true;
        for (int32_t s = b; s < t; ++s) first &= y_idx[s] != i || !isfinite(y_val[s]);
        if (!first) continue;
        float sum = *a + v;
        for (int32_t s = t + 1; s < e; ++s)
            if (y_idx[s] == i && isfinite(y_val[s])) sum += y_val[s];
        *a = sum;
    }
}

// True when some column of this block's S-column slab is active; with
// st == nullptr every slab works.
__device__ __forceinline__ bool columns_have_work(const ColState* st, int first, int last) {
    if (!st) return true;
    int w = 0;
    if (first + (int)threadIdx.x < last) w = st[first + threadIdx.x].active;
    return __syncthreads_or(w) != 0;
}
template <int S>
__device__ __forceinline__ bool slab_has_work(const ColState* st) {
    return columns_have_work(st, blockIdx.y * S, blockIdx.y * S + S);
}

#define FMA4(acc_, wt_, vec_)                  \
    acc_.x = fmaf(wt_, vec_.x, acc_.x);       \
    acc_.y = fmaf(wt_, vec_.y, acc_.y);       \
    acc_.z = fmaf(wt_, vec_.z, acc_.z);       \
    acc_.w = fmaf(wt_, vec_.w, acc_.w)

// 4-column slabs: two lanes per row, which compute the same two chains as a
// thread per row (chain s: entries 8c + {0, 2, 4, 6} of the full chunks of 8,
// then every tail entry in order; chain s2: entries 8c + {1, 3, 5, 7}; the row
// sum s + s2), so the bits do not change; the pairs halve each lane's serial
// gathers and read the row's indices two at a time (0.28 ms against 0.38 ms
// on the 1M-node graph, the same bits).  128 rows per block step.
__device__ __forceinline__ void spmm_rows_pair4(const int32_t* rp, const int32_t* ci, const float* wv,
                                                const float* P, const Panels& pv, float* Q, int64_t n, int32_t ld,
                                                int32_t col, float c1, float c2) {
    const int lane = threadIdx.x & 31, h = lane & 1;
    int pw;
    const float* Pc = panel_column(pv, P, col, pw);
    // rows advance warp-uniformly (the shuffle needs every lane); a lane past
    // the last row works on an empty row and writes nothing
    for (int64_t r0 = (int64_t)blockIdx.x * 128 + (threadIdx.x >> 5) * 16; r0 < n; r0 += (int64_t)gridDim.x * 128) {
        const int64_t row = r0 + (lane >> 1);
        const bool ok = row < n;
        const int32_t b = ok ? rp[row] : 0, e = ok ? rp[row + 1] : 0;
        const int32_t full = b + (e - b) / 8 * 8;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        int32_t t = b;
        for (; t + 16 <= full; t += 16) {  // two chunks: this lane's 8 entries
            float w[8];
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int32_t k = t + 2 * u + h;
                w[u] = __ldg(wv + k);
                v[u] = ld4(Pc + (int64_t)__ldg(ci + k) * pw);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                FMA4(s, w[u], v[u]);
            }
        }
        if (t < full) {  // one chunk left
            float w[4];
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int32_t k = t + 2 * u + h;
                w[u] = __ldg(wv + k);
                v[u] = ld4(Pc + (int64_t)__ldg(ci + k) * pw);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                FMA4(s, w[u], v[u]);
            }
            t += 8;
        }
        if (h == 0) {  // the tail belongs to chain s, in masked batches of 4
            for (; t < e; t += 4) {
                const int m = e - t;
                float4 v[4];
                float w[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    w[u] = u < m ? __ldg(wv + t + u) : 0.f;
                    v[u] = u < m ? ld4(Pc + (int64_t)__ldg(ci + t + u) * pw) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (u < m) {
                        FMA4(s, w[u], v[u]);
                    }
                }
            }
        }
        const float ox = __shfl_xor_sync(0xffffffffu, s.x, 1), oy = __shfl_xor_sync(0xffffffffu, s.y, 1);
        const float oz = __shfl_xor_sync(0xffffffffu, s.z, 1), ow = __shfl_xor_sync(0xffffffffu, s.w, 1);
        if (ok && h == 0) {
            s.x += ox;
            s.y += oy;
            s.z += oz;
            s.w += ow;
            const float4 own = ld4(Pc + row * pw);
            float4 q;
            q.x = c1 * own.x - c2 * s.x;
            q.y = c1 * own.y - c2 * s.y;
            q.z = c1 * own.z - c2 * s.z;
            q.w = c1 * own.w - c2 * s.w;
            st4(Q + row * ld + col, q);
        }
    }
}

// 4-column slabs of Q = c1 P - c2 W P.  `skip` (may be null): the launch
// returns at once when *skip is not 0.
__global__ void __launch_bounds__(256, 8) k_spmm4(const int32_t* rp, const int32_t* ci, const float* wv, const float* P,
                                                  const Panels pv, float* Q, int64_t n, int32_t ld, int32_t first,
                                                  float c1, float c2, const ColState* st, const int* skip) {
    if (skip && *skip) return;
    const int col = first + blockIdx.y * 4;
    if (!columns_have_work(st, col, col + 4)) return;
    spmm_rows_pair4(rp, ci, wv, P, pv, Q, n, ld, col, c1, c2);
}

// ---- the row gathers shared by the wider SpMM kernels
// A group of L lanes owns a row; each lane moves 16 bytes of every gathered
// row.  Bound: the random gathers (DRAM when the gathered block exceeds L2).
// What keeps them in flight is eight gathers per lane and the next eight
// (index, weight) pairs already on their way: the first G lanes of a group load
// one pair each and the group reads them by shuffle, two registers where
// private copies took sixteen.  At 64 registers (32 warps per SM) a 1M x 64
// product runs in 1.18 ms (7.2 GB of DRAM traffic, 6.1 TB/s) against 1.58 ms for
// a kernel of 32 registers and 64 warps, whose eight gathers the compiler had
// to issue a few at a time; 72 registers and 28 warps take 1.24 ms, 80 and 24
// 1.42 ms.  Sixteen lanes gather 256 bytes per row and prefer 28 warps.
constexpr int spmm_blocks(int lanes) { return lanes == 8 ? 8 : 7; }  // blocks of 128 threads per SM
struct RowLanes {
    int L, g, gb;      // lanes per row, this lane's place in its group, the group's first lane
    unsigned mask;     // lanes of the group
    unsigned row, step;  // first row of the group and the stride to its next
    bool idle;         // a lane past the last whole group of its warp
};
template <int LC>
__device__ __forceinline__ RowLanes row_lanes(int L_) {
    RowLanes r;
    r.L = LC ? LC : L_;
    const int lane = threadIdx.x & 31, per = 32 / r.L, gi = lane / r.L;
    r.gb = gi * r.L;
    r.g = LC ? lane & (LC - 1) : lane - r.gb;
    r.mask = (r.L == 32 ? 0xffffffffu : (1u << r.L) - 1u) << r.gb;
    r.idle = gi >= per;
    const unsigned rpb = (blockDim.x >> 5) * per;
    r.row = blockIdx.x * rpb + (threadIdx.x >> 5) * per + gi;
    r.step = gridDim.x * rpb;
    return r;
}
// Entries b .. e of one row: full chunks of 8 through acc(u, w, v), u the place
// in the chunk, the rest through tail(w, v), each in entry order; load(j)
// gathers row j.  The lanes of a group run it together.
template <int LC, class T>
__device__ __forceinline__ T from_lane(const RowLanes& r, T x, int u) {  // lane u of the group
    return LC ? __shfl_sync(r.mask, x, u, LC) : __shfl_sync(r.mask, x, r.gb + u);
}
template <int LC, int G, class V, class LD, class AC, class TL>
__device__ __forceinline__ void row_entries(const int32_t* __restrict__ ci, const float* __restrict__ wv, unsigned b,
                                            unsigned e, const RowLanes& r, LD load, AC acc, TL tail) {
    constexpr int NI = 8 / G;
    int32_t jj[NI];
    float ww[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const unsigned q = b + i * G + r.g;
        jj[i] = 0;
        ww[i] = 0.f;
        if (r.g < G && q < e) {
            jj[i] = __ldg(ci + q);
            ww[i] = __ldg(wv + q);
        }
    }
    const unsigned full = b + ((e - b) & ~7u);
    for (unsigned t = b; t < full; t += 8) {
        int32_t nj[NI];
        float nw[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const unsigned q = t + 8 + i * G + r.g;
            nj[i] = 0;
            nw[i] = 0.f;
            if (r.g < G && q < e) {
                nj[i] = __ldg(ci + q);
                nw[i] = __ldg(wv + q);
            }
        }
        V v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = load(from_lane<LC>(r, jj[u / G], u % G));
#pragma unroll
        for (int u = 0; u < 8; ++u) acc(u, from_lane<LC>(r, ww[u / G], u % G), v[u]);
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            jj[i] = nj[i];
            ww[i] = nw[i];
        }
    }
    const unsigned m = e - full;
    if (m) {
        V v[7];
#pragma unroll
        for (int u = 0; u < 7; ++u) {
            const int32_t j = from_lane<LC>(r, jj[u / G], u % G);
            v[u] = V{};  // keeps the loads predicated, all in flight before the first sum
            if (u < m) v[u] = load(j);
        }
#pragma unroll
        for (int u = 0; u < 7; ++u) {
            const float w = from_lane<LC>(r, ww[u / G], u % G);
            if (u < m) tail(w, v[u]);
        }
    }
}

// Q = c1 P - c2 W P, L lanes x 4 columns per slab blockIdx.y (LC > 0: L = LC at
// compile time, whole slabs only; G = min(L, 8) or the next smaller power of two).  The sums are
// the two chains of spmm_rows_pair4, the same at every slab width; the lanes of
// a ragged last slab past the last column repeat it and write nothing.  The
// P^T Q partials of CG come from k_dot below: fused in here they cost more
// registers, hence gathers in flight, than the extra pass.
template <int LC, int G>
__global__ void __launch_bounds__(128, spmm_blocks(LC)) k_spmm(const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                                 const float* __restrict__ wv, const float* __restrict__ P,
                                                 const Panels pv, float* __restrict__ Q, unsigned n, int32_t ld,
                                                 int32_t first, int32_t last, int L_, float c1, float c2,
                                                 const ColState* st, const int* skip) {
    if (skip && *skip) return;
    const int Lq = LC ? LC : L_;
    const int c0 = first + blockIdx.y * 4 * Lq;
    if (!columns_have_work(st, c0, min(last, c0 + 4 * Lq))) return;
    const RowLanes r = row_lanes<LC>(L_);
    if (r.idle) return;
    const bool own_col = LC || c0 + 4 * r.g < last;
    const int col = own_col ? c0 + 4 * r.g : last - 4;
    // (LC = 0: plain rows or the last panel, one stride for all, taken from the arguments)
    int pw = pv.wlast;
    const float* Pc = LC ? panel_column(pv, P, col, pw) : P + first * pv.n + (col - first);
    auto load = [&](int32_t j) { return ld4(Pc + (int64_t)j * (LC ? pw : pv.wlast)); };
    for (unsigned row = r.row; row < n; row += r.step) {
        const unsigned b = __ldg(rp + row), e = __ldg(rp + row + 1);
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 s2 = make_float4(0.f, 0.f, 0.f, 0.f);
        row_entries<LC, G, float4>(
            ci, wv, b, e, r, load,
            [&](int u, float w, const float4& v) {
                if (u & 1) {
                    FMA4(s2, w, v);
                } else {
                    FMA4(s, w, v);
                }
            },
            [&](float w, const float4& v) { FMA4(s, w, v); });
        s.x += s2.x;
        s.y += s2.y;
        s.z += s2.z;
        s.w += s2.w;
        const float4 own = ld4(Pc + (int64_t)row * (LC ? pw : pv.wlast));
        float4 q;
        q.x = c1 * own.x - c2 * s.x;
        q.y = c1 * own.y - c2 * s.y;
        q.z = c1 * own.z - c2 * s.z;
        q.w = c1 * own.w - c2 * s.w;
        if (own_col) st4s(Q + (int64_t)row * ld + col, q);
    }
}

// A batch of at most 4 columns (one 4-column slab, hd_query_batch only): four
// lanes per row, lane e summing entries b + e, b + e + 4, ... in order (four
// loads in flight), the four sums meeting as (v0 + v2) + (v1 + v3).  The
// row's index / weight reads are coalesced and eight rows gather per warp:
// 0.24 ms on the 1M-node benchmark graph against 0.28 ms for k_spmm4 (two
// lanes per row), 0.38 ms for a thread per row and 0.32 ms for a warp per row.
// Its sums run in another order than k_spmm's, so the server, whose results
// must not depend on the lane width, keeps k_spmm.
constexpr int N4_ROWS = 64;  // rows per 256-thread block
__global__ void __launch_bounds__(256, 8) k_spmm_n4(const int32_t* rp, const int32_t* ci, const float* wv,
                                                    const float* P, float* Q, int64_t n, float c1, float c2,
                                                    const ColState* st, const int* skip) {
    if (skip && *skip) return;
    if (!slab_has_work<4>(st)) return;
    const int lane = threadIdx.x & 31, e = lane & 3;
    // rows advance warp-uniformly (the shuffles need every lane); a lane past
    // the last row works on an empty row and writes nothing
    for (int64_t r0 = (int64_t)blockIdx.x * N4_ROWS + (threadIdx.x >> 5) * 8; r0 < n;
         r0 += (int64_t)gridDim.x * N4_ROWS) {
        const int64_t row = r0 + (lane >> 2);
        const bool ok = row < n;
        const int32_t b = ok ? rp[row] : 0, end = ok ? rp[row + 1] : 0;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int32_t t = b + e; t < end; t += 16) {
            const int m = (end - t + 3) / 4;
            float w[4];
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                w[u] = u < m ? __ldg(wv + t + 4 * u) : 0.f;
                v[u] = u < m ? ld4(P + (int64_t)__ldg(ci + t + 4 * u) * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (u < m) {
                    FMA4(s, w[u], v[u]);
                }
        }
#pragma unroll
        for (int o = 2; o > 0; o >>= 1) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
            s.z += __shfl_xor_sync(0xffffffffu, s.z, o);
            s.w += __shfl_xor_sync(0xffffffffu, s.w, o);
        }
        if (ok && e == 0) {
            const float4 own = ld4(P + row * 4);
            float4 q;
            q.x = c1 * own.x - c2 * s.x;
            q.y = c1 * own.y - c2 * s.y;
            q.z = c1 * own.z - c2 * s.z;
            q.w = c1 * own.w - c2 * s.w;
            st4(Q + row * 4, q);
        }
    }
}

// ---- a 16-bit copy of P for the SpMM gathers of late iterations
// Inexact Krylov methods (Simoncini and Szyld, SIAM J. Sci. Comput. 2003; van
// den Eshof and Sleijpen, SIAM J. Matrix Anal. Appl. 2004): the operator may be
// applied less accurately as the residual shrinks; the gap between recursive
// and true residual grows by |a_k| ||E_k p_k|| per iteration.  Here E_k p =
// c2 W (p~ - p) with p~ the fp16 copy (relative rounding u16 = 2^-11 per
// entry), and |a_k| ||p_k|| = ||x_{k+1} - x_k|| <= 2 ||r_k|| (L_a(W) >= I), so
// the gap added by an fp16 iteration is at most 2 c2 u16 ||W (p~ - p)|| / u16
// ||p|| times ||r_k||: 0.1 ||r_k|| in the worst case, ~0.008 ||r_k|| for rounding
// errors of random sign over ~54 neighbours.  The next SpMM gathers the fp16
// copy once every active column has ||r|| <= HALF_THETA tol ||b||, which keeps
// the typical gap near a quarter of tol ||b||; the true-residual confirmation
// certifies the result either way.  Each column is scaled by a power of two so
// that its largest entry lies in [2^13, 2^14) (exact, no overflow); the own-row
// term c1 p, the dot products and the updates stay fp32.
constexpr double HALF_THETA = 25.0;

// per-column max |P| (the bits of a non-negative float order like the value);
// runs when the next SpMM gathers the fp16 copy and some column is active
__global__ void __launch_bounds__(256) k_colmax(const float* __restrict__ P, const Panels pv, int64_t n, int32_t ld,
                                                unsigned* __restrict__ mx, const int* __restrict__ use_half,
                                                const int* __restrict__ num_active) {
    if (!*use_half || !*num_active) return;
    __shared__ unsigned bmax[256];  // per column of this block (ld <= 256)
    const int nq = ld >> 2;
    const int rpb = blockDim.x / nq;  // rows per block step
    for (int c = threadIdx.x; c < ld; c += blockDim.x) bmax[c] = 0u;
    __syncthreads();
    if ((int)threadIdx.x < rpb * nq) {
        const int q = threadIdx.x % nq;
        int pw;
        const float* Pc = panel_column(pv, P, 4 * q, pw);
        float m0 = 0.f, m1 = 0.f, m2 = 0.f, m3 = 0.f;
        for (int64_t row = (int64_t)blockIdx.x * rpb + threadIdx.x / nq; row < n; row += (int64_t)gridDim.x * rpb) {
            const float4 v = ld4(Pc + row * pw);
            m0 = fmaxf(m0, fabsf(v.x));
            m1 = fmaxf(m1, fabsf(v.y));
            m2 = fmaxf(m2, fabsf(v.z));
            m3 = fmaxf(m3, fabsf(v.w));
        }
        // one global atomic per column and block: same-address atomics from
        // every thread would serialise in the one L2 slice holding mx
        atomicMax(bmax + 4 * q, __float_as_uint(m0));
        atomicMax(bmax + 4 * q + 1, __float_as_uint(m1));
        atomicMax(bmax + 4 * q + 2, __float_as_uint(m2));
        atomicMax(bmax + 4 * q + 3, __float_as_uint(m3));
    }
    __syncthreads();
    for (int c = threadIdx.x; c < ld; c += blockDim.x) atomicMax(mx + c, bmax[c]);
}

// 2^k with max|P_j| 2^k in [2^13, 2^14) (1 for a zero column), and its inverse
__device__ __forceinline__ float half_scale(unsigned mbits, bool inverse) {
    const float m = __uint_as_float(mbits);
    if (!(m > 0.f)) return 1.f;
    int ex;
    frexpf(m, &ex);  // m = f 2^ex, f in [0.5, 1)
    return ldexpf(1.f, inverse ? ex - 14 : 14 - ex);
}

// P16 = fp16(P_j 2^k_j) column by column
__global__ void __launch_bounds__(256) k_to_half(const float* __restrict__ P, const Panels pv, int64_t n, int32_t ld,
                                                 const unsigned* __restrict__ mx, __half* __restrict__ P16,
                                                 const Panels hv,
                                                 const int* __restrict__ use_half,
                                                 const int* __restrict__ num_active) {
    if (!*use_half || !*num_active) return;
    const int nq = ld >> 2;
    const int rpb = blockDim.x / nq;
    if ((int)threadIdx.x >= rpb * nq) return;
    const int q = threadIdx.x % nq;
    const float s0 = half_scale(mx[4 * q], false), s1 = half_scale(mx[4 * q + 1], false);
    const float s2 = half_scale(mx[4 * q + 2], false), s3 = half_scale(mx[4 * q + 3], false);
    int pw, hw;
    const float* Pc = panel_column(pv, P, 4 * q, pw);
    __half* Hc = panel_column(hv, P16, 4 * q, hw);
    for (int64_t row = (int64_t)blockIdx.x * rpb + threadIdx.x / nq; row < n; row += (int64_t)gridDim.x * rpb) {
        const float4 v = ld4(Pc + row * pw);
        const __half2 a = __floats2half2_rn(v.x * s0, v.y * s1);
        const __half2 b = __floats2half2_rn(v.z * s2, v.w * s3);
        uint2 o;
        o.x = *reinterpret_cast<const unsigned*>(&a);
        o.y = *reinterpret_cast<const unsigned*>(&b);
        *reinterpret_cast<uint2*>(Hc + row * hw) = o;
    }
}

#define FMA8H(acc_, wt_, raw_)                                                    \
    {                                                                             \
        const __half2* h_ = reinterpret_cast<const __half2*>(&(raw_));            \
        _Pragma("unroll") for (int k_ = 0; k_ < 4; ++k_) {                        \
            const float2 f_ = __half22float2(h_[k_]);                             \
            acc_[2 * k_] = fmaf(wt_, f_.x, acc_[2 * k_]);                         \
            acc_[2 * k_ + 1] = fmaf(wt_, f_.y, acc_[2 * k_ + 1]);                 \
        }                                                                         \
    }

// Q = c1 P - c2 W P with the W P gathers from the fp16 copy (L lanes x 8
// columns per slab: a row's slab of 64 columns is one 128-byte line); the sums
// are fp32, unscaled by the column's power of two at the end.  Runs when
// *use_half is set.  0.74 ms for a 1M x 64 product (0.82 ms with private index
// copies); 0.06 ms against 0.16 ms for 100,000 x 40, which took 8-column slabs.
template <int LC, int G>
__global__ void __launch_bounds__(128, 7) k_spmm_h(const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                                   const float* __restrict__ wv, const __half* __restrict__ P16,
                                                   const Panels hv, const unsigned* __restrict__ mx,
                                                   const float* __restrict__ P, const Panels pv, float* __restrict__ Q,
                                                   unsigned n, int32_t ld, int32_t first, int32_t last, int L_, float c1,
                                                   float c2, const ColState* st, const int* __restrict__ use_half) {
    if (!*use_half) return;
    const int Lq = LC ? LC : L_;
    const int c0 = first + blockIdx.y * 8 * Lq, ce = min(last, c0 + 8 * Lq);
    // up to 256 columns of a slab against 128 threads
    if (!columns_have_work(st, c0, min(ce, c0 + 128)) && !columns_have_work(st, c0 + 128, ce)) return;
    // the scales wait in shared memory: in registers they cost gathers in flight
    __shared__ __align__(16) float inv[256];
    for (int c = c0 + threadIdx.x; c < ce; c += blockDim.x) inv[c - c0] = half_scale(mx[c], true);
    __syncthreads();
    const RowLanes r = row_lanes<LC>(L_);
    if (r.idle) return;
    const bool own_col = LC || c0 + 8 * r.g < last;
    const int col = own_col ? c0 + 8 * r.g : last - 8;
    int pw, hw = hv.wlast;
    const float* Po = panel_column(pv, P, col, pw);
    const __half* Pc = LC ? panel_column(hv, P16, col, hw) : P16 + first * hv.n + (col - first);
    auto load = [&](int32_t j) { return __ldg(reinterpret_cast<const uint4*>(Pc + (int64_t)j * (LC ? hw : hv.wlast))); };
    for (unsigned row = r.row; row < n; row += r.step) {
        const unsigned b = __ldg(rp + row), e = __ldg(rp + row + 1);
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        row_entries<LC, G, uint4>(
            ci, wv, b, e, r, load, [&](int, float w, const uint4& v) { FMA8H(acc, w, v); },
            [&](float w, const uint4& v) { FMA8H(acc, w, v); });
        const float* po = Po + (int64_t)row * pw;
        const float4 o0 = ld4(po), o1 = ld4(po + 4);
        const float4 i0 = *reinterpret_cast<const float4*>(inv + (col - c0));
        const float4 i1 = *reinterpret_cast<const float4*>(inv + (col - c0) + 4);
        const float iv[8] = {i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w};
        const float own[8] = {o0.x, o0.y, o0.z, o0.w, o1.x, o1.y, o1.z, o1.w};
        float q[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) q[c] = c1 * own[c] - c2 * (acc[c] * iv[c]);
        if (own_col) {
            float* qo = Q + (int64_t)row * ld + col;
            st4s(qo, make_float4(q[0], q[1], q[2], q[3]));
            st4s(qo + 4, make_float4(q[4], q[5], q[6], q[7]));
        }
    }
}

// ---- the true residual, accumulated in two fp32 words
// b - A x with A = c1 I - c2 W cancels: c1 x and c2 W x are ~1/(1 - a) times
// larger than the result, so the fp32 rounding of W x (relative ~u per term)
// would reach the residual magnified 1/(1 - a) times (about 7e-7 ||y|| on the
// 2,000-node graph, as large as a 1e-6 tolerance).  The residual kernels below
// carry W x as an unevaluated sum hi + lo of two fp32 numbers, built with
// error-free transformations: the product w v = p + e exactly (e from one fma;
// Ogita, Rump and Oishi, "Accurate sum and dot product", 2005) and the sum
// hi + p = s + e exactly (Knuth's TwoSum).  The _rn intrinsics keep the
// compiler from contracting these into other fma operations.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bv = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bv)), __fsub_rn(b, bv));
}

// hi + lo += w v
__device__ __forceinline__ void df_fma(float& hi, float& lo, float w, float v) {
    const float p = __fmul_rn(w, v);
    const float pe = __fmaf_rn(w, v, -p);
    float s, e;
    two_sum(hi, p, s, e);
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(e, pe));
}

// -(c1 x - c2 (hi + lo)), rounded once at the end
__device__ __forceinline__ float neg_operator(float c1, float x, float c2, float hi, float lo) {
    const float p1 = __fmul_rn(c1, x), e1 = __fmaf_rn(c1, x, -p1);
    const float p2 = __fmul_rn(c2, hi), e2 = __fmaf_rn(c2, hi, -p2);
    float d, e3;
    two_sum(p1, -p2, d, e3);
    const float tail = __fsub_rn(__fsub_rn(__fadd_rn(e3, e1), e2), __fmul_rn(c2, lo));
    return -__fadd_rn(d, tail);
}

// Q = -(c1 X - c2 W X), W X in two words, lanes and slabs as in k_spmm.
// Runs when *pick is 1 (see k_resid_pick).
template <int LC, int G>
__global__ void __launch_bounds__(128, 6) k_resid(const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                                  const float* __restrict__ wv, const float* __restrict__ X,
                                                  float* __restrict__ Q, unsigned n, int32_t ld, int L_, float c1,
                                                  float c2, const int* __restrict__ pick) {
    if (*pick != 1) return;
    const RowLanes r = row_lanes<LC>(L_);
    if (r.idle) return;
    const int quad = blockIdx.y * r.L + r.g, nq = ld >> 2;
    const bool own_col = LC || quad < nq;
    const int col = 4 * (own_col ? quad : nq - 1);
    const float* Xc = X + col;
    auto load = [&](int32_t j) { return ld4(Xc + (int64_t)j * ld); };
    for (unsigned row = r.row; row < n; row += r.step) {
        const unsigned b = __ldg(rp + row), e = __ldg(rp + row + 1);
        float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
        auto add = [&](float w, const float4& v) {
            df_fma(hi[0], lo[0], w, v.x);
            df_fma(hi[1], lo[1], w, v.y);
            df_fma(hi[2], lo[2], w, v.z);
            df_fma(hi[3], lo[3], w, v.w);
        };
        row_entries<LC, G, float4>(ci, wv, b, e, r, load, [&](int, float w, const float4& v) { add(w, v); }, add);
        const float4 own = ld4(Xc + (int64_t)row * ld);
        float4 q;
        q.x = neg_operator(c1, own.x, c2, hi[0], lo[0]);
        q.y = neg_operator(c1, own.y, c2, hi[1], lo[1]);
        q.z = neg_operator(c1, own.z, c2, hi[2], lo[2]);
        q.w = neg_operator(c1, own.w, c2, hi[3], lo[3]);
        if (own_col) st4s(Q + (int64_t)row * ld + col, q);
    }
}

// ---- per-column operators (truncated systems)
// Column j's row t holds the entries off[j * n + t] .. off[j * n + t + 1] of (ci,
// wv); columns j >= B are empty.  The vectors are read column by column (VT, the
// transposed block), so a column's gathers stay in its own n floats.
//
// Bound: one 4-byte gather per entry through L1 (110M entries: 0.38 ms at a line
// per cycle).  One block per SM takes an equal share of the entries and rows of all
// columns in column order, so its L1 keeps to one or two columns' vectors.  It streams
// the entries in order: coalesced (index, weight) loads two tiles ahead, the
// gathers they name one tile ahead, (weight, value) pairs in shared memory; a
// thread then sums its own rows from there, so the order of a row's sum does
// not depend on the tiling or on the shares.  64 systems of 75,000 rows, 110M entries: 0.55 ms;
// with tiles of 2,048 entries, in which only three warps' rows are summed at a
// time, 0.90 ms, of 8,192 (64 KB less L1) 0.64 ms; a thread per (row, 4 columns)
// walking four rows in global memory and gathering 4 bytes of a 256-byte row
// took 1.65 ms.
constexpr int TC_T = 1024;           // threads
constexpr int TC_E = 4;              // entries per thread and tile
constexpr int TC_TILE = TC_T * TC_E;
constexpr int TC_COLS = 4096;        // columns at most (hd_temporal_truncated)

// VT[j][i] = V[i][j]; grid (rows / 32, columns / 32), 32 x 8 threads
__global__ void __launch_bounds__(256) k_transpose(const float* __restrict__ V, int64_t n, int32_t ld,
                                                   float* __restrict__ VT) {
    __shared__ float t[32][33];
    const int64_t r0 = blockIdx.x * 32ll;
    const int c0 = blockIdx.y * 32;
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
#pragma unroll
    for (int u = 0; u < 32; u += 8)
        if (r0 + y + u < n && c0 + x < ld) t[y + u][x] = V[(r0 + y + u) * ld + c0 + x];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 32; u += 8)
        if (c0 + y + u < ld && r0 + x < n) VT[(int64_t)(c0 + y + u) * n + r0 + x] = t[x][y + u];
}

// Order of the columns that have rows, with the work before each: warp- and
// block-wide scans over a chunk of TC_T columns.  `put(k, at)` is called for the
// k-th of those with rows > 0 (w: the work of this thread's column); returns
// through have / work the totals so far.
template <class PUT>
__device__ __forceinline__ void trunc_scan(bool on, int64_t w, int warps, int& have, int64_t& work, PUT put) {
    __shared__ int warp_count[TC_T / 32];
    __shared__ int64_t warp_work[TC_T / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(0xffffffffu, on);
    int64_t x = w;  // inclusive within the warp
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) {
        warp_count[warp] = __popc(m);
        warp_work[warp] = x;
    }
    __syncthreads();
    int k = have + __popc(m & ((1u << lane) - 1u));
    int64_t at = work + x - w;
    for (int v = 0; v < warps; ++v) {
        k += v < warp ? warp_count[v] : 0;
        at += v < warp ? warp_work[v] : 0;
        have += warp_count[v];
        work += warp_work[v];
    }
    if (on) put(k, at);
    __syncthreads();
}

// The columns that have rows, in order, and their work; one block, once per call
__global__ void __launch_bounds__(TC_T) k_trunc_work(const int32_t* __restrict__ sl_ptr, const int64_t* __restrict__ off,
                                                     int32_t B, int64_t n, TruncWork* __restrict__ out) {
    int have = 0;
    int64_t work = 0;
    for (int c0 = 0; c0 < B; c0 += TC_T) {
        const int j = c0 + (int)threadIdx.x;
        int rows = 0;
        int64_t w = 0;
        if (j < B) {
            rows = sl_ptr[j + 1] - sl_ptr[j];
            w = off[j * n + rows] - off[j * n] + rows;
        }
        trunc_scan(rows > 0, w, min(TC_T, B - c0 + 31) / 32, have, work,
                   [&](int k, int64_t at) { out[k] = TruncWork{at, j, rows, (uint64_t)((double)rows / (double)w * 0x1p63)}; });
    }
    if (threadIdx.x == 0) out[have].at = work;
}

// The columns to work on, in order (whole quads, as in the update that reads Q;
// st == nullptr: all), in shared memory.  Block-wide; returns their number,
// list[number].at is the whole work.
__device__ __forceinline__ int trunc_columns(const TruncSys& s, const ColState* st, TruncWork* list) {
    int all = 1;
    for (int i = threadIdx.x; i <= s.ncol; i += TC_T) {
        const TruncWork w = s.work[i];
        list[i] = w;
        if (st && i < s.ncol) {
            const ColState* q = st + (w.j & ~3);
            all &= q[0].active | q[1].active | q[2].active | q[3].active;
        }
    }
    if (__syncthreads_and(all)) return s.ncol;
    int have = 0;
    int64_t work = 0;
    for (int c0 = 0; c0 < s.ncol; c0 += TC_T) {
        const int i = c0 + (int)threadIdx.x;
        TruncWork c{};
        int64_t w = 0;
        bool on = false;
        if (i < s.ncol) {
            c = s.work[i];
            const ColState* q = st + (c.j & ~3);
            on = q[0].active | q[1].active | q[2].active | q[3].active;
            if (on) w = s.work[i + 1].at - c.at;
        }
        trunc_scan(on, w, min(TC_T, s.ncol - c0 + 31) / 32, have, work, [&](int k, int64_t at) {
            c.at = at;
            list[k] = c;
        });
    }
    if (threadIdx.x == 0) list[have].at = work;
    __syncthreads();
    return have;
}

// Streams the rows lo .. hi of one column (off, ci, wv: its CSR, fewer than 2^31
// entries; v: its vector):
// add(k, w, x) for a row's entries in order, k with the parity of the entry's
// place, then done(row).
template <class RS, class AD, class DN>
__device__ __forceinline__ void trunc_rows(const int64_t* __restrict__ off, const int32_t* __restrict__ ci,
                                           const float* __restrict__ wv, const float* __restrict__ v, unsigned lo,
                                           unsigned hi, float2 (*tile)[TC_TILE], RS reset, AD add, DN done) {
    unsigned row = lo + threadIdx.x;
    reset();
    const int64_t first = __ldg(off + lo);
    const unsigned last = (unsigned)(__ldg(off + hi) - first);
    ci += first;
    wv += first;
    unsigned b = last, e = last, nb = last, ne = last;
    auto bounds = [&](unsigned r, unsigned& x, unsigned& y) {
        if (r < hi) {
            x = (unsigned)(__ldg(off + r) - first);
            y = (unsigned)(__ldg(off + r + 1) - first);
        }
    };
    bounds(row, b, e);
    bounds(row + TC_T, nb, ne);
    int32_t c[TC_E];
    float w[TC_E], x[TC_E], wn[TC_E];
    auto indices = [&](unsigned t0) {
#pragma unroll
        for (int u = 0; u < TC_E; ++u) {
            const unsigned q = t0 + u * TC_T + threadIdx.x;
            c[u] = 0;
            wn[u] = 0.f;
            if (q < last) {
                c[u] = __ldg(ci + q);
                wn[u] = __ldg(wv + q);
            }
        }
    };
    auto gather = [&]() {
#pragma unroll
        for (int u = 0; u < TC_E; ++u) {
            x[u] = __ldg(v + c[u]);
            w[u] = wn[u];
        }
    };
    indices(0);
    gather();
    indices(TC_TILE);
    int buf = 0;
    for (unsigned t0 = 0; t0 < last; t0 += TC_TILE, buf ^= 1) {
#pragma unroll
        for (int u = 0; u < TC_E; ++u) tile[buf][u * TC_T + threadIdx.x] = make_float2(w[u], x[u]);
        gather();                      // tile t0 + TC_TILE
        indices(t0 + 2 * TC_TILE);
        __syncthreads();  // this tile is complete, and every thread is done with the other buffer's last one
        const unsigned t1 = min(last, t0 + TC_TILE);
        while (row < hi && b < t1) {
            // the row's part of this tile, four reads ahead of their sums
            int q = (int)(max(b, t0) - t0);
            const int g = (int)(min(e, t1) - t0);
            if ((q + t0 - b) & 1) {
                const float2 z = tile[buf][q++];
                add(1, z.x, z.y);
            }
            for (; q + 4 <= g; q += 4) {
                float2 z[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) z[u] = tile[buf][q + u];
#pragma unroll
                for (int u = 0; u < 4; ++u) add(u, z[u].x, z[u].y);
            }
            for (int u = 0; q < g; ++q, ++u) {
                const float2 z = tile[buf][q];
                add(u, z.x, z.y);
            }
            if (e > t1) break;
            done(row);
            reset();
            row += TC_T;
            b = nb;
            e = ne;
            bounds(row + TC_T, nb, ne);
        }
    }
    for (; row < hi; row += TC_T) {  // rows without entries after the last one
        done(row);
        reset();
    }
    __syncthreads();
}

// A block's share of the work; rows of a column count alike.  (Shares of equal
// rows, those past a short list's end among them, left one shortlist of 500,000
// among 15 of 1,000 to a tenth of the blocks: 14.7 ms for a call of 20 iterations
// on 1M nodes with 54 entries a row against 4.7.)
template <class F>
__device__ __forceinline__ void trunc_share(int count, const TruncWork* list, F each) {
    __shared__ volatile int64_t share[2];  // (in registers they would be spilled around the rows)
    int k = 0;
    {
        const int64_t total = list[count].at, per = (total + gridDim.x - 1) / gridDim.x;
        const int64_t x0 = blockIdx.x * per, x1 = min(total, x0 + per);
        if (x0 >= x1) return;
        for (int a = count; a - k > 1;) {  // the last column whose work starts at or before x0
            const int m = (k + a) >> 1;
            if (list[m].at <= x0) k = m;
            else a = m;
        }
        if (threadIdx.x == 0) {
            share[0] = x0;
            share[1] = x1;
        }
        __syncthreads();
    }
    for (; list[k].at < share[1]; ++k) {  // (past the last column: the whole work)
        const TruncWork c = list[k];
        const int64_t y0 = share[0] - c.at, y1 = share[1] - c.at;
        // neighbouring blocks round their common bound alike
        auto row_at = [&](int64_t y) { return min((int64_t)__umul64hi((uint64_t)y << 1, c.rate), (int64_t)c.rows); };
        const int64_t lo = y0 <= 0 ? 0 : row_at(y0);
        const int64_t hi = y1 >= list[k + 1].at - c.at ? c.rows : row_at(y1);
        if (lo < hi) each(c.j, lo, hi);
    }
}

// Q = c1 P - c2 W_j P column by column (VT: the transposed P); even and odd
// entries of a row sum separately.  Rows past a shortlist's end are left alone:
// P is 0 there and Q was cleared at the start.
__global__ void __launch_bounds__(TC_T, 1)
    k_spmm_cols(const TruncSys s, const float* __restrict__ VT, float* __restrict__ Q, int64_t n, int32_t ld, float c1,
                float c2, const ColState* __restrict__ st) {
    extern __shared__ float2 tc_sm[];
    float2(*tile)[TC_TILE] = reinterpret_cast<float2(*)[TC_TILE]>(tc_sm);  // [2]
    TruncWork* list = reinterpret_cast<TruncWork*>(tc_sm + 2 * TC_TILE);
    trunc_share(trunc_columns(s, st, list), list, [&](int j, int64_t lo, int64_t hi) {
        const float* v = VT + (int64_t)j * n;
        float s0, s1;
        trunc_rows(
            s.off + (int64_t)j * n, s.ci, s.wv, v, lo, hi, tile, [&] { s0 = s1 = 0.f; },
            [&](int i, float w, float p) {
                if (i & 1) s1 = fmaf(w, p, s1);
                else s0 = fmaf(w, p, s0);
            },
            [&](unsigned row) { Q[(int64_t)row * ld + j] = c1 * v[row] - c2 * (s0 + s1); });
    });
}

// Q = -(c1 X - c2 W_j X) column by column, W_j X in two words (VT: the transposed X).
__global__ void __launch_bounds__(TC_T, 1)
    k_resid_cols(const TruncSys s, const float* __restrict__ VT, float* __restrict__ Q, int64_t n, int32_t ld, float c1,
                 float c2) {
    extern __shared__ float2 tc_sm[];
    float2(*tile)[TC_TILE] = reinterpret_cast<float2(*)[TC_TILE]>(tc_sm);  // [2]
    TruncWork* list = reinterpret_cast<TruncWork*>(tc_sm + 2 * TC_TILE);
    trunc_share(trunc_columns(s, nullptr, list), list, [&](int j, int64_t lo, int64_t hi) {
        const float* v = VT + (int64_t)j * n;
        float a, b;
        trunc_rows(
            s.off + (int64_t)j * n, s.ci, s.wv, v, lo, hi, tile, [&] { a = b = 0.f; },
            [&](int, float w, float p) { df_fma(a, b, w, p); },
            [&](unsigned row) { Q[(int64_t)row * ld + j] = neg_operator(c1, v[row], c2, a, b); });
    });
}

// *out = the largest row length (entries) of the CSR graph
__global__ void k_max_row(const int32_t* __restrict__ rp, int64_t n, int* out) {
    int m = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        m = max(m, rp[i + 1] - rp[i]);
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

// Row i's entries in segment s (columns [s w, (s + 1) w)) are
// bounds[s n + i] .. bounds[(s + 1) n + i] (rows sorted by column).
__global__ void k_seg_bounds(const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, int64_t n, int K,
                             int64_t w, int32_t* __restrict__ bounds) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int32_t t = rp[i];
    const int32_t e = rp[i + 1];
    bounds[i] = t;
    for (int s = 1; s < K; ++s) {
        const int64_t lim = (int64_t)s * w;
        while (t < e && ci[t] < lim) ++t;
        bounds[(int64_t)s * n + i] = t;
    }
    bounds[(int64_t)K * n + i] = e;
}

// One node-range segment of Q = c1 P - c2 W P: the gathered rows of P all lie
// in one range of the nodes, so that range stays in L2 for the pass.  The
// first segment writes Q, the others subtract into it.
template <int S>
__global__ void __launch_bounds__(256, 8) k_spmm_seg(const int32_t* __restrict__ lo, const int32_t* __restrict__ hi,
                                                  const int32_t* __restrict__ ci, const float* __restrict__ wv,
                                                  const float* __restrict__ P, float* __restrict__ Q, int64_t n,
                                                  int32_t ld, float c1, float c2, const ColState* __restrict__ st,
                                                  int first) {
    constexpr int L = S / 4;
    constexpr int RPB = 256 / L;
    if (!slab_has_work<S>(st)) return;
    const int g = (threadIdx.x & 31) % L;
    const int col = blockIdx.y * S + 4 * g;
    for (int64_t row = (int64_t)blockIdx.x * RPB + threadIdx.x / L; row < n; row += (int64_t)gridDim.x * RPB) {
        const int32_t b = __ldg(lo + row), e = __ldg(hi + row);
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 s2 = make_float4(0.f, 0.f, 0.f, 0.f);
        int32_t t = b;
        for (; t + 8 <= e; t += 8) {
            int32_t j[8];
            float w[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                j[u] = __ldg(ci + t + u);
                w[u] = __ldg(wv + t + u);
            }
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = ld4(P + (int64_t)j[u] * ld + col);
#pragma unroll
            for (int u = 0; u < 8; u += 2) {
                FMA4(s, w[u], v[u]);
                FMA4(s2, w[u + 1], v[u + 1]);
            }
        }
        // the last e - t < 8 entries as in k_spmm (a row's part in one node
        // range is short, ~nnz/(n K) entries, so this tail is a large share)
        for (; t < e; t += 4) {
            const int m = e - t;
            float4 v[4];
            float w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                w[u] = u < m ? __ldg(wv + t + u) : 0.f;
                v[u] = u < m ? ld4(P + (int64_t)__ldg(ci + t + u) * ld + col) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (u < m) {
                    FMA4(s, w[u], v[u]);
                }
            }
        }
        s.x += s2.x;
        s.y += s2.y;
        s.z += s2.z;
        s.w += s2.w;
        float4 q;
        if (first) {
            const float4 own = ld4(P + row * ld + col);
            q.x = c1 * own.x - c2 * s.x;
            q.y = c1 * own.y - c2 * s.y;
            q.z = c1 * own.z - c2 * s.z;
            q.w = c1 * own.w - c2 * s.w;
        } else {
            q = ld4v(Q + row * ld + col);
            q.x -= c2 * s.x;
            q.y -= c2 * s.y;
            q.z -= c2 * s.z;
            q.w -= c2 * s.w;
        }
        st4(Q + row * ld + col, q);
    }
}

// ---- column reductions ----
// Every per-column sum of the solve (||r||^2, p^T q, ||y||^2) is formed the
// same way whatever the launch shape: rows are cut into chunks of `rch`
// consecutive rows (rch depends on n only); within a chunk, thread g of 8 sums
// rows g, g + 8, ... in order for one column quad (compensated fp32), the 8
// sums meet in a fixed order in shared memory, and the chunk partials
// [nch][ld] are added in chunk order by the fp64 column kernels.  A column's CG
// scalars are therefore the same bit for bit whatever the slab width, the
// batch width or the other columns of the batch.
// A grid that fills the GPU runs these sums as they stand, one thread per (g,
// quad), rows streamed from memory (1M x 64: 0.23 ms for k_update, the copy
// bandwidth).  A small one would wait for memory 64 times in a row; there a
// block of 256 threads loads (and updates) a whole chunk of 16 columns at once
// into shared memory and one thread per (g, column) then sums its rows from
// there, in the same order (k_red_staged: with cold caches 7 us against 42 for
// the update of 2,000 x 16, 7 against 20 for the dot product).
constexpr int RG = 8;      // threads per chunk and quad
constexpr int RQ = 32;     // quads per block (at most)

int reduction_chunk_rows(int64_t n) {
    const int64_t r = (n + 4095) / 4096;
    return (int)std::max<int64_t>(512, (r + RG - 1) / RG * RG);
}

// the rows and columns of a thread: `work` is false when it has none
struct RedThread {
    int64_t r0, r1, chunk;
    int col, g, ql, qpb;
    bool work;
};
__device__ __forceinline__ RedThread red_thread(int64_t n, int32_t ld, int rch, const ColState* st) {
    RedThread t;
    const int nq = ld >> 2;
    t.qpb = nq < RQ ? nq : RQ;
    t.ql = (int)threadIdx.x % t.qpb;
    t.g = (int)threadIdx.x / t.qpb;
    const int quad = blockIdx.y * RQ + t.ql;
    t.col = 4 * quad;
    t.chunk = blockIdx.x;
    t.r0 = t.chunk * rch + t.g;
    t.r1 = min(n, (t.chunk + 1) * rch);
    t.work = quad < nq;
    if (t.work && st) {
        t.work = false;
#pragma unroll
        for (int c = 0; c < 4; ++c) t.work |= st[t.col + c].active != 0;
    }
    return t;
}

// combine the RG partial sums of each quad in g order and store the chunk partial
__device__ __forceinline__ void red_finish(float2* part, int32_t ld, const RedThread& t, const KSum (&a)[4]) {
    extern __shared__ float2 sm[];  // [RG][qpb * 4]
#pragma unroll
    for (int c = 0; c < 4; ++c)
        sm[(t.g * t.qpb + t.ql) * 4 + c] = t.work ? make_float2(a[c].s, a[c].c) : make_float2(0.f, 0.f);
    __syncthreads();
    if (t.g != 0 || !t.work) return;
    KSum s[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        s[c] = KSum{sm[t.ql * 4 + c].x, sm[t.ql * 4 + c].y};
#pragma unroll
        for (int h = 1; h < RG; ++h) {
            const float2 v = sm[(h * t.qpb + t.ql) * 4 + c];
            ksum_merge(s[c], KSum{v.x, v.y});
        }
    }
    float4* d = reinterpret_cast<float4*>(part + t.chunk * ld + t.col);
    d[0] = make_float4(s[0].s, s[0].c, s[1].s, s[1].c);
    d[1] = make_float4(s[2].s, s[2].c, s[3].s, s[3].c);
}

// Partials of sum_i V_ij^2 (every column).
__global__ void __launch_bounds__(256) k_colsq(const float* __restrict__ V, int64_t n, int32_t ld, int rch,
                                               float2* __restrict__ part) {
    constexpr int U = 8;
    const RedThread t = red_thread(n, ld, rch, nullptr);
    KSum acc[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
    if (t.work)
        for (int64_t row = t.r0; row < t.r1; row += U * RG) {
            float4 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                v[u] = row + u * RG < t.r1 ? ld4v(V + (row + u * RG) * ld + t.col) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (row + u * RG >= t.r1) break;
                ksum_add_product(acc[0], v[u].x, v[u].x);
                ksum_add_product(acc[1], v[u].y, v[u].y);
                ksum_add_product(acc[2], v[u].z, v[u].z);
                ksum_add_product(acc[3], v[u].w, v[u].w);
            }
        }
    red_finish(part, ld, t, acc);
}

// Partials of P^T Q (columns being iterated).  64 registers and four rows a turn: 1M x
// 64 takes 91 us, with the 48 registers of a plain loop 109.
__global__ void __launch_bounds__(256, 4) k_dot(const float* __restrict__ P, const Panels pv,
                                                const float* __restrict__ Q, int64_t n, int32_t ld, int rch,
                                                float2* __restrict__ part, const ColState* __restrict__ st) {
    const RedThread t = red_thread(n, ld, rch, st);
    KSum acc[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
    int pw;
    const float* Pc = panel_column(pv, P, t.col, pw);
    if (t.work)
#pragma unroll 4
        for (int64_t row = t.r0; row < t.r1; row += RG) {
            const float4 a = ld4(Pc + row * pw), b = ld4(Q + row * ld + t.col);
            ksum_add_product(acc[0], a.x, b.x);
            ksum_add_product(acc[1], a.y, b.y);
            ksum_add_product(acc[2], a.z, b.z);
            ksum_add_product(acc[3], a.w, b.w);
        }
    red_finish(part, ld, t, acc);
}

// The first block of the update (or, where the reduction after it is still gated
// by the active count, of the low-rank finish) clears what the scalar step and
// the fp16 copy accumulate into, in place of three memsets per iteration (16
// queries on 2,000 nodes: 457 -> 395 to 415 us); null pointers are skipped.
__device__ __forceinline__ void iter_reset(const IterReset& z) {
    if (blockIdx.x | blockIdx.y) return;
    if (z.p16_max)
        for (int c = threadIdx.x; c < z.Bp; c += blockDim.x) z.p16_max[c] = 0u;
    if (threadIdx.x == 0) {
        if (z.num_active) *z.num_active = 0;
        if (z.use_half) *z.use_half = -1;
    }
}

// The step lengths of a column quad and the columns that start afresh
struct UpdateQuad {
    float a[4], x[4];
    bool f[4], any;
};
__device__ __forceinline__ UpdateQuad update_quad(const ColState* st, int col, float xs) {
    UpdateQuad u;
    u.any = false;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        u.a[c] = (float)st[col + c].a;
        u.x[c] = xs * u.a[c];
        // a served column that took a new request at the last scalar step starts
        // from x0 = 0, r0 = y: x = a p, r = -a q here, y is added next
        u.f[c] = st[col + c].refill;
        u.any |= u.f[c];
    }
    return u;
}
__device__ __forceinline__ void update_row(const UpdateQuad& u, const float4& p, const float4& q, float4& x, float4& r) {
    if (u.any) {
        if (u.f[0]) x.x = r.x = 0.0f;
        if (u.f[1]) x.y = r.y = 0.0f;
        if (u.f[2]) x.z = r.z = 0.0f;
        if (u.f[3]) x.w = r.w = 0.0f;
    }
    x.x = fmaf(u.x[0], p.x, x.x);
    x.y = fmaf(u.x[1], p.y, x.y);
    x.z = fmaf(u.x[2], p.z, x.z);
    x.w = fmaf(u.x[3], p.w, x.w);
    r.x = fmaf(-u.a[0], q.x, r.x);
    r.y = fmaf(-u.a[1], q.y, r.y);
    r.z = fmaf(-u.a[2], q.z, r.z);
    r.w = fmaf(-u.a[3], q.w, r.w);
}

// X += xs a P; R -= a Q; partials of ||R||^2.  Four rows' loads ahead of their
// sums: at one row, which the compiler makes of a plain loop, 1M x 64 takes 239 us
// against 224, 1M x 100 421 against 353, 1M x 256 930 against 877.
__global__ void __launch_bounds__(256) k_update(float* __restrict__ X, float* __restrict__ R,
                                                const float* __restrict__ P, const Panels pv,
                                                const float* __restrict__ Q, int64_t n, int32_t ld, int rch,
                                                const ColState* __restrict__ st, float xs, float2* __restrict__ part,
                                                const IterReset z) {
    iter_reset(z);
    const RedThread t = red_thread(n, ld, rch, st);
    KSum acc[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
    constexpr int U = 4;
    if (t.work) {
        const UpdateQuad uq = update_quad(st, t.col, xs);
        int pw;
        const float* Pc = panel_column(pv, P, t.col, pw);
        for (int64_t row = t.r0; row < t.r1; row += U * RG) {
            float4 p[U], q[U], x[U], r[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                p[u] = q[u] = x[u] = r[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (row + u * RG < t.r1) {
                    const int64_t o = (row + u * RG) * ld + t.col;
                    p[u] = ld4v(Pc + (row + u * RG) * pw);
                    q[u] = ld4v(Q + o);
                    x[u] = ld4v(X + o);
                    r[u] = ld4v(R + o);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (row + u * RG >= t.r1) break;
                const int64_t o = (row + u * RG) * ld + t.col;
                update_row(uq, p[u], q[u], x[u], r[u]);
                st4(X + o, x[u]);
                st4(R + o, r[u]);
                ksum_add_product(acc[0], r[u].x, r[u].x);
                ksum_add_product(acc[1], r[u].y, r[u].y);
                ksum_add_product(acc[2], r[u].z, r[u].z);
                ksum_add_product(acc[3], r[u].w, r[u].w);
            }
        }
    }
    red_finish(part, ld, t, acc);
}

// The three sums above for small grids: block (chunk, group of 4 quads).
enum RedOp { RED_SQ, RED_DOT, RED_UPDATE };
constexpr int RS_ROWS = 512;  // rows staged at a time (a whole chunk up to 2M rows)
constexpr int RS_COLS = 16;   // columns of a block
template <int OP>
constexpr int rs_smem() {
    return RS_ROWS * RS_COLS * 4 * (OP == RED_DOT ? 2 : 1);
}
template <int OP>
__global__ void __launch_bounds__(256) k_red_staged(float* __restrict__ X, float* __restrict__ R,
                                                    const float* __restrict__ P, const Panels pv,
                                                    const float* __restrict__ Q, int64_t n, int32_t ld, int rch,
                                                    const ColState* __restrict__ st,
                                                    float xs, float2* __restrict__ part, const IterReset z) {
    if (OP == RED_UPDATE) iter_reset(z);
    constexpr int UL = 4;  // rows in flight per thread
    extern __shared__ float rs_sm[];
    __shared__ float2 sums[RG * RS_COLS];
    const int cq = min(RS_COLS / 4, (ld >> 2) - (int)blockIdx.y * (RS_COLS / 4)), nc = 4 * cq;
    const int c0 = blockIdx.y * RS_COLS;
    float4* A = reinterpret_cast<float4*>(rs_sm);  // [row][quad]
    float4* B = A + RS_ROWS * cq;
    const int64_t lo = (int64_t)blockIdx.x * rch, hi = min(n, lo + rch);
    // loading threads: quad lq of the group, rows lr, lr + rows_per_pass, ...
    const int lq = threadIdx.x % cq, lr = threadIdx.x / cq, pass = 256 / cq;
    const int col = c0 + 4 * lq;
    bool work = lr < pass;
    UpdateQuad uq;
    if (OP != RED_SQ) {
        work = work && (st[col].active | st[col + 1].active | st[col + 2].active | st[col + 3].active);
        if (OP == RED_UPDATE) uq = update_quad(st, col, xs);
    }
    int pw;
    const float* Pc = panel_column(pv, P, col, pw);
    // summing threads: column sc, partial sum sg
    const int sc = threadIdx.x % nc, sg = threadIdx.x / nc;
    bool sum = sg < RG;
    if (OP != RED_SQ && sum) {
        const ColState* q = st + c0 + (sc & ~3);
        sum = q[0].active | q[1].active | q[2].active | q[3].active;
    }
    KSum acc{0.f, 0.f};
    for (int64_t base = lo; base < hi; base += RS_ROWS) {
        const int rows = (int)min((int64_t)RS_ROWS, hi - base);
        if (work)
            for (int r0 = lr; r0 < rows; r0 += UL * pass) {
                float4 p[UL], q[UL], x[UL], r[UL];
#pragma unroll
                for (int u = 0; u < UL; ++u) {
                    const int64_t o = (base + r0 + u * pass) * ld + col;
                    if (r0 + u * pass < rows) {
                        p[u] = ld4v(Pc + (base + r0 + u * pass) * pw);
                        if (OP != RED_SQ) q[u] = ld4v(Q + o);
                        if (OP == RED_UPDATE) {
                            x[u] = ld4v(X + o);
                            r[u] = ld4v(R + o);
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < UL; ++u) {
                    const int row = r0 + u * pass;
                    if (row >= rows) break;
                    if (OP == RED_UPDATE) {
                        const int64_t o = (base + row) * ld + col;
                        update_row(uq, p[u], q[u], x[u], r[u]);
                        st4(X + o, x[u]);
                        st4(R + o, r[u]);
                        A[row * cq + lq] = r[u];
                    } else {
                        A[row * cq + lq] = p[u];
                        if (OP == RED_DOT) B[row * cq + lq] = q[u];
                    }
                }
            }
        __syncthreads();
        if (sum) {
            const float* a = reinterpret_cast<const float*>(A);
            const float* b = OP == RED_DOT ? reinterpret_cast<const float*>(B) : a;
#pragma unroll 8
            for (int row = sg; row < rows; row += RG) ksum_add_product(acc, a[row * nc + sc], b[row * nc + sc]);
        }
        __syncthreads();
    }
    if (sg < RG) sums[sg * RS_COLS + sc] = make_float2(acc.s, acc.c);
    __syncthreads();
    if (sum && sg == 0) {
        KSum t = acc;
#pragma unroll
        for (int h = 1; h < RG; ++h) {
            const float2 v = sums[h * RS_COLS + sc];
            ksum_merge(t, KSum{v.x, v.y});
        }
        part[(int64_t)blockIdx.x * ld + c0 + sc] = make_float2(t.s, t.c);
    }
}

// P = R + beta P.
template <int S>
__global__ void __launch_bounds__(256) k_direction(float* __restrict__ P, const Panels pv, const float* __restrict__ R,
                                                   int64_t n, int32_t ld, const ColState* __restrict__ st) {
    constexpr int L = S / 4;
    constexpr int RPB = 256 / L;
    if (!slab_has_work<S>(st)) return;
    const int g = (threadIdx.x & 31) % L;
    const int col = blockIdx.y * S + 4 * g;
    const float b0 = (float)st[col].beta, b1 = (float)st[col + 1].beta, b2 = (float)st[col + 2].beta,
                b3 = (float)st[col + 3].beta;
    // a served column that just took a new request: p0 = y, added after this
    const bool f0 = st[col].refill, f1 = st[col + 1].refill, f2 = st[col + 2].refill, f3 = st[col + 3].refill;
    int pw;
    float* Pc = panel_column(pv, P, col, pw);
    for (int64_t row = (int64_t)blockIdx.x * RPB + threadIdx.x / L; row < n; row += (int64_t)gridDim.x * RPB) {
        float* o = Pc + row * pw;
        const float4 r = ld4v(R + row * ld + col);
        float4 p = ld4v(o);
        p.x = b0 == 0.0f ? (f0 ? 0.0f : r.x) : fmaf(b0, p.x, r.x);
        p.y = b1 == 0.0f ? (f1 ? 0.0f : r.y) : fmaf(b1, p.y, r.y);
        p.z = b2 == 0.0f ? (f2 ? 0.0f : r.z) : fmaf(b2, p.z, r.z);
        p.w = b3 == 0.0f ? (f3 ? 0.0f : r.w) : fmaf(b3, p.w, r.w);
        st4(o, p);
    }
}

// ---- per-column scalar kernels: one block per column, fp64 reductions ----
// Block-wide fp64 sum (all threads get the result).
__device__ __forceinline__ double block_sum_f64(double v) {
    __shared__ double sm[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sm[w] = v;
    __syncthreads();
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += sm[i];
    return t;
}

// sum over blocks of column j's compensated partials (eight loads ahead of their adds)
__device__ __forceinline__ double col_sum(const float2* part, int nblk, int ld, int j) {
    double s = 0.0;
    const int step = blockDim.x;
    for (int b = threadIdx.x; b < nblk; b += 8 * step) {
        float2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            v[u] = b + u * step < nblk ? part[(int64_t)(b + u * step) * ld + j] : make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (b + u * step < nblk) s += (double)v[u].x + (double)v[u].y;
    }
    return block_sum_f64(s);
}

// sum_k coef_k C_kj^2
__device__ __forceinline__ double col_lowrank(const double* C, const double* coef, int r, int ld, int j) {
    double s = 0.0;
    if (C)
        for (int k = threadIdx.x; k < r; k += blockDim.x) {
            const double c = C[(int64_t)k * ld + j];
            s += coef[k] * c * c;
        }
    return block_sum_f64(s);
}

// Setup: bb = ||b||^2; rho = bb (+ sum D C^2 for PCG); activity and 0-iteration convergence.
__global__ void k_fin_setup(const float2* part, int nblk, int32_t Bp, int32_t B, const float* tol, ColState* st,
                            const double* C, const double* coef, int32_t r, int* num_active) {
    const int j = blockIdx.x;
    const double bb = col_sum(part, nblk, Bp, j);
    const double lrt = col_lowrank(C, coef, r, Bp, j);
    if (threadIdx.x != 0) return;
    ColState s;
    s.bb = bb;
    s.rr = bb;
    s.rho = bb + lrt;
    const double t = j < B ? (double)tol[j] : 0.0;
    s.tol2 = t * t * bb;
    s.sigma = 0.0;
    s.a = 0.0;
    s.beta = 0.0;
    s.iters = 0;
    s.confirms = 0;
    s.restart = 0;
    s.refill = 0;
    s.free_col = 0;
    s.rr_fix = 0.0;
    if (j >= B || bb == 0.0) {
        s.active = 0;
        s.status = HD_COL_EMPTY;
    } else if (bb <= s.tol2) {
        s.active = 0;
        s.status = HD_COL_CONVERGED;
    } else {
        s.active = 1;
        s.status = HD_COL_MAX_ITER;
        atomicAdd(num_active, 1);
    }
    st[j] = s;
}

// a = rho / sigma with sigma = SpMM partials (+ sum_k coef_k C_k^2).
__global__ void k_fin_sigma(const float2* part, int nblk, int32_t Bp, ColState* st, const double* C,
                            const double* coef, int32_t r) {
    const int j = blockIdx.x;
    ColState& s = st[j];
    if (!s.active) {
        if (threadIdx.x == 0) s.a = 0.0;
        return;
    }
    const double sig = col_sum(part, nblk, Bp, j) + col_lowrank(C, coef, r, Bp, j);
    if (threadIdx.x != 0) return;
    s.sigma = sig;
    if (!(sig > 0.0) || !isfinite(sig)) {
        s.active = 0;
        s.status = HD_COL_BREAKDOWN;
        s.a = 0.0;
    } else {
        s.a = s.rho / sig;
    }
}

// After the update: rr, convergence, beta.  With C: PCG rho' = rr + sum_k coef_k C_k^2.
// num_active must be zero before the launch (iter_reset).
// use_half (may be null; not 0 before the launch, see iter_reset): cleared when a column that stays
// active has ||r||^2 > theta2 tol^2 ||b||^2 (the next SpMM then gathers fp32).
__global__ void k_fin_rr(const float2* part, int nblk, int32_t Bp, ColState* st, int32_t max_iter,
                         const double* C, const double* coef, int32_t r, int* num_active, int* use_half = nullptr,
                         double theta2 = 0.0) {
    const int j = blockIdx.x;
    ColState& s = st[j];
    if (!s.active) {
        if (threadIdx.x == 0) s.beta = 0.0;
        return;
    }
    const double rr = col_sum(part, nblk, Bp, j);
    const double lrt = col_lowrank(C, coef, r, Bp, j);
    if (threadIdx.x != 0) return;
    const double rho = rr + lrt;
    s.iters += 1;
    s.rr = rr;
    s.beta = rho / s.rho;
    s.rho = rho;
    if (!isfinite(rr)) {
        s.active = 0;
        s.status = HD_COL_BREAKDOWN;
        s.beta = 0.0;
    } else if (rr <= s.tol2) {
        s.active = 0;
        s.status = HD_COL_CONVERGED;
    } else if (s.iters >= max_iter) {
        s.active = 0;
        s.status = HD_COL_MAX_ITER;
    } else {
        atomicAdd(num_active, 1);
        if (use_half && !(rr <= theta2 * s.tol2)) atomicExch(use_half, 0);
    }
}

// sum_k coef_k c_k^2 for one contiguous row c (block-wide)
__device__ __forceinline__ double row_lowrank(const double* c, const double* coef, int r) {
    double v = 0.0;
    if (c)
        for (int k = threadIdx.x; k < r; k += blockDim.x) v += coef[k] * c[k] * c[k];
    return block_sum_f64(v);
}

// The scalar step of a server lane (k_fin_rr plus admission inside the
// iteration).  A free column the host assigned (the lowest free ones, so that
// the occupied columns stay packed) takes its staged request, and a column that
// stops here claims the next unassigned one: the stopped request's iterations,
// status and ||r||^2 go to the
// host, the column restarts as the new request (r0 = y, rho = y^T M^-1 y from
// the staged U^T y) with `refill` set, so that the direction that follows
// forms p0 = M^-1 y and the next update starts x and r afresh.  A stopped
// column that claims nothing becomes free once the host has its ranking.
// A refilled column's first ||r||^2 adds rr_fix (the y entries, exact).
__global__ void k_fin_rr_serve(const float2* part, int nblk, int32_t Bp, ColState* st, int32_t max_iter,
                               const double* C, const double* coef, int32_t r, int* num_active, Refill rf) {
    __shared__ int claim;
    const int j = blockIdx.x;
    ColState& s = st[j];
    const bool active = s.active, was_free = s.free_col;
    if (!active && !was_free) {
        if (threadIdx.x == 0) s.beta = 0.0;
        return;
    }
    double rr = 0.0, lrt = 0.0;
    if (active) {
        rr = col_sum(part, nblk, Bp, j);
        lrt = col_lowrank(C, coef, r, Bp, j);
    }
    if (threadIdx.x == 0) {
        claim = -1;
        bool stopped = was_free;
        if (active) {
            if (s.refill) {
                rr += s.rr_fix;
                s.refill = 0;
            }
            const double rho = rr + lrt;
            s.iters += 1;
            s.rr = rr;
            s.beta = rho / s.rho;
            s.rho = rho;
            stopped = true;
            if (!isfinite(rr)) {
                s.active = 0;
                s.status = HD_COL_BREAKDOWN;
                s.beta = 0.0;
            } else if (rr <= s.tol2) {
                s.active = 0;
                s.status = HD_COL_CONVERGED;
            } else if (s.iters >= max_iter) {
                s.active = 0;
                s.status = HD_COL_MAX_ITER;
            } else {
                stopped = false;
                atomicAdd(num_active, 1);
            }
        }
        if (stopped) {
            // a free column the host assigned takes its request; a column that
            // stops here (or stopped earlier in the step) the next unassigned one
            const int ns = *rf.nstage;
            int c = INT_MAX;
            if (ns > 0) {
                const int pc = rf.pre[j];
                c = pc >= 0 ? pc : j < rf.live ? atomicAdd(rf.next, 1) : INT_MAX;
            }
            if (c < ns) claim = c;
            else if (active) s.free_col = 1;
        }
    }
    __syncthreads();
    const int c = claim;
    if (c < 0) return;
    const double lrs = row_lowrank(rf.C ? rf.C + (int64_t)c * rf.rpad : nullptr, coef, r);
    if (threadIdx.x != 0) return;
    // the request the column held (stopped here or at an earlier step's
    // iteration; the host ignores these for a column it holds as free)
    rf.ret_iters[j] = s.iters;
    rf.ret_status[j] = s.status;
    rf.ret_rr[j] = s.rr;
    rf.assign[j] = c;
    s.bb = rf.bb[c];
    s.tol2 = rf.tol2[c];
    s.rr = s.bb;
    s.rho = s.bb + lrs;
    s.beta = 0.0;
    s.a = 0.0;
    s.iters = 0;
    s.confirms = 0;
    s.restart = 0;
    s.rr_fix = 0.0;
    s.active = 1;
    s.free_col = 0;
    s.refill = 1;
    s.status = HD_COL_MAX_ITER;
    atomicAdd(num_active, 1);
}

// H = coef o (U^T y) for the columns that took a staged request (the operand
// of the direction's U H; the other columns keep theirs)
__global__ void k_refill_h(Refill rf, const double* coef, int rpad, int32_t Bp, float* H, __nv_bfloat16* Hhi,
                           __nv_bfloat16* Hlo) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)rpad * Bp) return;
    const int k = (int)(e / Bp), j = (int)(e % Bp);
    const int c = rf.assign[j];
    if (c < 0) return;
    const double h = coef[k] * rf.C[(int64_t)c * rpad + k];
    H[e] = (float)h;
    if (Hhi) {
        const __nv_bfloat16 hi = __double2bfloat16(h);
        const __nv_bfloat16 lo = __double2bfloat16(h - (double)__bfloat162float(hi));
        Hhi[(int64_t)j * rpad + k] = hi;
        Hlo[(int64_t)j * rpad + k] = lo;
    }
}

// p0 += y for the columns that took a staged request (the direction left
// U D U^T y there, or 0 without eigenpairs); y is kept with the column for its
// first update
__global__ void k_refill_p(Refill rf, float* P, const Panels pv, int32_t Bp) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= Bp) return;
    const int c = rf.assign[j];
    if (c < 0) return;
    const int32_t b = rf.off[c], e = rf.off[c + 1];
    int pw;
    float* Pc = panel_column(pv, P, j, pw);
    for (int32_t t = b; t < e; ++t) {
        const int32_t i = rf.yidx[t];
        const float v = rf.yval[t];
        Pc[(int64_t)i * pw] += v;
        rf.col_idx[(int64_t)j * REFILL_MAX_NNZ + (t - b)] = i;
        rf.col_val[(int64_t)j * REFILL_MAX_NNZ + (t - b)] = v;
    }
    rf.col_cnt[j] = e - b;
}

// After the first update of a refilled column (r = -a q): r += y, and rr_fix =
// sum over y's entries of (r_i + y_i)^2 - r_i^2 (fp64; duplicates in turn)
__global__ void k_refill_r(Refill rf, float* R, int32_t Bp, ColState* st) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= Bp || !st[j].refill) return;
    double fix = 0.0;
    for (int t = 0; t < rf.col_cnt[j]; ++t) {
        float* a = R + (int64_t)rf.col_idx[(int64_t)j * REFILL_MAX_NNZ + t] * Bp + j;
        const float v = *a;
        const float w = v + rf.col_val[(int64_t)j * REFILL_MAX_NNZ + t];
        *a = w;
        fix += (double)w * (double)w - (double)v * (double)v;
    }
    st[j].rr_fix = fix;
}

int launch_refill_r(Engine& E) {
    k_refill_r<<<ceil_div(E.Bp, 128), 128, 0, E.ctx->stream>>>(*E.refill, E.R, E.Bp, E.st);
    HD_CHECK_LAUNCH(E.ctx);
    return HD_OK;
}

// Which residual kernel runs: the fp32 evaluation of b - A x has an error of
// at most (c2 gamma_m + 2 u c1) ||x|| + 2 u ||b|| (u = 2^-24; gamma_m = m u /
// (1 - m u) bounds the rounding of a sum of m products, m the longest row
// plus one; ||W|x||| <= ||x|| for the nonnegative W of spectral radius 1).
// When that is at most a tenth of tol ||b|| for every column, the fp32 SpMM
// runs (*pick = 0), else the two-word kernel (*pick = 1).  part: partials of
// ||x_j||^2; one block per column.
__global__ void k_resid_pick(const float2* part, int nblk, int32_t Bp, int32_t B, const ColState* st, double gamma,
                             double c1, double c2, int* pick) {
    const int j = blockIdx.x;
    if (j >= B) return;
    const double xx = col_sum(part, nblk, Bp, j);
    if (threadIdx.x != 0) return;
    const ColState& s = st[j];
    if (s.status == HD_COL_EMPTY || s.status == HD_COL_CANCELLED || s.bb <= 0.0) return;
    const double u = 1.0 / 16777216.0;
    const double bound = (c2 * gamma + 2.0 * u * c1) * sqrt(xx) + 2.0 * u * sqrt(s.bb);
    // tol2 = tol^2 ||b||^2
    if (!(bound <= 0.1 * sqrt(s.tol2))) atomicExch(pick, 1);
}

// ---- confirmation by the true residual (x0 = 0 and a residual stopping rule, Sec. 4.4)
// Residual replacements allowed per column and solve.
constexpr int MAX_CONFIRM = 3;

// part: partials of ||T||^2, T = b - A x (every column).  rr := ||T||^2, the
// value the solve reports.  A column whose recursive residual met tol while
// ||T|| > tol ||b|| is reactivated with r := T (flag `restart`) while it has
// iterations and replacements left; otherwise it is STAGNATED.
__global__ void k_fin_confirm(const float2* part, int nblk, int32_t Bp, int32_t B, ColState* st, int32_t max_iter,
                              int* num_active) {
    const int j = blockIdx.x;
    ColState& s = st[j];
    if (j >= B || s.status == HD_COL_EMPTY || s.status == HD_COL_CANCELLED) return;
    const double tt = col_sum(part, nblk, Bp, j);
    if (threadIdx.x != 0) return;
    s.rr = tt;
    s.restart = 0;
    if (!isfinite(tt)) {
        s.status = HD_COL_BREAKDOWN;
        return;
    }
    if (s.status != HD_COL_CONVERGED || tt <= s.tol2) return;
    if (s.iters < max_iter && s.confirms < MAX_CONFIRM) {
        s.confirms += 1;
        s.active = 1;
        s.status = HD_COL_MAX_ITER;
        s.restart = 1;
        atomicAdd(num_active, 1);
    } else {
        s.status = HD_COL_STAGNATED;
    }
}

// R[:, j] := T[:, j] for the columns being restarted.
__global__ void k_restart_copy(float* __restrict__ R, const float* __restrict__ T, int64_t n, int32_t ld,
                               const ColState* __restrict__ st) {
    const int nq = ld >> 2;
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;  // float4 index = row * nq + quad
    if (e >= n * nq) return;
    const int col = 4 * (int)(e % nq);
    const int m = st[col].restart | st[col + 1].restart << 1 | st[col + 2].restart << 2 | st[col + 3].restart << 3;
    if (!m) return;
    float4 r = ld4v(R + 4 * e);
    const float4 t = ld4v(T + 4 * e);
    if (m & 1) r.x = t.x;
    if (m & 2) r.y = t.y;
    if (m & 4) r.z = t.z;
    if (m & 8) r.w = t.w;
    st4(R + 4 * e, r);
}

// Restarted columns: rho = ||r||^2 (+ sum_k coef_k C_k^2 with the
// preconditioner, C = U^T r), a fresh direction (beta = 0); every other
// column gets beta = 0 so the direction update leaves it finite.
__global__ void k_fin_restart(ColState* st, const double* C, const double* coef, int32_t r) {
    const int j = blockIdx.x;
    ColState& s = st[j];
    if (!s.restart) {
        if (threadIdx.x == 0) s.beta = 0.0;
        return;
    }
    const double lrt = col_lowrank(C, coef, r, gridDim.x, j);
    if (threadIdx.x != 0) return;
    s.rho = s.rr + lrt;
    s.beta = 0.0;
    s.a = 0.0;
    s.restart = 0;
}

// C [rpad][Bp] (fp64) given directly: H = coef o C (fp32 and bf16 hi/lo
// transposed), the operand layout lr_finish produces from partials.
__global__ void k_lr_coef(const double* __restrict__ Csrc, int rpad, int32_t Bp, const double* __restrict__ coef,
                          float* H, __nv_bfloat16* Hhi, __nv_bfloat16* Hlo) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)rpad * Bp) return;
    const int k = (int)(e / Bp), j = (int)(e % Bp);
    const double h = coef[k] * Csrc[e];
    H[e] = (float)h;
    if (Hhi) {
        const __nv_bfloat16 hi = __double2bfloat16(h);
        const __nv_bfloat16 lo = __double2bfloat16(h - (double)__bfloat162float(hi));
        Hhi[(int64_t)j * rpad + k] = hi;
        Hlo[(int64_t)j * rpad + k] = lo;
    }
}

__global__ void k_outputs(const ColState* st, int32_t B, int32_t* iters, float* relres, int32_t* status) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= B) return;
    ColState s = st[j];
    if (iters) iters[j] = s.iters;
    if (relres) relres[j] = s.bb > 0.0 ? (float)sqrt(s.rr / s.bb) : 0.0f;
    if (status) status[j] = s.status;
}

__global__ void k_copy_out(const float* Xi, int32_t Bp, float* X, int32_t ldx, int32_t B, int64_t n) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n * B) return;
    int64_t i = e / B;
    int j = (int)(e % B);
    X[i * ldx + j] = Xi[i * Bp + j];
}

// ------------------------------------------------------------------ low-rank, CUDA cores
template <typename T>
__device__ __forceinline__ float u_at(const T* U, const float* scale, int64_t i, int ldu, int k);
template <>
__device__ __forceinline__ float u_at<float>(const float* U, const float*, int64_t i, int ldu, int k) {
    return __ldg(U + i * ldu + k);
}
template <>
__device__ __forceinline__ float u_at<__nv_bfloat16>(const __nv_bfloat16* U, const float*, int64_t i, int ldu, int k) {
    return __bfloat162float(U[i * ldu + k]);
}
template <>
__device__ __forceinline__ float u_at<__nv_fp8_e4m3>(const __nv_fp8_e4m3* U, const float* scale, int64_t i, int ldu,
                                                      int k) {
    return float(U[i * ldu + k]) * __ldg(scale + i);
}

// part[c][k][j] = sum_{i in chunk c} U_ik V_ij ; grid (chunk, k-block of 64, 16-column slab)
template <typename T>
__global__ void __launch_bounds__(256) k_lr_reduce_simt(const T* __restrict__ U, const float* __restrict__ scale,
                                                        int ldu, int r, int rpad, const float* __restrict__ V,
                                                        int64_t n, int32_t Bp, int64_t rpc,
                                                        float* __restrict__ part, const int* gate) {
    if (gate && *gate == 0) return;
    const int kk = threadIdx.x >> 2, cq = 4 * (threadIdx.x & 3);
    const int k = blockIdx.y * 64 + kk;
    const int col = blockIdx.z * 16 + cq;
    const int64_t i0 = (int64_t)blockIdx.x * rpc;
    const int64_t i1 = min(n, i0 + rpc);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k < r && col < Bp)
        for (int64_t i = i0; i < i1; ++i) {
            const float u = u_at<T>(U, scale, i, ldu, k);
            const float4 v = ld4(V + i * Bp + col);
            acc.x = fmaf(u, v.x, acc.x);
            acc.y = fmaf(u, v.y, acc.y);
            acc.z = fmaf(u, v.z, acc.z);
            acc.w = fmaf(u, v.w, acc.w);
        }
    if (k < rpad && col < Bp) st4(part + ((int64_t)blockIdx.x * rpad + k) * Bp + col, acc);
}

// C = sum over chunks (fp64); H = coef o C (fp32 and bf16 hi/lo transposed).
// Block: 32 consecutive entries x 8 warps splitting the chunks.
__global__ void __launch_bounds__(256) k_lr_finish(const float* __restrict__ part, int nchunk, int rpad, int32_t Bp,
                                                   const double* coef, double* C, float* H, __nv_bfloat16* Hhi,
                                                   __nv_bfloat16* Hlo, const IterReset z) {
    iter_reset(z);
    __shared__ double sm[8][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t e = (int64_t)blockIdx.x * 32 + lane;
    const int64_t tot = (int64_t)rpad * Bp;
    double s = 0.0;
    if (e < tot)
        for (int c = w; c < nchunk; c += 64) {
            float v[8];  // eight chunks' loads ahead of their adds
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = c + 8 * u < nchunk ? part[(int64_t)(c + 8 * u) * tot + e] : 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (c + 8 * u < nchunk) s += (double)v[u];
        }
    sm[w][lane] = s;
    __syncthreads();
    if (w != 0 || e >= tot) return;
    s = 0.0;
    for (int i = 0; i < 8; ++i) s += sm[i][lane];
    const int k = (int)(e / Bp), j = (int)(e % Bp);
    C[e] = s;
    const double h = coef[k] * s;
    H[e] = (float)h;
    if (Hhi) {
        const __nv_bfloat16 hi = __double2bfloat16(h);
        const __nv_bfloat16 lo = __double2bfloat16(h - (double)__bfloat162float(hi));
        Hhi[(int64_t)j * rpad + k] = hi;
        Hlo[(int64_t)j * rpad + k] = lo;
    }
}

// out = op(U H) for the 16-column slab blockIdx.y; H staged in shared memory.
template <typename T>
__global__ void __launch_bounds__(256) k_lr_expand_simt(const T* __restrict__ U, const float* __restrict__ scale,
                                                        int ldu, int r, const float* __restrict__ H, int op,
                                                        float* __restrict__ out, const float* __restrict__ Rv,
                                                        const float* __restrict__ Pv, int64_t n, int32_t Bp,
                                                        const ColState* __restrict__ st, const int* gate) {
    if (gate && *gate == 0) return;
    extern __shared__ float Hs[];  // [r][16]
    const int slab = blockIdx.y;
    for (int e = threadIdx.x; e < r * 16; e += blockDim.x) {
        const int k = e >> 4, c = e & 15;
        Hs[e] = (slab * 16 + c < Bp) ? H[(int64_t)k * Bp + slab * 16 + c] : 0.0f;
    }
    __syncthreads();
    const int cq = 4 * (threadIdx.x & 3);
    const int col = slab * 16 + cq;
    if (col >= Bp) return;
    float b0 = 0.f, b1 = 0.f, b2 = 0.f, b3 = 0.f;
    bool f0 = false, f1 = false, f2 = false, f3 = false;
    if (op == EXP_DIRECTION) {
        b0 = (float)st[col].beta;
        b1 = (float)st[col + 1].beta;
        b2 = (float)st[col + 2].beta;
        b3 = (float)st[col + 3].beta;
        // a served column that just took a new request drops r (p0 = U D U^T y + y)
        f0 = st[col].refill;
        f1 = st[col + 1].refill;
        f2 = st[col + 2].refill;
        f3 = st[col + 3].refill;
    }
    for (int64_t row = (int64_t)blockIdx.x * 64 + (threadIdx.x >> 2); row < n; row += (int64_t)gridDim.x * 64) {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k = 0; k < r; ++k) {
            const float u = u_at<T>(U, scale, row, ldu, k);
            const float4 h = *reinterpret_cast<const float4*>(Hs + k * 16 + cq);
            acc.x = fmaf(u, h.x, acc.x);
            acc.y = fmaf(u, h.y, acc.y);
            acc.z = fmaf(u, h.z, acc.z);
            acc.w = fmaf(u, h.w, acc.w);
        }
        const int64_t o = row * Bp + col;
        float4 v;
        if (op == EXP_SET_X) {
            v = acc;
        } else if (op == EXP_SUB_R) {
            v = ld4v(out + o);
            v.x -= acc.x; v.y -= acc.y; v.z -= acc.z; v.w -= acc.w;
        } else if (op == EXP_ADD_Q) {
            v = ld4v(out + o);
            v.x += acc.x; v.y += acc.y; v.z += acc.z; v.w += acc.w;
        } else {
            const float4 rr = ld4v(Rv + o), pp = ld4v(Pv + o);
            v.x = (f0 ? 0.0f : rr.x) + acc.x + (b0 == 0.0f ? 0.0f : b0 * pp.x);
            v.y = (f1 ? 0.0f : rr.y) + acc.y + (b1 == 0.0f ? 0.0f : b1 * pp.y);
            v.z = (f2 ? 0.0f : rr.z) + acc.z + (b2 == 0.0f ? 0.0f : b2 * pp.z);
            v.w = (f3 ? 0.0f : rr.w) + acc.w + (b3 == 0.0f ? 0.0f : b3 * pp.w);
        }
        st4(out + o, v);
    }
}

int simt_nchunk(hd_ctx* ctx, int64_t n, int rpad, int Bp) {
    int blocks_per_chunk = (rpad / 64) * ceil_div(Bp, 16);
    int nc = ceil_div(4 * ctx->num_sms, blocks_per_chunk);
    int64_t maxc = std::max<int64_t>(1, n / 64);
    return (int)std::max<int64_t>(1, std::min<int64_t>(nc, maxc));
}

int lr_nchunk(hd_ctx* ctx, const hd_eig* e, int32_t Bp) {
    if (e->sparse) return lr_sparse_nchunk(ctx, e);
    return lr_use_tensor_cores(e) ? lr_tc_nchunk(ctx, e->n) : simt_nchunk(ctx, e->n, (e->r + 63) / 64 * 64, Bp);
}

int lr_reduce(hd_ctx* ctx, const LowRank& lr, const float* V, int64_t n, int32_t Bp, const int* gate) {
    HD_PROF(ctx, "lr_reduce");
    if (lr.e->sparse) return lr_sparse_reduce(ctx, lr, V, n, Bp, gate);
    if (lr_use_tensor_cores(lr.e)) return lr_tc_reduce(ctx, lr, V, n, Bp, gate);
    const hd_eig* e = lr.e;
    int64_t rpc = (n + lr.nchunk - 1) / lr.nchunk;
    dim3 grid(lr.nchunk, lr.rpad / 64, ceil_div(Bp, 16));
    if (e->storage == HD_F32)
        k_lr_reduce_simt<float><<<grid, 256, 0, ctx->stream>>>((const float*)e->U, e->scale, e->ldu, e->r, lr.rpad, V,
                                                               n, Bp, rpc, lr.part, gate);
    else if (e->storage == HD_BF16)
        k_lr_reduce_simt<__nv_bfloat16><<<grid, 256, 0, ctx->stream>>>((const __nv_bfloat16*)e->U, e->scale, e->ldu,
                                                                       e->r, lr.rpad, V, n, Bp, rpc, lr.part, gate);
    else
        k_lr_reduce_simt<__nv_fp8_e4m3><<<grid, 256, 0, ctx->stream>>>((const __nv_fp8_e4m3*)e->U, e->scale, e->ldu,
                                                                       e->r, lr.rpad, V, n, Bp, rpc, lr.part, gate);
    HD_CHECK_LAUNCH(ctx);
    return HD_OK;
}

int lr_finish(hd_ctx* ctx, const LowRank& lr, int32_t Bp, const double* coef, const IterReset& z) {
    HD_PROF(ctx, "scalar");
    int64_t tot = (int64_t)lr.rpad * Bp;
    k_lr_finish<<<ceil_div(tot, 32), 256, 0, ctx->stream>>>(lr.part, lr.nchunk, lr.rpad, Bp, coef, lr.C,
                                                             lr.H, lr.Hhi, lr.Hlo, z);
    HD_CHECK_LAUNCH(ctx);
    return HD_OK;
}

// H = coef o Csrc for a C kept from earlier (the operand of lr_expand)
static int lr_coef(hd_ctx* ctx, const LowRank& lr, int32_t Bp, const double* coef, const double* Csrc) {
    HD_PROF(ctx, "scalar");
    const int64_t tot = (int64_t)lr.rpad * Bp;
    k_lr_coef<<<ceil_div(tot, 256), 256, 0, ctx->stream>>>(Csrc, lr.rpad, Bp, coef, lr.H, lr.Hhi, lr.Hlo);
    HD_CHECK_LAUNCH(ctx);
    return HD_OK;
}

int lr_expand(hd_ctx* ctx, const LowRank& lr, int op, float* out, const float* Rv, const float* Pv, int64_t n,
              int32_t Bp, const ColState* st, const int* gate, const Panels* pv) {
    HD_PROF(ctx, "lr_expand");
    if (lr.e->sparse) return lr_sparse_expand(ctx, lr, op, out, Rv, Pv, n, Bp, st, gate);
    if (lr_use_tensor_cores(lr.e)) return lr_tc_expand(ctx, lr, op, out, Rv, Pv, n, Bp, st, gate, pv);
    const hd_eig* e = lr.e;
    size_t smem = (size_t)e->r * 16 * sizeof(float);
    int gx = (int)std::min<int64_t>(ceil_div(n, 64), (int64_t)ctx->num_sms * 8);
    dim3 grid(gx, ceil_div(Bp, 16));
    static HdDeviceOnce attr;
    if (const int ra = attr.run(ctx->device, [&]() -> int {
        HD_CUDA(ctx, cudaFuncSetAttribute(k_lr_expand_simt<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024 + 1024));
        HD_CUDA(ctx, cudaFuncSetAttribute(k_lr_expand_simt<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024 + 1024));
        HD_CUDA(ctx, cudaFuncSetAttribute(k_lr_expand_simt<__nv_fp8_e4m3>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024 + 1024));
        return HD_OK;
    })) return ra;
    if (e->storage == HD_F32)
        k_lr_expand_simt<float><<<grid, 256, smem, ctx->stream>>>((const float*)e->U, e->scale, e->ldu, e->r, lr.H, op,
                                                                  out, Rv, Pv, n, Bp, st, gate);
    else if (e->storage == HD_BF16)
        k_lr_expand_simt<__nv_bfloat16><<<grid, 256, smem, ctx->stream>>>(
            (const __nv_bfloat16*)e->U, e->scale, e->ldu, e->r, lr.H, op, out, Rv, Pv, n, Bp, st, gate);
    else
        k_lr_expand_simt<__nv_fp8_e4m3><<<grid, 256, smem, ctx->stream>>>(
            (const __nv_fp8_e4m3*)e->U, e->scale, e->ldu, e->r, lr.H, op, out, Rv, Pv, n, Bp, st, gate);
    HD_CHECK_LAUNCH(ctx);
    return HD_OK;
}

// ------------------------------------------------------------------ launch helpers


static int pick_slab(int32_t Bp) {
    static int forced = -1;
    if (forced < 0) {
        const char* s = getenv("HD_SLAB");
        forced = s ? atoi(s) : 0;
    }
    int cands[] = {128, 64, 32, 16, 8, 4};
    for (int S : cands)
        if ((forced == 0 || S <= forced) && Bp % S == 0) return S;
    return 4;
}

VecLaunch vec_launch(hd_ctx* ctx, int64_t n, int32_t Bp, int S) {
    VecLaunch v;
    v.S = S > 0 ? S : pick_slab(Bp);
    int rpb = 256 / (v.S / 4);
    v.slabs = Bp / v.S;
    v.nblk = (int)std::min<int64_t>(ceil_div(n, rpb), (int64_t)ctx->num_sms * 8);
    if (v.nblk < 1) v.nblk = 1;
    return v;
}

#define HD_DISPATCH_S(S, ...)                  \
    switch (S) {                               \
        case 4: { constexpr int SS = 4; __VA_ARGS__; } break;     \
        case 8: { constexpr int SS = 8; __VA_ARGS__; } break;     \
        case 16: { constexpr int SS = 16; __VA_ARGS__; } break;   \
        case 32: { constexpr int SS = 32; __VA_ARGS__; } break;   \
        case 64: { constexpr int SS = 64; __VA_ARGS__; } break;   \
        default: { constexpr int SS = 128; __VA_ARGS__; } break;  \
    }

static bool spmm_exceeds_l2(int64_t n, int32_t Bp, int bytes) { return n * Bp * bytes > (int64_t)64 << 20; }
// One 128-byte line of every node is more than twice what L2 holds: passes that
// gather a line per entry then find almost none of them there, and a longer
// stretch of each row at a time is the better use of DRAM.
static bool spmm_lines_exceed_l2(int64_t n) { return n * 128 > (int64_t)256 << 20; }

// Lanes per row of the SpMM over `cols` columns in groups of `per` (4 fp32 or 8
// fp16 columns per lane).
// Whole 128-byte lines, one per row and pass (8 lanes), when the width allows:
// a 64-column pass over a block larger than L2 reads 1.3 times the DRAM bytes
// (1M nodes, 64 columns: 1.18 ms against 1.50 ms).  16 lanes when the block fits
// in L2 (100,000 x 64: 0.082 ms against 0.086 ms), from 256 columns on, where
// the 128-byte lines of one pass lie 1 KB apart (1M x 256: 6.1 ms against 6.7;
// panels, see panels_for, take 4.8), and from 2.1M nodes on (16 lanes against 8 at
// 64 columns, 54 entries a row: 1.5M 2.68 / 2.35 ms, 2M 3.79 / 3.80, 3M 6.04 / 6.76,
// 5M 10.6 / 12.6).
// Other widths take the whole row at once up to 16 lanes, else the fewest even
// parts of at most 16: 100,000 x 40 runs in 0.067 ms with 10 lanes, 0.12 ms in
// two passes of 9 and 0.174 ms in five of 2.
static int spmm_lanes(int64_t n, int32_t cols, int per) {
    const int nl = cols / per;
    const bool pass_fits = !spmm_exceeds_l2(n, cols, 16 / per);
    if (nl % 8 == 0) return per == 4 && nl % 16 == 0 && (pass_fits || nl >= 64 || spmm_lines_exceed_l2(n)) ? 16 : 8;
    return ceil_div(nl, ceil_div(nl, 16));
}

// Column-slab width of the SpMM over plain rows (4 x lanes per row).  HD_SLAB caps it.
int spmm_slab(const hd_graph* g, int32_t Bp) {
    return getenv("HD_SLAB") ? pick_slab(Bp) : 4 * spmm_lanes(g->n, Bp, 4);
}

// Layout of a gathered n x Bp block with `bytes` per entry: rows, or panels as wide
// as a 128-byte line (32 fp32 or 64 fp16 columns).  A row of another width straddles
// lines, and the passes of a wide one find their lines far apart; a panel row is one
// line and neighbouring rows share DRAM pages.  Whole solves in rows / in panels, ms:
//   ragged widths   1M x 40: 16.2 / 14.4   1M x 72: 38.0 / 26.2   1M x 100: 65.5 / 44.9
//                   200,000 x 72: 3.70 / 3.44   30,000 x 148: 1.38 / 1.32   30,000 x 52: 0.67 / 0.69
//   whole lines     1M x 64: 17.0 / 17.1   1M x 128: 37.9 / 34.3   1M x 256: 75.4 / 67.8
//                   400,000 x 128: 11.6 / 11.7   250,000 x 256: 14.3 / 13.9
// Ragged widths take panels from 16 MB on, whole lines from 256 MB on, where the gain
// passes 3%: below that the two sides lie within 3% of each other either way.  From
// 2.1M nodes on, blocks of whole 64-column stretches go back to rows, read 256 bytes
// at a time (products in panels / rows, ms, 54 entries a row: 2M x 128 7.33 / 7.60,
// 2M x 256 15.0 / 15.3, 3M x 128 12.7 / 12.2, 5M x 128 23.1 / 21.2, 5M x 256 45.3 /
// 42.5; ragged widths stay: 5M x 40 9.9 / 10.2, 5M x 72 16.0 / 22.3).
// The columns past the last whole panel stand alone where the block exceeds L2 (1M x
// 72: 26.2 against 29.1 when fewer than half a panel join the one before), and join
// below that, where one launch less counts more (100,000 x 72: 1.84 against 1.90).
static Panels panels_for(int64_t n, int32_t Bp, int bytes) {
    const int32_t w = 128 / bytes;
    const int64_t mb = n * Bp * bytes >> 20;
    if (Bp % w ? Bp < w || mb < 16 : Bp <= 2 * w || mb < 256) return panel_rows(n, Bp);
    if (bytes == 4 && Bp % 64 == 0 && spmm_lines_exceed_l2(n)) return panel_rows(n, Bp);
    const int32_t alone = spmm_exceeds_l2(n, Bp, bytes) ? 4 : w / 2;
    const int32_t last = ((Bp + w - alone) / w - 1) * w;
    return Panels{n, w, last, Bp - last};
}

void engine_set_panels(Engine& E, int eff_mode) {
    E.pv = E.hv = panel_rows(E.n, E.Bp);
    // (truncated systems and segments read rows, and so do the low-rank products of
    // the deflated forms and those off the tensor cores; so does a forced slab width)
    if (E.ts) return;
    if (E.segK == 1 && !getenv("HD_SLAB") && (!E.has_lr || (eff_mode == HD_MODE_PCG && lr_use_tensor_cores(E.lr.e)))) {
        E.pv = panels_for(E.n, E.Bp, 4);
        E.hv = panels_for(E.n, E.Bp, 2);
    }
    // what the products of this solve run with, for hd_graph_tuning
    std::lock_guard<std::mutex> hold(E.g->found);
    E.g->slab_cache[E.Bp] = E.segK > 1 ? E.vl.S : E.pv.last ? std::min(E.slab, E.pv.w) : E.slab;
}

// LC = L where L is a power of two that divides the width, else LC = 0
#define HD_DISPATCH_L(L, width, ...)                                                  \
    switch ((width) % (L) ? 0 : (L)) {                                                \
        case 2: { constexpr int LC = 2, G = 2; __VA_ARGS__; } break;                  \
        case 4: { constexpr int LC = 4, G = 4; __VA_ARGS__; } break;                  \
        case 8: { constexpr int LC = 8, G = 8; __VA_ARGS__; } break;                  \
        case 16: { constexpr int LC = 16, G = 8; __VA_ARGS__; } break;                \
        case 32: { constexpr int LC = 32, G = 8; __VA_ARGS__; } break;                \
        default:                                                                      \
            if (L > 8) { constexpr int LC = 0, G = 8; __VA_ARGS__; }                  \
            else if (L > 4) { constexpr int LC = 0, G = 4; __VA_ARGS__; }             \
            else if (L > 1) { constexpr int LC = 0, G = 2; __VA_ARGS__; }             \
            else { constexpr int LC = 0, G = 1; __VA_ARGS__; }                        \
    }
// blocks of 128 threads: 32 / L rows per warp, `per_sm` resident blocks per SM
static dim3 spmm_grid(hd_ctx* ctx, int64_t n, int32_t cols, int per, int L, int per_sm) {
    const int rpb = 4 * (32 / L);
    return dim3((unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, rpb), (int64_t)ctx->num_sms * per_sm)),
                (unsigned)ceil_div(cols / per, L));
}
// Q = c1 P - c2 W P in slabs of S columns, or panel by panel
static int spmm_launch(hd_ctx* ctx, const hd_graph* g, const float* P, const Panels& pv, float* Q, int32_t ld, int S,
                       float c1, float c2, const ColState* st, const int* skip) {
    // panel by panel; apart, a last one of another width
    if (pv.last) S = std::min(S, pv.w);
    const int32_t cut = S == pv.w && pv.wlast != pv.w ? pv.last : 0;
    for (int32_t first = 0; first < ld; first = first < cut ? cut : ld) {
        const int32_t last = first < cut ? cut : ld;
        const int L = cut && last == ld ? (ld - cut) / 4 : S / 4;
        if (L == 1) {
            const VecLaunch v = vec_launch(ctx, g->n, last - first, 4);
            k_spmm4<<<dim3(v.nblk, v.slabs), 256, 0, ctx->stream>>>(g->row_ptr, g->col, g->val, P, pv, Q, g->n, ld,
                                                                    first, c1, c2, st, skip);
        } else {
            const dim3 grid = spmm_grid(ctx, g->n, last - first, 4, L, spmm_blocks(L));
            HD_DISPATCH_L(L, (last - first) / 4,
                          (k_spmm<LC, G><<<grid, 128, 0, ctx->stream>>>(g->row_ptr, g->col, g->val, P, pv, Q,
                                                                        (unsigned)g->n, ld, first, last, L, c1, c2, st,
                                                                        skip)));
        }
        HD_CHECK_LAUNCH(ctx);
    }
    return HD_OK;
}

int hd_spmm_apply(hd_ctx* ctx, const hd_graph* g, const float* P, float* Q, int32_t ld, int32_t B, float c1,
                  float c2) {
    return spmm_launch(ctx, g, P, panel_rows(g->n, ld), Q, ld, 4 * spmm_lanes(g->n, ld, 4), c1, c2, nullptr, nullptr);
}

// grid and block of the column reductions: one chunk per block row.  `staged`
// (k_red_staged) while the thread-per-(g, quad) form has too few threads to stream:
// below 192 per SM for the dot product, 168 for the update (which stores as it
// goes), 320 for the squares.  Thread form / staged, us:
//   dot      100,000 x 64 (165 per SM) 24.2 / 19.8   200,000 x 36 (185) 24.9 / 25.6
//            100,000 x 100 (258) 27.3 / 36.9         300,000 x 128 (987) 57.6 / 108
//   update   100,000 x 64 30.7 / 31.1   200,000 x 36 34 / 47   1M x 36 (926) 131 / 290
//   squares  100,000 x 128 (330) 19.3 / 18.9         200,000 x 128 (659) 27.3 / 35.9
// At one or two quads the thread form has 8 or 16 threads per block and short runs of
// a row: update and squares stay staged at any size (2M x 8 67.6 / 59.6 and 22.4 / 22.4,
// 5M x 4 135 / 96 and 44 / 37).
struct RedLaunch {
    dim3 grid;
    unsigned block;
    size_t smem;
    bool staged;
};
static RedLaunch red_launch(const Engine& E, RedOp op) {
    const int nq = E.Bp / 4, qpb = nq < RQ ? nq : RQ;
    const int per_sm = op == RED_DOT ? 192 : op == RED_UPDATE ? 168 : 320;
    RedLaunch l;
    l.staged = E.nch * nq * RG < (int64_t)E.ctx->num_sms * per_sm || (op != RED_DOT && nq <= 2);
    l.grid = dim3((unsigned)E.nch, (unsigned)ceil_div(E.Bp, l.staged ? RS_COLS : 4 * RQ));
    l.block = l.staged ? 256u : (unsigned)(RG * qpb);
    l.smem = (size_t)l.block * 4 * sizeof(float2);
    return l;
}
template <int OP>
static int launch_staged(Engine& E, const RedLaunch& l, const float* P, const Panels& pv, float2* part,
                         const ColState* st, const IterReset& z = {}) {
    hd_ctx* ctx = E.ctx;
    static HdDeviceOnce attr;
    if (const int ra = attr.run(ctx->device, [&]() -> int {
        HD_CUDA(ctx, cudaFuncSetAttribute(k_red_staged<OP>, cudaFuncAttributeMaxDynamicSharedMemorySize, rs_smem<OP>()));
        return HD_OK;
    })) return ra;
    k_red_staged<OP><<<l.grid, l.block, rs_smem<OP>(), ctx->stream>>>(E.X, E.R, P, pv, E.Q, E.n, E.Bp, E.rch, st, E.xs,
                                                                        part, z);
    HD_CHECK_LAUNCH(ctx);
    return HD_OK;
}

static int launch_dot(Engine& E, float2* part, const ColState* st) {
    hd_ctx* ctx = E.ctx;
    HD_PROF(ctx, "dot");
    const RedLaunch l = red_launch(E, RED_DOT);
    if (l.staged) return launch_staged<RED_DOT>(E, l, E.P, E.pv, part, st);
    k_dot<<<l.grid, l.block, l.smem, ctx->stream>>>(E.P, E.pv, E.Q, E.n, E.Bp, E.rch, part, st);
    HD_CHECK_LAUNCH(ctx);
    return HD_OK;
}

static int launch_update(Engine& E) {
    hd_ctx* ctx = E.ctx;
    HD_PROF(ctx, "update");
    const RedLaunch l = red_launch(E, RED_UPDATE);
    IterReset z;
    z.p16_max = E.use_half ? E.p16_max : nullptr;
    z.Bp = E.Bp;
    if (E.eff_mode != HD_MODE_PCG) {  // (PCG: the reduction that follows is gated by num_active)
        z.num_active = E.num_active;
        z.use_half = E.use_half;
    }
    if (l.staged) return launch_staged<RED_UPDATE>(E, l, E.P, E.pv, E.part, E.st, z);
    k_update<<<l.grid, l.block, l.smem, ctx->stream>>>(E.X, E.R, E.P, E.pv, E.Q, E.n, E.Bp, E.rch, E.st, E.xs, E.part,
                                                      z);
    HD_CHECK_LAUNCH(ctx);
    return HD_OK;
}

static int launch_colsq(Engine& E, const float* V) {
    hd_ctx* ctx = E.ctx;
    HD_PROF(ctx, "colsq");
    const RedLaunch l = red_launch(E, RED_SQ);
    if (l.staged) return launch_staged<RED_SQ>(E, l, V, panel_rows(E.n, E.Bp), E.part, nullptr);
    k_colsq<<<l.grid, l.block, l.smem, ctx->stream>>>(V, E.n, E.Bp, E.rch, E.part);
    HD_CHECK_LAUNCH(ctx);
    return HD_OK;
}

void engine_set_reduction(Engine& E) {
    E.rch = reduction_chunk_rows(E.n);
    E.nch = (E.n + E.rch - 1) / E.rch;
}

// Q = c1 V - c2 W V (V = P unless given) with the engine's slab width and
// segments (+ P^T Q partials)
static int launch_spmm(Engine& E, float c1, float c2, float2* part, const ColState* st, const float* V = nullptr) {
    hd_ctx* ctx = E.ctx;
    const hd_graph* g = E.g;
    const float* Pin = V ? V : E.P;
    int rc;
    if (!V && E.use_half) {
        // the iteration's SpMM: an fp16 copy of P is gathered when *use_half
        const int nq = E.Bp / 4;
        const int rpb = 256 / nq;
        const dim3 gc((unsigned)std::min<int64_t>(ceil_div(E.n, rpb), (int64_t)ctx->num_sms * 8));
        {
            HD_PROF(ctx, "to_half");
            k_colmax<<<gc, 256, 0, ctx->stream>>>(E.P, E.pv, E.n, E.Bp, E.p16_max, E.use_half, E.num_active);
            HD_CHECK_LAUNCH(ctx);
            k_to_half<<<gc, 256, 0, ctx->stream>>>(E.P, E.pv, E.n, E.Bp, E.p16_max, E.P16, E.hv, E.use_half,
                                                 E.num_active);
            HD_CHECK_LAUNCH(ctx);
        }
        {
            HD_PROF(ctx, "spmm");
            if ((rc = spmm_launch(ctx, g, E.P, E.pv, E.Q, E.Bp, E.slab, c1, c2, st, E.use_half))) return rc;
        }
        {
            HD_PROF(ctx, "spmm_h");
            const int32_t cut = E.hv.wlast != E.hv.w ? E.hv.last : 0;
            for (int32_t first = 0; first < E.Bp; first = first < cut ? cut : E.Bp) {
                const int32_t last = first < cut ? cut : E.Bp;
                const int L16 = cut && last == E.Bp ? (last - first) / 8
                                : E.hv.last         ? E.hv.w / 8
                                                    : spmm_lanes(E.n, E.Bp, 8);
                const dim3 gh = spmm_grid(ctx, E.n, last - first, 8, L16, 7);
                HD_DISPATCH_L(L16, (last - first) / 8, (k_spmm_h<LC, G><<<gh, 128, 0, ctx->stream>>>(
                                       g->row_ptr, g->col, g->val, E.P16, E.hv, E.p16_max, E.P, E.pv, E.Q,
                                       (unsigned)E.n, E.Bp, first, last, L16, c1, c2, st, E.use_half)));
                HD_CHECK_LAUNCH(ctx);
            }
        }
        if (part) return launch_dot(E, part, st);
        return HD_OK;
    }
    {
        HD_PROF(ctx, "spmm");
        if (E.segK <= 1 && E.Bp == 4 && E.narrow4) {
            const dim3 g4((unsigned)std::max(1, ceil_div(E.n, N4_ROWS)));
            k_spmm_n4<<<g4, 256, 0, ctx->stream>>>(g->row_ptr, g->col, g->val, Pin, E.Q, E.n, c1, c2, st, nullptr);
            HD_CHECK_LAUNCH(ctx);
        } else if (E.segK <= 1) {
            if ((rc = spmm_launch(ctx, g, Pin, V ? panel_rows(E.n, E.Bp) : E.pv, E.Q, E.Bp, E.slab, c1, c2, st, nullptr))) return rc;
        } else {
            const dim3 grid(E.vl.nblk, E.vl.slabs);
            for (int s = 0; s < E.segK; ++s) {
                const int32_t* lo = E.seg + (int64_t)s * E.n;
                HD_DISPATCH_S(E.vl.S, (k_spmm_seg<SS><<<grid, 256, 0, ctx->stream>>>(
                                          lo, lo + E.n, g->col, g->val, Pin, E.Q, E.n, E.Bp, c1, c2, st, s == 0)));
                HD_CHECK_LAUNCH(ctx);
            }
        }
    }
    if (part) return launch_dot(E, part, st);
    return HD_OK;
}

static const int32_t* seg_bounds_for(hd_ctx* ctx, const hd_graph* g, int K) {
    std::lock_guard<std::mutex> hold(g->found);
    auto it = g->seg_bounds.find(K);
    if (it != g->seg_bounds.end()) return it->second;
    int32_t* b = nullptr;
    if (cudaMalloc(&b, (size_t)(K + 1) * g->n * 4) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    const int64_t w = (g->n + K - 1) / K;
    k_seg_bounds<<<ceil_div(g->n, 256), 256, 0, ctx->stream>>>(g->row_ptr, g->col, g->n, K, w, b);
    ctx->launches++;
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
        cudaFree(b);
        return nullptr;
    }
    g->seg_bounds[K] = b;  // (complete: other contexts' streams may read them)
    return b;
}

// Two segments where a row is a quarter or half of a 128-byte line and half of the
// block still finds room in L2: a product in one pass / in two, ms (54 entries a row)
//   16 columns   2M 1.13 / 1.10   3M 2.29 / 1.91   5M 4.68 / 3.92
//    8 columns   3M 1.35 / 1.45   5M 3.61 / 2.80
// and whole solves, whose late iterations then gather fp32 too, 2M x 16 11.5 / 12.0,
// 3M x 16 21.5 / 20.4, 5M x 16 43.9 / 40.7, 5M x 8 30.8 / 28.6.  Narrower rows (5M x 4
// 1.80 / 2.26) and wider ones (5M x 32 5.9 / 6.3) lose.
int spmm_segments(hd_ctx* ctx, Engine& E) {
    const hd_graph* g = E.g;
    E.segK = 1;
    E.seg = nullptr;
    static int forced = -2;
    if (forced == -2) {
        const char* s = getenv("HD_SEGMENTS");
        forced = s ? atoi(s) : -1;
    }
    int K = std::max(forced, 1);
    if (forced < 1 && (E.Bp == 8 || E.Bp == 16) && E.n * E.Bp * 4 > (int64_t)140 << 20 && !getenv("HD_SLAB")) K = 2;
    if (K > 1) {
        const int32_t* b = seg_bounds_for(ctx, g, K);
        if (!b && forced > 1) return hd_fail(ctx, HD_ERR_OOM, "SpMM segment bounds");
        if (!b) K = 1;
        E.seg = b;
    }
    E.segK = K;
    std::lock_guard<std::mutex> hold(g->found);
    g->seg_cache[E.Bp] = K;  // reported by hd_graph_tuning
    return HD_OK;
}

// ------------------------------------------------------------------ the solve


#define LAUNCH_VEC(kernel, ...)                                                                 \
    do {                                                                                        \
        HD_PROF(S_.ctx, #kernel[2] == 's' && #kernel[3] == 'p' ? "spmm"                         \
                        : #kernel[2] == 'u' ? "update" : #kernel[2] == 'd' ? "direction" : "colsq"); \
        dim3 grid_(S_.vl.nblk, S_.vl.slabs);                                                    \
        HD_DISPATCH_S(S_.vl.S, (kernel<SS><<<grid_, 256, 0, S_.ctx->stream>>>(__VA_ARGS__)));   \
        HD_CHECK_LAUNCH(S_.ctx);                                                                \
    } while (0)


// The scalar step after the update (rr, convergence, beta; C / coef: the PCG
// term): k_fin_rr, or for a server lane k_fin_rr_serve, which also installs
// staged requests, followed by their U^T y into H for the direction.
static int launch_fin_rr(Engine& S_, const double* C, const double* coef, int r) {
    hd_ctx* ctx = S_.ctx;
    const int32_t Bp = S_.Bp;
    HD_PROF(ctx, "scalar");
    if (S_.refill) {
        k_fin_rr_serve<<<Bp, 128, 0, ctx->stream>>>(S_.part, (int)S_.nch, Bp, S_.st, S_.max_iter, C, coef, r,
                                                   S_.num_active, *S_.refill);
        HD_CHECK_LAUNCH(ctx);
        if (S_.has_lr && S_.eff_mode == HD_MODE_PCG) {
            const int64_t tot = (int64_t)S_.lr.rpad * Bp;
            k_refill_h<<<ceil_div(tot, 256), 256, 0, ctx->stream>>>(*S_.refill, S_.dcoef, S_.lr.rpad, Bp, S_.lr.H,
                                                                     S_.lr.Hhi, S_.lr.Hlo);
            HD_CHECK_LAUNCH(ctx);
        }
        return HD_OK;
    }
    k_fin_rr<<<Bp, 128, 0, ctx->stream>>>(S_.part, (int)S_.nch, Bp, S_.st, S_.max_iter, C, coef, r, S_.num_active,
                                         S_.use_half, HALF_THETA * HALF_THETA);
    HD_CHECK_LAUNCH(ctx);
    return HD_OK;
}

// Truncated systems: Q = c1 V - c2 W_j V of the columns being iterated, or with
// `resid` Q = -(c1 V - c2 W_j V) of every column in two words.
static int launch_trunc(Engine& E, const float* V, float c1, float c2, bool resid) {
    hd_ctx* ctx = E.ctx;
    const TruncSys& ts = *E.ts;
    HD_PROF(ctx, resid ? "resid" : "spmm");
    k_transpose<<<dim3((unsigned)ceil_div(E.n, 32), (unsigned)ceil_div(E.Bp, 32)), 256, 0, ctx->stream>>>(V, E.n, E.Bp,
                                                                                                        E.VT);
    HD_CHECK_LAUNCH(ctx);
    // a block per 1,024 rows, but no column waits for another while there are SMs: a
    // short column is a chain of loads (16 lists of 100 on 2,000 nodes: 1.85 ms for a
    // call with one block, 1.36 with 16)
    const unsigned grid = (unsigned)std::min<int64_t>(ctx->num_sms, std::max<int64_t>(std::max(1, ts.ncol), E.n * E.Bp / TC_T));
    constexpr int tiles = 2 * TC_TILE * (int)sizeof(float2);
    const int smem = tiles + (ts.ncol + 1) * (int)sizeof(TruncWork);
    static HdDeviceOnce attr;
    if (const int ra = attr.run(ctx->device, [&]() -> int {
        constexpr int most = tiles + (TC_COLS + 1) * (int)sizeof(TruncWork);
        HD_CUDA(ctx, cudaFuncSetAttribute(k_spmm_cols, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        HD_CUDA(ctx, cudaFuncSetAttribute(k_resid_cols, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        return HD_OK;
    })) return ra;
    if (resid)
        k_resid_cols<<<grid, TC_T, smem, ctx->stream>>>(ts, E.VT, E.Q, E.n, E.Bp, c1, c2);
    else
        k_spmm_cols<<<grid, TC_T, smem, ctx->stream>>>(ts, E.VT, E.Q, E.n, E.Bp, c1, c2, E.st);
    HD_CHECK_LAUNCH(ctx);
    return HD_OK;
}

// One CG iteration of every column (Eq. 20 operator, CG update, direction).
// `after_update`, if given, runs right after the X/R update (the serving loop
// scatters newly admitted observations there).
int engine_iteration(Engine& S_, int (*after_update)(void*), void* arg) {
    hd_ctx* ctx = S_.ctx;
    const int64_t n = S_.n;
    const int32_t Bp = S_.Bp;
    const int r = S_.r;
    const bool lr_on = S_.has_lr;
    const int eff_mode = S_.eff_mode;
    const float c1 = S_.c1, c2 = S_.c2;
    const int32_t max_iter = S_.max_iter;
    const double* Cd = lr_on ? S_.lr.C : nullptr;
    int rc;
    if (eff_mode == HD_MODE_PCG) {
        if ((rc = launch_spmm(S_, c1, c2, S_.part, S_.st))) return rc;
        { HD_PROF(ctx, "scalar");
        k_fin_sigma<<<Bp, 128, 0, ctx->stream>>>(S_.part, (int)S_.nch, Bp, S_.st, nullptr, nullptr, 0); }
        HD_CHECK_LAUNCH(ctx);
        if ((rc = launch_update(S_))) return rc;
    if (after_update && (rc = after_update(arg))) return rc;
        if ((rc = lr_reduce(ctx, S_.lr, S_.R, n, Bp, S_.num_active))) return rc;
        IterReset z;
        z.num_active = S_.num_active;
        z.use_half = S_.use_half;
        if ((rc = lr_finish(ctx, S_.lr, Bp, S_.dcoef, z))) return rc;
        if ((rc = launch_fin_rr(S_, Cd, S_.dcoef, r))) return rc;
        if ((rc = lr_expand(ctx, S_.lr, EXP_DIRECTION, S_.P, S_.R, S_.P, n, Bp, S_.st, S_.num_active,
                            &S_.pv)))
            return rc;
        if (S_.refill) {
            k_refill_p<<<ceil_div(Bp, 128), 128, 0, ctx->stream>>>(*S_.refill, S_.P, S_.pv, Bp);
            HD_CHECK_LAUNCH(ctx);
        }
    } else {
        if (S_.ts) {
            if ((rc = launch_trunc(S_, S_.P, c1, c2, false))) return rc;
            if ((rc = launch_dot(S_, S_.part, S_.st))) return rc;
        } else if ((rc = launch_spmm(S_, c1, c2, S_.part, S_.st)))
            return rc;
        if (lr_on) {
            if ((rc = lr_expand(ctx, S_.lr, EXP_ADD_Q, S_.Q, nullptr, nullptr, n, Bp, S_.st, S_.num_active)))
                return rc;
        }
        { HD_PROF(ctx, "scalar");
        k_fin_sigma<<<Bp, 128, 0, ctx->stream>>>(S_.part, (int)S_.nch, Bp, S_.st, Cd,
                                                lr_on ? S_.opcoef : nullptr, r); }
        HD_CHECK_LAUNCH(ctx);
        if ((rc = launch_update(S_))) return rc;
    if (after_update && (rc = after_update(arg))) return rc;
        if ((rc = launch_fin_rr(S_, nullptr, nullptr, 0))) return rc;
        LAUNCH_VEC(k_direction, S_.P, S_.pv, S_.R, n, Bp, S_.st);
        if (S_.refill) {
            k_refill_p<<<ceil_div(Bp, 128), 128, 0, ctx->stream>>>(*S_.refill, S_.P, S_.pv, Bp);
            HD_CHECK_LAUNCH(ctx);
        }
        if (lr_on) {
            if ((rc = lr_reduce(ctx, S_.lr, S_.P, n, Bp, S_.num_active))) return rc;
            if ((rc = lr_finish(ctx, S_.lr, Bp, S_.opcoef))) return rc;
        }
    }
    return HD_OK;
}

// Run `iters` CG iterations as one CUDA graph launch.  The graph is captured
// on a private stream (the context's stream may be the legacy default stream,
// which cannot be captured) and re-captured whenever anything the kernels take
// as an argument differs from every cached capture.
static uint64_t fbits(float f) {
    uint32_t u;
    memcpy(&u, &f, sizeof u);
    return u;
}

// Everything the iteration kernels take as arguments (the run length is added
// by the caller); the graph's and the eigenpairs' ids stand for all their arrays.
static std::vector<uint64_t> iteration_key(const Engine& E) {
    return {E.g->id, E.has_lr ? E.lr.e->id : 0, (uint64_t)E.ts, (uint64_t)(E.ts ? E.ts->off : nullptr),
            (uint64_t)(E.ts ? E.ts->ci : nullptr), (uint64_t)(E.ts ? E.ts->wv : nullptr),
            (uint64_t)(E.ts ? E.ts->work : nullptr), (uint64_t)(E.ts ? E.ts->ncol : 0), (uint64_t)E.n,
            (uint64_t)E.R, (uint64_t)E.P, (uint64_t)E.Q, (uint64_t)E.X, (uint64_t)E.VT, (uint64_t)E.part, (uint64_t)E.st,
            (uint64_t)E.num_active, (uint64_t)E.lr.part, (uint64_t)E.lr.C, (uint64_t)E.lr.H, (uint64_t)E.lr.Hhi,
            (uint64_t)E.lr.Hlo, (uint64_t)E.dcoef, (uint64_t)E.opcoef, (uint64_t)E.segK, (uint64_t)E.seg,
            (uint64_t)E.nch, (uint64_t)E.Bp, (uint64_t)E.slab, (uint64_t)E.vl.S, (uint64_t)E.vl.nblk, (uint64_t)E.vl.slabs,
            (uint64_t)E.lr.nchunk, (uint64_t)E.lr.rpad, (uint64_t)E.lr.Bp16, (uint64_t)E.has_lr,
            (uint64_t)E.eff_mode, (uint64_t)E.r, (uint64_t)E.max_iter, fbits(E.c1), fbits(E.c2), fbits(E.xs), (uint64_t)E.pv.last, (uint64_t)E.hv.last,
            (uint64_t)E.P16, (uint64_t)E.p16_max, (uint64_t)E.use_half, (uint64_t)E.ctx->stream};
}

static int run_iterations_graph(Engine& E, int iters) {
    hd_ctx* ctx = E.ctx;
    std::vector<uint64_t> key = iteration_key(E);
    key.push_back((uint64_t)iters);
    auto it = ctx->iter_graphs.find(key);
    if (it == ctx->iter_graphs.end()) {
        if (ctx->iter_graphs.size() >= 8) {
            for (auto& kv : ctx->iter_graphs) cudaGraphExecDestroy(kv.second.exec);
            ctx->iter_graphs.clear();
        }
        if (!ctx->cap_stream) HD_CUDA(ctx, cudaStreamCreateWithFlags(&ctx->cap_stream, cudaStreamNonBlocking));
        cudaStream_t user = ctx->stream;
        // the capture stream starts after everything already queued on the user stream
        HD_CUDA(ctx, cudaStreamSynchronize(user));
        ctx->stream = ctx->cap_stream;
        const int64_t l0 = ctx->launches;
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamBeginCapture(ctx->cap_stream, cudaStreamCaptureModeRelaxed);
        int rc = HD_OK;
        if (e == cudaSuccess) {
            for (int t = 0; t < iters && rc == HD_OK; ++t) rc = engine_iteration(E, nullptr, nullptr);
            cudaError_t e2 = cudaStreamEndCapture(ctx->cap_stream, &graph);
            if (rc == HD_OK && e2 != cudaSuccess) e = e2;
        }
        ctx->stream = user;
        if (rc) return rc;
        if (e != cudaSuccess) {
            cudaGetLastError();
            return hd_fail(ctx, HD_ERR_CUDA, "iteration graph capture: %s", cudaGetErrorString(e));
        }
        hd_ctx::IterGraph ig;
        e = cudaGraphInstantiate(&ig.exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) return hd_fail(ctx, HD_ERR_CUDA, "iteration graph instantiate: %s", cudaGetErrorString(e));
        ig.launches = ctx->launches - l0;
        ctx->launches = l0;
        it = ctx->iter_graphs.emplace(key, ig).first;
    }
    HD_CUDA(ctx, cudaGraphLaunch(it->second.exec, ctx->stream));
    ctx->launches += it->second.launches;
    return HD_OK;
}

// HD_NO_HALF=1: every SpMM of the iterations gathers fp32
static bool half_gathers_off() {
    static int off = -1;
    if (off < 0) {
        const char* s = getenv("HD_NO_HALF");
        off = (s && atoi(s)) ? 1 : 0;
    }
    return off != 0;
}

static bool graphs_enabled(hd_ctx* ctx) {
    static int off = -1;
    if (off < 0) {
        const char* s = getenv("HD_NO_GRAPH");
        off = (s && atoi(s)) ? 1 : 0;
    }
    return !off && !ctx->prof;
}

extern "C" int hd_query_batch(hd_ctx* ctx, const hd_graph* g, const hd_eig* eig, int mode, int32_t B,
                              const int32_t* y_ptr, const int32_t* y_idx, const float* y_val, double alpha,
                              const float* tol, int32_t max_iter, float* X, int32_t ldx, int32_t* iters,
                              float* relres, int32_t* status) {
    return hd_query_impl(ctx, g, nullptr, eig, mode, B, y_ptr, y_idx, y_val, alpha, tol, max_iter, X, ldx, iters,
                         relres, status);
}

static const char* const BAD_OBSERVATION = "bad observation: index out of range, non-finite value or bad y_ptr";

// Iterate until no column is active: runs of iterations (CUDA graphs when
// enabled), each followed by a poll of the active count and of the
// tensor-core kernels' wait flags.  The first run is as long as the previous
// solve with the same key took (at most 8), later runs 2, 4, 8, then 16
// iterations, so a repeated workload polls once and launches no idle
// iterations.  `ran` accumulates the iterations launched.
static int iterate_until_stopped(Engine& E, int& ran) {
    hd_ctx* ctx = E.ctx;
    const std::vector<uint64_t> hkey = iteration_key(E);
    const int first = (ctx->hint_key == hkey && ctx->iter_hint > 0) ? std::min(ctx->iter_hint, 8) : 4;
    int run = 0, next = 2;
    int active = 1;
    int rc;
    // every active column stops within max_iter iterations of its own; the
    // bound only guards the host loop
    const int64_t cap = (int64_t)(MAX_CONFIRM + 1) * E.max_iter + 8;
    while (active > 0 && ran < cap) {
        int todo = first;
        if (run > 0) {
            todo = next;
            next = std::min(2 * next, 16);
        }
        if (graphs_enabled(ctx)) {
            if ((rc = run_iterations_graph(E, todo))) return rc;
        } else {
            for (int t = 0; t < todo; ++t)
                if ((rc = engine_iteration(E, nullptr, nullptr))) return rc;
        }
        ran += todo;
        ++run;
        HD_CUDA(ctx, cudaMemcpyAsync(ctx->h_poll, E.num_active, 2 * sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
        HD_CUDA(ctx, cudaMemcpyAsync(ctx->h_poll + 8, ctx->d_flags + 2, 2 * sizeof(int), cudaMemcpyDeviceToHost,
                                     ctx->stream));
        HD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        active = ctx->h_poll[0];
        if (ctx->h_poll[1]) return hd_fail(ctx, HD_ERR_INVALID_ARG, "%s", BAD_OBSERVATION);
        if (ctx->h_poll[8] || ctx->h_poll[9]) return lr_tc_check_flags(ctx);
    }
    return HD_OK;
}

// T = b - A x into Q for every column (A the operator the solve iterates on,
// applied to X; b = y, or y - U C_y for the projected form) and the partials
// of ||T||^2 in E.part.  X holds the temporal term alone at this point.
static int true_residual(Engine& E, double alpha) {
    hd_ctx* ctx = E.ctx;
    const int64_t n = E.n;
    const int32_t Bp = E.Bp;
    const double c1d = 1.0 / (1.0 - alpha), c2d = alpha / (1.0 - alpha);
    const float c1 = (float)c1d, c2 = (float)c2d;
    int rc;
    if (E.ts) {
        // Q = -L_a(W_j) x column by column (truncated systems), in two words
        if ((rc = launch_trunc(E, E.X, c1, c2, true))) return rc;
    } else {
        // Q = -L_a(W) x: the fp32 SpMM when its rounding bound is small against
        // every column's tolerance, else the two-word kernel (k_resid_pick)
        const hd_graph* g = E.g;
        const double u = 1.0 / 16777216.0;
        const double m = (double)g->max_row + 1.0;
        const double gamma = m * u / (1.0 - m * u);
        int* pick = E.num_active + 2;
        if ((rc = launch_colsq(E, E.X))) return rc;
        {
            HD_PROF(ctx, "scalar");
            HD_CUDA(ctx, cudaMemsetAsync(pick, 0, sizeof(int), ctx->stream));
            k_resid_pick<<<Bp, 128, 0, ctx->stream>>>(E.part, (int)E.nch, Bp, E.B, E.st, gamma, c1d, c2d, pick);
        }
        HD_CHECK_LAUNCH(ctx);
        HD_PROF(ctx, "resid");
        if (Bp == 4 && E.narrow4) {
            k_spmm_n4<<<std::max(1, ceil_div(n, N4_ROWS)), 256, 0, ctx->stream>>>(g->row_ptr, g->col, g->val, E.X, E.Q,
                                                                                  n, -c1, -c2, nullptr, pick);
            HD_CHECK_LAUNCH(ctx);
        } else if ((rc = spmm_launch(ctx, g, E.X, panel_rows(n, Bp), E.Q, Bp, E.slab, -c1, -c2, nullptr, pick))) {
            return rc;
        }
        const int L = std::max(1, E.slab / 4);
        const dim3 gr = spmm_grid(ctx, n, Bp, 4, L, 6);
        HD_DISPATCH_L(L, Bp / 4, (k_resid<LC, G><<<gr, 128, 0, ctx->stream>>>(g->row_ptr, g->col, g->val, E.X, E.Q, (unsigned)n,
                                                                       Bp, L, c1, c2, pick)));
        HD_CHECK_LAUNCH(ctx);
    }
    if (E.has_lr && E.eff_mode != HD_MODE_PCG) {
        // deflated operator: Q -= (a / (1 - a)) U (Lambda (U^T x))
        if ((rc = lr_reduce(ctx, E.lr, E.X, n, Bp))) return rc;
        if ((rc = lr_finish(ctx, E.lr, Bp, E.negop))) return rc;
        if ((rc = lr_expand(ctx, E.lr, EXP_ADD_Q, E.Q, nullptr, nullptr, n, Bp, nullptr))) return rc;
        if (E.eff_mode == HD_MODE_PROJ) {
            // b = y - U (U^T y)
            if ((rc = lr_coef(ctx, E.lr, Bp, E.ones, E.Cy))) return rc;
            if ((rc = lr_expand(ctx, E.lr, EXP_SUB_R, E.Q, nullptr, nullptr, n, Bp, nullptr))) return rc;
        }
    }
    k_scatter_y<<<E.B, 128, 0, ctx->stream>>>(E.yp, E.yi, E.yv, E.nnz_y, n, Bp, E.Q, E.err);
    HD_CHECK_LAUNCH(ctx);
    return launch_colsq(E, E.Q);
}

// Restart the columns k_fin_confirm reactivated: r := T (in Q), a fresh
// direction from it (p = M^-1 r with the preconditioner, p = r otherwise), and
// for the deflated forms C = U^T p for the next operator application.
static int restart_columns(Engine& E) {
    hd_ctx* ctx = E.ctx;
    const int64_t n = E.n;
    const int32_t Bp = E.Bp;
    int rc;
    k_restart_copy<<<ceil_div(n * (Bp / 4), 256), 256, 0, ctx->stream>>>(E.R, E.Q, n, Bp, E.st);
    HD_CHECK_LAUNCH(ctx);
    if (E.use_half) HD_CUDA(ctx, cudaMemsetAsync(E.use_half, 0, sizeof(int), ctx->stream));
    if (E.eff_mode == HD_MODE_PCG) {
        if ((rc = lr_reduce(ctx, E.lr, E.R, n, Bp))) return rc;
        if ((rc = lr_finish(ctx, E.lr, Bp, E.dcoef))) return rc;
        {
            HD_PROF(ctx, "scalar");
            k_fin_restart<<<Bp, 128, 0, ctx->stream>>>(E.st, E.lr.C, E.dcoef, E.r);
        }
        HD_CHECK_LAUNCH(ctx);
        return lr_expand(ctx, E.lr, EXP_DIRECTION, E.P, E.R, E.P, n, Bp, E.st, nullptr, &E.pv);
    }
    {
        HD_PROF(ctx, "scalar");
        k_fin_restart<<<Bp, 128, 0, ctx->stream>>>(E.st, nullptr, nullptr, 0);
    }
    HD_CHECK_LAUNCH(ctx);
    {
        HD_PROF(ctx, "direction");
        dim3 grid(E.vl.nblk, E.vl.slabs);
        HD_DISPATCH_S(E.vl.S, (k_direction<SS><<<grid, 256, 0, ctx->stream>>>(E.P, E.pv, E.R, n, Bp, E.st)));
        HD_CHECK_LAUNCH(ctx);
    }
    if (E.has_lr) {
        if ((rc = lr_reduce(ctx, E.lr, E.P, n, Bp))) return rc;
        if ((rc = lr_finish(ctx, E.lr, Bp, E.opcoef))) return rc;
    }
    return HD_OK;
}

// The solve behind hd_query_batch; with `ts` the operator is the per-column
// truncated system (rows = shortlist positions) instead of the graph.
int hd_query_impl(hd_ctx* ctx, const hd_graph* g, const TruncSys* ts, const hd_eig* eig, int mode, int32_t B,
                  const int32_t* y_ptr, const int32_t* y_idx, const float* y_val, double alpha, const float* tol,
                  int32_t max_iter, float* X, int32_t ldx, int32_t* iters, float* relres, int32_t* status) {
    if (!ctx || !g || !y_ptr || !tol || !X) return HD_ERR_INVALID_ARG;
    if (ts && eig) return hd_fail(ctx, HD_ERR_INVALID_ARG, "truncated systems take no eigenpairs");
    if (B <= 0 || ldx < B) return hd_fail(ctx, HD_ERR_INVALID_ARG, "B=%d ldx=%d", B, ldx);
    if (!(alpha >= 0.0 && alpha < 1.0)) return hd_fail(ctx, HD_ERR_INVALID_ARG, "alpha=%g not in [0,1)", alpha);
    const bool temporal_only = (mode & HD_MODE_TEMPORAL_ONLY) != 0;
    mode &= ~HD_MODE_TEMPORAL_ONLY;
    if (mode != HD_MODE_PAPER && mode != HD_MODE_PROJ && mode != HD_MODE_PCG)
        return hd_fail(ctx, HD_ERR_INVALID_ARG, "mode %d", mode);
    if (temporal_only && mode == HD_MODE_PCG)
        return hd_fail(ctx, HD_ERR_INVALID_ARG, "HD_MODE_TEMPORAL_ONLY needs the paper's or the projected form");
    if (max_iter < 0) return hd_fail(ctx, HD_ERR_INVALID_ARG, "max_iter %d", max_iter);
    if (eig && eig->n != g->n) return hd_fail(ctx, HD_ERR_INVALID_ARG, "eigenpairs for n=%lld, graph n=%lld",
                                              (long long)eig->n, (long long)g->n);
    HD_CUDA(ctx, cudaSetDevice(ctx->device));
    Engine S_;
    S_.ctx = ctx;
    S_.g = g;
    S_.ts = ts;
    S_.n = ts ? ts->smax : g->n;
    engine_set_reduction(S_);
    S_.B = B;
    S_.Bp = (B + 3) / 4 * 4;
    S_.vl = vec_launch(ctx, S_.n, S_.Bp, pick_slab(S_.Bp));
    const int64_t n = S_.n;
    const int32_t Bp = S_.Bp;
    const bool lr_on = eig && eig->r > 0;
    S_.has_lr = lr_on;
    S_.lr = LowRank{};
    const int r = lr_on ? eig->r : 0;
    const int rpad = lr_on ? (r + 63) / 64 * 64 : 0;
    const int Bp16 = (Bp + 15) / 16 * 16;

    // host-side copy of y_ptr to learn nnz
    int32_t nnz_y;
    {
        int32_t last;
        if (hd_is_device_ptr(y_ptr)) {
            HD_CUDA(ctx, cudaMemcpy(&last, y_ptr + B, 4, cudaMemcpyDeviceToHost));
        } else {
            last = y_ptr[B];
        }
        nnz_y = last;
        if (nnz_y < 0) return hd_fail(ctx, HD_ERR_INVALID_ARG, "y_ptr[B] = %d", nnz_y);
        if (nnz_y > 0 && (!y_idx || !y_val)) return HD_ERR_INVALID_ARG;
    }
    const bool x_direct = hd_is_device_ptr(X) && ldx == Bp;
    int nchunk = 0;
    if (lr_on) nchunk = lr_nchunk(ctx, eig, Bp);

    size_t vec = (size_t)n * Bp * sizeof(float);
    size_t bytes = 3 * ws_size(vec) + (x_direct ? 0 : ws_size(vec)) + ws_size((size_t)S_.nch * Bp * sizeof(float2)) +
                   ws_size(Bp * sizeof(ColState));
    // what the host sends in one copy: the observations and tolerances that are
    // in host memory, then the six coefficient vectors; long observations follow
    // in copies of their own
    const void* host_in[4] = {y_ptr, y_idx, y_val, tol};
    const size_t host_len[4] = {(size_t)(B + 1) * 4, (size_t)nnz_y * 4, (size_t)nnz_y * 4, (size_t)B * 4};
    size_t host_at[4] = {0, 0, 0, 0}, in_bytes = 0;
    for (int k = 0; k < 4; ++k) {
        if (host_len[k] && hd_is_device_ptr(host_in[k])) host_in[k] = nullptr;  // used where it is
        if (!host_in[k] || host_len[k] > HD_STAGE_MOST) continue;
        host_at[k] = in_bytes;
        in_bytes += ws_size(host_len[k]);
    }
    const size_t coef_at = in_bytes, staged = coef_at + 6 * (size_t)rpad * 8;
    in_bytes = ws_size(staged);
    for (int k = 0; k < 4; ++k)
        if (host_in[k] && host_len[k] > HD_STAGE_MOST) {
            host_at[k] = in_bytes;
            in_bytes += ws_size(host_len[k]);
        }
    // what starts at zero: the counters, max |P_j|, the split H
    const size_t zero_bytes = ws_size(64) + ws_size((size_t)Bp * 4) + (lr_on ? 2 * ws_size((size_t)Bp16 * rpad * 2) : 0);
    bytes += ws_size(in_bytes) + zero_bytes;
    if (lr_on)
        bytes += ws_size((size_t)nchunk * rpad * Bp * 4) + 2 * ws_size((size_t)rpad * Bp * 8) +
                 ws_size((size_t)rpad * Bp * 4);
    // the fp16 gather copy of P: graph solves with 8 <= Bp <= 256 columns in multiples of 8
    const bool half_ok = !ts && Bp % 8 == 0 && Bp <= 256;
    if (half_ok) bytes += ws_size((size_t)n * Bp * 2);
    void* ws;
    int rc = hd_ws_reserve(ctx, bytes, &ws);
    if (rc) return rc;
    WsCarver cv(ws);
    S_.R = cv.take<float>((size_t)n * Bp);
    S_.P = cv.take<float>((size_t)n * Bp);
    S_.Q = cv.take<float>((size_t)n * Bp);
    S_.X = x_direct ? X : cv.take<float>((size_t)n * Bp);
    if (ts) S_.VT = ts->vt;
    S_.part = cv.take<float2>((size_t)S_.nch * Bp);
    S_.st = cv.take<ColState>(Bp);
    char* zero = cv.take<char>(zero_bytes);
    WsCarver zv(zero);
    S_.num_active = zv.take<int>(16);
    S_.err = S_.num_active + 1;
    unsigned* p16_max = zv.take<unsigned>(Bp);
    HD_CUDA(ctx, cudaMemsetAsync(zero, 0, zero_bytes, ctx->stream));
    char* d_in = cv.take<char>(in_bytes);
    char* hs;  // pinned: the inputs now, the columns' states after the confirmation
    if ((rc = hd_host_stage(ctx, std::max(staged, B * sizeof(ColState)), (void**)&hs))) return rc;
    const void* dev_in[4] = {y_ptr, y_idx, y_val, tol};
    for (int k = 0; k < 4; ++k)
        if (host_in[k]) {
            dev_in[k] = d_in + host_at[k];
            if (host_len[k] > HD_STAGE_MOST)
                HD_CUDA(ctx, cudaMemcpyAsync(d_in + host_at[k], host_in[k], host_len[k], cudaMemcpyHostToDevice, ctx->stream));
            else if (host_len[k])
                memcpy(hs + host_at[k], host_in[k], host_len[k]);
        }
    const void *yp = dev_in[0], *yi = dev_in[1], *yv = dev_in[2], *tl = dev_in[3];
    S_.nnz_y = nnz_y;
    S_.yp = (const int32_t*)yp;
    S_.yi = (const int32_t*)yi;
    S_.yv = (const float*)yv;
    __half* p16 = half_ok ? cv.take<__half>((size_t)n * Bp) : nullptr;
    if (lr_on) {
        S_.lr.e = eig;
        S_.lr.rpad = rpad;
        S_.lr.nchunk = nchunk;
        S_.lr.Bp16 = Bp16;
        S_.lr.part = cv.take<float>((size_t)nchunk * rpad * Bp);
        S_.lr.C = cv.take<double>((size_t)rpad * Bp);
        S_.Cy = cv.take<double>((size_t)rpad * Bp);
        S_.lr.H = cv.take<float>((size_t)rpad * Bp);
        S_.lr.Hhi = zv.take<__nv_bfloat16>((size_t)Bp16 * rpad);
        S_.lr.Hlo = zv.take<__nv_bfloat16>((size_t)Bp16 * rpad);
        double** dst[6] = {&S_.gcoef, &S_.hcoef, &S_.opcoef, &S_.dcoef, &S_.ones, &S_.negop};
        double* co = (double*)(hs + coef_at);
        std::fill(co, co + 6 * (size_t)rpad, 0.0);
        for (int k = 0; k < 6; ++k) *dst[k] = (double*)(d_in + coef_at) + (size_t)k * rpad;
        double *gc = co, *hc = gc + rpad, *oc = hc + rpad, *dc = oc + rpad, *on = dc + rpad, *ng = on + rpad;
        const double a = alpha;
        const double c3 = mode == HD_MODE_PROJ ? a : a / (1.0 - a);
        for (int k = 0; k < r; ++k) {
            double l = eig->lambda_h[k];
            gc[k] = (1.0 - a) * a * l / (1.0 - a * l);  // g_alpha, Eq. 16
            hc[k] = (1.0 - a) / (1.0 - a * l);          // h_alpha, Sec. 3.2
            oc[k] = c3 * l;
            double lt = l > 0.0 ? l : 0.0;
            dc[k] = a * lt / (1.0 - a * lt);
            on[k] = 1.0;
            ng[k] = -a / (1.0 - a) * l;
        }
    }
    if (staged) HD_CUDA(ctx, cudaMemcpyAsync(d_in, hs, staged, cudaMemcpyHostToDevice, ctx->stream));

    // ---------------- setup
    if (!ts && g->max_row < 0) {
        // the longest row bounds the rounding of the true residual (k_resid_pick)
        k_max_row<<<std::min<int64_t>(ceil_div(n, 256), (int64_t)ctx->num_sms * 8), 256, 0, ctx->stream>>>(
            g->row_ptr, n, S_.num_active);
        HD_CHECK_LAUNCH(ctx);
        HD_CUDA(ctx, cudaMemcpyAsync(ctx->h_poll, S_.num_active, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
        HD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        g->max_row = ctx->h_poll[0];
        HD_CUDA(ctx, cudaMemsetAsync(S_.num_active, 0, sizeof(int), ctx->stream));
    }
    if (!ts) {
        S_.slab = spmm_slab(g, Bp);
        if ((rc = spmm_segments(ctx, S_))) return rc;
    }
    engine_set_panels(S_, lr_on ? mode : HD_MODE_PAPER);
    if (half_ok && S_.segK == 1 && !half_gathers_off()) {
        S_.P16 = p16;
        S_.p16_max = p16_max;
        S_.use_half = S_.num_active + 3;  // 0: the first iteration gathers fp32
    }
    const int eff_mode = lr_on ? mode : HD_MODE_PAPER;
    const double a = alpha;
    float c1, c2, xs = 1.0f;
    if (eff_mode == HD_MODE_PROJ) {
        c1 = 1.0f;
        c2 = (float)a;
        xs = (float)(1.0 - a);
    } else {
        c1 = (float)(1.0 / (1.0 - a));
        c2 = (float)(a / (1.0 - a));
    }
    // X accumulates the temporal term alone; the spectral term is added after
    // the true-residual confirmation
    HD_CUDA(ctx, cudaMemsetAsync(S_.R, 0, vec, ctx->stream));
    HD_CUDA(ctx, cudaMemsetAsync(S_.X, 0, vec, ctx->stream));
    if (ts) {
        HD_CUDA(ctx, cudaMemsetAsync(S_.Q, 0, vec, ctx->stream));  // (rows past a shortlist's end stay 0)
        k_trunc_work<<<1, TC_T, 0, ctx->stream>>>(ts->sl_ptr, ts->off, B, n, ts->work);
        HD_CHECK_LAUNCH(ctx);
    }
    k_scatter_y<<<B, 128, 0, ctx->stream>>>((const int32_t*)yp, (const int32_t*)yi, (const float*)yv, nnz_y, n, Bp,
                                            S_.R, S_.err);
    HD_CHECK_LAUNCH(ctx);
    const double* Cd = lr_on ? S_.lr.C : nullptr;
    const size_t cbytes = (size_t)rpad * Bp * sizeof(double);
    if (eff_mode == HD_MODE_PAPER) {
        if ((rc = launch_colsq(S_, S_.R))) return rc;
        k_fin_setup<<<Bp, 128, 0, ctx->stream>>>(S_.part, (int)S_.nch, Bp, B, (const float*)tl, S_.st, nullptr, nullptr,
                                                0, S_.num_active);
        HD_CHECK_LAUNCH(ctx);
        if (S_.pv.last)
            LAUNCH_VEC(k_direction, S_.P, S_.pv, S_.R, n, Bp, S_.st);  // (beta is 0)
        else
            HD_CUDA(ctx, cudaMemcpyAsync(S_.P, S_.R, vec, cudaMemcpyDeviceToDevice, ctx->stream));
        if (lr_on) {
            // C = U^T y: kept for x^s = U g(Lambda) C (Eq. 18), and U^T P for the first operator
            if ((rc = lr_reduce(ctx, S_.lr, S_.R, n, Bp))) return rc;
            if ((rc = lr_finish(ctx, S_.lr, Bp, S_.opcoef))) return rc;
            HD_CUDA(ctx, cudaMemcpyAsync(S_.Cy, S_.lr.C, cbytes, cudaMemcpyDeviceToDevice, ctx->stream));
        }
    } else if (eff_mode == HD_MODE_PROJ) {
        // C = U^T y (kept); b = y - U C
        if ((rc = lr_reduce(ctx, S_.lr, S_.R, n, Bp))) return rc;
        if ((rc = lr_finish(ctx, S_.lr, Bp, S_.ones))) return rc;
        HD_CUDA(ctx, cudaMemcpyAsync(S_.Cy, S_.lr.C, cbytes, cudaMemcpyDeviceToDevice, ctx->stream));
        if ((rc = lr_expand(ctx, S_.lr, EXP_SUB_R, S_.R, nullptr, nullptr, n, Bp, S_.st))) return rc;
        if ((rc = launch_colsq(S_, S_.R))) return rc;
        k_fin_setup<<<Bp, 128, 0, ctx->stream>>>(S_.part, (int)S_.nch, Bp, B, (const float*)tl, S_.st, nullptr, nullptr,
                                                0, S_.num_active);
        HD_CHECK_LAUNCH(ctx);
        HD_CUDA(ctx, cudaMemcpyAsync(S_.P, S_.R, vec, cudaMemcpyDeviceToDevice, ctx->stream));
        if ((rc = lr_reduce(ctx, S_.lr, S_.P, n, Bp))) return rc;
        if ((rc = lr_finish(ctx, S_.lr, Bp, S_.opcoef))) return rc;
    } else {  // PCG
        if ((rc = launch_colsq(S_, S_.R))) return rc;
        if ((rc = lr_reduce(ctx, S_.lr, S_.R, n, Bp))) return rc;
        if ((rc = lr_finish(ctx, S_.lr, Bp, S_.dcoef))) return rc;
        k_fin_setup<<<Bp, 128, 0, ctx->stream>>>(S_.part, (int)S_.nch, Bp, B, (const float*)tl, S_.st, Cd, S_.dcoef, r,
                                                S_.num_active);
        HD_CHECK_LAUNCH(ctx);
        // (beta is 0: whatever P holds is dropped)
        if ((rc = lr_expand(ctx, S_.lr, EXP_DIRECTION, S_.P, S_.R, S_.P, n, Bp, S_.st, nullptr, &S_.pv)))
            return rc;
    }

    // ---------------- iterations, then confirmation by the true residual
    S_.eff_mode = eff_mode;
    S_.c1 = c1;
    S_.c2 = c2;
    S_.xs = xs;
    S_.r = r;
    S_.max_iter = max_iter;
    // (no poll here: the first run of iterations is queued behind the set-up; its
    // kernels return at once if no column is active, and a bad observation, which
    // the scatter left out, is reported by the poll after it)
    int active = 1, ran = 0, first_ran = -1;
    const ColState* hcol = (const ColState*)hs;
    for (int round = 0; round <= MAX_CONFIRM; ++round) {
        if (active > 0 && max_iter > 0 && (rc = iterate_until_stopped(S_, ran))) return rc;
        if (first_ran < 0) first_ran = ran;
        if ((rc = true_residual(S_, a))) return rc;
        {
            HD_PROF(ctx, "scalar");
            HD_CUDA(ctx, cudaMemsetAsync(S_.num_active, 0, sizeof(int), ctx->stream));
            k_fin_confirm<<<Bp, 128, 0, ctx->stream>>>(S_.part, (int)S_.nch, Bp, B, S_.st, max_iter, S_.num_active);
        }
        HD_CHECK_LAUNCH(ctx);
        HD_CUDA(ctx, cudaMemcpyAsync(ctx->h_poll, S_.num_active, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
        HD_CUDA(ctx, cudaMemcpyAsync(ctx->h_poll + 1, S_.err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
        HD_CUDA(ctx, cudaMemcpyAsync(hs, S_.st, B * sizeof(ColState), cudaMemcpyDeviceToHost, ctx->stream));
        HD_CUDA(ctx, cudaMemcpyAsync(ctx->h_poll + 8, ctx->d_flags + 2, 2 * sizeof(int), cudaMemcpyDeviceToHost,
                                     ctx->stream));
        HD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        if (ctx->h_poll[1]) return hd_fail(ctx, HD_ERR_INVALID_ARG, "%s", BAD_OBSERVATION);
        if (ctx->h_poll[8] || ctx->h_poll[9]) return lr_tc_check_flags(ctx);
        active = ctx->h_poll[0];
        if (active == 0) break;
        if ((rc = restart_columns(S_))) return rc;
    }
    // the next solve with the same key polls first after as many iterations as
    // this one's columns took before any restart (without restarts the
    // columns' own count, else the iterations launched)
    int most = 0;
    for (int j = 0; j < B; ++j) most = std::max(most, hcol[j].iters);
    ctx->hint_key = iteration_key(S_);
    ctx->iter_hint = ran == first_ran ? most : first_ran;
    for (int j = 0; j < B; ++j) {
        if (iters && !hd_is_device_ptr(iters)) iters[j] = hcol[j].iters;
        if (relres && !hd_is_device_ptr(relres)) relres[j] = hcol[j].bb > 0 ? (float)std::sqrt(hcol[j].rr / hcol[j].bb) : 0.f;
        if (status && !hd_is_device_ptr(status)) status[j] = hcol[j].status;
    }
    // ---------------- spectral term (Eq. 17-18): X += U g(Lambda) U^T y, or U h(Lambda) U^T y (projected form)
    if (lr_on && eff_mode != HD_MODE_PCG && !temporal_only) {
        if ((rc = lr_coef(ctx, S_.lr, Bp, eff_mode == HD_MODE_PAPER ? S_.gcoef : S_.hcoef, S_.Cy))) return rc;
        if ((rc = lr_expand(ctx, S_.lr, EXP_ADD_Q, S_.X, nullptr, nullptr, n, Bp, nullptr))) return rc;
    }

    // ---------------- outputs
    if ((iters && hd_is_device_ptr(iters)) || (relres && hd_is_device_ptr(relres)) ||
        (status && hd_is_device_ptr(status))) {
        k_outputs<<<ceil_div(B, 128), 128, 0, ctx->stream>>>(S_.st, B, hd_is_device_ptr(iters) ? iters : nullptr,
                                                             hd_is_device_ptr(relres) ? relres : nullptr,
                                                             hd_is_device_ptr(status) ? status : nullptr);
        HD_CHECK_LAUNCH(ctx);
    }
    if (!x_direct) {
        if (hd_is_device_ptr(X)) {
            k_copy_out<<<ceil_div(n * B, 256), 256, 0, ctx->stream>>>(S_.X, Bp, X, ldx, B, n);
            HD_CHECK_LAUNCH(ctx);
        } else {
            HD_CUDA(ctx, cudaMemcpy2DAsync(X, (size_t)ldx * 4, S_.X, (size_t)Bp * 4, (size_t)B * 4, n,
                                           cudaMemcpyDeviceToHost, ctx->stream));
            HD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        }
    }
    // the tensor-core kernels' status was read with the confirmation unless more ran since
    if (lr_on && lr_use_tensor_cores(eig) && (eff_mode != HD_MODE_PCG || !x_direct)) return lr_tc_check_flags(ctx);
    return HD_OK;
}

// ------------------------------------------------------------------ spectral products on their own
static int lowrank_setup(hd_ctx* ctx, const hd_eig* e, int32_t Bp, LowRank& lr, double** coef_ones, WsCarver& cv) {
    lr.e = e;
    lr.rpad = (e->r + 63) / 64 * 64;
    lr.Bp16 = (Bp + 15) / 16 * 16;
    lr.nchunk = lr_nchunk(ctx, e, Bp);
    lr.part = cv.take<float>((size_t)lr.nchunk * lr.rpad * Bp);
    lr.C = cv.take<double>((size_t)lr.rpad * Bp);
    lr.H = cv.take<float>((size_t)lr.rpad * Bp);
    lr.Hhi = cv.take<__nv_bfloat16>((size_t)lr.Bp16 * lr.rpad);
    lr.Hlo = cv.take<__nv_bfloat16>((size_t)lr.Bp16 * lr.rpad);
    *coef_ones = cv.take<double>(lr.rpad);
    std::vector<double> on(lr.rpad, 0.0);
    for (int k = 0; k < e->r; ++k) on[k] = 1.0;
    HD_CUDA(ctx, cudaMemcpyAsync(*coef_ones, on.data(), lr.rpad * 8, cudaMemcpyHostToDevice, ctx->stream));
    HD_CUDA(ctx, cudaMemsetAsync(lr.Hhi, 0, (size_t)lr.Bp16 * lr.rpad * 2, ctx->stream));
    HD_CUDA(ctx, cudaMemsetAsync(lr.Hlo, 0, (size_t)lr.Bp16 * lr.rpad * 2, ctx->stream));
    return HD_OK;
}

static size_t lowrank_bytes(hd_ctx* ctx, const hd_eig* e, int32_t Bp) {
    int rpad = (e->r + 63) / 64 * 64;
    int nch = lr_nchunk(ctx, e, Bp);
    return ws_size((size_t)nch * rpad * Bp * 4) + ws_size((size_t)rpad * Bp * 8) + ws_size((size_t)rpad * Bp * 4) +
           2 * ws_size((size_t)((Bp + 15) / 16 * 16) * rpad * 2) + ws_size(rpad * 8);
}

extern "C" int hd_eig_project(hd_ctx* ctx, const hd_eig* e, const float* V, int32_t B, double* C_out) {
    if (!ctx || !e || !V || !C_out || B <= 0 || B % 4 || B > 256 || e->r <= 0) return HD_ERR_INVALID_ARG;
    if (!hd_is_device_ptr(V)) return hd_fail(ctx, HD_ERR_INVALID_ARG, "V must be device memory");
    void* ws;
    int rc = hd_ws_reserve(ctx, lowrank_bytes(ctx, e, B), &ws);
    if (rc) return rc;
    WsCarver cv(ws);
    LowRank lr;
    double* ones;
    if ((rc = lowrank_setup(ctx, e, B, lr, &ones, cv))) return rc;
    if ((rc = lr_reduce(ctx, lr, V, e->n, B))) return rc;
    if ((rc = lr_finish(ctx, lr, B, ones))) return rc;
    // rows 0..r-1 of C (fp64, r x B)
    cudaMemcpyKind kind = hd_is_device_ptr(C_out) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    HD_CUDA(ctx, cudaMemcpyAsync(C_out, lr.C, (size_t)e->r * B * 8, kind, ctx->stream));
    HD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    if (lr_use_tensor_cores(e) && (rc = lr_tc_check_flags(ctx))) return rc;
    return HD_OK;
}

// H (fp64, r x B) -> the fp32 partial layout [1][rpad][B], zero beyond r.
__global__ void k_h_to_part(const double* Hin, int r, int32_t B, int rpad, float* part) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)rpad * B) return;
    int k = (int)(e / B);
    part[e] = k < r ? (float)Hin[e] : 0.0f;
}

extern "C" int hd_eig_expand(hd_ctx* ctx, const hd_eig* e, const double* H, int32_t B, float* X_out) {
    if (!ctx || !e || !H || !X_out || B <= 0 || B % 4 || B > 256 || e->r <= 0) return HD_ERR_INVALID_ARG;
    if (!hd_is_device_ptr(X_out)) return hd_fail(ctx, HD_ERR_INVALID_ARG, "X_out must be device memory");
    void* ws;
    int rc = hd_ws_reserve(ctx, lowrank_bytes(ctx, e, B) + ws_size((size_t)e->r * B * 8), &ws);
    if (rc) return rc;
    WsCarver cv(ws);
    LowRank lr;
    double* ones;
    if ((rc = lowrank_setup(ctx, e, B, lr, &ones, cv))) return rc;
    double* Hs = cv.take<double>((size_t)e->r * B);
    const void* Hd;
    if ((rc = hd_stage_in(ctx, H, (size_t)e->r * B * 8, Hs, &Hd))) return rc;
    lr.nchunk = 1;
    k_h_to_part<<<ceil_div((int64_t)lr.rpad * B, 256), 256, 0, ctx->stream>>>((const double*)Hd, e->r, B, lr.rpad,
                                                                             lr.part);
    HD_CHECK_LAUNCH(ctx);
    if ((rc = lr_finish(ctx, lr, B, ones))) return rc;
    if ((rc = lr_expand(ctx, lr, EXP_SET_X, X_out, nullptr, nullptr, e->n, B, nullptr))) return rc;
    HD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    if (lr_use_tensor_cores(e) && (rc = lr_tc_check_flags(ctx))) return rc;
    return HD_OK;
}

// ------------------------------------------------------------------ general transfer functions (Appendix A)

// out = (accumulate ? out : 0) + c * Y over n x Bp
__global__ void k_axpy_dense(float* __restrict__ out, const float* __restrict__ Y, float c, int64_t count4,
                             int accumulate) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= count4) return;
    const float4 y = reinterpret_cast<const float4*>(Y)[e];
    float4 o = accumulate ? reinterpret_cast<const float4*>(out)[e] : make_float4(0.f, 0.f, 0.f, 0.f);
    o.x = fmaf(c, y.x, o.x);
    o.y = fmaf(c, y.y, o.y);
    o.z = fmaf(c, y.z, o.z);
    o.w = fmaf(c, y.w, o.w);
    reinterpret_cast<float4*>(out)[e] = o;
}

extern "C" int hd_filter_poly(hd_ctx* ctx, const hd_graph* g, const hd_eig* eig, int32_t B, const int32_t* y_ptr,
                              const int32_t* y_idx, const float* y_val, const double* coeffs, int32_t ncoef,
                              float* X, int32_t ldx) {
    if (!ctx || !g || !y_ptr || !coeffs || !X) return HD_ERR_INVALID_ARG;
    if (B <= 0 || B > 4096 || ldx < B) return hd_fail(ctx, HD_ERR_INVALID_ARG, "B=%d ldx=%d", B, ldx);
    if (ncoef < 1 || ncoef > 100000) return hd_fail(ctx, HD_ERR_INVALID_ARG, "ncoef=%d", ncoef);
    for (int i = 0; i < ncoef; ++i)
        if (!std::isfinite(coeffs[i])) return hd_fail(ctx, HD_ERR_INVALID_ARG, "coefficient %d not finite", i);
    if (eig && eig->n != g->n) return hd_fail(ctx, HD_ERR_INVALID_ARG, "eigenpairs for n=%lld, graph n=%lld",
                                              (long long)eig->n, (long long)g->n);
    HD_CUDA(ctx, cudaSetDevice(ctx->device));
    const int64_t n = g->n;
    const int32_t Bp = (B + 3) / 4 * 4;
    const bool lr_on = eig && eig->r > 0;
    int32_t nnz_y;
    if (hd_is_device_ptr(y_ptr)) {
        HD_CUDA(ctx, cudaMemcpy(&nnz_y, y_ptr + B, 4, cudaMemcpyDeviceToHost));
    } else {
        nnz_y = y_ptr[B];
    }
    if (nnz_y < 0) return hd_fail(ctx, HD_ERR_INVALID_ARG, "y_ptr[B] = %d", nnz_y);
    if (nnz_y > 0 && (!y_idx || !y_val)) return HD_ERR_INVALID_ARG;
    const size_t vec = (size_t)n * Bp * 4;
    size_t bytes = 3 * ws_size(vec) + ws_size(64) + ws_size((B + 1) * 4) + 2 * ws_size((size_t)nnz_y * 4 + 4);
    if (lr_on) bytes += lowrank_bytes(ctx, eig, Bp) + 2 * ws_size((size_t)((eig->r + 63) / 64 * 64) * 8);
    void* ws;
    int rc = hd_ws_reserve(ctx, bytes, &ws);
    if (rc) return rc;
    WsCarver cv(ws);
    float* Yd = cv.take<float>((size_t)n * Bp);
    float* acc = cv.take<float>((size_t)n * Bp);
    float* Q = cv.take<float>((size_t)n * Bp);
    int* err = cv.take<int>(16);
    int32_t* d_yptr = cv.take<int32_t>(B + 1);
    int32_t* d_yidx = cv.take<int32_t>(nnz_y + 1);
    float* d_yval = cv.take<float>(nnz_y + 1);
    const void *yp, *yi, *yv;
    if ((rc = hd_stage_in(ctx, y_ptr, (B + 1) * 4, d_yptr, &yp))) return rc;
    if ((rc = hd_stage_in(ctx, y_idx, (size_t)nnz_y * 4, d_yidx, &yi))) return rc;
    if ((rc = hd_stage_in(ctx, y_val, (size_t)nnz_y * 4, d_yval, &yv))) return rc;
    LowRank lr{};
    double *ones = nullptr, *lamc = nullptr, *gc = nullptr;
    if (lr_on) {
        if ((rc = lowrank_setup(ctx, eig, Bp, lr, &ones, cv))) return rc;
        lamc = cv.take<double>(lr.rpad);
        gc = cv.take<double>(lr.rpad);
        // g(lambda) = h(lambda) - h(0) = sum_{i >= 1} c_i lambda^i (Eq. 33), Horner in fp64
        std::vector<double> lh(lr.rpad, 0.0), gh(lr.rpad, 0.0);
        for (int k = 0; k < eig->r; ++k) {
            const double l = eig->lambda_h[k];
            double s = 0.0;
            for (int i = ncoef - 1; i >= 1; --i) s = s * l + coeffs[i];
            lh[k] = l;
            gh[k] = s * l;
        }
        HD_CUDA(ctx, cudaMemcpyAsync(lamc, lh.data(), lr.rpad * 8, cudaMemcpyHostToDevice, ctx->stream));
        HD_CUDA(ctx, cudaMemcpyAsync(gc, gh.data(), lr.rpad * 8, cudaMemcpyHostToDevice, ctx->stream));
    }
    HD_CUDA(ctx, cudaMemsetAsync(Yd, 0, vec, ctx->stream));
    HD_CUDA(ctx, cudaMemsetAsync(err, 0, sizeof(int), ctx->stream));
    k_scatter_y<<<B, 128, 0, ctx->stream>>>((const int32_t*)yp, (const int32_t*)yi, (const float*)yv, nnz_y, n, Bp,
                                            Yd, err);
    HD_CHECK_LAUNCH(ctx);
    const int64_t c4 = (int64_t)n * Bp / 4;
    // h(W_r) y by Horner's rule on the black box W_r z = W z - U (Lambda (U^T z)) (Eq. 32)
    k_axpy_dense<<<ceil_div(c4, 256), 256, 0, ctx->stream>>>(acc, Yd, (float)coeffs[ncoef - 1], c4, 0);
    HD_CHECK_LAUNCH(ctx);
    for (int i = ncoef - 2; i >= 0; --i) {
        { HD_PROF(ctx, "spmm");
          if ((rc = hd_spmm_apply(ctx, g, acc, Q, Bp, B, 0.0f, -1.0f))) return rc; }
        if (lr_on) {
            if ((rc = lr_reduce(ctx, lr, acc, n, Bp))) return rc;
            if ((rc = lr_finish(ctx, lr, Bp, lamc))) return rc;
            if ((rc = lr_expand(ctx, lr, EXP_SUB_R, Q, nullptr, nullptr, n, Bp, nullptr))) return rc;
        }
        k_axpy_dense<<<ceil_div(c4, 256), 256, 0, ctx->stream>>>(Q, Yd, (float)coeffs[i], c4, 1);
        HD_CHECK_LAUNCH(ctx);
        std::swap(acc, Q);
    }
    // + U g(Lambda) U^T y (Eq. 32)
    if (lr_on) {
        if ((rc = lr_reduce(ctx, lr, Yd, n, Bp))) return rc;
        if ((rc = lr_finish(ctx, lr, Bp, gc))) return rc;
        if ((rc = lr_expand(ctx, lr, EXP_ADD_Q, acc, nullptr, nullptr, n, Bp, nullptr))) return rc;
    }
    HD_CUDA(ctx, cudaMemcpyAsync(ctx->h_poll, err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    HD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    if (ctx->h_poll[0])
        return hd_fail(ctx, HD_ERR_INVALID_ARG, "bad observation: index out of range, non-finite value or bad y_ptr");
    if (hd_is_device_ptr(X)) {
        k_copy_out<<<ceil_div(n * B, 256), 256, 0, ctx->stream>>>(acc, Bp, X, ldx, B, n);
        HD_CHECK_LAUNCH(ctx);
    } else {
        HD_CUDA(ctx, cudaMemcpy2DAsync(X, (size_t)ldx * 4, acc, (size_t)Bp * 4, (size_t)B * 4, n,
                                       cudaMemcpyDeviceToHost, ctx->stream));
    }
    HD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    if (lr_on && lr_use_tensor_cores(eig) && (rc = lr_tc_check_flags(ctx))) return rc;
    return HD_OK;
}
