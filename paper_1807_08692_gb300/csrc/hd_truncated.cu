// Temporal filtering on truncated graphs, "Temporal†" (Sec. 3.1, Sec. 5.1,
// Table 1): for query j only the shortlist S_j of database items is kept, the
// affinity restricted to S_j x S_j is normalised again by its own degrees,
// W_j = D_j^-1/2 A_{S_j S_j} D_j^-1/2, and L_alpha(W_j) x_j = y_j is solved by
// the same multi-column CG as the full query (one system per column).
//
// The affinity is recovered from the stored graph as A_ik = W_ik / (d_i^-1/2
// d_k^-1/2).  Building the B systems:
//   bits[j]    = S_j as a bitmap of n bits, which a block keeps in shared memory:
//                most entries of a row are outside S_j, and a test there costs
//                no trip to L2
//   pos[j][i]  = (position of id i in S_j, d_i^-1/2) for the ids of S_j: one
//                gather per kept entry.  Columns share up to 512 MB of it in
//                turn (64 on 1M nodes at once), a bitmap of B n / 8 bytes is
//                all that grows with B n
//   row (j, t) = the entries of A's row S_j[t] whose column is in S_j, in the
//                graph's column order, with their local positions
//   counts (bitmap tests alone), offsets by an exclusive scan of them, entries
//   and subgraph degrees, then the values rescaled by the subgraph's D^-1/2 on
//   both sides.  64 shortlists of 75,000 on 1M nodes: 3.7 ms (2.5 of them the
//   fill, one row per warp in flight) against 4.3 ms when both passes looked every
//   entry up in pos and called the allocator sixteen times.
// Observations outside the shortlist are dropped (index 0, value 0).
#include <algorithm>
#include <cmath>
#include <vector>

#include "hd_solve.cuh"

namespace {

// thread (t, j): S_j's bitmap, and pos[j][S_j[t]] = (t, D^-1/2) of the first `placed`
// columns; bad ids and duplicates raise the error flag
__global__ void k_ts_mark(const int32_t* sl_ptr, const int32_t* sl_idx, const float* dinv, int64_t n, int2* pos,
                          int32_t placed, uint32_t* bits, int64_t words, int* err) {
    const int j = blockIdx.y;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int32_t b = sl_ptr[j], e = sl_ptr[j + 1];
    if (t >= e - b) return;
    const int32_t i = sl_idx[b + t];
    if (i < 0 || i >= n) {
        atomicExch(err, 1);
        return;
    }
    const uint32_t bit = 1u << (i & 31);
    if (atomicOr(&bits[(int64_t)j * words + (i >> 5)], bit) & bit) atomicExch(err, 2);
    if (j < placed) pos[(int64_t)j * n + i] = make_int2((int32_t)t, __float_as_int(dinv[i]));
}
// the same positions for a later group of columns (ids already checked)
__global__ void k_ts_place(const int32_t* sl_ptr, const int32_t* sl_idx, const float* dinv, int64_t n, int2* pos) {
    const int j = blockIdx.y;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int32_t b = sl_ptr[j], e = sl_ptr[j + 1];
    if (t >= e - b) return;
    const int32_t i = sl_idx[b + t];
    pos[(int64_t)j * n + i] = make_int2((int32_t)t, __float_as_int(dinv[i]));
}

// Both passes over the rows: a block takes an equal share of all shortlists' rows
// in column order; a warp takes up to 32 rows at a time (fewer where a column's part
// of the share is short, so that all warps have some), reads their bounds side by
// side and then each row's columns, two per lane, one row ahead of the tests.
constexpr int TS_T = 1024;
constexpr int TS_SMEM_WORDS = 50 * 1024;  // bitmaps up to 200 KB (1.6M nodes) go to shared memory
constexpr int64_t TS_POS_BYTES = (int64_t)512 << 20;  // position maps at a time (at least one column's)

// For the rows lo .. hi of one column: row.rows32(t, valid, i) with each lane's own
// row t (id i, -1 for an empty one) of the next 32, then for the r-th of them
// begin(r), entries(q, k, kept) per 64 columns (two per lane, at q and q + 32)
// and end(r), at last flush(t0, rows).
template <class ROW>
__device__ __forceinline__ void ts_rows(const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
                                        const int32_t* __restrict__ sl, int64_t n, int64_t lo, int64_t hi,
                                        const uint32_t* bits, ROW row) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (int)min((int64_t)32, (hi - lo + TS_T / 32 - 1) / (TS_T / 32));
    for (int64_t t0 = lo + per * warp; t0 < hi; t0 += per * (TS_T / 32)) {
        const int rows = (int)min((int64_t)per, hi - t0);
        const int64_t mine = t0 + lane;
        int32_t i = lane < rows ? __ldg(sl + mine) : -1;
        if (i >= n) i = -1;  // out of range (flagged by k_ts_mark): an empty row
        const int32_t b = i >= 0 ? __ldg(rp + i) : 0, e = i >= 0 ? __ldg(rp + i + 1) : 0;
        int32_t k[2], nk[2];
        auto columns = [&](int32_t q0, int32_t end, int32_t (&x)[2]) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int32_t q = q0 + 32 * u + lane;
                x[u] = q < end ? __ldg(col + q) : -1;
            }
        };
        columns(__shfl_sync(0xffffffffu, b, 0), __shfl_sync(0xffffffffu, e, 0), nk);
        row.rows32(mine, lane < rows, i);
        for (int r = 0; r < rows; ++r) {
            const int32_t rb = __shfl_sync(0xffffffffu, b, r), re = __shfl_sync(0xffffffffu, e, r);
            const int r1 = min(r + 1, 31);
            const int32_t xb = __shfl_sync(0xffffffffu, b, r1), xe = __shfl_sync(0xffffffffu, e, r1);
            k[0] = nk[0];
            k[1] = nk[1];
            if (r + 1 < rows) columns(xb, xe, nk);
            row.begin(r);
            for (int32_t q0 = rb; q0 < re; q0 += 64) {
                if (q0 != rb) columns(q0, re, k);
                bool keep[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) keep[u] = k[u] >= 0 && (bits[k[u] >> 5] >> (k[u] & 31) & 1u);
                row.entries(q0 + lane, k, keep);
            }
            row.end(r);
        }
        row.flush(t0, rows);
    }
}
// A block's share of the rows, with the column's bitmap in shared memory if it fits
template <class F>
__device__ __forceinline__ void ts_share(int32_t B, const int32_t* __restrict__ sl_ptr, const uint32_t* bits,
                                         int64_t words, uint32_t* sm, F each) {
    const int32_t first = __ldg(sl_ptr);
    const int64_t total = (int64_t)__ldg(sl_ptr + B) - first, per = (total + gridDim.x - 1) / gridDim.x;
    const int64_t g0 = blockIdx.x * per, g1 = min(total, g0 + per);
    if (g0 >= g1) return;
    int j = 0;  // the column of row g0: the last whose rows start at or before it
    for (int a = B; a - j > 1;) {
        const int m = (j + a) >> 1;
        if (__ldg(sl_ptr + m) - first <= g0) j = m;
        else a = m;
    }
    for (int64_t g = g0; g < g1; ++j) {
        const int64_t at = (int64_t)__ldg(sl_ptr + j) - first, end = (int64_t)__ldg(sl_ptr + j + 1) - first;
        const int64_t lo = g - at, hi = min(end, g1) - at;
        if (lo >= hi) continue;  // an empty shortlist
        const uint32_t* bj = bits + j * words;
        if (words <= TS_SMEM_WORDS) {
            __syncthreads();
            for (int64_t w = threadIdx.x; w < words; w += TS_T) sm[w] = __ldg(bj + w);
            __syncthreads();
            bj = sm;
        }
        each(j, lo, hi, bj);
        g += hi - lo;
    }
}

// cnt[j][t]: entries of row t of column j
struct CountRow {
    int32_t* cnt;
    int c, mine;
    __device__ __forceinline__ void rows32(int64_t, bool, int32_t) {}
    __device__ __forceinline__ void begin(int) { c = 0; }
    __device__ __forceinline__ void entries(int32_t, const int32_t (&)[2], const bool (&keep)[2]) {
        c += __popc(__ballot_sync(0xffffffffu, keep[0])) + __popc(__ballot_sync(0xffffffffu, keep[1]));
    }
    __device__ __forceinline__ void end(int r) {
        if ((threadIdx.x & 31) == r) mine = c;
    }
    __device__ __forceinline__ void flush(int64_t t0, int rows) {
        const int lane = threadIdx.x & 31;
        if (lane < rows) cnt[t0 + lane] = mine;
    }
};
__global__ void __launch_bounds__(TS_T, 1) k_ts_count(const int32_t* rp, const int32_t* col, const int32_t* sl_ptr,
                                                      const int32_t* sl_idx, int32_t B, int64_t n, int64_t smax,
                                                      const uint32_t* bits, int64_t words, int32_t* cnt) {
    extern __shared__ uint32_t ts_sm[];
    ts_share(B, sl_ptr, bits, words, ts_sm, [&](int j, int64_t lo, int64_t hi, const uint32_t* bj) {
        CountRow row;
        row.cnt = cnt + j * smax;
        row.mine = 0;
        ts_rows(rp, col, sl_idx + sl_ptr[j], n, lo, hi, bj, row);
    });
}

// The kept entries with their local column, in order, values A_ik (scaled by
// k_ts_scale), and the subgraph degree of every row.
struct FillRow {
    const float *val, *dinv;
    const int2* pj;
    const int64_t* off;
    int32_t* ci;
    float *wv, *deg;
    float di, d, mine, di32;
    int64_t at, at32;
    __device__ __forceinline__ void rows32(int64_t t, bool valid, int32_t i) {
        at32 = valid ? __ldg(off + t) : 0;
        di32 = i >= 0 ? __ldg(dinv + i) : 0.f;
    }
    __device__ __forceinline__ void begin(int r) {
        at = __shfl_sync(0xffffffffu, at32, r);
        di = __shfl_sync(0xffffffffu, di32, r);
        d = 0.f;
    }
    __device__ __forceinline__ void entries(int32_t q, const int32_t (&k)[2], const bool (&keep)[2]) {
        const uint32_t below = (1u << (threadIdx.x & 31)) - 1u;
        int2 u[2];
        float v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            u[h] = make_int2(0, 0);
            v[h] = 0.f;
            if (keep[h]) {
                u[h] = __ldg(pj + k[h]);
                v[h] = __ldg(val + q + 32 * h);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float a = keep[h] ? v[h] / (di * __int_as_float(u[h].y)) : 0.f;
            d += a;
            const uint32_t kb = __ballot_sync(0xffffffffu, keep[h]);
            if (keep[h]) {
                const int64_t o = at + __popc(kb & below);
                ci[o] = u[h].x;
                wv[o] = a;
            }
            at += __popc(kb);
        }
    }
    __device__ __forceinline__ void end(int r) {
        for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if ((threadIdx.x & 31) == r) mine = d;
    }
    __device__ __forceinline__ void flush(int64_t t0, int rows) {
        const int lane = threadIdx.x & 31;
        if (lane < rows) deg[t0 + lane] = mine;
    }
};
__global__ void __launch_bounds__(TS_T, 1)
    k_ts_fill(const int32_t* rp, const int32_t* col, const float* val, const float* dinv, const int32_t* sl_ptr,
              const int32_t* sl_idx, int32_t B, int64_t n, int64_t smax, const int2* pos, const uint32_t* bits,
              int64_t words, const int64_t* off, int32_t* ci, float* wv, float* deg) {
    extern __shared__ uint32_t ts_sm[];
    ts_share(B, sl_ptr, bits, words, ts_sm, [&](int j, int64_t lo, int64_t hi, const uint32_t* bj) {
        FillRow row;
        row.val = val;
        row.dinv = dinv;
        row.pj = pos + (int64_t)j * n;
        row.off = off + j * smax;
        row.ci = ci;
        row.wv = wv;
        row.deg = deg + j * smax;
        row.mine = 0.f;
        ts_rows(rp, col, sl_idx + sl_ptr[j], n, lo, hi, bj, row);
    });
}

// wv = D^-1/2 A D^-1/2 of the subgraphs: eight lanes per row, four entries of each
// lane in flight
__global__ void __launch_bounds__(256) k_ts_scale(const int64_t* __restrict__ off, const int32_t* __restrict__ ci, float* wv,
                                                  const float* __restrict__ sdinv, int64_t rows, int64_t smax) {
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3;
    if (w >= rows) return;
    const int64_t b = off[w], e = off[w + 1];
    const float* sj = sdinv + w / smax * smax;
    const float si = sdinv[w];
    for (int64_t q0 = b + (threadIdx.x & 7); q0 < e; q0 += 32) {
        float a[4], x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t q = q0 + 8 * u;
            a[u] = x[u] = 0.f;
            if (q < e) {
                a[u] = wv[q];
                x[u] = __ldg(sj + __ldg(ci + q));
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (q0 + 8 * u < e) wv[q0 + 8 * u] = si * a[u] * x[u];
    }
}

__global__ void k_ts_sdinv(const float* deg, int64_t count, float* sdinv) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e < count) sdinv[e] = deg[e] > 0.0f ? 1.0f / sqrtf(deg[e]) : 0.0f;
}

// observations of column j -> local positions (outside S_j: position 0, value 0)
__global__ void k_ts_map_y(const int32_t* y_ptr, const int32_t* y_idx, const float* y_val, int32_t B, int64_t n,
                           const int2* pos, const uint32_t* bits, int64_t words, int32_t* y_loc, float* y_lv,
                           int* err) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= B) return;
    for (int32_t q = y_ptr[j]; q < y_ptr[j + 1]; ++q) {
        const int32_t i = y_idx[q];
        if (i < 0 || i >= n || !isfinite(y_val[q])) {
            atomicExch(err, 3);
            y_loc[q] = 0;
            y_lv[q] = 0.0f;
            continue;
        }
        const bool in = bits[j * words + (i >> 5)] >> (i & 31) & 1u;
        const int32_t u = in ? pos[(int64_t)j * n + i].x : -1;
        y_loc[q] = u >= 0 ? u : 0;
        y_lv[q] = u >= 0 ? y_val[q] : 0.0f;
    }
}

// exclusive scan, part 1: sums of 1024-element blocks
__global__ void k_scan_sums(const int32_t* in, int64_t count, int64_t* bsum) {
    __shared__ int64_t sm[32];
    const int64_t e = blockIdx.x * 1024ll + threadIdx.x;
    int64_t v = e < count ? in[e] : 0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t s = 0;
        for (int w = 0; w < 32; ++w) s += sm[w];
        bsum[blockIdx.x] = s;
    }
}

// part 2: out[e] = boff[block] + sum of in[block start .. e - 1]; out[count] = total
__global__ void k_scan_apply(const int32_t* in, int64_t count, const int64_t* boff, int64_t* out) {
    __shared__ int64_t sm[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t e = blockIdx.x * 1024ll + threadIdx.x;
    const int64_t v = e < count ? in[e] : 0;
    int64_t x = v;  // inclusive scan within the warp
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sm[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int64_t s = sm[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        sm[lane] = s;  // inclusive over warps
    }
    __syncthreads();
    const int64_t before = boff[blockIdx.x] + (warp > 0 ? sm[warp - 1] : 0) + x - v;
    if (e < count) out[e] = before;
    if (e == count - 1) out[count] = before + v;
}

}  // namespace

extern "C" int hd_temporal_truncated(hd_ctx* ctx, const hd_graph* g, int32_t B, const int32_t* sl_ptr,
                                     const int32_t* sl_idx, const int32_t* y_ptr, const int32_t* y_idx,
                                     const float* y_val, double alpha, const float* tol, int32_t max_iter, float* X,
                                     int32_t ldx, int32_t* iters, float* relres, int32_t* status) {
    if (!ctx || !g || !sl_ptr || !sl_idx || !y_ptr || !tol || !X || B <= 0 || B > 4096) return HD_ERR_INVALID_ARG;
    HD_CUDA(ctx, cudaSetDevice(ctx->device));
    const int64_t n = g->n;
    // shortlist sizes on the host
    std::vector<int32_t> hp(B + 1);
    if (hd_is_device_ptr(sl_ptr)) {
        HD_CUDA(ctx, cudaMemcpy(hp.data(), sl_ptr, (B + 1) * 4, cudaMemcpyDeviceToHost));
    } else {
        std::copy(sl_ptr, sl_ptr + B + 1, hp.begin());
    }
    int64_t smax = 0;
    for (int j = 0; j < B; ++j) {
        if (hp[j + 1] < hp[j] || hp[j] < 0) return hd_fail(ctx, HD_ERR_INVALID_ARG, "shortlist pointers not monotone");
        smax = std::max<int64_t>(smax, hp[j + 1] - hp[j]);
    }
    if (smax <= 0) return hd_fail(ctx, HD_ERR_INVALID_ARG, "empty shortlists");
    if (smax > n) return hd_fail(ctx, HD_ERR_INVALID_ARG, "shortlist longer than the graph");
    if (ldx < B) return hd_fail(ctx, HD_ERR_INVALID_ARG, "ldx=%d < B=%d", ldx, B);
    const int64_t nsl = hp[B];
    int32_t nnz_y;
    if (hd_is_device_ptr(y_ptr)) {
        HD_CUDA(ctx, cudaMemcpy(&nnz_y, y_ptr + B, 4, cudaMemcpyDeviceToHost));
    } else {
        nnz_y = y_ptr[B];
    }
    if (nnz_y < 0 || (nnz_y > 0 && (!y_idx || !y_val))) return HD_ERR_INVALID_ARG;
    const int64_t rows = (int64_t)B * smax;
    const int64_t nblk = (rows + 1023) / 1024;

    // the systems live in the context's auxiliary workspaces (the solve below uses
    // the main one): [0] everything whose size is known now, [1] the entries
    size_t bytes0 = 0;
    auto part0 = [&](size_t bytes) {
        const size_t at = bytes0;
        bytes0 += ws_size(bytes ? bytes : 16);
        return at;
    };
    auto release = [&]() {
        cudaStreamSynchronize(ctx->stream);
        hd_aux_trim(ctx);
    };
    int rc = HD_OK;
#define TS_TRY(x)         \
    do {                  \
        if ((rc = (x))) { \
            release();    \
            return rc;    \
        }                 \
    } while (0)
#define TS_CUDA(x) TS_TRY(hd_check_cuda(ctx, (x), #x, __FILE__, __LINE__))
#define TS_LAUNCH() TS_TRY(hd_check_launch(ctx, __FILE__, __LINE__))
    int32_t *d_slp, *d_sli, *cnt, *d_yp, *d_yi, *y_loc;
    float *d_yv, *y_lv, *deg, *sdinv;
    int64_t *bsum, *off;
    int* err;
    const size_t at_d_slp = part0((B + 1) * 4);
    const size_t at_d_sli = part0((size_t)nsl * 4);
    // pos, cnt, deg and sdinv are done with when the solve starts, which keeps its
    // transposed operand there (4 bytes a row and padded column)
    const int32_t group = (int32_t)std::max<int64_t>(1, std::min<int64_t>(B, TS_POS_BYTES / (8 * n)));
    const size_t at_pos = part0((size_t)group * n * 8);
    const size_t at_cnt = part0((size_t)rows * 4);
    const size_t at_deg = part0((size_t)rows * 4);
    const size_t at_sdinv = part0((size_t)rows * 4);
    bytes0 = std::max(bytes0, at_pos + ws_size((size_t)smax * ((B + 3) / 4 * 4) * 4));
    const int64_t words = (n + 31) / 32;
    const size_t at_bits = part0((size_t)B * words * 4);
    const size_t at_work = part0((size_t)(B + 1) * sizeof(TruncWork));
    const size_t at_bsum = part0((size_t)nblk * 8);
    const size_t at_off = part0((size_t)(rows + 1) * 8);
    const size_t at_d_yp = part0((B + 1) * 4);
    const size_t at_d_yi = part0((size_t)nnz_y * 4);
    const size_t at_d_yv = part0((size_t)nnz_y * 4);
    const size_t at_y_loc = part0((size_t)nnz_y * 4);
    const size_t at_y_lv = part0((size_t)nnz_y * 4);
    const size_t at_err = part0(16);
    void* aux;
    TS_TRY(hd_aux_reserve(ctx, 0, bytes0, &aux));
    d_slp = (int32_t*)((char*)aux + at_d_slp);
    d_sli = (int32_t*)((char*)aux + at_d_sli);
    int2* pos = (int2*)((char*)aux + at_pos);
    uint32_t* bits = (uint32_t*)((char*)aux + at_bits);
    cnt = (int32_t*)((char*)aux + at_cnt);
    deg = (float*)((char*)aux + at_deg);
    sdinv = (float*)((char*)aux + at_sdinv);
    TruncWork* work = (TruncWork*)((char*)aux + at_work);
    bsum = (int64_t*)((char*)aux + at_bsum);
    off = (int64_t*)((char*)aux + at_off);
    d_yp = (int32_t*)((char*)aux + at_d_yp);
    d_yi = (int32_t*)((char*)aux + at_d_yi);
    d_yv = (float*)((char*)aux + at_d_yv);
    y_loc = (int32_t*)((char*)aux + at_y_loc);
    y_lv = (float*)((char*)aux + at_y_lv);
    err = (int*)((char*)aux + at_err);
    auto copy_in = [&](void* dst, const void* src, size_t bytes) -> int {
        if (!bytes) return HD_OK;
        return hd_check_cuda(ctx, cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, ctx->stream), "copy in",
                             __FILE__, __LINE__);
    };
    TS_TRY(copy_in(d_slp, hp.data(), (B + 1) * 4));
    TS_TRY(copy_in(d_sli, sl_idx, (size_t)nsl * 4));
    TS_TRY(copy_in(d_yp, y_ptr, (B + 1) * 4));
    TS_TRY(copy_in(d_yi, y_idx, (size_t)nnz_y * 4));
    TS_TRY(copy_in(d_yv, y_val, (size_t)nnz_y * 4));
    TS_CUDA(cudaMemsetAsync(err, 0, 16, ctx->stream));
    TS_CUDA(cudaMemsetAsync(bits, 0, (size_t)B * words * 4, ctx->stream));
    if (nsl - hp[0] < rows) {  // rows past a shortlist's end: no entries, degree 0
        TS_CUDA(cudaMemsetAsync(cnt, 0, (size_t)rows * 4, ctx->stream));
        TS_CUDA(cudaMemsetAsync(deg, 0, (size_t)rows * 4, ctx->stream));
    }
    const size_t smem = words <= TS_SMEM_WORDS ? (size_t)words * 4 : 0;
    const unsigned grid = (unsigned)std::min<int64_t>(ctx->num_sms, std::max<int64_t>(B, rows / 256));
    static HdDeviceOnce attr;
    TS_TRY(attr.run(ctx->device, [&]() -> int {
        HD_CUDA(ctx, cudaFuncSetAttribute(k_ts_count, cudaFuncAttributeMaxDynamicSharedMemorySize, TS_SMEM_WORDS * 4));
        HD_CUDA(ctx, cudaFuncSetAttribute(k_ts_fill, cudaFuncAttributeMaxDynamicSharedMemorySize, TS_SMEM_WORDS * 4));
        return HD_OK;
    }));
    {
        HD_PROF(ctx, "trunc_build");
        k_ts_mark<<<dim3((unsigned)((smax + 255) / 256), B), 256, 0, ctx->stream>>>(d_slp, d_sli, g->dinv, n, pos,
                                                                                    group, bits, words, err);
        TS_LAUNCH();
        k_ts_count<<<grid, TS_T, smem, ctx->stream>>>(g->row_ptr, g->col, d_slp, d_sli, B, n, smax, bits, words, cnt);
        TS_LAUNCH();
        k_scan_sums<<<(unsigned)nblk, 1024, 0, ctx->stream>>>(cnt, rows, bsum);
        TS_LAUNCH();
    }
    std::vector<int64_t> hb(nblk);
    TS_CUDA(cudaMemcpyAsync(hb.data(), bsum, (size_t)nblk * 8, cudaMemcpyDeviceToHost, ctx->stream));
    TS_CUDA(cudaMemcpyAsync(ctx->h_poll, err, 4, cudaMemcpyDeviceToHost, ctx->stream));
    TS_CUDA(cudaStreamSynchronize(ctx->stream));
    if (ctx->h_poll[0]) {
        const int e = ctx->h_poll[0];
        release();
        return hd_fail(ctx, HD_ERR_INVALID_ARG, e == 2 ? "duplicate id in a shortlist" : "shortlist id out of range");
    }
    int64_t run = 0;
    for (int64_t b = 0; b < nblk; ++b) {
        const int64_t s = hb[b];
        hb[b] = run;
        run += s;
    }
    const int64_t nnz = run;
    TS_CUDA(cudaMemcpyAsync(bsum, hb.data(), (size_t)nblk * 8, cudaMemcpyHostToDevice, ctx->stream));
    int32_t* ci;
    float* wv;
    TS_TRY(hd_aux_reserve(ctx, 1, 2 * ws_size((size_t)nnz * 4 + 4), &aux));
    ci = (int32_t*)aux;
    wv = (float*)((char*)aux + ws_size((size_t)nnz * 4 + 4));
    {
        HD_PROF(ctx, "trunc_build");
        k_scan_apply<<<(unsigned)nblk, 1024, 0, ctx->stream>>>(cnt, rows, bsum, off);
        TS_LAUNCH();
        for (int32_t j0 = 0; j0 < B; j0 += group) {
            const int32_t cols = std::min(group, B - j0);
            if (j0) {
                k_ts_place<<<dim3((unsigned)((smax + 255) / 256), cols), 256, 0, ctx->stream>>>(d_slp + j0, d_sli,
                                                                                             g->dinv, n, pos);
                TS_LAUNCH();
            }
            k_ts_fill<<<grid, TS_T, smem, ctx->stream>>>(g->row_ptr, g->col, g->val, g->dinv, d_slp + j0, d_sli, cols, n,
                                                         smax, pos, bits + j0 * words, words, off + j0 * smax, ci, wv,
                                                         deg + j0 * smax);
            TS_LAUNCH();
            k_ts_map_y<<<ceil_div(cols, 128), 128, 0, ctx->stream>>>(d_yp + j0, d_yi, d_yv, cols, n, pos,
                                                                    bits + j0 * words, words, y_loc, y_lv, err);
            TS_LAUNCH();
        }
        k_ts_sdinv<<<ceil_div(rows, 256), 256, 0, ctx->stream>>>(deg, rows, sdinv);
        TS_LAUNCH();
        k_ts_scale<<<ceil_div(rows * 8, 256), 256, 0, ctx->stream>>>(off, ci, wv, sdinv, rows, smax);
        TS_LAUNCH();
    }
    TruncSys ts;
    ts.sl_ptr = d_slp;
    ts.work = work;
    for (int j = 0; j < B; ++j) ts.ncol += hp[j + 1] > hp[j];
    ts.off = off;
    ts.ci = ci;
    ts.wv = wv;
    ts.smax = smax;
    ts.vt = (float*)pos;
    rc = hd_query_impl(ctx, g, &ts, nullptr, HD_MODE_PAPER, B, d_yp, y_loc, y_lv, alpha, tol, max_iter, X, ldx, iters,
                       relres, status);
    if (!rc) {
        TS_CUDA(cudaMemcpyAsync(ctx->h_poll, err, 4, cudaMemcpyDeviceToHost, ctx->stream));
        TS_CUDA(cudaStreamSynchronize(ctx->stream));
        if (ctx->h_poll[0]) rc = hd_fail(ctx, HD_ERR_INVALID_ARG, "bad observation: index out of range or non-finite value");
    }
    release();
    return rc;
#undef TS_LAUNCH
#undef TS_CUDA
#undef TS_TRY
}
