// k-NN search and graph construction (Sec. 3; Sec. 5.1).
//
// Similarities s = q^T x are accumulated in fp32: bf16 descriptors on the 5th
// generation tensor cores (tcgen05.mma, TMA-fed shared memory, accumulators in
// TMEM) with the per-row top-k selection fused into the TMEM epilogue, so the
// n x n similarity matrix never leaves the SM; fp32 descriptors on CUDA cores
// (exact fp32 products).  Neighbour lists are ordered by decreasing s, ties to
// the smaller database index; self is excluded when the query set is the
// database.  The graph keeps weight max(s, 0)^gamma, symmetrised (union or
// mutual), then W = D^-1/2 A D^-1/2.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>

#include <cudaTypedefs.h>

#include "hd_internal.cuh"
#include "tc.cuh"

int hd_graph_alloc_internal(hd_ctx* ctx, int64_t n, int64_t nnz, hd_graph** out);
void hd_graph_free_internal(hd_graph* g);

// ------------------------------------------------------------------ tensor maps
int hd_make_tmap_2d(CUtensorMap* map, const void* base, int elem_bytes, uint64_t rows, uint64_t cols,
                    uint64_t ld_elems, uint32_t box_rows, uint32_t box_cols, int swizzle128) {
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        cudaDriverEntryPointQueryResult q;
        void* fn = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn)
            return -1;
        encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    }
    CUtensorMapDataType dt = elem_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                             : elem_bytes == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                                               : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    cuuint64_t gdim[2] = {cols, rows};
    cuuint64_t gstride[1] = {ld_elems * (uint64_t)elem_bytes};
    cuuint32_t box[2] = {box_cols, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = encode(map, dt, 2, const_cast<void*>(base), gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        swizzle128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : -2;
}

constexpr int KMAX = 64;  // neighbours per list

// ------------------------------------------------------------------ top-k selection
// A (similarity, id) pair is one 64-bit key, ordered like the lists (larger
// similarity first, then smaller id); 0 is the empty entry, below every real
// one.  Adding +0 turns -0 into +0, which compares equal to it.
constexpr int KBUF = 64;      // buffered candidates per row
constexpr int KBUF_LD = KBUF + 1;

__device__ __forceinline__ uint64_t knn_key(float s, int64_t id) {
    return ((uint64_t)float_key(s + 0.0f) << 32) | (uint64_t)(~(uint32_t)id);
}
__device__ __forceinline__ float key_sim(uint64_t key) { return key ? key_float((uint32_t)(key >> 32)) : -INFINITY; }
__device__ __forceinline__ int32_t key_id(uint64_t key) { return key ? (int32_t)(~(uint32_t)key) : -1; }

// Warp-wide lists of 64 keys: entry 32 r + lane in register r.
// One compare-exchange with the lane `stride` away; the lane keeps the larger
// key when `up` and the smaller otherwise.
__device__ __forceinline__ uint64_t key_exchange(uint64_t v, int stride, bool up) {
    const uint64_t o = __shfl_xor_sync(0xffffffffu, v, stride);
    return ((v > o) == up) ? v : o;
}
// a bitonic list of 64 -> descending
__device__ __forceinline__ void merge64(uint64_t& c0, uint64_t& c1, int lane) {
    const uint64_t hi = c0 > c1 ? c0 : c1, lo = c0 > c1 ? c1 : c0;
    c0 = hi;
    c1 = lo;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1) {
        c0 = key_exchange(c0, st, !(lane & st));
        c1 = key_exchange(c1, st, !(lane & st));
    }
}
// any list of 64 -> descending (bitonic sort)
__device__ __forceinline__ void sort64(uint64_t& b0, uint64_t& b1, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int st = size >> 1; st > 0; st >>= 1) {
            // register 1 sorts the other way at size 32, which makes the pair bitonic
            const bool d0 = size == 32 ? true : !(lane & size);
            const bool d1 = size == 32 ? false : !(lane & size);
            b0 = key_exchange(b0, st, d0 == !(lane & st));
            b1 = key_exchange(b1, st, d1 == !(lane & st));
        }
    }
    merge64(b0, b1, lane);
}
// the 64 largest keys of two descending lists, descending, into a
__device__ __forceinline__ void take64(uint64_t& a0, uint64_t& a1, uint64_t b0, uint64_t b1, int lane) {
    const uint64_t r1 = __shfl_xor_sync(0xffffffffu, b1, 31), r0 = __shfl_xor_sync(0xffffffffu, b0, 31);
    a0 = a0 > r1 ? a0 : r1;
    a1 = a1 > r0 ? a1 : r0;
    merge64(a0, a1, lane);
}

// Merge a row's `cnt` buffered candidates (shared memory) into its list of 64
// keys (global scratch, descending).  Warp-collective; returns the similarity of
// the k-th entry, -inf while there are fewer.
__device__ __forceinline__ float knn_flush(uint64_t* list, const uint64_t* buf, int cnt, int k, int lane) {
    uint64_t a0 = list[lane], a1 = list[lane + 32];
    uint64_t b0 = lane < cnt ? buf[lane] : 0ull, b1 = lane + 32 < cnt ? buf[lane + 32] : 0ull;
    sort64(b0, b1, lane);
    take64(a0, a1, b0, b1, lane);
    list[lane] = a0;
    list[lane + 32] = a1;
    return key_sim(__shfl_sync(0xffffffffu, k > 32 ? a1 : a0, (k - 1) & 31));
}

// The same for at most 32 candidates held as (similarity bits, id) pairs.
__device__ __forceinline__ float knn_flush32(uint64_t* list, const uint64_t* buf, int cnt, int k, int lane) {
    uint64_t a0 = list[lane], a1 = list[lane + 32];
    uint64_t b = 0ull;
    if (lane < cnt) {
        const uint64_t raw = buf[lane];
        b = knn_key(__uint_as_float((uint32_t)raw), (int64_t)(raw >> 32));
    }
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
        for (int st = size >> 1; st > 0; st >>= 1) b = key_exchange(b, st, (size == 32 || !(lane & size)) == !(lane & st));
    // the list's lower half against the candidates, smallest first: bitonic again
    const uint64_t r = __shfl_xor_sync(0xffffffffu, b, 31);
    a1 = a1 > r ? a1 : r;
    merge64(a0, a1, lane);
    list[lane] = a0;
    list[lane + 32] = a1;
    return key_sim(__shfl_sync(0xffffffffu, k > 32 ? a1 : a0, (k - 1) & 31));
}

// The k best of a query's per-segment lists: one block per query, each warp
// merges every eighth segment, warp 0 the eight results.
__global__ void __launch_bounds__(256) k_knn_merge(const uint64_t* __restrict__ part, int nseg, int64_t nq, int k,
                                                   int32_t* __restrict__ idx_out, float* __restrict__ sim_out) {
    __shared__ uint64_t sh[8][64];
    const int64_t q = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint64_t a0 = 0ull, a1 = 0ull;
    for (int s = warp; s < nseg; s += 8) {
        const uint64_t* p = part + ((int64_t)s * nq + q) * k;
        const uint64_t b0 = lane < k ? __ldg(p + lane) : 0ull, b1 = lane + 32 < k ? __ldg(p + lane + 32) : 0ull;
        take64(a0, a1, b0, b1, lane);
    }
    sh[warp][lane] = a0;
    sh[warp][lane + 32] = a1;
    __syncthreads();
    if (warp) return;
    for (int w = 1; w < 8; ++w) take64(a0, a1, sh[w][lane], sh[w][lane + 32], lane);
    if (lane < k) {
        idx_out[q * k + lane] = key_id(a0);
        sim_out[q * k + lane] = key_sim(a0);
    }
    if (lane + 32 < k) {
        idx_out[q * k + lane + 32] = key_id(a1);
        sim_out[q * k + lane + 32] = key_sim(a1);
    }
}

// ------------------------------------------------------------------ search arguments
// A work item is one block of queries against one segment of the database: all
// of it when there are enough query blocks to fill the GPU, else a share, the
// per-segment lists meeting in k_knn_merge.  Items are numbered with the query
// block fastest, so the blocks of one wave read the same database tiles.
struct KnnArgs {
    int64_t n, nq;
    int d, k, excl;
    int nwork;         // query blocks
    int nseg, tps;     // database segments and tiles per segment
    uint64_t* lists;   // running lists of 64: [gridDim.x][rows of a query block], twice for the bf16 kernel
    uint64_t* part;    // [nseg][nq][k] per-segment results (nseg > 1)
    int32_t* idx_out;  // [nq][k] (nseg == 1)
    float* sim_out;
};

// the final list of a row (entries lane and lane + 32 of each lane): the result
// itself, or the segment's part of it
__device__ __forceinline__ void knn_store(const KnnArgs& a, int seg, int64_t row, uint64_t x0, uint64_t x1, int lane) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        const uint64_t key = h ? x1 : x0;
        if (c >= a.k) continue;
        if (a.nseg > 1) {
            a.part[((int64_t)seg * a.nq + row) * a.k + c] = key;
        } else {
            a.idx_out[row * a.k + c] = key_id(key);
            a.sim_out[row * a.k + c] = key_sim(key);
        }
    }
}

// ------------------------------------------------------------------ fp32 kNN on CUDA cores
// Exact fp32 products: every similarity is one chain of fused multiply-adds in
// the order of the dimensions, whatever the tile.  16 x 16 threads hold a tile
// of 16 TM queries x 128 database rows, TM x 8 per thread (multiply-adds packed
// two by two run at half the rate and need their operand doubled: 15.6 ms for
// 38,912 x 256 against 14.8).  16 dimensions at a time go through
// double-buffered shared memory, loaded into registers one step ahead.
// TM = 8 when there are more than 64 queries; fewer queries take the smallest
// tile that holds them, so that no product is formed for padding.
//
// Bound: the FP32 pipe (127 ms of fused multiply-adds for the lists of 100,000 x
// 512; 210 ms for the whole graph, from 407 ms with a 64 x 64 tile, 4 x 4 per
// thread, and one thread inserting per row; 64 queries against 100,000 x 512:
// 0.40 ms, from 101.5 ms on one SM).  Candidates above a row's threshold are
// appended to 64 slots of shared memory (32 columns of a row at a time), merged
// as in k_knn_tc.
namespace knnf {
constexpr int BN = 128;      // database rows per tile
constexpr int FK = 16;       // dimensions per step
constexpr int BLD = BN + 4;  // leading dimension of the transposed tiles (16-byte rows)
template <int TM>
struct Cfg {
    static constexpr int BM = 16 * TM;
    static constexpr int ALD = BM + 4;
    static constexpr int AV = (BM * FK / 4 + 255) / 256;  // float4 loads per thread and step
    static constexpr size_t SMEM = 2 * (size_t)FK * (ALD + BLD) * 4 + (size_t)BM * KBUF_LD * 8 + BM * 12;
};

// four dimensions of one row (zero past the end)
__device__ __forceinline__ float4 load4(const float* p, int64_t row, int64_t rows, int d, int c, bool vec) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row >= rows || c >= d) return v;
    const float* q = p + row * d + c;
    if (vec) return __ldg(reinterpret_cast<const float4*>(q));
    v.x = __ldg(q);
    if (c + 1 < d) v.y = __ldg(q + 1);
    if (c + 2 < d) v.z = __ldg(q + 2);
    if (c + 3 < d) v.w = __ldg(q + 3);
    return v;
}
__device__ __forceinline__ void put4(float* t, int ld, int c, int r, float4 v) {
    t[c * ld + r] = v.x;
    t[(c + 1) * ld + r] = v.y;
    t[(c + 2) * ld + r] = v.z;
    t[(c + 3) * ld + r] = v.w;
}
// the tile row of a thread's i-th query: groups of four rows, 64 apart
template <int TM>
__device__ __forceinline__ int tile_row(int ty, int i) {
    return TM >= 4 ? (i >> 2) * 64 + ty * 4 + (i & 3) : ty * TM + i;
}
__device__ __forceinline__ int tile_col(int tx, int j) { return (j >> 2) * 64 + tx * 4 + (j & 3); }
}  // namespace knnf

template <int TM>
__global__ void __launch_bounds__(256, 2)
    k_knn_f32(const float* __restrict__ X, const float* __restrict__ Q, const KnnArgs a, const int vec) {
    using namespace knnf;
    using C = Cfg<TM>;
    constexpr int BM = C::BM, ALD = C::ALD, AV = C::AV;
    extern __shared__ __align__(16) uint8_t smem_f[];
    float* As = reinterpret_cast<float*>(smem_f);           // [2][FK][ALD]
    float* Bs = As + 2 * FK * ALD;                          // [2][FK][BLD]
    uint64_t* bufs = reinterpret_cast<uint64_t*>(Bs + 2 * FK * BLD);  // [BM][KBUF_LD]
    float* tau = reinterpret_cast<float*>(bufs + BM * KBUF_LD);       // [BM]
    float* kth = tau + BM;                                            // [BM]
    int* cnt = reinterpret_cast<int*>(kth + BM);                      // [BM]
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, warp = tid >> 5, lane = tid & 31;
    const int ntile = (int)((a.n + BN - 1) / BN), nk = (a.d + FK - 1) / FK, nitem = a.nwork * a.nseg;
    uint64_t* lists = a.lists + (int64_t)blockIdx.x * BM * 64;

    for (int item = blockIdx.x; item < nitem; item += gridDim.x) {
        const int w = item % a.nwork, seg = item / a.nwork, t0 = seg * a.tps, t1 = min(ntile, t0 + a.tps);
        const int64_t q0 = (int64_t)w * BM;
        for (int r = warp; r < BM; r += 8) {
            lists[r * 64 + lane] = 0ull;
            lists[r * 64 + lane + 32] = 0ull;
        }
        if (tid < BM) {
            tau[tid] = kth[tid] = q0 + tid < a.nq ? -INFINITY : INFINITY;  // a row past the last query takes nothing
            cnt[tid] = 0;
        }
        float4 ar[AV], br[2];
        auto fetch = [&](int t, int kc) {
#pragma unroll
            for (int u = 0; u < AV; ++u) {
                const int e = tid + u * 256;
                if (BM * FK / 4 >= 256 || e < BM * FK / 4) ar[u] = load4(Q, q0 + (e >> 2), a.nq, a.d, kc * FK + (e & 3) * 4, vec);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int e = tid + u * 256;
                br[u] = load4(X, (int64_t)t * BN + (e >> 2), a.n, a.d, kc * FK + (e & 3) * 4, vec);
            }
        };
        auto stash = [&](int b) {
#pragma unroll
            for (int u = 0; u < AV; ++u) {
                const int e = tid + u * 256;
                if (BM * FK / 4 >= 256 || e < BM * FK / 4) put4(As + b * FK * ALD, ALD, (e & 3) * 4, e >> 2, ar[u]);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int e = tid + u * 256;
                put4(Bs + b * FK * BLD, BLD, (e & 3) * 4, e >> 2, br[u]);
            }
        };
        fetch(t0, 0);
        stash(0);
        __syncthreads();
        int b = 0;
        for (int t = t0; t < t1; ++t) {
            float acc[TM][8];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
            for (int kc = 0; kc < nk; ++kc, b ^= 1) {
                const bool more = kc + 1 < nk || t + 1 < t1;
                if (more) fetch(kc + 1 < nk ? t : t + 1, kc + 1 < nk ? kc + 1 : 0);
                const float* at = As + b * FK * ALD;
                const float* bt = Bs + b * FK * BLD + tx * 4;
#pragma unroll
                for (int c = 0; c < FK; ++c) {
                    const float4 b0 = *reinterpret_cast<const float4*>(bt + c * BLD);
                    const float4 b1 = *reinterpret_cast<const float4*>(bt + c * BLD + 64);
                    float av[TM];
#pragma unroll
                    for (int i = 0; i < TM; i += 4) {
                        const float* p = at + c * ALD + tile_row<TM>(ty, i);
                        if constexpr (TM >= 4) {
                            const float4 v = *reinterpret_cast<const float4*>(p);
                            av[i] = v.x;
                            av[i + 1] = v.y;
                            av[i + 2] = v.z;
                            av[i + 3] = v.w;
                        } else {
#pragma unroll
                            for (int u = 0; u < TM; ++u) av[u] = p[u];
                        }
                    }
#pragma unroll
                    for (int i = 0; i < TM; ++i) {
                        const float bb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
                        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(av[i], bb[j], acc[i][j]);
                    }
                }
                if (more) stash(b ^ 1);
                __syncthreads();
            }
            // ---- candidates of this tile, 32 columns of every row at a time: what lies
            // above the threshold, which starts at the k-th similarity so far.  The four
            // steps interleave their columns, so a step can meet an id smaller than one
            // that an earlier step of this tile put in the list; a merge in mid-tile
            // therefore leaves the threshold just below the new k-th similarity, equals
            // are taken too and the lists' order decides (a comparison of ids per
            // candidate instead cost 1 to 5% of the kernel)
            bool merged = false;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                int most = 0;
                const int64_t id0 = (int64_t)t * BN + tile_col(tx, 2 * j);
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    const int r = tile_row<TM>(ty, i);
                    const float th = tau[r];
                    const float v[2] = {acc[i][2 * j], acc[i][2 * j + 1]};
#pragma unroll
                    for (int u = 0; u < 2; ++u)
                        if (v[u] > th && id0 + u < a.n && !(a.excl && id0 + u == q0 + r)) {
                            const int p = atomicAdd(&cnt[r], 1);
                            bufs[r * KBUF_LD + p] = knn_key(v[u], id0 + u);
                            most = max(most, p + 1);
                        }
                }
                if (__syncthreads_or(most > KBUF - 32)) {
                    merged = true;
                    for (int r = warp; r < BM; r += 8) {
                        const int rc = cnt[r];
                        __syncwarp();
                        if (rc <= KBUF - 32) continue;
                        const float s = knn_flush(lists + r * 64, bufs + r * KBUF_LD, rc, a.k, lane);
                        if (lane == 0) {
                            kth[r] = s;
                            tau[r] = nextafterf(s, -INFINITY);
                            cnt[r] = 0;
                        }
                    }
                    __syncthreads();
                }
            }
            if (merged && tid < BM) tau[tid] = kth[tid];  // (read again after the next tile's barriers)
        }
        __syncthreads();
        for (int r = warp; r < BM; r += 8) {
            if (q0 + r >= a.nq) break;
            if (cnt[r] > 0) knn_flush(lists + r * 64, bufs + r * KBUF_LD, cnt[r], a.k, lane);
            knn_store(a, seg, q0 + r, lists[r * 64 + lane], lists[r * 64 + lane + 32], lane);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ bf16 tcgen05 kNN
// 128 queries x 256 database rows per tile, items as above.
//
// Bound: the tensor cores when there are many queries, the stream of the
// database when there are few (64 queries against 1M x 2048: 0.80 ms for the
// whole observation, 0.60 ms at the copy bandwidth; 43.4 ms with one block per
// query block).
//
// Selection: two epilogue threads per query row, each with half of a tile's
// columns and a list of its own (merged at the end of the item).  A thread keeps
// a threshold (its k-th best so far, from the last merge); what beats it is
// appended to 32 slots of shared memory by predicated stores, 16 columns at a
// time, and when a row holds more than 16 its warp sorts them and merges them
// into the row's list by shuffles.  With one or two warps per scheduler the
// epilogue lives off straight-line code: the lists of 250,000 x 512 at k = 50
// take 47 ms, 34 at the tensor cores' rate; with one thread per row and a branch
// per column it took 73 ms, bound by the epilogue at any depth, and with every
// insertion a walk of the list in global memory 409 ms.  (Reading a chunk ahead
// from TMEM gains nothing: 49 ms.)
namespace knntc {
constexpr int BM = 128, BN = 256, BK = 64, STAGES = 3;
constexpr int A_BYTES = BM * BK * 2;   // 16 KB
constexpr int B_BYTES = BN * BK * 2;   // 32 KB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int CHUNK = 16;            // columns between two looks at the buffers
constexpr int TBUF = 32, TBUF_LD = TBUF + 1;
constexpr int BUF_BYTES = 2 * BM * TBUF_LD * 8;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + BUF_BYTES + 1024 + 256;
constexpr int EPI = 256;             // epilogue threads: two per query row
constexpr int THREADS = 64 + EPI;
}  // namespace knntc

__global__ void __launch_bounds__(knntc::THREADS, 1)
    k_knn_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmX, const KnnArgs a,
             int* __restrict__ err) {
    using namespace knntc;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* bufs = (uint64_t*)(smem + STAGES * STAGE_BYTES);  // [2][128][TBUF_LD]
    uint64_t* full = bufs + 2 * BM * TBUF_LD;
    uint64_t* empty = full + STAGES;
    uint64_t* acc_full = empty + STAGES;
    uint64_t* acc_empty = acc_full + 2;
    uint64_t* drain = acc_empty + 2;
    uint32_t* tmem_slot = (uint32_t*)(drain + 1);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nkb = (a.d + BK - 1) / BK;
    const int ntile = (int)((a.n + BN - 1) / BN);
    const int nitem = a.nwork * a.nseg;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&acc_full[b], 1);
            tc::mbar_init(&acc_empty[b], EPI);
        }
        tc::mbar_init(drain, 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
    }
    if (warp == 1) tc::tmem_alloc<512>(tmem_slot);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ---------------- TMA producer
        if (lane == 0) {
            tc::prefetch_tmap(&tmQ);
            tc::prefetch_tmap(&tmX);
            uint32_t it = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < nitem && ok; item += gridDim.x) {
                const int w = item % a.nwork, t0 = item / a.nwork * a.tps, t1 = min(ntile, t0 + a.tps);
                for (int t = t0; t < t1 && ok; ++t)
                    for (int kb = 0; kb < nkb; ++kb, ++it) {
                        int s = it % STAGES;
                        uint32_t ph = (it / STAGES) & 1;
                        if (!tc::mbar_wait(&empty[s], ph ^ 1, abort_flag)) {
                            ok = false;
                            break;
                        }
                        uint8_t* sa = smem + s * STAGE_BYTES;
                        tc::mbar_arrive_expect_tx(&full[s], STAGE_BYTES);
                        tc::tma_load_2d(sa, &tmQ, &full[s], kb * BK, w * BM);
                        tc::tma_load_2d(sa + A_BYTES, &tmX, &full[s], kb * BK, t * BN);
                    }
            }
            if (!ok) {
                *abort_flag = 1;
                atomicExch(err, 1);
            }
            // drain: the latest load issued into each stage must land before the CTA may exit
            for (uint32_t j = 0; j < (uint32_t)STAGES && j < it; ++j) {
                uint32_t last = it - 1 - j;
                tc::mbar_wait(&full[last % STAGES], (last / STAGES) & 1, nullptr, 200000000ull);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer
        if (lane == 0) {
            constexpr uint32_t IDESC = tc::idesc_bf16(BM, BN, 0, 0);
            uint32_t it = 0, tcount = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < nitem && ok; item += gridDim.x) {
                const int t0 = item / a.nwork * a.tps, t1 = min(ntile, t0 + a.tps);
                for (int t = t0; t < t1 && ok; ++t, ++tcount) {
                    int ab = tcount & 1;
                    uint32_t aph = (tcount >> 1) & 1;
                    if (!tc::mbar_wait(&acc_empty[ab], aph ^ 1, abort_flag)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after_sync();
                    uint32_t dt = tmem + ab * BN;
                    for (int kb = 0; kb < nkb; ++kb, ++it) {
                        int s = it % STAGES;
                        uint32_t ph = (it / STAGES) & 1;
                        if (!tc::mbar_wait(&full[s], ph, abort_flag)) {
                            ok = false;
                            break;
                        }
                        tc::fence_after_sync();
                        uint32_t sa = tc::smem_u32(smem + s * STAGE_BYTES);
                        uint32_t sb = sa + A_BYTES;
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
                            uint64_t ad = tc::smem_desc(sa + kk * 32, 16, 1024, tc::SWIZZLE_128B);
                            uint64_t bd = tc::smem_desc(sb + kk * 32, 16, 1024, tc::SWIZZLE_128B);
                            tc::mma_bf16(dt, ad, bd, IDESC, (kb | kk) ? 1u : 0u);
                        }
                        tc::mma_commit(&empty[s]);
                    }
                    if (ok) tc::mma_commit(&acc_full[ab]);
                }
            }
            if (!ok) {
                *abort_flag = 1;
                atomicExch(err, 2);
                // wait for every MMA this thread issued before TMEM is released
                tc::mma_commit(drain);
                tc::mbar_wait(drain, 0, nullptr, 200000000ull);
            }
        }
    } else {
        // ---------------- epilogue: warps 2..9; the TMEM lanes (rows) of a warp are
        // those of its quarter, its columns those of its half
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        uint64_t* lists = a.lists + (((int64_t)blockIdx.x * 2 + half) * BM + quarter * 32) * 64;  // this warp's 32 rows
        uint64_t* wbuf = bufs + (half * BM + quarter * 32) * TBUF_LD;
        const uint32_t slot0 = tc::smem_u32(wbuf + lane * TBUF_LD);
        uint32_t tcount = 0;
        bool ok = true;
        for (int item = blockIdx.x; item < nitem && ok; item += gridDim.x) {
            const int w = item % a.nwork, seg = item / a.nwork, t0 = seg * a.tps, t1 = min(ntile, t0 + a.tps);
            const int64_t row0 = (int64_t)w * BM + quarter * 32, row = row0 + lane;
            for (int c = lane; c < 32 * 64; c += 32) lists[c] = 0ull;
            float tau = row < a.nq ? -INFINITY : INFINITY;  // a row past the last query takes nothing
            uint32_t slot = slot0;
            for (int t = t0; t < t1; ++t, ++tcount) {
                int ab = tcount & 1;
                uint32_t aph = (tcount >> 1) & 1;
                // one answer per warp: the collectives below need every lane
                if (!__all_sync(0xffffffffu, tc::mbar_wait(&acc_full[ab], aph, abort_flag))) {
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16) + ab * BN + half * (BN / 2);
#pragma unroll 1
                for (int c = 0; c < BN / 2; c += CHUNK) {
                    float v[CHUNK];
                    tc::tmem_ld16(acc + c, v);
                    tc::tmem_ld_wait16(v);
                    const int64_t base = (int64_t)t * BN + half * (BN / 2) + c;
                    // columns past the database, and the row itself, take no part
                    if (base + CHUNK > a.n) {
#pragma unroll
                        for (int i = 0; i < CHUNK; ++i)
                            if (base + i >= a.n) v[i] = -INFINITY;
                    }
                    if (a.excl && base >> 5 == row0 >> 5) {
#pragma unroll
                        for (int i = 0; i < CHUNK; ++i)
                            if (base + i == row) v[i] = -INFINITY;
                    }
                    float m[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
                    for (int i = 4; i < CHUNK; ++i) m[i & 3] = fmaxf(m[i & 3], v[i]);
                    if (__any_sync(0xffffffffu, fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])) > tau)) {
#pragma unroll
                        for (int i = 0; i < CHUNK; ++i)
                            asm volatile(
                                "{\n .reg .pred p;\n setp.gt.f32 p, %1, %2;\n"
                                " @p st.shared.v2.b32 [%0], {%3, %4};\n @p add.u32 %0, %0, 8;\n}"
                                : "+r"(slot)
                                : "f"(v[i]), "f"(tau), "r"(__float_as_uint(v[i])), "r"((uint32_t)(base + i))
                                : "memory");
                        const int cnt = (int)(slot - slot0) >> 3;
                        unsigned need = __ballot_sync(0xffffffffu, cnt > TBUF - CHUNK);
                        if (need) {
                            __syncwarp();
                            while (need) {
                                const int r = __ffs(need) - 1;
                                need &= need - 1;
                                const float th = knn_flush32(lists + r * 64, wbuf + r * TBUF_LD,
                                                             __shfl_sync(0xffffffffu, cnt, r), a.k, lane);
                                if (lane == r) {
                                    tau = th;
                                    slot = slot0;
                                }
                            }
                            __syncwarp();
                        }
                    }
                }
                tc::fence_before_sync();
                tc::mbar_arrive(&acc_empty[ab]);
            }
            if (!ok) {
                *abort_flag = 1;
                atomicExch(err, 3);
            }
            __syncwarp();
            const int left = (int)(slot - slot0) >> 3;
            for (int r = 0; r < 32; ++r) {
                const int rc = __shfl_sync(0xffffffffu, left, r);
                if (rc > 0) knn_flush32(lists + r * 64, wbuf + r * TBUF_LD, rc, a.k, lane);
            }
            // the two halves of a row meet: each warp stores 16 rows of its quarter
            asm volatile("bar.sync 1, %0;" ::"n"(EPI) : "memory");
            const uint64_t* other = a.lists + (((int64_t)blockIdx.x * 2 + (half ^ 1)) * BM + quarter * 32) * 64;
            for (int r = 16 * half; r < 16 * half + 16; ++r) {
                if (row0 + r >= a.nq) break;
                uint64_t x0 = lists[r * 64 + lane], x1 = lists[r * 64 + lane + 32];
                take64(x0, x1, other[r * 64 + lane], other[r * 64 + lane + 32], lane);
                knn_store(a, seg, row0 + r, x0, x1, lane);
            }
            // one answer for all eight warps: the flag may rise between two warps' reads of
            // it, and a warp that went on alone would wait at the next barrier for ever
            ok = !tc::bar_any<1, EPI>(!ok || *abort_flag);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc<512>(tmem);
    }
}

// ------------------------------------------------------------------ launch plan
// Query blocks of `bm` rows against `ntile` database tiles on `slots` resident
// blocks: the number of database segments that gives the shortest schedule, an
// item costing its tiles plus about `fixed` tiles of start-up (thresholds that
// start at -inf let more candidates through, plus the merge).  More segments
// than 304 or more than 16,384 keys per query to merge are not considered.
struct KnnPlan {
    int nwork, nseg, tps, grid;
};
static KnnPlan knn_plan(int64_t nq, int64_t ntile, int bm, int slots, int k, int fixed) {
    KnnPlan p;
    p.nwork = ceil_div(nq, bm);
    const int most = (int)std::min<int64_t>(std::min<int64_t>(ntile, 304), 16384 / k);
    int64_t best = INT64_MAX;
    for (int s = 1; s <= most; ++s) {
        const int64_t tps = (ntile + s - 1) / s;
        if (s > 1 && (ntile + tps - 1) / tps < s) continue;  // a segment without tiles
        const int64_t cost = (((int64_t)p.nwork * s + slots - 1) / slots) * (tps + (s > 1 ? fixed : 0));
        if (cost < best) {
            best = cost;
            p.nseg = s;
            p.tps = (int)tps;
        }
    }
    p.grid = (int)std::min<int64_t>((int64_t)p.nwork * p.nseg, slots);
    return p;
}
// queries per thread of the fp32 kernel: the smallest tile that holds them all
static int knn_f32_tm(int64_t nq) { return nq <= 16 ? 1 : nq <= 32 ? 2 : nq <= 64 ? 4 : 8; }
static int knn_bm(int64_t nq, int dtype) { return dtype == HD_F32 ? 16 * knn_f32_tm(nq) : knntc::BM; }
static KnnPlan knn_plan_for(const hd_ctx* ctx, int64_t n, int64_t nq, int k, int dtype) {
    if (dtype == HD_F32)
        return knn_plan(nq, (n + knnf::BN - 1) / knnf::BN, knn_bm(nq, dtype), 2 * ctx->num_sms, k, 2);
    return knn_plan(nq, (n + knntc::BN - 1) / knntc::BN, knntc::BM, ctx->num_sms, k, 4);
}

static size_t knn_list_keys(const KnnPlan& p, int64_t nq, int dtype) {
    return (size_t)p.grid * knn_bm(nq, dtype) * (dtype == HD_BF16 ? 2 : 1) * 64;
}

// Workspace bytes hd_knn_impl needs for a search (its `scratch`).
static size_t knn_scratch_bytes(const hd_ctx* ctx, int64_t n, int64_t nq, int32_t k, int dtype) {
    if (k < 1 || k > KMAX || nq <= 0 || n <= 0) return 256;
    const KnnPlan p = knn_plan_for(ctx, n, nq, k, dtype);
    return ws_size(knn_list_keys(p, nq, dtype) * 8) + (p.nseg > 1 ? ws_size((size_t)p.nseg * nq * k * 8) : 0);
}

// Enqueue a search on the context's stream; `scratch` holds knn_scratch_bytes.
// The caller synchronises and then reads the wait status with hd_knn_status.
static int hd_knn_impl(hd_ctx* ctx, const void* Xd, int64_t n, int32_t d, int dtype, const void* Qd, int64_t nq,
                       int32_t k, int exclude_self, int32_t* idx_d, float* sim_d, void* scratch) {
    ctx->h_poll[1] = 0;
    if (k < 1 || k > KMAX) return hd_fail(ctx, HD_ERR_INVALID_ARG, "k=%d outside [1, %d]", k, KMAX);
    if (nq <= 0 || n <= 0) return HD_OK;
    if (dtype != HD_F32 && dtype != HD_BF16) return hd_fail(ctx, HD_ERR_INVALID_ARG, "dtype %d", dtype);
    if (dtype == HD_BF16 && d % 8)
        return hd_fail(ctx, HD_ERR_INVALID_ARG, "bf16 descriptors need d %% 8 == 0 (d=%d)", d);
    const KnnPlan p = knn_plan_for(ctx, n, nq, k, dtype);
    KnnArgs a;
    a.n = n;
    a.nq = nq;
    a.d = d;
    a.k = k;
    a.excl = exclude_self;
    a.nwork = p.nwork;
    a.nseg = p.nseg;
    a.tps = p.tps;
    WsCarver cv(scratch);
    a.lists = cv.take<uint64_t>(knn_list_keys(p, nq, dtype));
    a.part = p.nseg > 1 ? cv.take<uint64_t>((size_t)p.nseg * nq * k) : nullptr;
    a.idx_out = idx_d;
    a.sim_out = sim_d;
    HD_PROF(ctx, "knn");
    if (dtype == HD_F32) {
        // float4 loads need 16-byte rows
        const int vec = d % 4 == 0 && ((uintptr_t)Xd & 15) == 0 && ((uintptr_t)Qd & 15) == 0;
        static HdDeviceOnce attr_f;
        if (const int ra = attr_f.run(ctx->device, [&]() -> int {
            HD_CUDA(ctx, cudaFuncSetAttribute(k_knn_f32<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)knnf::Cfg<1>::SMEM));
            HD_CUDA(ctx, cudaFuncSetAttribute(k_knn_f32<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)knnf::Cfg<2>::SMEM));
            HD_CUDA(ctx, cudaFuncSetAttribute(k_knn_f32<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)knnf::Cfg<4>::SMEM));
            HD_CUDA(ctx, cudaFuncSetAttribute(k_knn_f32<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)knnf::Cfg<8>::SMEM));
            return HD_OK;
        })) return ra;
        const float *X = (const float*)Xd, *Q = (const float*)Qd;
        switch (knn_f32_tm(nq)) {
            case 1: k_knn_f32<1><<<p.grid, 256, knnf::Cfg<1>::SMEM, ctx->stream>>>(X, Q, a, vec); break;
            case 2: k_knn_f32<2><<<p.grid, 256, knnf::Cfg<2>::SMEM, ctx->stream>>>(X, Q, a, vec); break;
            case 4: k_knn_f32<4><<<p.grid, 256, knnf::Cfg<4>::SMEM, ctx->stream>>>(X, Q, a, vec); break;
            default: k_knn_f32<8><<<p.grid, 256, knnf::Cfg<8>::SMEM, ctx->stream>>>(X, Q, a, vec); break;
        }
        HD_CHECK_LAUNCH(ctx);
    } else {
        using namespace knntc;
        CUtensorMap tq, tx;
        if (hd_make_tmap_2d(&tq, Qd, 2, nq, d, d, BM, BK, 1) || hd_make_tmap_2d(&tx, Xd, 2, n, d, d, BN, BK, 1))
            return hd_fail(ctx, HD_ERR_CUDA, "cuTensorMapEncodeTiled failed");
        static HdDeviceOnce attr;
        if (const int ra = attr.run(ctx->device, [&]() -> int {
            HD_CUDA(ctx, cudaFuncSetAttribute(k_knn_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
            return HD_OK;
        })) return ra;
        HD_CUDA(ctx, cudaMemsetAsync(ctx->d_flags + 1, 0, sizeof(int), ctx->stream));
        k_knn_tc<<<p.grid, THREADS, SMEM_BYTES, ctx->stream>>>(tq, tx, a, ctx->d_flags + 1);
        HD_CHECK_LAUNCH(ctx);
        HD_CUDA(ctx, cudaMemcpyAsync(ctx->h_poll + 1, ctx->d_flags + 1, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    }
    if (p.nseg > 1) {
        k_knn_merge<<<(unsigned)nq, 256, 0, ctx->stream>>>(a.part, p.nseg, nq, k, idx_d, sim_d);
        HD_CHECK_LAUNCH(ctx);
    }
    return HD_OK;
}

// after a synchronisation: did the search's bounded waits all end?
static int hd_knn_status(hd_ctx* ctx) {
    if (ctx->h_poll[1]) return hd_fail(ctx, HD_ERR_TIMEOUT, "k-NN tensor-core pipeline wait timed out (%d)", ctx->h_poll[1]);
    return HD_OK;
}

// ------------------------------------------------------------------ symmetrisation
__device__ __forceinline__ float edge_weight(float s, float gamma) {
    float m = fmaxf(s, 0.0f);
    return gamma == 3.0f ? m * m * m : powf(m, gamma);
}

// For each directed entry i -> j: is i in j's list (reciprocal), and j's weight for it.
__global__ void k_recip(const int32_t* idx, const float* sim, int64_t n, int k, float gamma, int8_t* recip,
                        float* wrev, int32_t* extra) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n * k) return;
    int64_t i = e / k;
    int32_t j = idx[e];
    float w = j >= 0 ? edge_weight(sim[e], gamma) : 0.0f;
    int8_t found = 0;
    float wr = 0.0f;
    if (j >= 0 && w > 0.0f) {
        for (int u = 0; u < k; ++u)
            if (idx[(int64_t)j * k + u] == (int32_t)i) {
                float w2 = edge_weight(sim[(int64_t)j * k + u], gamma);
                if (w2 > 0.0f) {
                    found = 1;
                    wr = w2;
                }
                break;
            }
        if (!found) atomicAdd(&extra[j], 1);
    }
    recip[e] = found;
    wrev[e] = wr;
}

__global__ void k_rowlen(const int32_t* idx, const float* sim, const int8_t* recip, const int32_t* extra, int64_t n,
                         int k, float gamma, int sym, int32_t* len, int32_t* own) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int c = 0;
    for (int u = 0; u < k; ++u) {
        int64_t e = i * k + u;
        bool valid = idx[e] >= 0 && edge_weight(sim[e], gamma) > 0.0f;
        if (valid && (sym == HD_SYM_UNION || recip[e])) ++c;
    }
    own[i] = c;
    len[i] = c + (sym == HD_SYM_UNION ? extra[i] : 0);
}

__global__ void k_fill(const int32_t* idx, const float* sim, const int8_t* recip, const float* wrev,
                       const int32_t* row_ptr, const int32_t* own, int32_t* cursor, int64_t n, int k, float gamma,
                       int sym, int32_t* col, float* val) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int32_t pos = row_ptr[i];
    for (int u = 0; u < k; ++u) {
        int64_t e = i * k + u;
        int32_t j = idx[e];
        float w = j >= 0 ? edge_weight(sim[e], gamma) : 0.0f;
        if (!(w > 0.0f)) continue;
        if (recip[e]) {
            col[pos] = j;
            val[pos] = sym == HD_SYM_UNION ? fmaxf(w, wrev[e]) : fminf(w, wrev[e]);
            ++pos;
        } else if (sym == HD_SYM_UNION) {
            col[pos] = j;
            val[pos] = w;
            ++pos;
            int32_t q = row_ptr[j] + own[j] + atomicAdd(&cursor[j], 1);
            col[q] = (int32_t)i;
            val[q] = w;
        }
    }
}

int hd_graph_from_lists(hd_ctx* ctx, int64_t n, int32_t k, const int32_t* idx_d, const float* sim_d, float gamma,
                        int sym, hd_graph** out) {
    size_t nk = (size_t)n * k;
    // temporaries: the context's second auxiliary block (the neighbour lists are in the first)
    void* aux;
    int rc = hd_aux_reserve(ctx, 1, ws_size(nk) + ws_size(nk * 4) + 4 * ws_size(n * 4), &aux);
    if (rc) return rc;
    WsCarver cv(aux);
    int8_t* recip = cv.take<int8_t>(nk);
    float* wrev = cv.take<float>(nk);
    int32_t *extra = cv.take<int32_t>(n), *len = cv.take<int32_t>(n), *own = cv.take<int32_t>(n), *cursor = cv.take<int32_t>(n);
    HD_CUDA(ctx, cudaMemsetAsync(extra, 0, n * 4, ctx->stream));
    HD_CUDA(ctx, cudaMemsetAsync(cursor, 0, n * 4, ctx->stream));
    k_recip<<<ceil_div(nk, 256), 256, 0, ctx->stream>>>(idx_d, sim_d, n, k, gamma, recip, wrev, extra);
    HD_CHECK_LAUNCH(ctx);
    k_rowlen<<<ceil_div(n, 256), 256, 0, ctx->stream>>>(idx_d, sim_d, recip, extra, n, k, gamma, sym, len, own);
    HD_CHECK_LAUNCH(ctx);
    std::vector<int32_t> h_len(n), h_ptr(n + 1);
    HD_CUDA(ctx, cudaMemcpyAsync(h_len.data(), len, n * 4, cudaMemcpyDeviceToHost, ctx->stream));
    HD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    int64_t acc = 0;
    int32_t longest = 0;
    for (int64_t i = 0; i < n; ++i) {
        h_ptr[i] = (int32_t)acc;
        acc += h_len[i];
        longest = std::max(longest, h_len[i]);
    }
    h_ptr[n] = (int32_t)acc;
    if (acc >= (1ll << 31)) return hd_fail(ctx, HD_ERR_INVALID_ARG, "graph too large: nnz=%lld", (long long)acc);
    hd_graph* g;
    rc = hd_graph_alloc_internal(ctx, n, acc, &g);
    if (rc) return rc;
    HD_CUDA(ctx, cudaMemcpyAsync(g->row_ptr, h_ptr.data(), (n + 1) * 4, cudaMemcpyHostToDevice, ctx->stream));
    k_fill<<<ceil_div(n, 256), 256, 0, ctx->stream>>>(idx_d, sim_d, recip, wrev, g->row_ptr, own, cursor, n, k, gamma,
                                                      sym, g->col, g->val);
    HD_CHECK_LAUNCH(ctx);
    rc = hd_sort_rows(ctx, g->row_ptr, g->col, g->val, n, longest);
    if (!rc) rc = hd_normalize_graph(ctx, g);
    const int rs = hd_check_cuda(ctx, cudaStreamSynchronize(ctx->stream), "graph", __FILE__, __LINE__);
    if (!rc) rc = rs;
    if (rc) {
        hd_graph_free_internal(g);
        return rc;
    }
    *out = g;
    return HD_OK;
}

// ------------------------------------------------------------------ C ABI
static int stage_matrix(hd_ctx* ctx, const void* p, size_t bytes, void** owned, const void** dev) {
    *owned = nullptr;
    if (hd_is_device_ptr(p)) {
        *dev = p;
        return HD_OK;
    }
    HD_CUDA(ctx, cudaMalloc(owned, bytes));
    HD_CUDA(ctx, cudaMemcpyAsync(*owned, p, bytes, cudaMemcpyHostToDevice, ctx->stream));
    *dev = *owned;
    return HD_OK;
}

extern "C" {

int hd_knn(hd_ctx* ctx, const void* X, int64_t n, int32_t d, int dtype, const void* Q, int64_t nq, int32_t k,
           int exclude_self, int32_t* idx_out, float* sim_out) {
    if (!ctx || !X || !Q || !idx_out || !sim_out || n <= 0 || nq <= 0 || d <= 0) return HD_ERR_INVALID_ARG;
    if (dtype != HD_F32 && dtype != HD_BF16) return hd_fail(ctx, HD_ERR_INVALID_ARG, "dtype %d", dtype);
    if (k < 1 || k > KMAX) return hd_fail(ctx, HD_ERR_INVALID_ARG, "k=%d outside [1, %d]", k, KMAX);
    HD_CUDA(ctx, cudaSetDevice(ctx->device));
    size_t es = dtype == HD_F32 ? 4 : 2;
    void *ox, *oq;
    const void *xd, *qd;
    int rc = stage_matrix(ctx, X, (size_t)n * d * es, &ox, &xd);
    if (!rc) rc = stage_matrix(ctx, Q, (size_t)nq * d * es, &oq, &qd);
    if (rc) return rc;
    // results that go to the host pass through the workspace, behind the search's own part of it
    const bool dev_out = hd_is_device_ptr(idx_out) && hd_is_device_ptr(sim_out);
    const size_t need = knn_scratch_bytes(ctx, n, nq, k, dtype), out_bytes = (size_t)nq * k * 4;
    void* ws = nullptr;
    rc = hd_ws_reserve(ctx, ws_size(need) + (dev_out ? 0 : 2 * ws_size(out_bytes)), &ws);
    if (!rc) {
        int32_t* idd = dev_out ? idx_out : (int32_t*)((char*)ws + ws_size(need));
        float* sdd = dev_out ? sim_out : (float*)((char*)ws + ws_size(need) + ws_size(out_bytes));
        rc = hd_knn_impl(ctx, xd, n, d, dtype, qd, nq, k, exclude_self, idd, sdd, ws);
        if (!rc && !dev_out)
            rc = hd_check_cuda(ctx, cudaMemcpyAsync(idx_out, idd, out_bytes, cudaMemcpyDefault, ctx->stream),
                               "neighbour ids", __FILE__, __LINE__);
        if (!rc && !dev_out)
            rc = hd_check_cuda(ctx, cudaMemcpyAsync(sim_out, sdd, out_bytes, cudaMemcpyDefault, ctx->stream),
                               "similarities", __FILE__, __LINE__);
    }
    const int rs = hd_check_cuda(ctx, cudaStreamSynchronize(ctx->stream), "k-NN search", __FILE__, __LINE__);
    if (!rc) rc = rs;
    if (!rc) rc = hd_knn_status(ctx);
    if (ox) cudaFree(ox);
    if (oq) cudaFree(oq);
    return rc;
}

int hd_build_graph(hd_ctx* ctx, const void* X, int64_t n, int32_t d, int dtype, int32_t k, float gamma, int sym,
                   hd_graph** out) {
    if (!ctx || !X || !out || n <= 1 || d <= 0 || k < 1 || k >= n) return HD_ERR_INVALID_ARG;
    if (sym != HD_SYM_UNION && sym != HD_SYM_MUTUAL) return hd_fail(ctx, HD_ERR_INVALID_ARG, "sym %d", sym);
    if (dtype != HD_F32 && dtype != HD_BF16) return hd_fail(ctx, HD_ERR_INVALID_ARG, "dtype %d", dtype);
    *out = nullptr;
    HD_CUDA(ctx, cudaSetDevice(ctx->device));
    size_t es = dtype == HD_F32 ? 4 : 2;
    void* ox;
    const void* xd;
    int rc = stage_matrix(ctx, X, (size_t)n * d * es, &ox, &xd);
    if (rc) return rc;
    int32_t* idx = nullptr;
    float* sim = nullptr;
    void *ws, *aux;
    rc = k > KMAX ? hd_fail(ctx, HD_ERR_INVALID_ARG, "k=%d outside [1, %d]", k, KMAX)
                  : hd_aux_reserve(ctx, 0, 2 * ws_size((size_t)n * k * 4), &aux);
    if (!rc) {
        idx = (int32_t*)aux;
        sim = (float*)((char*)aux + ws_size((size_t)n * k * 4));
        rc = hd_ws_reserve(ctx, knn_scratch_bytes(ctx, n, n, k, dtype), &ws);
    }
    if (!rc) rc = hd_knn_impl(ctx, xd, n, d, dtype, xd, n, k, 1, idx, sim, ws);
    if (!rc) rc = hd_check_cuda(ctx, cudaStreamSynchronize(ctx->stream), "k-NN search", __FILE__, __LINE__);
    if (!rc) rc = hd_knn_status(ctx);
    if (!rc) rc = hd_graph_from_lists(ctx, n, k, idx, sim, gamma, sym, out);
    cudaStreamSynchronize(ctx->stream);
    hd_aux_trim(ctx);
    if (ox) cudaFree(ox);
    return rc;
}

int hd_observe(hd_ctx* ctx, const void* X, int64_t n, int32_t d, int dtype, const void* Q, int32_t nq, int32_t k_y,
               float gamma, int32_t* y_ptr, int32_t* y_idx, float* y_val) {
    if (!ctx || !X || !Q || !y_ptr || !y_idx || !y_val || nq <= 0 || k_y < 1 || k_y > n) return HD_ERR_INVALID_ARG;
    std::vector<int32_t> li((size_t)nq * k_y);
    std::vector<float> ls((size_t)nq * k_y);
    int rc = hd_knn(ctx, X, n, d, dtype, Q, nq, k_y, 0, li.data(), ls.data());
    if (rc) return rc;
    std::vector<int32_t> ptr(nq + 1), ids;
    std::vector<float> vals;
    ptr[0] = 0;
    for (int32_t q = 0; q < nq; ++q) {
        std::vector<std::pair<int32_t, float>> row;
        for (int u = 0; u < k_y; ++u) {
            int32_t j = li[(size_t)q * k_y + u];
            float s = ls[(size_t)q * k_y + u];
            float m = s > 0.0f ? s : 0.0f;
            float w = gamma == 3.0f ? m * m * m : powf(m, gamma);
            if (j >= 0 && w > 0.0f) row.push_back({j, w});
        }
        std::sort(row.begin(), row.end(), [](auto& a, auto& b) { return a.first < b.first; });
        for (auto& e : row) {
            ids.push_back(e.first);
            vals.push_back(e.second);
        }
        ptr[q + 1] = (int32_t)ids.size();
    }
    auto put = [&](void* dst, const void* src, size_t bytes) -> int {
        if (!bytes) return HD_OK;
        cudaMemcpyKind kd = hd_is_device_ptr(dst) ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost;
        HD_CUDA(ctx, cudaMemcpy(dst, src, bytes, kd));
        return HD_OK;
    };
    if ((rc = put(y_ptr, ptr.data(), ptr.size() * 4))) return rc;
    if ((rc = put(y_idx, ids.data(), ids.size() * 4))) return rc;
    if ((rc = put(y_val, vals.data(), vals.size() * 4))) return rc;
    return HD_OK;
}

}  // extern "C"
