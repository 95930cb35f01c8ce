// Sort and Merge stages shared by the workspaces that keep their accumulation array and all array
// in global memory (Algorithm 1 with integer labels, Sec. 5.2): a stable LSD radix sort of 64-bit
// labels with the values carried along, the reduction of runs of equal labels in insertion
// order, and the driver that feeds the products in rounds of the accumulation array's capacity.
// Included by the translation units that instantiate it.
#pragma once
#include <type_traits>

#include "common.cuh"

namespace spws {

constexpr int OT = 256;                 // threads of the element-wise kernels
constexpr u64 ABSENT_LABEL = ~0ull;     // a numbered product that does not exist (sorts last, dropped)

static int grid_for(const LaunchCtx& c, i64 work_items, int per_block) {
    i64 want = (work_items + per_block - 1) / per_block;
    const i64 cap = (i64)c.sm_count * 16;
    if (want > cap) want = cap;
    return (int)(want < 1 ? 1 : want);
}

// ---- stable LSD radix sort, 8 bits per pass -------------------------------------------------
// The digits of all passes are counted in one reading of the keys; a pass is then one launch: a
// block takes the next tile of RS_TILE consecutive elements, ranks them among equal digits (warp w
// owns the w-th contiguous slice of the tile and walks it 32 elements at a time, so "block, warp,
// step, lane" is the input order), learns from the tiles before it how many of each digit precede
// (a decoupled look-back per digit: the single-pass scheme of Merrill and Garland, and of Adinets
// and Merrill's "Onesweep"), puts the tile in digit order in shared memory and lets every digit's
// elements leave as one contiguous run.  One reading and one writing per pass; a histogram, a scan over
// (digit, block) and a scatter per pass read the keys twice and launch five kernels (a call that sorts 43e6
// products of SpTTM 9.0 ms, 8.0 ms like this and with the run reduction below).
constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_STEPS = 8;                             // 32-element steps per warp (16: 128 registers, half the warps, 15 % slower)
constexpr int RS_TILE = RS_WARPS * RS_STEPS * 32;       // 2048
constexpr int RS_PASSES = 8;

// counts and tickets at the start of the sort temporaries, followed by one status word per tile and digit
struct SortHead {
    int hist[RS_PASSES][256];
    int ticket[RS_PASSES];
};
static size_t sort_head_bytes() { return (sizeof(SortHead) + 255) & ~(size_t)255; }

// Digits of the labels a block writes, for a kernel of 256 threads: start, add for every label, flush.
struct DigitCounts {
    int h[RS_PASSES][256];
    __device__ __forceinline__ void start(int passes) {
        for (int p = 0; p < passes; ++p) h[p][threadIdx.x] = 0;
        __syncthreads();
    }
    __device__ __forceinline__ void add(u64 key, int passes) {
        for (int p = 0; p < passes; ++p, key >>= 8) atomicAdd(&h[p][(unsigned)key & 255u], 1);
    }
    __device__ __forceinline__ void flush(int passes, SortHead* head) {
        __syncthreads();
        for (int p = 0; p < passes; ++p)
            if (h[p][threadIdx.x]) atomicAdd(&head->hist[p][threadIdx.x], h[p][threadIdx.x]);
    }
};

static __global__ void __launch_bounds__(RS_THREADS) radix_hist_kernel(const u64* __restrict__ keys, i64 n, int passes, SortHead* __restrict__ head) {
    __shared__ int s_h[RS_PASSES][256];
    for (int p = 0; p < passes; ++p) s_h[p][threadIdx.x] = 0;
    __syncthreads();
    for (i64 t = (i64)blockIdx.x * RS_THREADS + threadIdx.x; t < n; t += (i64)gridDim.x * RS_THREADS) {
        u64 k = keys[t];
        for (int p = 0; p < passes; ++p, k >>= 8) atomicAdd(&s_h[p][(unsigned)k & 255u], 1);
    }
    __syncthreads();
    for (int p = 0; p < passes; ++p)
        if (s_h[p][threadIdx.x]) atomicAdd(&head->hist[p][threadIdx.x], s_h[p][threadIdx.x]);
}

// K: labels of 32 or 64 bits.  `numbered`: the first pass over elements whose values are their places.
template <typename K, typename T, bool VALUES>
__global__ void __launch_bounds__(RS_THREADS) radix_pass_kernel(const K* __restrict__ keys, const T* __restrict__ vals, bool numbered, i64 n, int pass,
                                                                SortHead* __restrict__ head, u64* __restrict__ status, DevCtl* ctl,
                                                                K* __restrict__ keys_out, T* __restrict__ vals_out) {
    __shared__ int s_cnt[RS_WARPS][256];        // elements with the digit in this warp's slice, then their start inside the digit's part
    __shared__ int s_start[256];                // start of the digit's part inside the tile
    __shared__ i64 s_goff[256];
    __shared__ int s_ws[33];
    __shared__ int s_tile;
    __shared__ K s_key[RS_TILE];
    __shared__ T s_val[VALUES ? RS_TILE : 1];
    constexpr bool numbers = std::is_same<T, int>::value;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, shift = 8 * pass;
    if constexpr (sizeof(K) == 4) chained_start();        // (not for long sorts, which are none the faster for it)
    if (threadIdx.x == 0) s_tile = atomicAdd(&head->ticket[pass], 1);
    for (int d = lane; d < 256; d += 32) s_cnt[warp][d] = 0;
    __syncthreads();
    const int tile = s_tile;
    const i64 base = (i64)tile * RS_TILE + (i64)warp * (RS_STEPS * 32);
    K key[RS_STEPS];
    int rank[RS_STEPS];
#pragma unroll
    for (int st = 0; st < RS_STEPS; ++st) {
        const i64 t = base + st * 32 + lane;
        key[st] = t < n ? keys[t] : (K)~0ull;
    }
#pragma unroll
    for (int st = 0; st < RS_STEPS; ++st) {
        const bool live = base + st * 32 + lane < n;
        const unsigned d = (unsigned)(key[st] >> shift) & 255u;
        // lanes of this step with the same digit (lanes past the end form their own group)
        const unsigned peers = __match_any_sync(0xffffffffu, live ? d : 256u);
        const int before = __popc(peers & ((1u << lane) - 1u));
        int old = 0;
        if (live && before == 0) {                       // first lane of a group books the group's slots
            old = s_cnt[warp][d];
            s_cnt[warp][d] = old + __popc(peers);
        }
        old = __shfl_sync(0xffffffffu, old, __ffs(peers) - 1);
        rank[st] = old + before;
        __syncwarp();
    }
    __syncthreads();
    // thread d: start of each warp's share of digit d inside the digit's part of the tile, the start of
    // that part inside the tile, and the digit's place in the output
    int tile_total;
    {
        const int d = threadIdx.x;                       // RS_THREADS == 256 digits
        int run = 0;
        for (int w = 0; w < RS_WARPS; ++w) { const int c = s_cnt[w][d]; s_cnt[w][d] = run; run += c; }
        u64* const mine = status + (i64)tile * 256 + d;
        look_publish(mine, 2 * pass + (tile == 0 ? 2 : 1), run);
        const int start = block_excl_scan<RS_THREADS>(run, s_ws, tile_total);
        int all;
        const int digit0 = block_excl_scan<RS_THREADS>(head->hist[pass][d], s_ws, all);
        i64 before = 0;
        if (tile > 0) {
            before = look_back<sizeof(K) == 4 ? 4 : 1>(status + d, 256, tile, pass, ctl);      // (four cost the other registers)
            look_publish(mine, 2 * pass + 2, before + run);
        }
        s_start[d] = start;
        s_goff[d] = digit0 + before - start;             // global position of staged slot i of digit d = s_goff[d] + i
    }
    __syncthreads();
#pragma unroll
    for (int st = 0; st < RS_STEPS; ++st) {
        const i64 t = base + st * 32 + lane;
        if (t < n) {
            const unsigned d = (unsigned)(key[st] >> shift) & 255u;
            const int at = s_start[d] + s_cnt[warp][d] + rank[st];
            s_key[at] = key[st];
            if (VALUES) s_val[at] = numbers && numbered ? (T)t : vals[t];
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < tile_total; i += RS_THREADS) {
        const K k = s_key[i];
        const i64 at = s_goff[(unsigned)(k >> shift) & 255u] + i;
        keys_out[at] = k;
        if (VALUES) vals_out[at] = s_val[i];
    }
}

static size_t sort_scratch_bytes(i64 n) {
    const i64 nblocks = (n + RS_TILE - 1) / RS_TILE;
    return sort_head_bytes() + 8 * 256 * (size_t)(nblocks > 0 ? nblocks : 1);
}

// Sorts n (label, value) pairs by label; `bits` = number of significant label bits.  Input in
// (k0, v0), the other buffer in (k1, v1); *in_first tells which pair holds the result.  `counted`: the caller has cleared
// `tmp`, and its kernel that wrote the labels has counted their digits (DigitCounts).
// `numbered`: the values are the elements' places, and v0 is not read.
template <typename K, typename T, bool VALUES>
static cudaError_t radix_sort_t(const LaunchCtx& c, i64 n, int bits, K* k0, T* v0, K* k1, T* v1, char* tmp, bool* in_first, bool counted = false, bool numbered = false) {
    *in_first = true;
    if (n <= 1) return cudaSuccess;
    const int nblocks = (int)((n + RS_TILE - 1) / RS_TILE);
    const int passes = (bits + 7) / 8;
    SortHead* head = reinterpret_cast<SortHead*>(tmp);
    u64* status = reinterpret_cast<u64*>(tmp + sort_head_bytes());
    if constexpr (sizeof(K) == 8) if (!counted) {
        const cudaError_t e = cudaMemsetAsync(tmp, 0, sort_scratch_bytes(n), c.stream);
        if (e != cudaSuccess) return e;
        const int hist_blocks = 4 * c.sm_count;
        radix_hist_kernel<<<nblocks < hist_blocks ? nblocks : hist_blocks, RS_THREADS, 0, c.stream>>>(k0, n, passes, head);
        ++c.launches;
    }
    K *ki = k0, *ko = k1;
    T *vi = v0, *vo = v1;
    for (int pass = 0; pass < passes; ++pass) {
        if constexpr (sizeof(K) == 4) {
            const cudaError_t e = launch_chained(c, radix_pass_kernel<K, T, VALUES>, nblocks, RS_THREADS, 0, ki, vi, numbered && pass == 0, n, pass, head, status, c.ctl, ko, vo);
            if (e != cudaSuccess) return e;
        } else {
            radix_pass_kernel<K, T, VALUES><<<nblocks, RS_THREADS, 0, c.stream>>>(ki, vi, numbered && pass == 0, n, pass, head, status, c.ctl, ko, vo);
            ++c.launches;
        }
        K* tk = ki; ki = ko; ko = tk;
        T* tv = vi; vi = vo; vo = tv;
        *in_first = !*in_first;
    }
    return cudaGetLastError();
}

// ---- Merge (reduce runs of equal labels) and Compress ----------------------------------------
// One pass over the sorted labels: the first entry of a run of equal labels finds its place among
// the distinct labels (tiles hand the running count on as above), writes the label there and
// (VALUES) the run's sum in insertion order.  Absent products carry the largest label and are no
// run.  Heads, their three-launch scan and the reduction were separate passes before.
constexpr int RR_ITEMS = 16;
constexpr int RR_TILE = OT * RR_ITEMS;

template <typename T, bool VALUES>
__global__ void __launch_bounds__(OT) reduce_runs_kernel(const u64* __restrict__ keys, const T* __restrict__ vals, i64 n, int* __restrict__ ticket,
                                                         u64* __restrict__ status, DevCtl* ctl, u64* __restrict__ ukeys,
                                                         T* __restrict__ uvals, i64* __restrict__ cnt_out) {
    __shared__ u64 s_key[OT * (RR_ITEMS + 1)];
    __shared__ unsigned short s_at[RR_TILE];
    __shared__ int s_ws[33];
    __shared__ int s_tile;
    __shared__ i64 s_before;
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1);
    __syncthreads();
    const int tile = s_tile;
    // the tile's labels, read across the block and handed to each thread as RR_ITEMS consecutive ones
    // (one word of padding per thread keeps the strided reading clear of bank conflicts)
    const i64 tile0 = (i64)tile * RR_TILE;
#pragma unroll
    for (int x = 0; x < RR_ITEMS; ++x) {
        const int i = x * OT + threadIdx.x;
        s_key[i + i / RR_ITEMS] = tile0 + i < n ? keys[tile0 + i] : ABSENT_LABEL;
    }
    __syncthreads();
    u64* const key = s_key + threadIdx.x * (RR_ITEMS + 1);
    unsigned head = 0;
    u64 prev = threadIdx.x > 0 ? key[-2] : (tile0 > 0 ? keys[tile0 - 1] : ABSENT_LABEL);
#pragma unroll
    for (int x = 0; x < RR_ITEMS; ++x) {
        const u64 k = key[x];
        if (k != ABSENT_LABEL && k != prev) head |= 1u << x;
        prev = k;
    }
    int total;
    const int excl = block_excl_scan<OT>(__popc(head), s_ws, total);
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0) look_publish(status + tile, tile == 0 ? 2 : 1, total);
        i64 before = 0;
        if (tile > 0) {
            before = look_back_warp(status, tile, 0, ctl);
            if (threadIdx.x == 0) look_publish(status + tile, 2, before + total);
        }
        if (threadIdx.x == 0) {
            s_before = before;
            if ((i64)(tile + 1) * RR_TILE >= n) *cnt_out = before + total;
        }
    }
    // the heads' places in the tile, packed, so that consecutive threads sum and write consecutive runs
    int slot = excl;
#pragma unroll
    for (int x = 0; x < RR_ITEMS; ++x)
        if ((head >> x) & 1u) s_at[slot++] = (unsigned short)(threadIdx.x * RR_ITEMS + x);
    __syncthreads();
    for (int i = threadIdx.x; i < total; i += OT) {
        const int p = s_at[i];
        const u64 k = s_key[p + p / RR_ITEMS];
        ukeys[s_before + i] = k;
        if (VALUES) {
            T sum = vals[tile0 + p];
            for (i64 y = tile0 + p + 1; y < n; ++y) {
                const int z = (int)min(y - tile0, (i64)RR_TILE);
                if ((z < RR_TILE ? s_key[z + z / RR_ITEMS] : keys[y]) != k) break;
                sum = add_rn(sum, vals[y]);
            }
            uvals[s_before + i] = sum;
        }
    }
}

// Sort + reduce n entries that start at (k, v); the other buffer of the same size is (k2, v2).
// The duplicate-free result is written to whichever of the two buffers the sorted sequence did
// not end in, and the caller learns which.  The number of distinct labels goes to *cnt_dev and is
// read back.
template <typename T, bool VALUES>
static cudaError_t sort_reduce_t(const LaunchCtx& c, i64 n, int label_bits, u64* k, T* v, u64* k2, T* v2, char* sort_tmp, i64* cnt_dev,
                                 i64* cnt_host_pinned, bool* result_in_first) {
    bool first = true;
    cudaError_t e = radix_sort_t<u64, T, VALUES>(c, n, label_bits, k, v, k2, v2, sort_tmp, &first);
    if (e != cudaSuccess) return e;
    u64* ks = first ? k : k2;
    T* vs = first ? v : v2;
    u64* ku = first ? k2 : k;
    T* vu = first ? v2 : v;
    if ((e = cudaMemsetAsync(cnt_dev, 0, sizeof(i64), c.stream)) != cudaSuccess) return e;
    if (n > 0) {
        const int tiles = (int)((n + RR_TILE - 1) / RR_TILE);
        SortHead* head = reinterpret_cast<SortHead*>(sort_tmp);
        u64* status = reinterpret_cast<u64*>(sort_tmp + sort_head_bytes());
        if ((e = cudaMemsetAsync(sort_tmp, 0, sort_head_bytes() + 8 * (size_t)tiles, c.stream)) != cudaSuccess) return e;
        reduce_runs_kernel<T, VALUES><<<tiles, OT, 0, c.stream>>>(ks, vs, n, &head->ticket[0], status, c.ctl, ku, vu, cnt_dev);
        ++c.launches;
    }
    if ((e = cudaMemcpyAsync(cnt_host_pinned, cnt_dev, sizeof(i64), cudaMemcpyDeviceToHost, c.stream)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(c.stream)) != cudaSuccess) return e;
    *result_in_first = !first;
    return cudaGetLastError();
}

// One pass of a sparse workspace over P numbered products, in rounds of `cap` (Algorithm 1: when
// the accumulation array is full it is sorted and reduced on its own, then united with the all
// array; the entry that found it full opens the next round).  `expand(t0, n, keys, vals)` enqueues
// the kernel that appends the products with ordinals [t0, t0 + n); a product may be marked absent
// with the all-ones label, which sorts last and is dropped.
// Buffers: two (label, value) arrays of N = P + (cap < P ? cap : 0) entries, sort temporaries.  On return *result_first tells which array holds the
// duplicate-free result; its length is in *nnz_host_pinned.
template <typename T, bool VALUES, typename Expand>
static cudaError_t ism_rounds_t(const LaunchCtx& c, Expand expand, i64 P, i64 cap, int label_bits,
                                u64* kA, T* vA, u64* kB, T* vB, char* sort_tmp, i64* nnz_dev, i64* nnz_host_pinned, bool* result_first) {
    u64 *kc = kA, *ko = kB;             // kc/vc: the buffer that holds the all array (n_all entries, sorted, duplicate-free)
    T *vc = vA, *vo = vB;
    i64 n_all = 0;
    *nnz_host_pinned = 0;
    const size_t vsz = VALUES ? sizeof(T) : 0;
    for (i64 t0 = 0; t0 < P; t0 += cap) {
        const i64 n_new = (P - t0 < cap) ? P - t0 : cap;
        // Insert: the round's products behind the all array
        cudaError_t e = expand(t0, n_new, kc + n_all, VALUES ? vc + n_all : (T*)nullptr);
        if (e != cudaSuccess) return e;
        // Sort + reduce of the accumulation array alone
        bool in_first = true;
        e = sort_reduce_t<T, VALUES>(c, n_new, label_bits, kc + n_all, VALUES ? vc + n_all : nullptr, ko + n_all,
                                     VALUES ? vo + n_all : nullptr, sort_tmp, nnz_dev, nnz_host_pinned, &in_first);
        if (e != cudaSuccess) return e;
        const i64 n_acc = *nnz_host_pinned;
        if (n_all == 0) {
            // nothing to unite with: the reduced accumulation array is the all array
            if (!in_first) { u64* tk = kc; kc = ko; ko = tk; T* tv = vc; vc = vo; vo = tv; }
            n_all = n_acc;
            continue;
        }
        if (!in_first) {                // bring the reduced accumulation array behind the all array
            if ((e = cudaMemcpyAsync(kc + n_all, ko + n_all, 8 * (size_t)n_acc, cudaMemcpyDeviceToDevice, c.stream)) != cudaSuccess) return e;
            if (VALUES && (e = cudaMemcpyAsync(vc + n_all, vo + n_all, vsz * (size_t)n_acc, cudaMemcpyDeviceToDevice, c.stream)) != cudaSuccess) return e;
        }
        // Merge: all array first, so that a label in both sums as all + accumulated
        e = sort_reduce_t<T, VALUES>(c, n_all + n_acc, label_bits, kc, vc, ko, vo, sort_tmp, nnz_dev, nnz_host_pinned, &in_first);
        if (e != cudaSuccess) return e;
        if (!in_first) { u64* tk = kc; kc = ko; ko = tk; T* tv = vc; vc = vo; vo = tv; }
        n_all = *nnz_host_pinned;
    }
    *nnz_host_pinned = n_all;
    *result_first = (kc == kA);
    return cudaGetLastError();
}

}  // namespace spws
