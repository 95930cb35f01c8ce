// Insert-sort-merge workspace: 4, 8 or 16 lanes per output row of at most 32, 64 or 128 products, a warp per row of
// at most 1024, a CTA per row beyond (Algorithm 1; the accumulation array is shared memory and is never full because
// the symbolic upper bound sized it; coordinate-sort policy, Sec. 5.2).
//   Insert : product t of the row (loop order k, then j) is appended at slot t: its value stays
//            there, and the packed word (j, t) enters the sort (accumulation indexing, Sec. 5.1:
//            only integers move).  The word is 32 bits (j << log2 CAP | t) when the column count
//            leaves room for it, else 64 bits (j << 32 | t).
//   Sort   : bitonic sort of the packed words (lexicographic on (j, t), hence stable).
//   Merge  : runs of equal j are reduced in slot order and written at row_ptr[i] + rank.
#include <algorithm>
#include "common.cuh"

namespace spws {

template <int CAP> struct Log2 { static constexpr int value = 1 + Log2<CAP / 2>::value; };
template <> struct Log2<1> { static constexpr int value = 0; };

// packed (column, slot) words
template <typename P, int CAP> struct Pack;
template <int CAP> struct Pack<u64, CAP> {
    static __device__ __forceinline__ u64 make(int col, int slot) { return ((u64)(unsigned)col << 32) | (unsigned)slot; }
    static __device__ __forceinline__ unsigned key(u64 p) { return (unsigned)(p >> 32); }
    static __device__ __forceinline__ unsigned slot(u64 p) { return (unsigned)p; }
    static __device__ __forceinline__ u64 sentinel() { return ~0ull; }
};
template <int CAP> struct Pack<unsigned, CAP> {
    static constexpr int LG = Log2<CAP>::value;
    static __device__ __forceinline__ unsigned make(int col, int slot) { return ((unsigned)col << LG) | (unsigned)slot; }
    static __device__ __forceinline__ unsigned key(unsigned p) { return p >> LG; }
    static __device__ __forceinline__ unsigned slot(unsigned p) { return p & (unsigned)(CAP - 1); }
    static __device__ __forceinline__ unsigned sentinel() { return ~0u; }
};

template <typename T, typename P, int CAP, int THREADS, bool NUMERIC>
__global__ void __launch_bounds__(THREADS) ism_smem_kernel(const int* __restrict__ perm, DevCtl* __restrict__ ctl, int cls,
                                                           int counter_slot, i64 above, Csr A, Csr B, const i64* __restrict__ ub,
                                                           int* __restrict__ cnt, const i64* __restrict__ rowptr, int* __restrict__ Ccrd,
                                                           T* __restrict__ Cval) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typedef Pack<P, CAP> PK;
    T* vals = reinterpret_cast<T*>(smem_raw);                             // CAP (numeric only)
    P* packed = reinterpret_cast<P*>(vals + (NUMERIC ? CAP : 0));         // CAP
    i64* e_qs = reinterpret_cast<i64*>(smem_raw + (((NUMERIC ? sizeof(T) * CAP : 0) + sizeof(P) * CAP + 7) & ~(size_t)7));   // THREADS
    T* e_a = reinterpret_cast<T*>(e_qs + THREADS);                        // THREADS
    int* e_off = reinterpret_cast<int*>(e_a + THREADS);                   // THREADS + 1
    int* ws = e_off + THREADS + 1;                                        // 33
    __shared__ int s_next;

    if (ctl->status != 0) return;
    int off, n;
    class_range(ctl, cls, off, n);
    const int* __restrict__ rows = perm + off;
    const T* __restrict__ Aval = (const T*)A.val;
    const T* __restrict__ Bval = (const T*)B.val;
    const int tid = threadIdx.x;

    for (;;) {
        __syncthreads();
        if (tid == 0) s_next = atomicAdd(&ctl->work_counter[counter_slot], 1);
        __syncthreads();
        const int r = s_next;
        if (r >= n) break;
        const int row = rows[r];
        if (ub[row] <= above) continue;                 // the warp kernel's rows
        const i64 ps = A.pos[row], pe = A.pos[row + 1];

        // ---- Insert
        int total = 0;
        for (i64 p0 = ps; p0 < pe; p0 += THREADS) {
            const i64 p = p0 + tid;
            int len = 0;
            i64 qs = 0;
            T a = 0;
            if (p < pe) {
                const int k = __ldg(A.crd + p);
                if ((unsigned)k < (unsigned)B.nrows) {
                    qs = __ldg(B.pos + k);
                    len = (int)(__ldg(B.pos + k + 1) - qs);
                }
                if (NUMERIC) a = __ldg(Aval + p);
            }
            int chunk_total;
            const int excl = block_excl_scan<THREADS>(len, ws, chunk_total);
            e_off[tid] = excl;
            e_qs[tid] = qs;
            if (NUMERIC) e_a[tid] = a;
            if (tid == 0) e_off[THREADS] = chunk_total;
            __syncthreads();
            const int nE = (int)min((i64)THREADS, pe - p0);
            if (total + chunk_total > CAP) chunk_total = CAP - total;     // cannot happen for a correctly classed row
            for (int t = tid; t < chunk_total; t += THREADS) {
                int lo = 0, hi = nE;
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (e_off[mid] <= t) lo = mid; else hi = mid;
                }
                const i64 q = e_qs[lo] + (t - e_off[lo]);
                const int slot = total + t;
                packed[slot] = PK::make(__ldg(B.crd + q), slot);
                if (NUMERIC) vals[slot] = mul_rn(e_a[lo], __ldg(Bval + q));
            }
            total += chunk_total;
            __syncthreads();
        }
        int n2 = 1;
        while (n2 < total) n2 <<= 1;
        for (int t = total + tid; t < n2; t += THREADS) packed[t] = PK::sentinel();
        __syncthreads();

        // ---- Sort
        for (int k = 2; k <= n2; k <<= 1) {
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int t = tid; t < (n2 >> 1); t += THREADS) {
                    const int i = 2 * t - (t & (j - 1));
                    const int l = i + j;
                    const P x = packed[i], y = packed[l];
                    const bool up = (i & k) == 0;
                    if ((x > y) == up) { packed[i] = y; packed[l] = x; }
                }
                __syncthreads();
            }
        }

        // ---- Merge
        const int chunk = (total + THREADS - 1) / THREADS;
        const int x0 = min(total, tid * chunk), x1 = min(total, x0 + chunk);
        int heads = 0;
        for (int x = x0; x < x1; ++x)
            heads += (x == 0) || (PK::key(packed[x]) != PK::key(packed[x - 1]));
        int row_cnt;
        int rank = block_excl_scan<THREADS>(heads, ws, row_cnt);
        if (!NUMERIC) {
            if (tid == 0) cnt[row] = row_cnt;
        } else {
            const i64 out0 = rowptr[row];
            for (int x = x0; x < x1; ++x) {
                const unsigned key = PK::key(packed[x]);
                if (x != 0 && key == PK::key(packed[x - 1])) continue;
                T sum = vals[PK::slot(packed[x])];
                for (int y = x + 1; y < total && PK::key(packed[y]) == key; ++y)
                    sum = add_rn(sum, vals[PK::slot(packed[y])]);
                Ccrd[out0 + rank] = (int)key;
                Cval[out0 + rank] = sum;
                ++rank;
            }
        }
    }
}

// ---------------------------------------------------------------------------------------
// A warp per row, the sort in registers.  Lane l holds E packed words; comparisons over a distance
// below E stay inside the lane, longer ones cost one shuffle per word, and no barrier is left: a
// network in shared memory took about 12 warp instructions per product and 55 barriers at 1024
// products, this one about 2.7.  Bound by instruction issue.
//   Insert : 32 A entries at a time; a group of lanes per entry (as many as the mean B row has
//            entries) writes the products of its B row at their slots.
//   Sort   : E = 6, 8, 12, 16, 24 or 32 words per lane, the smallest network that holds the row (four for the few rows of up to
//            128 products that go along with longer ones).
//   Merge  : the sorted words go back to shared memory, the places of the run heads are packed, and
//            one lane per run sums it in slot order.
//   Of rows of more than 256 products the counting pass leaves the sorted words in scratch when there is room
// (coalesced: word x of lane l at x * lanes + l, lanes past the last word left out), and the numeric pass then only
// fetches the values: 8e4 rows of 674 products, f32: count 507 -> 578 us, numeric 871 -> 400 us; 2e5 rows
// of 470, f64: 154 -> 210 and 494 -> 225 us.  Shorter rows gain nothing, their sort is a small part of the work.
// Stencil 41 x 37 x 53 (f32, 674 products a row): count 1714 -> 508 us, numeric 1905 -> 863 us against a CTA per
// row.  With sizes of three times a power of two, long merges as loops and lane groups found by shifts: count 578 -> 384 us
// on the stencil (372 since; numeric 370, 309 since), 210 -> 172 us on the rows of 470; 143-product rows (3e4): 44 -> 36
// and 55 -> 49 us.
//   Where outputs are at most half of the products and B rows fill a warp, the counting pass leaves the places of the products
// among the outputs and ism_rank_kernel adds: stencil 41 x 37 x 53, f32, count 374 -> 400 us, numeric 309 -> 135 (of it 11 for
// the rows at its edges); 40^3, f64, 300 -> 321 and 296 -> 138.  Not with words of 64 bits, whose counting kernel would slow
// down (60000 rows of 600 products, f64: 881 -> 895 us).  The line at half of the products: 40000 rows of 18 B rows of 32, f32, a call at 2 products an output, where
// few rows rank, 438 -> 443, at 2.1 436 -> 408, at 3 426 -> 340; of 35 B rows of 17 (a step of the adding kernel fills half a warp) 538 -> 529, 530 -> 477, 519 -> 404; of
// 10 of 64, f64, at 2 466 -> 473.  A hash set of the columns before the sort instead: 348 us, and 786 for
// a numeric pass that looks its products up in it.
// ---------------------------------------------------------------------------------------
constexpr int IW_WARPS = 4;

template <typename P>
__device__ __forceinline__ void sort_pair(P& a, P& b) {
    const P lo = min(a, b), hi = max(a, b);
    a = lo;
    b = hi;
}

// Ascending bitonic sort of G * E words by each group of G lanes, element index = lane of the group * E + x, E = 2^a or
// 3 * 2^a.  Every merge starts with the mirrored comparison (i against i ^ (k - 1) within its k), so all comparisons point the same way; with
// a factor of three the merges end at triples, which three comparisons sort.
template <typename P, int E, int G = 32>
__device__ __forceinline__ void warp_sort(P (&w)[E]) {
    constexpr int BASE = E % 3 == 0 ? 3 : 1;
    const int lane = threadIdx.x & 31;
    auto triples = [&]() {
        if (BASE == 3) {
#pragma unroll
            for (int x = 0; x + 2 < E; x += 3) {
                sort_pair(w[x], w[x + 1]);
                sort_pair(w[x + 1], w[x + 2]);
                sort_pair(w[x], w[x + 1]);
            }
        }
    };
    // the last stages of a merge: bitonic runs of up to E words inside a lane
    auto lane_merge = [&](int k) {
#pragma unroll
        for (int j = k >> 1; j >= BASE; j >>= 1)
#pragma unroll
            for (int x = 0; x < E; ++x)
                if (x % (2 * j) < j) sort_pair(w[x], w[x + j]);
        triples();
    };
    triples();
#pragma unroll
    for (int k = 2 * BASE; k <= E; k <<= 1) {
#pragma unroll
        for (int x = 0; x < E; ++x)
            if (x % k < k / 2) sort_pair(w[x], w[x / k * k + k - 1 - x % k]);
        lane_merge(k / 2);
    }
    // merges across m lanes; the long ones stay loops: a kernel whose warps run several unrolled networks of
    // 16 .. 32 words outgrows the instruction cache (counting 2e5 rows of 257 .. 1024 products: 300 us against 172; 8e4
    // rows of 674: 456 against 384; of up to 8 words the unrolled ones are faster, 50 against 55 us)
    constexpr int U = E > 8 ? 1 : 5;
#pragma unroll U
    for (int m = 2; m <= G; m <<= 1) {
        const bool low_half = (lane & (m >> 1)) == 0;
#pragma unroll
        for (int x = 0; x < (E + 1) / 2; ++x) {
            const int y = E - 1 - x;
            const P ox = __shfl_xor_sync(0xffffffffu, w[y], m - 1);
            if (y != x) {
                const P oy = __shfl_xor_sync(0xffffffffu, w[x], m - 1);
                w[y] = low_half ? min(w[y], oy) : max(w[y], oy);
            }
            w[x] = low_half ? min(w[x], ox) : max(w[x], ox);
        }
#pragma unroll U
        for (int d = m >> 2; d > 0; d >>= 1) {
            const bool low = (lane & d) == 0;
#pragma unroll
            for (int x = 0; x < E; ++x) {
                const P other = __shfl_xor_sync(0xffffffffu, w[x], d);
                w[x] = low ? min(w[x], other) : max(w[x], other);
            }
        }
        lane_merge(E);
    }
}

// one word of padding per 32 keeps both the strided and the per-lane consecutive accesses conflict-free
__device__ __forceinline__ int padded(int i) { return i + (i >> 5); }

// What the counting pass keeps of a row whose outputs are at most half of its products and whose B rows fill a warp, instead of the
// sorted words: the distinct columns, then every product's place among them (16 bits, loop order).  The numeric pass adds one
// B row after the other, whose products go to different outputs, and reads no columns.
constexpr i64 ORDER_RANKS = 1ll << 61;                  // flag above the offset of such a row (no flag of a dense row's)

// Sorts the row's packed words and counts its distinct columns; numeric: leaves the sorted words in `packed`
// and the places of the run heads in `heads`.  `order` (may be null): numeric: the words as sorted before;
// else receives them, or (*ranks, when the row is of that kind and may_rank) the columns and places.  (Without RANKS at once: words that
// live across the count of the heads cost the kernel spills.)
template <typename PK, typename P, int E, bool NUMERIC, bool RANKS>
__device__ __forceinline__ int sort_row(P* packed, unsigned short* heads, int total, P* order, bool may_rank, bool* ranks) {
    const int lane = threadIdx.x & 31;
    P w[E];
    const int lanes = order_lanes(total, E);
    if (NUMERIC && order) {
#pragma unroll
        for (int x = 0; x < E; ++x) w[x] = lane < lanes ? order[x * lanes + lane] : PK::sentinel();
    } else {
#pragma unroll
        for (int x = 0; x < E; ++x) {
            const int i = x * 32 + lane;
            w[x] = i < total ? packed[padded(i)] : PK::sentinel();
        }
        warp_sort<P, E>(w);
        if (!NUMERIC && !RANKS && order && lane < lanes) {
#pragma unroll
            for (int x = 0; x < E; ++x) order[x * lanes + lane] = w[x];
        }
    }
    const P before = __shfl_up_sync(0xffffffffu, w[E - 1], 1);
    unsigned head = 0;
#pragma unroll
    for (int x = 0; x < E; ++x) {
        const bool first = x == 0 ? (lane == 0 || PK::key(w[x]) != PK::key(before)) : PK::key(w[x]) != PK::key(w[x > 0 ? x - 1 : 0]);
        if (w[x] != PK::sentinel() && first) head |= 1u << x;
    }
    const int mine = __popc(head);
    // (where rows may rank the sum alone, before the words are left: with the scan the kernel spills more)
    constexpr bool SUM = !NUMERIC && RANKS;
    const int incl = SUM ? 0 : warp_incl_scan(mine);
    const int n = SUM ? __reduce_add_sync(0xffffffffu, mine) : __shfl_sync(0xffffffffu, incl, 31);
    if (NUMERIC) {
        __syncwarp();
        int at = incl - mine;
#pragma unroll
        for (int x = 0; x < E; ++x) {
            packed[padded(lane * E + x)] = w[x];
            if ((head >> x) & 1u) heads[at++] = (unsigned short)(lane * E + x);
        }
        __syncwarp();
    } else if (RANKS && order) {
        if (may_rank && 2 * n <= total) {
            __syncwarp();
            unsigned* const cols = reinterpret_cast<unsigned*>(packed);
            unsigned short* const place = reinterpret_cast<unsigned short*>(cols + n);
            int at = warp_incl_scan(mine) - mine - 1;
#pragma unroll
            for (int x = 0; x < E; ++x)
                if (w[x] != PK::sentinel()) {
                    if ((head >> x) & 1u) cols[++at] = PK::key(w[x]);
                    place[PK::slot(w[x])] = (unsigned short)at;
                }
            __syncwarp();
            // (whole quads: the room of a row, like that of its packed words, is a multiple of 16 bytes)
            for (int i = lane; 4 * i < n + (total + 1) / 2; i += 32) reinterpret_cast<uint4*>(order)[i] = reinterpret_cast<const uint4*>(packed)[i];
            __syncwarp();
            *ranks = true;
        } else if (lane < lanes) {
#pragma unroll
            for (int x = 0; x < E; ++x) order[x * lanes + lane] = w[x];
        }
    }
    return n;
}

// ---------------------------------------------------------------------------------------
// Rows of at most 32, 64 or 128 products: G = 4, 8 or 16 lanes per row, eight products per lane at most, so that a warp works
// on eight, four or two of them at a time.
//   Insert : G entries at a time; lane l takes the products l, l + G, .. of those entries, whose owners it finds by a search
//            among the running counts.
//   Sort   : six or eight words per lane in registers; with four lanes a row two or four where no row of the warp has more.
//            The narrower the group, the more of the network stays inside the lanes.
//   Merge  : as below: the sorted words and the places of the run heads go to shared memory, a lane per run.
// Every step of the way to a row's products is a load that waits for the one before: several rows per warp and some 40 warps
// keep enough of them in flight, and a block for every 128 lanes' rows spares fetching ahead (persistent blocks: numeric 80 us
// where these take 75).  Bound by the integer pipe (half of the instructions, a warp every two cycles).  A warp per row
// against this, count + numeric: 2e5 rows of 59 products, f32, 123 + 148 and 92 + 128 us; 1.6e5 fibres of 110, 95 + 108 and 64 + 93
// us; 1.9e5 rows of 82, f64, 137 + 178 and 99 + 144 us.  Rows of at most 32 products had as many lanes as products before: 1.2e5
// rows of 16 .. 24, f64, 22 + 45 and 12 + 40 us; 65536 rows of 16 whose B rows come from memory, 18 + 25 and 16 + 26 us.
// Words of 64 bits (four lanes: from 2^27 columns on): 2.6e5 rows of 16 products, f32, 28 + 38 us, where the register kernel with
// columns relative to the row's first took 40 + 48; words of 32 bits 18 + 30.
// ---------------------------------------------------------------------------------------
constexpr int IG_THREADS = 128;

template <typename T, bool NUMERIC> struct GroupEntry { i64 q; T a; };          // start of the B row less the products before it
template <typename T> struct GroupEntry<T, false> { i64 q; };

template <int G> __host__ __device__ constexpr int group_words() { return 8 * G + G / 4 + G; }     // packed words of a row, with room against bank conflicts
template <typename T, typename P, int G, bool NUMERIC>
__host__ __device__ constexpr int group_row_bytes() {
    return (int)sizeof(GroupEntry<T, NUMERIC>) * G + (NUMERIC ? (int)sizeof(T) * 9 * G : 0) + (int)sizeof(P) * group_words<G>() + (NUMERIC ? 8 * G : 0);
}
template <typename T, typename P, bool NUMERIC> constexpr int group_blocks() { return sizeof(P) == 8 ? 8 : NUMERIC && sizeof(T) == 8 ? 10 : 12; }

// Sorts a row's packed words and counts its distinct columns; numeric: leaves the sorted words in `packed` and the places of the
// run heads in `heads`.  For all lanes of a warp together.
template <typename PK, typename P, int E, int G, bool NUMERIC>
__device__ __forceinline__ int sort_group(P* packed, unsigned char* heads, int total, int gl) {
    P w[E];
#pragma unroll
    for (int x = 0; x < E; ++x) {
        const int i = x * G + gl;
        w[x] = i < total ? packed[padded(i)] : PK::sentinel();
    }
    warp_sort<P, E, G>(w);
    const P before = __shfl_up_sync(0xffffffffu, w[E - 1], 1, G);
    unsigned head = 0;
#pragma unroll
    for (int x = 0; x < E; ++x) {
        const bool first = x == 0 ? (gl == 0 || PK::key(w[x]) != PK::key(before)) : PK::key(w[x]) != PK::key(w[x > 0 ? x - 1 : 0]);
        if (w[x] != PK::sentinel() && first) head |= 1u << x;
    }
    const int mine = __popc(head);
    int incl = mine;
#pragma unroll
    for (int d = 1; d < G; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, d, G);
        if (gl >= d) incl += t;
    }
    if (NUMERIC) {
        __syncwarp();
        int at = incl - mine;
#pragma unroll
        for (int x = 0; x < E; ++x) {
            packed[padded(gl * E + x)] = w[x];
            if ((head >> x) & 1u) heads[at++] = (unsigned char)(gl * E + x);
        }
        __syncwarp();
    }
    return __shfl_sync(0xffffffffu, incl, G - 1, G);
}

template <typename T, typename P, int G, bool NUMERIC>
__global__ void __launch_bounds__(IG_THREADS, (group_blocks<T, P, NUMERIC>())) ism_group_kernel(const int* __restrict__ rows, int n, const DevCtl* __restrict__ ctl,
                                                                                               Csr A, Csr B, int* __restrict__ cnt,
                                                                                               const i64* __restrict__ rowptr, int* __restrict__ Ccrd,
                                                                                               T* __restrict__ Cval) {
    constexpr int CAP = 8 * G, ROWS = IG_THREADS / G;
    typedef Pack<P, CAP> PK;
    typedef GroupEntry<T, NUMERIC> Entry;
    __shared__ __align__(16) unsigned char smem[ROWS * group_row_bytes<T, P, G, NUMERIC>()];
    const int gl = threadIdx.x % G, group = threadIdx.x / G;
    Entry* const entry = reinterpret_cast<Entry*>(smem) + group * G;
    T* const vals = reinterpret_cast<T*>(smem + ROWS * G * sizeof(Entry)) + group * (NUMERIC ? 9 * G : 0);
    P* const packed = reinterpret_cast<P*>(smem + ROWS * G * (sizeof(Entry) + (NUMERIC ? 9 * sizeof(T) : 0))) + group * group_words<G>();
    unsigned char* const heads = smem + ROWS * (G * (sizeof(Entry) + (NUMERIC ? 9 * sizeof(T) : 0)) + sizeof(P) * group_words<G>()) + group * (NUMERIC ? CAP : 0);
    const T* __restrict__ Aval = (const T*)A.val;
    const T* __restrict__ Bval = (const T*)B.val;
    const int r = chained_start(blockIdx.x * ROWS + group);
    not_before(ctl);
    if (ctl->status != 0) return;
    if ((r & ~(32 / G - 1)) >= n) return;           // (whole warps)
    int row = 0;
    i64 ps = 0, pe = 0;
    if (r < n) {
        row = __ldg(rows + r);
        ps = __ldg(A.pos + row);
        pe = __ldg(A.pos + row + 1);
    }
    // ---- Insert
    int total = 0;
    for (i64 p0 = ps; __any_sync(0xffffffffu, p0 < pe); p0 += G) {
        const i64 p = p0 + gl;
        i64 qs = 0;
        int len = 0;
        T a = 0;
        if (p < pe) {
            const int k = __ldg(A.crd + p);
            if (NUMERIC) a = __ldg(Aval + p);
            if ((unsigned)k < (unsigned)B.nrows) {
                qs = __ldg(B.pos + k);
                len = max((int)(__ldg(B.pos + k + 1) - qs), 0);
            }
        }
        int incl = len;
#pragma unroll
        for (int d = 1; d < G; d <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, d, G);
            if (gl >= d) incl += t;
        }
        const int excl = incl - len;
        const int chunk = min(__shfl_sync(0xffffffffu, incl, G - 1, G), CAP - total);      // (a correctly classed row fits)
        entry[gl].q = qs - excl;
        if constexpr (NUMERIC) entry[gl].a = a;
        __syncwarp();
        const int most = __reduce_max_sync(0xffffffffu, max(chunk, 0));
        for (int u0 = 0; u0 < most; u0 += 4 * G) {
            int col[4];
            T v[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                // the last entry whose running count is <= u
                const int u = u0 + x * G + gl;
                int e = 0;
#pragma unroll
                for (int s = G / 2; s >= 1; s >>= 1) {
                    const int before = __shfl_sync(0xffffffffu, excl, e + s, G);
                    if (before <= u) e += s;
                }
                if (u < chunk) {
                    const Entry d = entry[e];
                    col[x] = __ldg(B.crd + d.q + u);
                    if constexpr (NUMERIC) v[x] = mul_rn(d.a, __ldg(Bval + d.q + u));
                }
            }
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const int u = u0 + x * G + gl, slot = total + u;
                if (u < chunk) {
                    packed[padded(slot)] = PK::make(col[x], slot);
                    if (NUMERIC) vals[slot] = v[x];
                }
            }
        }
        total += max(chunk, 0);
        __syncwarp();
    }
    // ---- Sort
    int distinct;
    const int longest = __reduce_max_sync(0xffffffffu, total);
    if (G == 4 && longest <= 2 * G) distinct = sort_group<PK, P, 2, G, NUMERIC>(packed, heads, total, gl);
    else if (G == 4 && longest <= 4 * G) distinct = sort_group<PK, P, 4, G, NUMERIC>(packed, heads, total, gl);
    else if (longest > 6 * G) distinct = sort_group<PK, P, 8, G, NUMERIC>(packed, heads, total, gl);
    else distinct = sort_group<PK, P, 6, G, NUMERIC>(packed, heads, total, gl);
    // ---- Merge
    if (r < n) {
        if (!NUMERIC) {
            if (gl == 0) cnt[row] = distinct;
        } else {
            const i64 out0 = __ldg(rowptr + row);
            for (int h = gl; h < distinct; h += G) {
                const int x0 = heads[h], x1 = h + 1 < distinct ? (int)heads[h + 1] : total;
                const P w = packed[padded(x0)];
                T sum = vals[PK::slot(w)];
                for (int x = x0 + 1; x < x1; ++x) sum = add_rn(sum, vals[PK::slot(packed[padded(x)])]);
                Ccrd[out0 + h] = (int)PK::key(w);
                Cval[out0 + h] = sum;
            }
        }
    }
}

// blocks an SM is to hold (the compiler would keep several of the networks below in registers at once)
template <typename T, typename P, int CAP, bool NUMERIC>
constexpr int iw_blocks() {
    if (CAP <= 256) return sizeof(P) == 8 || (NUMERIC && sizeof(T) == 8) ? 9 : 12;
    return sizeof(P) == 8 ? 3 : NUMERIC && sizeof(T) == 8 ? 5 : 7;
}

// RANKS: counting: rows may leave their products' places; numeric: some have, and are passed over.
template <typename T, typename P, int CAP, bool NUMERIC, bool RANKS>
__global__ void __launch_bounds__(IW_WARPS * 32, (iw_blocks<T, P, CAP, NUMERIC>())) ism_warp_kernel(const int* __restrict__ perm, int first_cls, int cls, int small_cap, DevCtl* __restrict__ ctl, int counter_slot,
                                                                 Csr A, Csr B, const i64* __restrict__ ub, i64* __restrict__ order_off, char* order_arena,
                                                                 size_t order_bytes, int* __restrict__ cnt,
                                                                 const i64* __restrict__ rowptr, int* __restrict__ Ccrd, T* __restrict__ Cval, int launch_slots) {
    typedef Pack<P, CAP> PK;
    const int slots = CAP > 256 ? launch_slots : CAP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // per warp, `slots` products: values, packed words (one of padding per 32), places of the run heads
    const int padded_slots = slots + slots / 32;
    T* const vals = reinterpret_cast<T*>(smem_raw) + warp * (NUMERIC ? slots : 0);
    P* const packed = reinterpret_cast<P*>(smem_raw + (NUMERIC ? (int)sizeof(T) * slots * IW_WARPS : 0)) + warp * padded_slots;
    unsigned short* const heads = reinterpret_cast<unsigned short*>(smem_raw + ((NUMERIC ? (int)sizeof(T) * slots : 0) + (int)sizeof(P) * padded_slots) * IW_WARPS) + warp * slots;
    chained_start();
    if (ctl->status != 0) return;
    // the rows of the classes first_cls .. cls, one range of perm (with a table of ranges, or the range as arguments, the kernels
    // spill: counting / numeric, rows of 200 products 85 / 123 us, now 83 / 116; stencil 41 x 37 x 53 by ISM, f32, 376 / 317 and 372 / 309)
    int off, n;
    class_range(ctl, first_cls, off, n);
    for (int c = first_cls + 1; c <= cls; ++c) n += ctl->class_count[c];
    const int* __restrict__ rows = perm + off;
    const T* __restrict__ Aval = (const T*)A.val;
    const T* __restrict__ Bval = (const T*)B.val;
    // The way to a row is a chain of loads (its number, its place in perm, its fields, its A entries, their B rows).  AHEAD:
    // the number and the fields of the next row are fetched between the steps of this one.  Worth its registers in the numeric
    // pass of rows beyond 256 products, where few warps are resident (8e4 rows of 674, f32, 20 warps on an SM, 369 -> 345 us).
    // Not below: numeric, f64, 6e4 rows of 200 products on 2^16 columns 123 us with it and 116 without, on 2^25 267 and 253,
    // 1e5 rows of 250 222 and 213.
    constexpr bool AHEAD = NUMERIC && CAP > 256;
    int row, row_n = -1, products, products_n = 0;
    i64 ps, pe, ps_n = 0, pe_n = 0;
    // (from the last row on: those of the largest class first)
    auto take = [&](int r) { row_n = r < n ? __ldg(rows + (n - 1 - r)) : -1; };
    auto fields = [&]() {
        if (row_n < 0) return;
        products_n = (int)min(__ldg(ub + row_n), (i64)0x7fffffff);
        ps_n = __ldg(A.pos + row_n);
        pe_n = __ldg(A.pos + row_n + 1);
    };
    auto next = [&]() {
        int r = 0;
        if (lane == 0) r = atomicAdd(&ctl->work_counter[counter_slot], 1);
        take(__shfl_sync(0xffffffffu, r, 0));
        fields();
    };
    if (AHEAD) next();
    for (;;) {
        if (!AHEAD) next();
        if (row_n < 0) break;
        row = row_n;
        products = products_n;
        ps = ps_n;
        pe = pe_n;
        if (products > slots) {                                    // the CTA kernel's rows
            if (AHEAD) next();
            continue;
        }
        int r_n = 0;
        if (AHEAD && lane == 0) r_n = atomicAdd(&ctl->work_counter[counter_slot], 1);
        P* order = nullptr;
        const bool kept = CAP > 256 && order_arena && products > small_cap;     // a row of CLS_ISM_SMEM: it leaves its order
        if (kept) {
            i64 at = -1;
            if (NUMERIC) {
                at = order_off[row];
                if (RANKS && at >= 0 && (at & ORDER_RANKS)) {      // ism_rank_kernel's row
                    take(__shfl_sync(0xffffffffu, r_n, 0));
                    fields();
                    continue;
                }
            } else if (lane == 0) {
                const u64 bytes = (u64)order_words_of(products) * sizeof(P);
                at = (i64)atomicAdd(&ctl->order_used, bytes);
                if ((u64)at + bytes > order_bytes) at = -1;
            }
            if (!NUMERIC) at = __shfl_sync(0xffffffffu, at, 0);
            if (at >= 0) order = reinterpret_cast<P*>(order_arena + at);
        }
        const bool sorted = CAP > 256 && NUMERIC && order;
        const int lg = pick_group_log(products, pe - ps), gs = 1 << lg;
        const int g = lane >> lg, gl = lane & (gs - 1), ng = 32 >> lg;

        // ---- Insert
        int total = 0;
        for (i64 p0 = ps; p0 < pe; p0 += 32) {
            int len = 0;
            i64 qs = 0;
            T a = 0;
            if (p0 + lane < pe) {
                const int k = __ldg(A.crd + p0 + lane);
                if (NUMERIC) a = __ldg(Aval + p0 + lane);
                if ((unsigned)k < (unsigned)B.nrows) {
                    qs = __ldg(B.pos + k);
                    len = (int)(__ldg(B.pos + k + 1) - qs);
                }
            }
            const int incl = warp_incl_scan(len);
            const int base = total + incl - len;
            const int nE = (int)min((i64)32, pe - p0);
            for (int i = 0; i < nE; i += 2 * ng) {
                // two entries per group, the first element of both loaded before either is stored
                const int e0 = i + g, e1 = min(i + ng + g, 31);
                const i64 q0 = __shfl_sync(0xffffffffu, qs, e0), q1 = __shfl_sync(0xffffffffu, qs, e1);
                const int l0 = __shfl_sync(0xffffffffu, len, e0), b0 = __shfl_sync(0xffffffffu, base, e0);
                const int l1r = __shfl_sync(0xffffffffu, len, e1), b1 = __shfl_sync(0xffffffffu, base, e1);
                const int l1 = i + ng + g < 32 ? l1r : 0;
                T a0 = 0, a1 = 0;
                if (NUMERIC) { a0 = __shfl_sync(0xffffffffu, a, e0); a1 = __shfl_sync(0xffffffffu, a, e1); }
                int c0 = 0, c1 = 0;
                T v0 = 0, v1 = 0;
                if (gl < l0) { if (!sorted) c0 = __ldg(B.crd + q0 + gl); if (NUMERIC) v0 = __ldg(Bval + q0 + gl); }
                if (gl < l1) { if (!sorted) c1 = __ldg(B.crd + q1 + gl); if (NUMERIC) v1 = __ldg(Bval + q1 + gl); }
                auto put = [&](int slot, int col, T v) {
                    if (slot < slots) {                          // always so for a correctly classed row
                        if (!sorted) packed[padded(slot)] = PK::make(col, slot);
                        if (NUMERIC) vals[slot] = v;
                    }
                };
                if (gl < l0) put(b0 + gl, c0, mul_rn(a0, v0));
                for (int t = gl + gs; t < l0; t += gs) put(b0 + t, sorted ? 0 : __ldg(B.crd + q0 + t), NUMERIC ? mul_rn(a0, __ldg(Bval + q0 + t)) : (T)0);
                if (gl < l1) put(b1 + gl, c1, mul_rn(a1, v1));
                for (int t = gl + gs; t < l1; t += gs) put(b1 + t, sorted ? 0 : __ldg(B.crd + q1 + t), NUMERIC ? mul_rn(a1, __ldg(Bval + q1 + t)) : (T)0);
            }
            total += __shfl_sync(0xffffffffu, incl, 31);
        }
        total = min(total, slots);
        __syncwarp();
        if (AHEAD) take(__shfl_sync(0xffffffffu, r_n, 0));

        // ---- Sort
        int distinct;
        const int e = words_per_lane<CAP>(total);
        if (total != products) order = nullptr;             // (a malformed B row)
        P* const keep = CAP > 256 ? order : nullptr;
        bool ranks = false;
        if (!NUMERIC && !RANKS && kept && lane == 0) order_off[row] = order ? (i64)(reinterpret_cast<char*>(order) - order_arena) : -1;
        if constexpr (CAP <= 256) {
            switch (e) {
                case 4: distinct = sort_row<PK, P, 4, NUMERIC, RANKS>(packed, heads, total, keep, gs == 32, &ranks); break;
                case 6: distinct = sort_row<PK, P, 6, NUMERIC, RANKS>(packed, heads, total, keep, gs == 32, &ranks); break;
                default: distinct = sort_row<PK, P, 8, NUMERIC, RANKS>(packed, heads, total, keep, gs == 32, &ranks); break;
            }
        } else {
            switch (e) {
                case 8: distinct = sort_row<PK, P, 8, NUMERIC, RANKS>(packed, heads, total, keep, gs == 32, &ranks); break;
                case 12: distinct = sort_row<PK, P, 12, NUMERIC, RANKS>(packed, heads, total, keep, gs == 32, &ranks); break;
                case 16: distinct = sort_row<PK, P, 16, NUMERIC, RANKS>(packed, heads, total, keep, gs == 32, &ranks); break;
                case 24: distinct = sort_row<PK, P, 24, NUMERIC, RANKS>(packed, heads, total, keep, gs == 32, &ranks); break;
                default: distinct = sort_row<PK, P, 32, NUMERIC, RANKS>(packed, heads, total, keep, gs == 32, &ranks); break;
            }
        }
        if (!NUMERIC && RANKS && kept && lane == 0) order_off[row] = order ? (i64)(reinterpret_cast<char*>(order) - order_arena) | (ranks ? ORDER_RANKS : 0) : -1;
        if (!NUMERIC && RANKS && ranks && lane == 0) atomicAdd(&ctl->n_ranked, 1);

        if (AHEAD) fields();

        // ---- Merge
        if (!NUMERIC) {
            if (lane == 0) cnt[row] = distinct;
        } else {
            const i64 out0 = __ldg(rowptr + row);
            for (int h = lane; h < distinct; h += 32) {
                const int x0 = heads[h], x1 = h + 1 < distinct ? (int)heads[h + 1] : total;
                const P w = packed[padded(x0)];
                T sum = vals[PK::slot(w)];
                for (int x = x0 + 1; x < x1; ++x) sum = add_rn(sum, vals[PK::slot(packed[padded(x)])]);
                Ccrd[out0 + h] = (int)PK::key(w);
                Cval[out0 + h] = sum;
            }
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------------------
// Numeric pass of the rows whose products' places the counting pass has kept: a warp per row, its lanes across one B row after the
// other, so that no two lanes add into one output and every output is summed in loop order.  Bound by the chains of loads that lead
// to a row's B rows: a block for every four rows, four B rows in flight, and shared memory for the outputs alone, so that 40 .. 48
// warps are on an SM (as a path of ism_warp_kernel, at 28 warps, two B rows in flight 246 us, four 211).  Where few rows of the class
// have kept places, a warp looks at `step` rows side by side.
// ---------------------------------------------------------------------------------------
// start of the B row and its length, place of the entry's first product, A value
template <typename T> struct __align__(16) RankEntry { u64 row; T a; int at; };

template <typename T>
__global__ void __launch_bounds__(IW_WARPS * 32, sizeof(T) == 8 ? 10 : 12) ism_rank_kernel(const int* __restrict__ rows, int n_rows, const DevCtl* __restrict__ ctl, Csr A, Csr B,
                                                                                          const i64* __restrict__ ub, const i64* __restrict__ order_off,
                                                                                          const char* __restrict__ order_arena, const i64* __restrict__ rowptr,
                                                                                          int* __restrict__ Ccrd, T* __restrict__ Cval, int most, int step) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (ctl->status != 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    RankEntry<T>* const entry = reinterpret_cast<RankEntry<T>*>(smem_raw) + warp * 32;
    T* const vals = reinterpret_cast<T*>(smem_raw + sizeof(RankEntry<T>) * 32 * IW_WARPS) + warp * most;
    const T* __restrict__ Aval = (const T*)A.val;
    const T* __restrict__ Bval = (const T*)B.val;
    const i64 r = (i64)(blockIdx.x * IW_WARPS + warp) * step + lane;
    int my_row = 0, my_products = 0;
    i64 my_off = -1;
    if (lane < step && r < n_rows) {
        my_row = __ldg(rows + r);
        my_off = __ldg(order_off + my_row);
        my_products = (int)__ldg(ub + my_row);
    }
    // (others are ism_warp_kernel's rows, or a CTA's, of which nothing has written order_off: at most a class's 4096 products)
    for (unsigned todo = __ballot_sync(0xffffffffu, my_products <= ISM_WARP_MAX && my_off >= 0 && (my_off & ORDER_RANKS)); todo; todo &= todo - 1) {
        const int src = __ffs(todo) - 1;
        const int row = __shfl_sync(0xffffffffu, my_row, src), products = __shfl_sync(0xffffffffu, my_products, src);
        const i64 off = __shfl_sync(0xffffffffu, my_off, src);
        const i64 ps = __ldg(A.pos + row), pe = __ldg(A.pos + row + 1), out0 = __ldg(rowptr + row);
        const int n = min((int)(__ldg(rowptr + row + 1) - out0), most);
        const unsigned* __restrict__ cols = reinterpret_cast<const unsigned*>(order_arena + (off & ~ORDER_RANKS));
        const unsigned short* __restrict__ place = reinterpret_cast<const unsigned short*>(cols + n);
        for (int x = lane; x < n; x += 32) {
            Ccrd[out0 + x] = (int)__ldg(cols + x);
            vals[x] = (T)-0.0;                              // (the sum of nothing that leaves the sign of a first zero)
        }
        int total = 0;
        for (i64 p0 = ps; p0 < pe; p0 += 32) {
            RankEntry<T> mine;
            mine.row = 0;
            mine.a = 0;
            if (p0 + lane < pe) {
                const int k = __ldg(A.crd + p0 + lane);
                mine.a = __ldg(Aval + p0 + lane);
                if ((unsigned)k < (unsigned)B.nrows) {
                    const i64 qs = __ldg(B.pos + k);
                    mine.row = (u64)qs << 16 | (u64)min(__ldg(B.pos + k + 1) - qs, (i64)products);
                }
            }
            const int len = (int)(mine.row & 0xffffu), incl = warp_incl_scan(len);
            mine.at = min(total + incl - len, products - len);          // (the lengths add up to the products)
            __syncwarp();
            entry[lane] = mine;
            __syncwarp();
            const bool longer = __any_sync(0xffffffffu, len > 32);
            const int nE = (int)min((i64)32, pe - p0);
            for (int e = 0; e < nE; e += 4) {               // (length 0 past the last entry)
                T v[4];
                int x[4];
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    const RankEntry<T> d = entry[e + y];
                    x[y] = -1;
                    v[y] = 0;
                    if (lane < (int)(d.row & 0xffffu)) { x[y] = __ldg(place + d.at + lane); v[y] = mul_rn(d.a, __ldg(Bval + (d.row >> 16) + lane)); }
                }
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    if (x[y] >= 0) vals[x[y]] = add_rn(vals[x[y]], v[y]);
                    if (longer) {
                        const RankEntry<T> d = entry[e + y];
                        for (int t = 32 + lane; t < (int)(d.row & 0xffffu); t += 32) {
                            const int z = __ldg(place + d.at + t);
                            vals[z] = add_rn(vals[z], mul_rn(d.a, __ldg(Bval + (d.row >> 16) + t)));
                        }
                    }
                    __syncwarp();
                }
            }
            total += __shfl_sync(0xffffffffu, incl, 31);
        }
        for (int x = lane; x < n; x += 32) Cval[out0 + x] = vals[x];
        __syncwarp();
    }
}

template <typename T, typename P, int CAP, int THREADS>
static size_t smem_bytes(bool numeric) {
    return (((numeric ? sizeof(T) * CAP : 0) + sizeof(P) * CAP + 7) & ~(size_t)7) + sizeof(i64) * THREADS + sizeof(T) * THREADS +
           sizeof(int) * (THREADS + 1 + 33) + 16;
}

template <typename T, typename P, int CAP, int THREADS, bool NUMERIC>
static cudaError_t launch_k(const LaunchCtx& c, int cls, int n_host, const Csr& A, const Csr& B,
                            const i64* rowptr, int* Ccrd, void* Cval) {
    const size_t smem = smem_bytes<T, P, CAP, THREADS>(NUMERIC);
    const int slot = NUMERIC ? ISM_CTA_NUM_SLOT : ISM_CTA_SLOT;
    cudaError_t e;
    int per_sm = 0;
    auto k = ism_smem_kernel<T, P, CAP, THREADS, NUMERIC>;
    if ((e = resident_blocks((const void*)k, THREADS, smem, &per_sm)) != cudaSuccess) return e;
    i64 grid = (i64)c.sm_count * (per_sm > 0 ? per_sm : 1);
    if (n_host >= 0 && n_host < grid) grid = n_host > 0 ? n_host : 1;
    k<<<(int)grid, THREADS, smem, c.stream>>>(c.tab.perm, c.ctl, cls, slot, (i64)ISM_WARP_MAX, A, B, c.tab.ub, c.tab.cnt, rowptr, Ccrd, (T*)Cval);
    ++c.launches;
    return cudaGetLastError();
}

template <typename T, typename P, int CAP, bool NUMERIC>
static cudaError_t launch_warp_k(const LaunchCtx& c, const IsmLaunch& l, const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval) {
    // room for the largest row of the launch, where it is known: more warps fit (numeric, 8e4 rows of up to 729 products,
    // f32: 345 us at 1024 slots, 312 us at 768 and seven blocks per SM; f64 435 -> 299 us)
    const int slots = CAP > 256 && c.max_ub_smem > 0 && c.max_ub_smem < CAP ? 32 * words_per_lane<CAP>((int)c.max_ub_smem) : CAP;
    const size_t smem = (size_t)IW_WARPS * ((NUMERIC ? (sizeof(T) + sizeof(short)) * slots : 0) + sizeof(P) * (slots + slots / 32));
    cudaError_t e;
    int per_sm = 0;
    // (words of 64 bits: as before, for the sake of their registers)
    constexpr bool MAY = CAP > 256 && sizeof(P) == 4;
    const bool ranks = MAY && (NUMERIC ? c.order && c.n_ranked > 0 : c.may_rank);
    auto k = ranks ? ism_warp_kernel<T, P, CAP, NUMERIC, MAY> : ism_warp_kernel<T, P, CAP, NUMERIC, false>;
    if ((e = resident_blocks((const void*)k, IW_WARPS * 32, smem, &per_sm)) != cudaSuccess) return e;
    i64 grid = (i64)c.sm_count * (per_sm > 0 ? per_sm : 1);
    const int n = l.n, cls = l.level == 4 ? CLS_ISM_SMEM : CLS_ISM_SMEM_S;
    const i64 want = ((i64)n + IW_WARPS - 1) / IW_WARPS;
    if (want < grid) grid = want > 0 ? want : 1;
    return launch_chained(c, k, grid, IW_WARPS * 32, smem, c.tab.perm, l.first_cls, cls, c.prm.smem_small_cap, c.ctl, cls + (NUMERIC ? NUM_SLOT : 0), A, B, c.tab.ub,
                          c.tab.bm_off, c.order, c.order_bytes, c.tab.cnt, rowptr, Ccrd, (T*)Cval, slots);
}

// Packed words are 32 bits wide when (column, slot) fits below the all-ones sentinel.
template <int CAP>
static bool narrow(const Csr& B) { return (i64)B.ncols < (1ll << (32 - Log2<CAP>::value)); }

size_t order_bytes_of(i64 words, i64 max_products, i64 ncols) {
    if (max_products <= 256) return 0;                  // (sorted again: their kernel keeps no order)
    return (size_t)words * (ncols < (1ll << (32 - Log2<ISM_WARP_MAX>::value)) ? 4 : 8);     // wide words from 2^22 columns on
}

template <typename T, typename P, int G, bool NUMERIC>
static cudaError_t launch_group_k(const LaunchCtx& c, const IsmLaunch& l, const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval) {
    constexpr int ROWS = IG_THREADS / G;
    const int n = l.n;
    return launch_chained(c, ism_group_kernel<T, P, G, NUMERIC>, ((i64)n + ROWS - 1) / ROWS, IG_THREADS, 0, l.rows, n, c.ctl, A, B, c.tab.cnt, rowptr, Ccrd, (T*)Cval);
}

template <typename T, int G>
static cudaError_t launch_group(const LaunchCtx& c, bool numeric, const IsmLaunch& l, const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval) {
    // (the count does not depend on the value type)
    if (narrow<8 * G>(B))
        return numeric ? launch_group_k<T, unsigned, G, true>(c, l, A, B, rowptr, Ccrd, Cval)
                       : launch_group_k<float, unsigned, G, false>(c, l, A, B, rowptr, Ccrd, Cval);
    return numeric ? launch_group_k<T, u64, G, true>(c, l, A, B, rowptr, Ccrd, Cval)
                   : launch_group_k<float, u64, G, false>(c, l, A, B, rowptr, Ccrd, Cval);
}

template <typename T, int CAP>
static cudaError_t launch_warp(const LaunchCtx& c, bool numeric, const IsmLaunch& l, const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval) {
    if (narrow<CAP>(B))
        return numeric ? launch_warp_k<T, unsigned, CAP, true>(c, l, A, B, rowptr, Ccrd, Cval)
                       : launch_warp_k<T, unsigned, CAP, false>(c, l, A, B, rowptr, Ccrd, Cval);
    return numeric ? launch_warp_k<T, u64, CAP, true>(c, l, A, B, rowptr, Ccrd, Cval)
                   : launch_warp_k<T, u64, CAP, false>(c, l, A, B, rowptr, Ccrd, Cval);
}

template <typename T>
static cudaError_t launch_t(const LaunchCtx& c, bool numeric, const IsmLaunch& l, const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval) {
    if (l.level == 0) return launch_group<T, 4>(c, numeric, l, A, B, rowptr, Ccrd, Cval);
    if (l.level == 1) return launch_group<T, 8>(c, numeric, l, A, B, rowptr, Ccrd, Cval);
    if (l.level == 2) return launch_group<T, 16>(c, numeric, l, A, B, rowptr, Ccrd, Cval);
    // (the full class when its largest row is that small: fewer registers and less shared memory per warp)
    i64 most = l.level == 3 ? 256 : c.prm.smem_cap;
    if (l.level == 4 && c.max_ub_smem > 0 && c.max_ub_smem < most) most = c.max_ub_smem;
    if (most <= 256) return launch_warp<T, 256>(c, numeric, l, A, B, rowptr, Ccrd, Cval);
    cudaError_t e = cudaSuccess;
    bool rest = true;
    if (numeric && c.order && c.n_ranked > 0) {
        const int outputs = (int)std::min(most, (i64)ISM_WARP_MAX) / 2;             // (at most half of the products)
        const size_t smem = IW_WARPS * (sizeof(T) * outputs + 32 * sizeof(RankEntry<T>));
        int per_sm = 0;
        if ((e = resident_blocks((const void*)ism_rank_kernel<T>, IW_WARPS * 32, smem, &per_sm)) != cudaSuccess) return e;
        // (two rows a warp: 40000 rows of 576 products of which few, of 595 of which a third rank, f32, a call 443.5 and 534 us with one, 443 and 529
        // with two, 445 and 538 with four, 457 and 534 with up to 32, a warp's ranked rows one after the other; without places 438 and 538)
        const int step = 2 * c.n_ranked <= l.own ? 2 : 1, rows = IW_WARPS * step;
        ism_rank_kernel<T><<<(l.own + rows - 1) / rows, IW_WARPS * 32, smem, c.stream>>>(l.rows + (l.n - l.own), l.own, c.ctl, A, B, c.tab.ub, c.tab.bm_off, c.order, rowptr,
                                                                                        Ccrd, (T*)Cval, outputs, step);
        ++c.launches;
        rest = c.n_ranked < l.own;
        // the rows of smaller classes that go along with these
        if (!rest && l.n > l.own) e = launch_warp<T, 256>(c, numeric, IsmLaunch{3, l.first_cls, l.rows, l.n - l.own, l.n - l.own}, A, B, rowptr, Ccrd, Cval);
    }
    if (e == cudaSuccess && rest) e = launch_warp<T, ISM_WARP_MAX>(c, numeric, l, A, B, rowptr, Ccrd, Cval);
    if (e != cudaSuccess || most <= ISM_WARP_MAX || !rest) return e;
    // rows of 1025 .. 4096 products: a CTA each (a counter of their own: the two kernels share the class);
    // under `auto` they are counted through a hash set of their columns, which needs no order
    const int n = l.own;
    if (!numeric && c.prm.policy == 2) return launch_hash(c, false, CLS_ISM_SMEM, n, A, B, rowptr, Ccrd, Cval);
    if (narrow<4096>(B))
        return numeric ? launch_k<T, unsigned, 4096, 256, true>(c, CLS_ISM_SMEM, n, A, B, rowptr, Ccrd, Cval)
                       : launch_k<T, unsigned, 4096, 256, false>(c, CLS_ISM_SMEM, n, A, B, rowptr, Ccrd, Cval);
    return numeric ? launch_k<T, u64, 4096, 256, true>(c, CLS_ISM_SMEM, n, A, B, rowptr, Ccrd, Cval)
                   : launch_k<T, u64, 4096, 256, false>(c, CLS_ISM_SMEM, n, A, B, rowptr, Ccrd, Cval);
}

cudaError_t launch_ism(const LaunchCtx& c, bool numeric, const IsmLaunch& l, const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval) {
    return c.is_f64 ? launch_t<double>(c, numeric, l, A, B, rowptr, Ccrd, Cval) : launch_t<float>(c, numeric, l, A, B, rowptr, Ccrd, Cval);
}

// A kernel takes any row with fewer products than its own as well, at more instructions a row, and a launch for a handful of rows
// costs 4 .. 10 us: a kernel with no more than ISM_FEW rows leaves them to the next larger one that has rows of its own.  Stencil
// 41 x 37 x 53, 3e3 rows at its edges: a call 824 us with a launch for each class, 796 us.  2000 rows each of 16, 60, 100 and
// 200 products go along with 2100 rows of 400 in 23 + 29 us, and with 50 such rows in 16 + 23, where a kernel each (no lane
// groups then) took 29 + 39 and 24 + 30; 2000 rows of 16 beside 3e4 of 900: 207 + 268 us, 211 + 274.
constexpr i64 ISM_FEW = 2048;
int ism_launches(const LaunchCtx& c, IsmLaunch* out) {
    const i64* const rows = c.class_rows;
    const i64 n[ISM_LEVELS] = {rows[CLS_ISM_REG8] + rows[CLS_ISM_REG16] + rows[CLS_ISM_REG], rows[CLS_ISM_GROUP8], rows[CLS_ISM_GROUP16], rows[CLS_ISM_SMEM_S],
                               rows[CLS_ISM_SMEM]};
    const int cls[ISM_LEVELS] = {CLS_ISM_REG8, CLS_ISM_GROUP8, CLS_ISM_GROUP16, CLS_ISM_SMEM_S, CLS_ISM_SMEM};
    i64 first[ISM_LEVELS] = {rows[CLS_EMPTY]};          // the levels follow one another in perm
    for (int k = 1; k < ISM_LEVELS; ++k) first[k] = first[k - 1] + n[k - 1];
    int made = 0;
    for (int at = ISM_LEVELS - 1, from; at >= 0; at = from) {
        from = at - 1;
        if (n[at] == 0) continue;
        while (from >= 0 && n[from] <= ISM_FEW) --from;
        const i64 start = first[from + 1];
        out[made++] = IsmLaunch{at, cls[from + 1], c.tab.perm + start, (int)(first[at] + n[at] - start), (int)n[at]};
    }
    for (int k = 0; 2 * k < made - 1; ++k) std::swap(out[k], out[made - 1 - k]);
    return made;
}

}  // namespace spws
