// Shared device-side definitions of the spws kernels (sm_100a).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace spws {

typedef long long i64;
typedef unsigned long long u64;

constexpr int NCLASS = 15;
// Row classes = the workspace a row (or (i,j) fibre) is routed to in the symbolic pass.
enum RowClass : int {
    CLS_EMPTY = 0,      // no intermediate product
    CLS_ISM_REG8 = 1,   // insert-sort-merge by 4 lanes per row, two words per lane (<= 8 products)
    CLS_ISM_REG16 = 2,  // ... four words per lane (<= 16 products)
    CLS_ISM_REG = 3,    // ... six or eight words per lane (<= 32 products)
    // (the sparse classes in the order of their products: rows of several go to one launch as one range of perm)
    CLS_ISM_GROUP8 = 4, // insert-sort-merge of at most 64 products by 8 lanes per row
    CLS_ISM_GROUP16 = 5,    // ... of 65 .. 128 products by 16 lanes
    CLS_ISM_SMEM_S = 6, // insert-sort-merge of 129 .. 256 products, one warp per row
    CLS_ISM_SMEM = 7,   // insert-sort-merge in shared memory, full CTA
    CLS_DENSE_WARP = 8, // dense workspace (occupancy bitmap), one warp per row
    CLS_DENSE_HUB = 9,  // dense workspace, CTA units, rows of at least DENSE_HUB_UB products (told apart in the statistics)
    CLS_DENSE_CTA = 10, // dense workspace, CTA units
    CLS_ISM_GLOBAL = 11,    // accumulation array in shared memory, all array in global memory
    CLS_HASH_S = 12,    // hash table in shared memory (reduction at insert time), small CTA
    CLS_HASH = 13,      // hash table in shared memory, full CTA
    CLS_COPY = 14       // one A entry picking a B row of at most COPY_MAX entries: the result is that row, scaled
};
constexpr int NUM_SLOT = 16;   // work_counter[cls] in the symbolic pass, work_counter[NUM_SLOT + cls] in the numeric pass
constexpr int CEIL_SLOT = 32;  // work_counter[CEIL_SLOT + cls] in the gather-only (iteration-only) kernels
constexpr int EMIT_SLOT = 48;  // work_counter slot of the coordinate emission of the CTA dense route
constexpr int BW_SLOT = 49;    // work_counter slot of the word-list build
constexpr int WARP_SLOT = 52;  // work_counter slots of the lists of the warp dense route: numeric, gather-only
constexpr int CEIL_WARP_SLOT = 54;
constexpr int BW_WARP_SLOT = 56; // as BW_SLOT, for the rows a warp takes
constexpr int ISM_CTA_SLOT = 50; // work_counter slots of the CTA kernel of the shared-memory ISM, symbolic and numeric
constexpr int ISM_CTA_NUM_SLOT = 51;
constexpr int N_WORK_COUNTERS = 64;
// index of a class in the public statistics (the register classes are reported as one, and so are the small ISM ones)
__host__ __device__ inline int public_class(int cls) { return cls == CLS_EMPTY ? 0 : (cls <= CLS_ISM_REG || cls == CLS_COPY) ? 1 : cls <= CLS_ISM_SMEM_S ? 2 : cls - 4; }
constexpr int N_PUBLIC_CLASS = 10;
constexpr int HASH_SMALL_CAP = 1024;       // products of a row the small / the full hash workspace takes
constexpr int HASH_CAP = 4096;
constexpr int ISM_WARP_MAX = 1024;         // products of a row the warp kernel of the shared-memory ISM takes

// Capacities fixed at compile time.
constexpr int DENSE_WARP_BM_WORDS = 1024;  // bitmap words a warp-per-row workspace may span (32768 columns)
constexpr int DENSE_WARP_ACC = 256;        // outputs a warp-per-row numeric workspace may hold ...
constexpr int DENSE_WARP_ACC2 = 1024;      // ... and the larger one that `auto` gives rows of more outputs
constexpr int N_WARP_LISTS = 2;            // rows of the warp numeric kernel by those capacities
constexpr int DENSE_WARP_MAX_UB = 4096;    // products a single warp is given at most
constexpr i64 DENSE_HUB_UB = 1ll << 17;    // products from which a row counts as a hub
constexpr int DENSE_MAX_SPAN_WORDS = 16384;// 2^19 columns: the widest bitmap (8 bytes per word with its rank) one CTA holds
// Word lists of long B rows (symbolic pass of the CTA dense route): a B row with at least
// BW_MIN_LEN entries whose entries share bitmap words is also kept as (word index, bits) pairs,
// so that a row that picks it sets one word per pair instead of one bit per entry.
constexpr int COPY_MAX = 256;        // entries of the B row a copied row may pick (eight lanes copy a row)
constexpr int LONG_A_ROW = 1024;     // entries of an A row beyond which a whole CTA computes its bounds
constexpr int BW_MIN_LEN = 256;
constexpr i64 BW_MAX_NNZ = 1ll << 26;      // lists are built only for a B with at most this many entries

enum DevStatus : int {
    DEV_OK = 0,
    DEV_NONCANONICAL = 4,
    DEV_SCRATCH_TOO_SMALL = 5,
    DEV_WORKSPACE_TOO_LARGE = 6,
    DEV_INTERNAL_OVERFLOW = 8
};

// Control block at the start of the scratch buffer (zeroed when a symbolic pass starts).
struct DevCtl {
    i64 nnz;
    i64 products;
    i64 max_ub;
    i64 max_ub_global;      // largest product count among CLS_ISM_GLOBAL rows
    i64 max_ub_smem;        // largest product count among CLS_ISM_SMEM rows (sizes that kernel's launch)
    i64 kept[2];            // TTM: surviving slices (level 0) and fibres (level 1)
    u64 bm_words;           // words of the bitmap arena that the dense rows take (counted by the bounds kernel)
    u64 bm_words_used;      // words handed out so far
    u64 order_words;        // words the sorted CLS_ISM_SMEM rows of up to ISM_WARP_MAX products have (counted by the bounds kernel)
    u64 order_used;         // bytes handed out of their arena
    int n_ranked;           // rows that left their products' places instead of their sorted words
    int status;
    int n_units;            // numeric dense CTA units (row, share of its entries)
    int units_of[7];        // units per bucket of rows (counted by the binning, without the rows that outgrow a warp) ...
    int unit_cursor[7];     // ... and units numbered so far
    int sym_units[2];       // symbolic dense CTA units: shares of split rows, whole rows
    int n_warp_rows[N_WARP_LISTS];  // numeric dense warp rows by the accumulator they need
    int max_span_words;     // widest bitmap among the dense rows
    int max_warp_cnt[N_WARP_LISTS]; // most outputs of a row on each list
    int n_long, n_longest;  // B rows with at least BW_MIN_LEN / BW_BLOCK_ROW entries (candidates for a word list, by a warp / a block)
    int rows_done, slices_done;                 // blocks that have finished
    int rows_ticket, slices_ticket;             // tiles handed out
    int* host_status;       // HostBlock::late (null before the first publication)
    int class_count[NCLASS];
    int class_cursor[NCLASS];
    int work_counter[N_WORK_COUNTERS];   // dynamic work distribution; cleared before each pass
    i64 class_products[NCLASS];
    i64 class_nnz[N_PUBLIC_CLASS];
    i64 dense_warp_products, dense_warp_nnz;   // share of the dense rows the warp numeric kernel takes
};

struct ClassParams {
    int policy;             // spws_policy_t
    int reg_cap;            // CLS_ISM_REG: products <= reg_cap
    int smem_small_cap;     // CLS_ISM_GROUP8, CLS_ISM_GROUP16 and CLS_ISM_SMEM_S (at most 256)
    int smem_cap;           // CLS_ISM_SMEM
    int unit_outputs;       // accumulator capacity of a dense CTA unit
    int max_span_words;     // dense allowed up to this many bitmap words
    float span_words_per_product;
    int unit_cap;           // entries available in the unit table
    int unit_products;      // products a dense CTA unit takes at least; 0: by the job's size
    u64 bm_arena_words;     // capacity of the bitmap arena
    int warp_outputs;       // most outputs of a row that stays with a warp
};

// Scratch of the forms whose first operand is put in output-row order (rowwise.cu).
struct RowwiseBufs {
    u64 *kA, *kB;               // labels of the entries, two buffers for the sort (32 bits each where they fit)
    int *entry[2], *pick;       // numbers of the entries, two buffers; the row that each picks
    char* sort_tmp;
    i64* pos;                   // the reordered operand
    int* crd;
    int* src;
    u64* row_key;               // output-row labels (coordinate-form results)
};

struct Csr {
    const i64* pos;
    const int* crd;
    const void* val;
    int nrows;
    int ncols;
};

// A CSF 3-tensor on the device (three compressed levels).
struct Csf3Dev {
    const i64* pos1;    // n0 + 1
    const i64* pos2;    // n1 + 1
    const int* crd0;
    const int* crd1;
    const int* crd2;
    const void* val;
    int n0, n1;
    i64 nnz;
};

// Per-row tables in scratch.
struct RowTables {
    i64* ub;
    int* cnt;
    int* jmin;
    int* jmax;
    unsigned char* cls;
    int* perm;
    i64* bm_off;        // word offset of the row's bitmap in the arena (dense classes); byte offset of its sorted words (CLS_ISM_SMEM)
    unsigned* bm_arena;
    int* warp_rows;     // numeric: rows handled by the warp-per-row dense kernel: list 0 from the front, list 1 from the back
    int* row_unit0;     // first CTA unit of a row: symbolic (split rows), then numeric
    int* unit_row;      // row of a CTA unit: symbolic (shares of split rows from the front, whole rows from the back), then numeric
};

// Products one dense CTA unit should take: `least`, or more when the whole job is so large that the unit table (rows + 2^19
// entries) would not hold that many units.  By default (least = 0) 2^16 (power law on 2^18 vertices: units of 2^17 products
// cost the accumulation kernel 10 % more, of 2^18 products 35 %, of 2^15 8 %), less in small jobs, so that no block is left alone with the
// last units: a 2048th of the products, 2^13 at least (accumulation in units of 2^16 / 2^15 / 2^14 / 2^13, us: power law on 1500
// vertices 26 / 25 / 21 / 18, 4001 52 / 51 / 38 / 34, 8001 (f64) 142 / 124 / 100 / 93, 16381 191 / 182 / 188 / 208, 60000 1580 / 1562 / 1582 / 1725).
// `total_products` is the sum over the rows that the binning saw: the table and the kernels that
// walk it must divide by the same number.
__host__ __device__ inline i64 dense_unit_products(i64 total_products, int least) {
    const i64 need = (total_products + (1ll << 19) - 1) >> 19;
    i64 unit = least;
    if (least == 0) {
        unit = total_products >> 11;
        if (unit < (1ll << 13)) unit = 1ll << 13;
        if (unit > (1ll << 16)) unit = 1ll << 16;
    }
    return need > unit ? need : unit;
}
// The order in which CTA units are taken.  With few of them the heaviest rows come first, by powers of two of the
// row's products (2^17 and more, 2^16, .., 2^13, fewer, rows that outgrew a warp), so that the last units
// taken are small: power law on 16381 vertices, 4e3 units, accumulation 362 -> 310 us (of the kernel as it was; 251
// today).  With many, units
// are numbered in row order and taken in runs of UNIT_RUN whose order is scattered: rows of like weight
// tend to be neighbours (the hubs of a graph first of all), and a mixture overlaps what heavy and light
// rows wait for: power law on 2^18 vertices, 1.4e5 units, coordinates 4200 -> 3860 us and accumulation
// 14350 -> 14050 us against heaviest first (runs of 64 .. 1024 units within 0.3 %).
constexpr int UNIT_BUCKETS = 7;
static_assert(sizeof(DevCtl::units_of) == 4 * UNIT_BUCKETS, "a counter per bucket");
constexpr int UNIT_FEW = 1 << 14;       // (about 55 units per CTA)
constexpr int UNIT_RUN = 256;
__device__ __forceinline__ int unit_bucket(i64 ub) { return ub >= (1ll << 17) ? 0 : ub < (1ll << 13) ? 5 : __clz((int)ub) - 14; }
__device__ __forceinline__ int unit_at(int t, int n) {
    const unsigned runs = (unsigned)n / UNIT_RUN, run = (unsigned)t / UNIT_RUN;
    if (n < UNIT_FEW || run >= runs) return t;
    return (int)((u64)run * 2654435761ull % runs) * UNIT_RUN + (int)((unsigned)t % UNIT_RUN);      // (a prime: a permutation of the runs)
}
__host__ __device__ inline int dense_units_of_row(i64 ub, i64 unit_products) {
    const i64 n = (ub + unit_products - 1) / unit_products;
    return (int)(n < 1 ? 1 : n);
}

// Symbolic CTA units: a row with more than a 4096th of the products of its kind (about a quarter of what a block of a full grid
// takes in all) is shared by several blocks, which otherwise wait for the one that has it (a 2048th / 16384th: power law on 2^18
// vertices 2806 / 2644 us, 2621 like this), but not below 4096 products (8192 / 2048: 4001 vertices 31 / 25 us, 21 like this;
// 1500 vertices 27 / 16, 20).
constexpr i64 SYM_PART_LEAST = 4096;
inline i64 sym_part_products(i64 cta_products) { return cta_products >> 12 > SYM_PART_LEAST ? cta_products >> 12 : SYM_PART_LEAST; }
__device__ __forceinline__ int sym_parts_of_row(i64 ub, i64 part_products) { return (int)((ub + part_products - 1) / part_products); }

// What a plan keeps in pinned host memory: the control block as last read back, and one slot per
// block of the counting kernels, which write their partial sums there and the host adds up.
constexpr int COUNT_BLOCKS = 256;
// The device writes every 4-byte word of the control block together with the number of the publication, so that
// the host sees word by word what has arrived and no fence has to come before a last word.
constexpr int CTL_WORDS = sizeof(DevCtl) / 4;
struct HostBlock {
    DevCtl ctl;             // as the host last received it
    int late;               // status raised after the first publication of a pass, which clears it
    int pad[31];
    u64 words[CTL_WORDS];   // number of the publication above a word of the control block
    u64 partial[2 * COUNT_BLOCKS];
};

// The first error wins; it is also written to the plan's pinned block once that is known.
__device__ __forceinline__ void raise_status(DevCtl* ctl, int s) {
    if (atomicCAS(&ctl->status, 0, s) == 0 && ctl->host_status) *(volatile int*)ctl->host_status = s;
}

// Start of a kernel that launch_chained() enqueues: waits until all that came before it in the stream is done and what it wrote is
// there; then the blocks of the kernel launched next may be placed as room comes free.  No load on the read-only path may be moved
// above the wait: its address comes from the number that is returned (the one given), from a pointer that has passed not_before(),
// or from what was loaded or counted since.  (All pointers through the wait cost the bounds kernel registers: stencil of 2^18
// rows 47 -> 50 us.)
__device__ __forceinline__ int chained_start(int x = 0) {
    asm volatile("griddepcontrol.wait;" : "+r"(x) : : "memory");
    asm volatile("griddepcontrol.launch_dependents;" : : : "memory");
    return x;
}
template <typename P> __device__ __forceinline__ void not_before(P& p) { asm volatile("" : "+l"(p) : : "memory"); }
__device__ __forceinline__ void not_before(Csr& m) { not_before(m.pos); not_before(m.crd); }

// Copies the control block to pinned host memory, which the host polls (a whole block of threads, after the counters are
// final): it goes on about 5 us before a stream synchronisation would let it.  A system-wide fence before a single number
// cost the publishing kernel 4 us (row pointer of 2048 rows: 10.4 us with it, 6.4 us with a number in every word).
__device__ __forceinline__ void publish_ctl(const DevCtl* ctl, HostBlock* host, int seq) {
    for (int w = threadIdx.x; w < CTL_WORDS; w += blockDim.x)
        *(volatile u64*)&host->words[w] = (u64)(unsigned)seq << 32 | reinterpret_cast<volatile const unsigned*>(ctl)[w];
}

// True in every thread of the last of `blocks` blocks to come here; all earlier blocks' writes are visible to it.
__device__ __forceinline__ bool last_block(int* done, int blocks) {
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done, 1) == blocks - 1;
    __syncthreads();
    if (s_last) __threadfence();
    return s_last != 0;
}

// ---- running sums handed from tile to tile ---------------------------------------------------
// A tile of a single-pass scan publishes one 64-bit word: a tag above 56 bits of count.  The tag of a
// pass is 2 * pass + 1 while the word holds the tile's own count and 2 * pass + 2 once it holds the
// count of all tiles up to it, so one clearing serves all the passes of a sort.  Tiles are numbered
// by a ticket taken when a block starts, hence every tile that is waited for is running or done; a
// wait that does not end after LOOK_LIMIT polls raises the status word and goes on with what it has
// (too small a count, so that every index stays inside the arrays).
constexpr int LOOK_SHIFT = 56;
constexpr u64 LOOK_MASK = (1ull << LOOK_SHIFT) - 1;
constexpr int LOOK_LIMIT = 1 << 22;

__device__ __forceinline__ void look_publish(u64* word, int tag, i64 count) {
    *(volatile u64*)word = ((u64)tag << LOOK_SHIFT) | (u64)count;
}

// Sum of the counts of the tiles before `tile` (one word per tile, `stride` words apart): a single
// thread walks back until it meets a running sum, WORDS a step, loaded side by side (tiles that start together find few
// running sums; sorting 7e5 entries, three passes, 52 us a word at a time, 43 us with four).
template <int WORDS>
__device__ __forceinline__ i64 look_back(const u64* words, int stride, int tile, int pass, DevCtl* ctl) {
    i64 sum = 0;
    int polls = 0;
    for (int t = tile - 1; t >= 0;) {
        u64 w[WORDS];
#pragma unroll
        for (int x = 0; x < WORDS; ++x) w[x] = *(const volatile u64*)(words + (i64)max(t - x, 0) * stride);
#pragma unroll
        for (int x = 0; x < WORDS; ++x) {
            const int tag = (int)(w[x] >> LOOK_SHIFT);
            if (tag <= 2 * pass) {                              // not there yet: again from this one
                if (++polls >= LOOK_LIMIT) { raise_status(ctl, DEV_INTERNAL_OVERFLOW); return sum; }
                break;
            }
            sum += (i64)(w[x] & LOOK_MASK);
            if (tag == 2 * pass + 2) return sum;
            --t;                                                // (the first tile's sum is a running one: t >= 0)
        }
    }
    return sum;
}

// The same for a whole warp: 32 predecessors per step.  Every lane returns the sum.
__device__ __forceinline__ i64 look_back_warp(const u64* words, int tile, int pass, DevCtl* ctl) {
    const int lane = threadIdx.x & 31;
    i64 sum = 0;
    int polls = 0;
    for (int t0 = tile - 1; t0 >= 0; t0 -= 32) {
        const int t = t0 - lane;
        u64 w = (u64)(2 * pass + 2) << LOOK_SHIFT;              // before the first tile: a running sum of nothing
        for (;;) {
            if (t >= 0) w = *(const volatile u64*)(words + t);
            if (__all_sync(0xffffffffu, (int)(w >> LOOK_SHIFT) > 2 * pass)) break;
            if (++polls >= LOOK_LIMIT) {
                if (lane == 0) raise_status(ctl, DEV_INTERNAL_OVERFLOW);
                return sum;
            }
        }
        const unsigned ends = __ballot_sync(0xffffffffu, (int)(w >> LOOK_SHIFT) == 2 * pass + 2);
        const int last = ends ? __ffs(ends) - 1 : 31;           // the nearest running sum ends the walk
        i64 v = lane <= last ? (i64)(w & LOOK_MASK) : 0;
        for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
        sum += v;
        if (ends) break;
    }
    return sum;
}


// ---- warp-per-row insert-sort-merge: words each lane holds for a row of `total` words, lanes whose words are
// kept in scratch, and the words kept of a row that the kernel for up to ISM_WARP_MAX products sorts
template <int CAP>
__host__ __device__ __forceinline__ int words_per_lane(int total) {
    if (CAP <= 256) return total <= 128 ? 4 : total <= 192 ? 6 : 8;
    return total <= 384 ? (total <= 256 ? 8 : 12) : total <= 512 ? 16 : total <= 768 ? 24 : 32;
}
__host__ __device__ __forceinline__ int order_lanes(int total, int e) { return ((total + e - 1) / e + 7) & ~7; }
__host__ __device__ __forceinline__ int order_words_of(int total) {
    const int e = words_per_lane<ISM_WARP_MAX>(total);
    return e * order_lanes(total, e);
}

// Rows of class `cls` are perm[off, off + n).
__device__ __forceinline__ void class_range(const DevCtl* ctl, int cls, int& off, int& n) {
    off = 0;
    for (int c = 0; c < cls; ++c) off += ctl->class_count[c];
    n = ctl->class_count[cls];
}

__device__ __forceinline__ int warp_incl_scan(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += t;
    }
    return v;
}

// Exclusive scan over a block of THREADS threads; `ws` needs 33 ints; every thread gets `total`.
template <int THREADS>
__device__ __forceinline__ int block_excl_scan(int v, int* ws, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int incl = warp_incl_scan(v);
    __syncthreads();                       // ws may still be read from a previous call
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int s = (lane < THREADS / 32) ? ws[lane] : 0;
        const int si = warp_incl_scan(s);
        if (lane < THREADS / 32) ws[lane] = si - s;
        if (lane == 31) ws[32] = si;
    }
    __syncthreads();
    total = ws[32];
    return ws[warp] + incl - v;
}

// Sum over the block, valid in thread 0; `ws` needs one word per warp.
template <int THREADS>
__device__ __forceinline__ i64 block_sum(i64 v, i64* ws) {
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < THREADS / 32; ++w) v += ws[w];
    return v;
}

// First position in crd[lo, hi) whose coordinate is >= c (rows are sorted).
__device__ __forceinline__ i64 lower_bound_crd(const int* __restrict__ crd, i64 lo, i64 hi, i64 c) {
    while (lo < hi) {
        const i64 mid = (lo + hi) >> 1;
        if ((i64)__ldg(crd + mid) < c) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// lanes per A entry: the smallest power of two >= the mean B-row segment length
__device__ __forceinline__ int pick_group_log(i64 ub, i64 entries) {
    return (ub > entries) + (ub > 2 * entries) + (ub > 4 * entries) + (ub > 8 * entries) + (ub > 16 * entries);
}

// Products are formed as a rounded multiply followed by rounded adds (no contraction), so the
// routes that sum in product order reproduce a plain sequential sum bit for bit.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }

// ---- launchers (defined in the .cu files) ------------------------------------------------
struct LaunchCtx {
    cudaStream_t stream;
    int sm_count;
    DevCtl* ctl;
    ClassParams prm;
    RowTables tab;
    int is_f64;
    int dense_smem_words;    // bitmap words the CTA dense kernels reserve (from ncols)
    char* rest;              // scratch after the fixed tables: bitmap arena, sorted words, then the ISM-global arena
    size_t rest_bytes;
    char* order;             // arena of sorted words (null: every pass sorts)
    size_t order_bytes;
    int may_rank;            // counting: rows may leave their products' places; n_ranked: numeric, such rows of the pass
    int n_ranked;
    int global_cap;          // accumulation-array capacity of CLS_ISM_GLOBAL
    HostBlock* host;         // the plan's pinned block: receives the control block ...
    int seq;                 // ... as publication `seq` (class sizes) and `seq` + 1 (row pointer)
    u64* look;               // one word per tile of the kernels that hand running sums on ...
    int n_look;              // ... cleared by the binning kernel
    i64 unit_nnz;            // numeric: outputs of a dense CTA unit's row on average, shared out among its units ...
    i64 b_bytes;             // ... and coordinates and values of B
    i64 max_ub_smem;         // largest product count of a CLS_ISM_SMEM row when known (0: unknown)
    const i64* class_rows;   // rows per class, once they are binned
    uint2* bw;               // word lists of long B rows, indexed like B's entries (null: not built)
    int* bw_long;            // the long B rows, in arrival order
    int bw_long_cap;
    int4* brow;                 // per B row: first column, last column, length (null: not kept)
    mutable int launches;    // kernels enqueued through this context
    int chain;               // kernels that begin with chained_start() may be launched so that their blocks are placed while the one before ends
};

// Enqueues a kernel that begins with chained_start().  Chained, the gap between two kernels (1.3 .. 2.5 us) all but goes: 2048 rows of 64 products
// 63.7 -> 55.1 us a call, 30011 rows of 143 142 -> 135, 65536 rows over 2^26 columns 108.7 -> 101.2.  Not on forked streams, where the host takes some 9 us for such a
// launch behind an event, and the waiting blocks take room that other kernels have use for (fibres of 110 products 419 -> 432), nor
// while the stream is being captured.
template <typename... P, typename... A>
inline cudaError_t launch_chained(const LaunchCtx& c, void (*kernel)(P...), i64 grid, int threads, size_t smem, A... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c.stream;
    cfg.attrs = &at;
    cfg.numAttrs = c.chain ? 1 : 0;
    ++c.launches;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Blocks of `kernel` that fit one SM with `smem` bytes of dynamic shared memory, for which the kernel is made ready.
cudaError_t resident_blocks(const void* kernel, int threads, size_t smem, int* per_sm);

// setup.cu
cudaError_t launch_validate(const LaunchCtx& c, const Csr& A, const Csr& B, i64 nnzA, i64 nnzB);
// clear_ctl: the control block is cleared by the first kernel
cudaError_t launch_row_bounds(const LaunchCtx& c, const Csr& A, const Csr& B, i64 nnzA, bool clear_ctl);
// symbolic units of the CTA rows; word lists of long B rows
// (products: of the CTA rows)
cudaError_t launch_cta_prepare(const LaunchCtx& c, i64 products, const Csr& B);
// (also publishes the class sizes to the host)
cudaError_t launch_bin_rows(const LaunchCtx& c, int m);
// row pointer, numeric routing of the dense rows, outputs per class
cudaError_t launch_finish_rows(const LaunchCtx& c, int m, bool any_dense, i64* rowptr);
// the same for the fibres of a 3-tensor, with C's upper levels; sfp: n_i + 1 words of scratch
cudaError_t launch_finish_fibres(const LaunchCtx& c, int n_i, int n_ij, bool any_dense, const i64* Apos1, const int* Acrd0, const int* Acrd1,
                                 i64* rowptr_raw, i64* sfp, i64* Cpos0, int* Ccrd0, i64* Cpos1, int* Ccrd1, i64* Cpos2);
size_t look_words(i64 rows, i64 slices);
// exclusive scan of n counts into n + 1 positions
cudaError_t launch_scan_counts(const LaunchCtx& c, const int* cnt, int n, i64* out, i64* block_sums, i64* total_out);
// class kernels: n_host < 0 means "size the grid for any count"
cudaError_t launch_copy_rows(const LaunchCtx& c, const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval);
// The insert-sort-merge rows of up to smem_cap products by the kernels that take them: 4, 8 or 16 lanes per row (at most 32, 64 or
// 128 products), a warp per row (256), the kernels of the full class.
constexpr int ISM_LEVELS = 5;
// One launch: its rows lie one after the other in perm, the `own` rows of its level behind those of lower levels.
struct IsmLaunch {
    int level, first_cls;
    const int* rows;
    int n, own;
};
// the launches for the rows as binned (at most ISM_LEVELS, lowest level first); returns their number
int ism_launches(const LaunchCtx& c, IsmLaunch* out);
cudaError_t launch_ism(const LaunchCtx& c, bool numeric, const IsmLaunch& l, const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval);
// scratch that keeps the sorted words of the rows of the warp-per-row ISM from the counting pass to the numeric one;
// words: DevCtl::order_words, max_products: of a CLS_ISM_SMEM row
size_t order_bytes_of(i64 words, i64 max_products, i64 ncols);
// max_span_words: widest dense row of the pass
cudaError_t launch_dense_sym_warp(const LaunchCtx& c, int max_span_words, const Csr& A, const Csr& B);
cudaError_t launch_dense_sym_cta(const LaunchCtx& c, i64 products, const Csr& A, const Csr& B);
// chk_idx / chk_val non-null: the gather-only form of the same kernel (workspace stripped, checksums out).
// n[], max_cnt[]: rows on each list and their largest output counts
cudaError_t launch_dense_num_warp(const LaunchCtx& c, const int* n, const int* max_cnt, int m, int max_span_words, const Csr& A, const Csr& B,
                                  const i64* rowptr, int* Ccrd, void* Cval, u64* chk_idx = nullptr, double* chk_val = nullptr);
// phase 0: write the coordinates and clear the value segments several units add into; 1: accumulate.
// total_products: products of all rows of the pass, as the control block had them when the units were numbered
cudaError_t launch_dense_num_cta(const LaunchCtx& c, int phase, int n_units_host, int max_span_words, i64 total_products,
                                 const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval,
                                 u64* chk_idx = nullptr, double* chk_val = nullptr);
cudaError_t launch_ism_global(const LaunchCtx& c, bool numeric, int n_host, const Csr& A, const Csr& B,
                              const i64* rowptr, int* Ccrd, void* Cval);
cudaError_t launch_hash(const LaunchCtx& c, bool numeric, int cls, int n_host, const Csr& A, const Csr& B, const i64* rowptr,
                        int* Ccrd, void* Cval);

// outer.cu: second-order workspaces of the outer-product form
cudaError_t launch_outer_counts(const LaunchCtx& c, const Csr& At, const Csr& B, int* cnt);
size_t outer_sort_scratch_bytes(i64 n);
cudaError_t launch_outer_ism(const LaunchCtx& c, bool numeric, const Csr& At, const Csr& B, const i64* koff, i64 P, i64 cap, i64 J,
                             int label_bits, u64* kA, void* vA, u64* kB, void* vB, char* sort_tmp, i64* nnz_dev, i64* nnz_host_pinned,
                             bool* result_first);
cudaError_t launch_coo_pos(const LaunchCtx& c, const u64* ukeys, i64 nnz, i64 m, i64 J, i64* pos);
cudaError_t launch_coo_out(const LaunchCtx& c, const u64* ukeys, const void* uvals, i64 nnz, i64 J, int* Ccrd, void* Cval);
cudaError_t launch_outer_dense(const LaunchCtx& c, bool numeric, const Csr& At, const Csr& B, const i64* koff, i64 P, i64 m, i64 J,
                               unsigned* dbits, void* dvals, int* cnt, const i64* pos, int* Ccrd, void* Cval);
// number of products; partial[0 .. *blocks) (pinned host memory, cleared by the caller) receives one sum per block, plus one
cudaError_t launch_outer_total(const LaunchCtx& c, const Csr& At, const Csr& B, u64* partial, int* blocks);
// higher.cu: the higher-order scatters with coordinate-form output
// (and partial[COUNT_BLOCKS ..] another)
cudaError_t launch_higher_total(const LaunchCtx& c, int form, const Csf3Dev& B, const Csr& C, u64* partial, int* blocks);
cudaError_t launch_higher_setup(const LaunchCtx& c, int form, const Csf3Dev& B, const Csr& C, int* fib_of, int* slice_of, int* cnt);
cudaError_t launch_higher_ism(const LaunchCtx& c, bool numeric, int form, const Csf3Dev& B, const Csr& C, const Csr& D, const int* fib_of,
                              const int* slice_of, const i64* eoff, i64 P, i64 cap, u64 d1, u64 d2, int label_bits, u64* kA, void* vA,
                              u64* kB, void* vB, char* sort_tmp, i64* nnz_dev, i64* nnz_host_pinned, bool* result_first);
cudaError_t launch_higher_unpack(const LaunchCtx& c, int order, const u64* ukeys, const void* uvals, i64 nnz, u64 d1, u64 d2, int* o0,
                                 int* o1, int* o2, void* oval, bool interleaved);

// rowwise.cu: the same forms taken row by row
size_t rw_sort_bytes(i64 n);
// (first of all: clears the control block and the temporaries of a sort of n entries)
cudaError_t launch_rw_clear(const LaunchCtx& c, i64 n, char* sort_tmp);
cudaError_t launch_rw_outer(const LaunchCtx& c, const Csr& At, i64 n, const Csr& B, i64 nnzB, int bits, const RowwiseBufs& b);
// d0, d1: extents of the coordinates of a label
cudaError_t launch_rw_csf(const LaunchCtx& c, int form, const Csf3Dev& B, u64 d0, u64 d1, i64 m, int bits, const RowwiseBufs& b);
cudaError_t launch_rw_values(const LaunchCtx& c, const void* val, const int* src, i64 n, void* out);
cudaError_t launch_rw_fibre_rows(const LaunchCtx& c, bool values, const Csf3Dev& B, const Csr& C, const Csr& D, int* cnt, i64* fpos, int* fcrd,
                                 void* fval, i64* block_sums);
cudaError_t launch_rw_coords(const LaunchCtx& c, int order, const i64* rowptr, const u64* row_key, i64 m, i64 nnz, u64 d, const int* cols, int* o0,
                             int* o1, int* o2, bool interleaved);

}  // namespace spws
