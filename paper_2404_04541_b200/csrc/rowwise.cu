// The scatters of second and third order taken row by row.
//
// When a form's first operand is put in the order of the output rows, the reduction variable moves
// next to the last index and every output row owns a first-order workspace (Sec. 2.2), whose rows
// the row-wise kernels count and fill.  Only the stored ENTRIES of the first operand are sorted
// (label = output row, stable, so a row keeps its entries in loop order), never the products, and
// nothing of size I x J is touched:
//   outer      C(i,j)   = A(k,i) B(k,j)          rows i,      entry (k,i)   picks row k of B
//   SpTTM      A(i,j,l) = B(k,i,j) C(k,l)        rows (i,j),  entry (k,i,j) picks row k of C
//   SpTTM-I    A(k,j,l) = B(k,i,j) C(i,l)        rows (k,j),  entry (k,i,j) picks row i of C
//   SpMTTKRP   A(i,j)   = B(k,l,i) C(k,j) D(l,j) rows i,      entry (k,l,i) picks row (k,l) of F,
//              F((k,l),j) = C(k,j) D(l,j) formed once per stored fibre (k,l)
// The reordered operand is a CSR matrix in scratch: pos, crd (the picked row), src (where the entry's
// value stands in the operand as given, so that a numeric pass reads the values of its own call).
#include <algorithm>

#include "sortmerge.cuh"

namespace spws {

// The last r in [lo, hi) with pos[r] <= p (pos[lo] <= p < pos[hi]).
__device__ __forceinline__ int owner_row(const i64* __restrict__ pos, int lo, int hi, i64 p) {
    while (hi - lo > 1) {
        const int mid = (int)(((i64)lo + hi) >> 1);
        if (__ldg(pos + mid) <= p) lo = mid; else hi = mid;
    }
    return lo;
}

// The same by a whole warp, 32 probes a step: a block looks for the owners of its tile among all rows first (the keys of 1e6 entries
// in 5e5 fibres 31 us by halves, 27 us like this; of 7e5 in 5e4 rows 23 and 18).  Inside [lo, hi) whatever the offsets, as by halves.
__device__ __forceinline__ int owner_row_warp(const i64* __restrict__ pos, int lo, int hi, i64 p) {
    const int lane = threadIdx.x & 31;
    while (hi - lo > 1) {
        const int step = (int)(((unsigned)(hi - lo) + 31u) >> 5);
        const i64 at = lo + (i64)lane * step;
        const int n = max(__popc(__ballot_sync(0xffffffffu, at < hi && __ldg(pos + at) <= p)), 1);
        hi = (int)min((i64)hi, lo + (i64)n * step);
        lo += (n - 1) * step;
    }
    return lo;
}

constexpr int RK_ITEMS = 4;
constexpr int RK_TILE = OT * RK_ITEMS;

// Output-row label (K: 32 bits where they hold it) and picked row of every entry; a block takes a tile of
// consecutive entries, so the owners of its first and last entry bound every search.  B's columns
// are checked on the way (the row kernels look at the ends of a row only).
template <typename K>
__global__ void __launch_bounds__(OT) rw_keys_outer_kernel(Csr At, i64 n, Csr B, i64 nnzB, K* __restrict__ keys, int* __restrict__ pick,
                                                           int passes, SortHead* head, DevCtl* ctl) {
    __shared__ int s_lo, s_hi;
    __shared__ DigitCounts s_digits;
    bool bad = false;
    chained_start();
    not_before(At);
    not_before(B);
    s_digits.start(passes);
    for (i64 q = (i64)blockIdx.x * OT + threadIdx.x; q < nnzB; q += (i64)gridDim.x * OT) bad |= (unsigned)__ldg(B.crd + q) >= (unsigned)B.ncols;
    for (i64 t0 = (i64)blockIdx.x * RK_TILE; t0 < n; t0 += (i64)gridDim.x * RK_TILE) {
        __syncthreads();
        if (threadIdx.x < 32) {
            const int r = owner_row_warp(At.pos, 0, At.nrows, t0);
            if (threadIdx.x == 0) s_lo = r;
        } else if (threadIdx.x < 64) {
            const int r = owner_row_warp(At.pos, 0, At.nrows, min(n, t0 + RK_TILE) - 1);
            if (threadIdx.x == 32) s_hi = r + 1;
        }
        __syncthreads();
        for (int x = 0; x < RK_ITEMS; ++x) {
            const i64 p = t0 + x * OT + threadIdx.x;
            if (p >= n) break;
            const int i = __ldg(At.crd + p);
            bad |= (unsigned)i >= (unsigned)At.ncols;
            keys[p] = (K)(unsigned)i;
            s_digits.add((u64)(unsigned)i, passes);
            pick[p] = owner_row(At.pos, s_lo, s_hi, p);
        }
    }
    s_digits.flush(passes, head);
    if (bad) raise_status(ctl, DEV_NONCANONICAL);
}

// form: 0 SpTTM, 1 SpTTM-I, 2 SpMTTKRP.  Label: a * d1 + b of coordinates below d0 and d1 (forms 0, 1), a alone (form 2), which are
// checked on the way: a label cut to 32 bits would be another row's.
// pos[0 .. m] := nnz on the way (rw_sparse_rows_kernel writes the rows there are).
template <typename K>
__global__ void __launch_bounds__(OT) rw_keys_csf_kernel(int form, Csf3Dev B, u64 d0, u64 d1, K* __restrict__ keys, int* __restrict__ picks, int passes,
                                                         SortHead* head, i64* __restrict__ pos, i64 m, DevCtl* ctl) {
    __shared__ int s_f[2], s_s[2];
    __shared__ DigitCounts s_digits;
    bool bad = false;
    chained_start();
    not_before(B.pos1);
    not_before(B.pos2);
    not_before(B.crd0);
    not_before(B.crd1);
    not_before(B.crd2);
    s_digits.start(passes);
    for (i64 i = (i64)blockIdx.x * OT + threadIdx.x; i <= m; i += (i64)gridDim.x * OT) pos[i] = B.nnz;
    for (i64 t0 = (i64)blockIdx.x * RK_TILE; t0 < B.nnz; t0 += (i64)gridDim.x * RK_TILE) {
        __syncthreads();
        if (threadIdx.x < 64) {
            const int which = threadIdx.x >> 5;
            const int f = owner_row_warp(B.pos2, 0, B.n1, which == 0 ? t0 : min(B.nnz, t0 + RK_TILE) - 1);
            const int s = owner_row_warp(B.pos1, 0, B.n0, f);
            if ((threadIdx.x & 31) == 0) { s_f[which] = f; s_s[which] = s; }
        }
        __syncthreads();
        for (int x = 0; x < RK_ITEMS; ++x) {
            const i64 e = t0 + x * OT + threadIdx.x;
            if (e >= B.nnz) break;
            const int f = owner_row(B.pos2, s_f[0], s_f[1] + 1, e);
            const u64 c2 = (u64)(unsigned)__ldg(B.crd2 + e);
            u64 key = c2, pick = (u64)(unsigned)f;
            if (form != 2) {
                const u64 c1 = (u64)(unsigned)__ldg(B.crd1 + f);
                const u64 c0 = (u64)(unsigned)__ldg(B.crd0 + owner_row(B.pos1, s_s[0], s_s[1] + 1, f));
                const u64 a = form == 0 ? c1 : c0;
                key = a * d1 + c2;
                pick = form == 0 ? c0 : c1;
                bad |= a >= d0 || c2 >= d1;
            } else {
                bad |= c2 >= d0;
            }
            keys[e] = (K)key;
            s_digits.add(key, passes);
            picks[e] = (int)pick;
        }
    }
    s_digits.flush(passes, head);
    if (bad) raise_status(ctl, DEV_NONCANONICAL);
}

// CSR result: the reordered operand has one row per output row; pos by binary search in the sorted labels.
template <typename K>
__global__ void __launch_bounds__(OT) rw_dense_rows_kernel(const K* __restrict__ keys, const int* __restrict__ entry, const int* __restrict__ pick, i64 n, i64 m,
                                                           i64* __restrict__ pos, int* __restrict__ crd, int* __restrict__ src) {
    const i64 stride = (i64)gridDim.x * OT, t0 = (i64)blockIdx.x * OT + threadIdx.x;
    chained_start();
    not_before(keys);
    not_before(entry);
    not_before(pick);
    for (i64 i = t0; i <= m; i += stride) {
        i64 lo = 0, hi = n;
        while (lo < hi) {
            const i64 mid = (lo + hi) >> 1;
            if ((u64)keys[mid] < (u64)i) lo = mid + 1; else hi = mid;
        }
        pos[i] = lo;
    }
    for (i64 p = t0; p < n; p += stride) {
        const int e = entry[p];
        crd[p] = pick[(unsigned)e];
        src[p] = e;
    }
}

// Coordinate-form result: only the labels that occur become rows, in order (row r has label row_key[r]);
// pos was filled with n, so the rows past the last label are empty.  Tiles hand the number of rows
// on as in reduce_runs_kernel.  More than m labels mean a coordinate out of its range.
// (1024 tiles of 1e6 entries: 22.7 us at six blocks an SM, 17.6 with all of them resident)
template <typename K>
__global__ void __launch_bounds__(OT, 8) rw_sparse_rows_kernel(const K* __restrict__ keys, const int* __restrict__ entry, const int* __restrict__ pick, i64 n, i64 m,
                                                            int* __restrict__ ticket, u64* __restrict__ status, DevCtl* ctl,
                                                            u64* __restrict__ row_key, i64* __restrict__ pos, int* __restrict__ crd,
                                                            int* __restrict__ src) {
    __shared__ u64 s_edge[RK_ITEMS][OT / 32];
    __shared__ int s_ws[33];
    __shared__ int s_tile;
    __shared__ i64 s_before;
    chained_start();
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1);
    __syncthreads();
    const int tile = s_tile;
    const i64 t0 = (i64)tile * RK_TILE;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    u64 key[RK_ITEMS];
#pragma unroll
    for (int x = 0; x < RK_ITEMS; ++x) {
        const i64 p = t0 + x * OT + threadIdx.x;
        key[x] = p < n ? (u64)keys[p] : ABSENT_LABEL;
        if (p < n) {
            const int e = entry[p];
            crd[p] = pick[(unsigned)e];
            src[p] = e;
        }
        if (lane == 31) s_edge[x][warp] = key[x];
    }
    __syncthreads();
    // heads before this thread's in the tile = heads of the earlier rounds of OT entries + of its round
    int rank[RK_ITEMS], total = 0;
    bool head[RK_ITEMS];
#pragma unroll
    for (int x = 0; x < RK_ITEMS; ++x) {
        u64 prev = __shfl_up_sync(0xffffffffu, key[x], 1);
        if (lane == 0) {
            if (warp > 0) prev = s_edge[x][warp - 1];
            else if (x > 0) prev = s_edge[x - 1][OT / 32 - 1];
            else prev = t0 > 0 ? (u64)keys[t0 - 1] : ABSENT_LABEL;
        }
        head[x] = key[x] != ABSENT_LABEL && key[x] != prev;
        int round;
        rank[x] = total + block_excl_scan<OT>(head[x], s_ws, round);
        total += round;
    }
    if (warp == 0) {
        if (lane == 0) look_publish(status + tile, tile == 0 ? 2 : 1, total);
        i64 before = 0;
        if (tile > 0) {
            before = look_back_warp(status, tile, 0, ctl);
            if (lane == 0) look_publish(status + tile, 2, before + total);
        }
        if (lane == 0) s_before = before;
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < RK_ITEMS; ++x)
        if (head[x]) {
            const i64 r = s_before + rank[x];
            if (r >= m) { raise_status(ctl, DEV_NONCANONICAL); continue; }
            row_key[r] = key[x];
            pos[r] = t0 + x * OT + threadIdx.x;
        }
}

template <typename T>
__global__ void __launch_bounds__(OT) rw_values_kernel(const T* __restrict__ val, const int* __restrict__ src, i64 n, T* __restrict__ out) {
    for (i64 p = (i64)blockIdx.x * OT + threadIdx.x; p < n; p += (i64)gridDim.x * OT) out[p] = __ldg(val + (unsigned)src[p]);
}

// Rows of F (SpMTTKRP): a warp per stored fibre (k,l) walks the shorter of C's row k and D's row l and
// looks every column up in the longer one.  PASS 0 counts, 1 writes the columns, 2 the products.
template <typename T, int PASS>
__global__ void __launch_bounds__(OT) rw_fibre_rows_kernel(Csf3Dev B, Csr C, Csr D, int* __restrict__ cnt, const i64* __restrict__ fpos,
                                                           int* __restrict__ fcrd, T* __restrict__ fval, DevCtl* ctl) {
    const int lane = threadIdx.x & 31;
    for (i64 f = ((i64)blockIdx.x * OT + threadIdx.x) >> 5; f < B.n1; f += ((i64)gridDim.x * OT) >> 5) {
        const int k = __ldg(B.crd0 + owner_row(B.pos1, 0, B.n0, f)), l = __ldg(B.crd1 + f);
        if ((unsigned)k >= (unsigned)C.nrows || (unsigned)l >= (unsigned)D.nrows) {
            raise_status(ctl, DEV_NONCANONICAL);
            if (PASS == 0 && lane == 0) cnt[f] = 0;
            continue;
        }
        i64 s0 = __ldg(C.pos + k), s1 = __ldg(C.pos + k + 1), g0 = __ldg(D.pos + l), g1 = __ldg(D.pos + l + 1);
        const int* __restrict__ scrd = C.crd;
        const int* __restrict__ gcrd = D.crd;
        const T* __restrict__ sval = (const T*)C.val;
        const T* __restrict__ gval = (const T*)D.val;
        if (s1 - s0 > g1 - g0) {
            i64 t = s0; s0 = g0; g0 = t;
            t = s1; s1 = g1; g1 = t;
            scrd = D.crd; gcrd = C.crd;
            sval = (const T*)D.val; gval = (const T*)C.val;
        }
        int found = 0;
        i64 out = PASS > 0 ? fpos[f] : 0;
        for (i64 q0 = s0; q0 < s1; q0 += 32) {
            const i64 q = q0 + lane;
            const int col = q < s1 ? __ldg(scrd + q) : -1;
            const i64 at = q < s1 ? lower_bound_crd(gcrd, g0, g1, col) : g1;
            const bool hit = at < g1 && __ldg(gcrd + at) == col;
            const unsigned hits = __ballot_sync(0xffffffffu, hit);
            if (PASS > 0 && hit) {
                const i64 o = out + __popc(hits & ((1u << lane) - 1u));
                if (PASS == 1) fcrd[o] = col;
                else fval[o] = mul_rn(__ldg(sval + q), __ldg(gval + at));
            }
            found += __popc(hits);
            out += __popc(hits);
        }
        if (PASS == 0 && lane == 0) cnt[f] = found;
    }
}

// Coordinates of a coordinate-form result from its row pointer, row labels and columns.  A block takes a run of
// tiles of RC_TILE consecutive entries: the first entry of every row in the tile leaves the row's
// coordinates in shared memory, a running maximum hands each entry the place of its row's first one,
// and a thread writes the coordinates of its eight consecutive entries.  The rows of a tile are read 256 at a time from where
// the tile before ended.  Bound by HBM and the four barriers of a tile.
// 43e6 entries of three coordinates: 333 us for three arrays with a search per entry and 883 us to interleave
// them; interleaved 276 us with two searches per tile, 198 us without them and 165 us with whole lines per store
// (516 MB out, 172 MB in).  As many blocks as are resident, a run of tiles each: 139 us, with 16 an SM 164.
constexpr int RC_ITEMS = 8;
constexpr int RC_TILE = OT * RC_ITEMS;

template <int ORDER, bool INTERLEAVED>
__global__ void __launch_bounds__(OT) rw_coords_kernel(const i64* __restrict__ rowptr, const u64* __restrict__ row_key, i64 m, i64 nnz, u64 d,
                                                       const int* __restrict__ cols, int* __restrict__ o0, int* __restrict__ o1,
                                                       int* __restrict__ o2) {
    __shared__ int s_c0[RC_TILE], s_c1[ORDER == 3 ? RC_TILE : 1];
    __shared__ __align__(16) unsigned short s_head[RC_TILE];    // entry i: i when a row starts there, else 0; zero between tiles
    __shared__ __align__(16) int s_out[INTERLEAVED ? ORDER * RC_TILE : 4];
    __shared__ int s_lo, s_warp[OT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool vec = (((u64)o0 | (INTERLEAVED ? 0 : (u64)o1 | (u64)o2)) & 15) == 0;      // 16-byte stores
    const i64 tiles = (nnz + RC_TILE - 1) / RC_TILE;
    const i64 first = tiles * blockIdx.x / gridDim.x, last = tiles * (blockIdx.x + 1) / gridDim.x;
    for (int i = tid; i < RC_TILE; i += OT) s_head[i] = 0;
    if (tid == 0 && first < last) s_lo = owner_row(rowptr, 0, (int)m, first * RC_TILE);
    for (i64 tile = first; tile < last; ++tile) {
        const i64 t0 = tile * RC_TILE, t1 = min(nnz, t0 + RC_TILE);
        const int i0 = tid * RC_ITEMS;
        const bool whole = vec && t0 + RC_TILE <= nnz;
        int col[RC_ITEMS];
        if (whole) {
            *reinterpret_cast<int4*>(col) = __ldg(reinterpret_cast<const int4*>(cols + t0 + i0));
            *reinterpret_cast<int4*>(col + 4) = __ldg(reinterpret_cast<const int4*>(cols + t0 + i0) + 1);
        }
        __syncthreads();
        const int lo = s_lo;                            // a row that starts at or before t0, none but empty ones between
        __syncthreads();
        for (i64 r0 = lo;; r0 += OT) {
            const i64 r = r0 + tid;
            bool inside = false;
            if (r < m) {
                const i64 a = __ldg(rowptr + r), b = __ldg(rowptr + r + 1);
                inside = a < t1;
                if (inside && b > t0 && b > a) {
                    const int i = (int)max(a - t0, (i64)0);     // (the first row may have begun before the tile)
                    const u64 key = __ldg(row_key + r);
                    s_c0[i] = ORDER == 3 ? (int)(key / d) : (int)key;
                    if (ORDER == 3) s_c1[i] = (int)(key % d);
                    s_head[i] = (unsigned short)i;
                }
                if (inside && b >= t1) s_lo = (int)r;           // the next tile starts here
            }
            if (!__syncthreads_or(tid == OT - 1 && inside)) break;
        }
        int h[RC_ITEMS];
        const uint4 hv = reinterpret_cast<const uint4*>(s_head)[tid];
        reinterpret_cast<uint4*>(s_head)[tid] = make_uint4(0, 0, 0, 0);
        h[0] = hv.x & 0xffff; h[1] = hv.x >> 16; h[2] = hv.y & 0xffff; h[3] = hv.y >> 16;
        h[4] = hv.z & 0xffff; h[5] = hv.z >> 16; h[6] = hv.w & 0xffff; h[7] = hv.w >> 16;
#pragma unroll
        for (int x = 1; x < RC_ITEMS; ++x) h[x] = max(h[x], h[x - 1]);
        int incl = h[RC_ITEMS - 1];
#pragma unroll
        for (int e = 1; e < 32; e <<= 1) incl = max(incl, __shfl_up_sync(0xffffffffu, incl, e));
        if (lane == 31) s_warp[warp] = incl;
        int before = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) before = 0;
        __syncthreads();
        for (int w = 0; w < warp; ++w) before = max(before, s_warp[w]);
        if (whole) {
            int out[RC_ITEMS * ORDER];                      // entry by entry, or array by array
#pragma unroll
            for (int x = 0; x < RC_ITEMS; ++x) {
                const int at = max(h[x], before);
                out[INTERLEAVED ? x * ORDER : x] = s_c0[at];
                if (ORDER == 3) out[INTERLEAVED ? x * ORDER + 1 : x + RC_ITEMS] = s_c1[at];
                out[INTERLEAVED ? x * ORDER + ORDER - 1 : x + (ORDER - 1) * RC_ITEMS] = col[x];
            }
            constexpr int QUADS = RC_ITEMS * ORDER / 4;
            if (INTERLEAVED) {                              // through shared memory, so that a warp stores whole lines
#pragma unroll
                for (int y = 0; y < QUADS; ++y)
                    reinterpret_cast<int4*>(s_out)[tid * QUADS + y] = make_int4(out[4 * y], out[4 * y + 1], out[4 * y + 2], out[4 * y + 3]);
                __syncwarp();
                int4* const to = reinterpret_cast<int4*>(o0 + t0 * ORDER) + warp * (32 * QUADS);
#pragma unroll
                for (int y = 0; y < QUADS; ++y) to[y * 32 + lane] = reinterpret_cast<const int4*>(s_out)[warp * (32 * QUADS) + y * 32 + lane];
                __syncwarp();
            } else {
#pragma unroll
                for (int y = 0; y < QUADS; ++y)
                    *reinterpret_cast<int4*>((y < 2 ? o0 : y < 4 ? o1 : o2) + t0 + i0 + 4 * (y & 1)) = make_int4(out[4 * y], out[4 * y + 1], out[4 * y + 2], out[4 * y + 3]);
            }
        } else {
#pragma unroll
            for (int x = 0; x < RC_ITEMS; ++x) {
                const i64 t = t0 + i0 + x;
                if (t >= t1) break;
                const int at = max(h[x], before);
                const i64 o = INTERLEAVED ? t * ORDER : t;
                o0[o] = s_c0[at];
                if (ORDER == 3) (INTERLEAVED ? o0 + 1 : o1)[o] = s_c1[at];
                (INTERLEAVED ? o0 + ORDER - 1 : ORDER == 3 ? o2 : o1)[o] = __ldg(cols + t);
            }
        }
    }
}

// ---- host side --------------------------------------------------------------------------------
// (what the sort needs, then the ticket and the words of rw_sparse_rows_kernel: cleared together)
size_t rw_sort_bytes(i64 n) { return sort_scratch_bytes(n) + 8 * (size_t)((n + RK_TILE - 1) / RK_TILE + 1); }

static int passes_of(int bits) { return (bits + 7) / 8; }

// Sorts the entries by output row and writes the reordered operand (all but its values).  `sparse`: a row per
// label that occurs (at most m), labels to row_key; otherwise a row per label value.  The kernel that wrote the labels has
// counted their digits (a kernel of its own for that, one for `pos` and their clearing took 10 .. 18 us a call).
// Only the labels and 32-bit entry numbers move (the picked row is fetched at the end), labels of 32 bits where they fit: 1e6 entries
// of 22 bits in three passes 79 us with labels, picked rows and entries in 16 bytes, 57 us like this; 7e5 of 18 bits 62 and 46.
template <typename K>
static cudaError_t rw_reorder(const LaunchCtx& c, i64 n, i64 m, int bits, bool sparse, const RowwiseBufs& b) {
    cudaError_t e;
    bool first = true;
    K *const k0 = reinterpret_cast<K*>(b.kA), *const k1 = reinterpret_cast<K*>(b.kB);
    if (n == 1 && (e = cudaMemsetAsync(b.entry[0], 0, sizeof(int), c.stream)) != cudaSuccess) return e;      // (nothing to sort)
    if ((e = radix_sort_t<K, int, true>(c, n, bits, k0, b.entry[0], k1, b.entry[1], b.sort_tmp, &first, true, true)) != cudaSuccess) return e;
    const K* ks = first ? k0 : k1;
    const int* es = first ? b.entry[0] : b.entry[1];
    if (!sparse) return launch_chained(c, rw_dense_rows_kernel<K>, grid_for(c, n > m ? n : m + 1, OT), OT, 0, ks, es, b.pick, n, m, b.pos, b.crd, b.src);
    if (n == 0) return cudaSuccess;
    const int tiles = (int)((n + RK_TILE - 1) / RK_TILE);
    u64* const words = reinterpret_cast<u64*>(b.sort_tmp + sort_scratch_bytes(n));
    return launch_chained(c, rw_sparse_rows_kernel<K>, tiles, OT, 0, ks, es, b.pick, n, m, reinterpret_cast<int*>(words), words + 1, c.ctl, b.row_key, b.pos, b.crd, b.src);
}

template <typename K>
static cudaError_t rw_outer_t(const LaunchCtx& c, const Csr& At, i64 n, const Csr& B, i64 nnzB, int bits, const RowwiseBufs& b) {
    const cudaError_t e = launch_chained(c, rw_keys_outer_kernel<K>, grid_for(c, std::max(n, nnzB), RK_TILE), OT, 0, At, n, B, nnzB, reinterpret_cast<K*>(b.kA), b.pick,
                                         passes_of(bits), reinterpret_cast<SortHead*>(b.sort_tmp), c.ctl);
    return e != cudaSuccess ? e : rw_reorder<K>(c, n, At.ncols, bits, false, b);
}

// Clears the control block and the sort's temporaries (a memset each took the host 3 .. 4 us more).
__global__ void __launch_bounds__(OT) rw_clear_kernel(int* __restrict__ ctl, int n_ctl, int4* __restrict__ tmp, i64 n_tmp) {
    chained_start();
    const i64 t0 = (i64)blockIdx.x * OT + threadIdx.x, stride = (i64)gridDim.x * OT;
    for (i64 i = t0; i < n_ctl; i += stride) ctl[i] = 0;
    for (i64 i = t0; i < n_tmp; i += stride) tmp[i] = make_int4(0, 0, 0, 0);
}

cudaError_t launch_rw_clear(const LaunchCtx& c, i64 n, char* tmp) {
    const i64 quads = (i64)(rw_sort_bytes(n) + 15) / 16;           // (its room is a multiple of 256 bytes)
    return launch_chained(c, rw_clear_kernel, grid_for(c, quads, OT), OT, 0, reinterpret_cast<int*>(c.ctl), (int)(sizeof(DevCtl) / 4), reinterpret_cast<int4*>(tmp), quads);
}

cudaError_t launch_rw_outer(const LaunchCtx& c, const Csr& At, i64 n, const Csr& B, i64 nnzB, int bits, const RowwiseBufs& b) {
    return rw_outer_t<unsigned>(c, At, n, B, nnzB, bits, b);        // (a row number)
}

template <typename K>
static cudaError_t rw_csf_t(const LaunchCtx& c, int form, const Csf3Dev& B, u64 d0, u64 d1, i64 m, int bits, const RowwiseBufs& b) {
    const cudaError_t e = launch_chained(c, rw_keys_csf_kernel<K>, grid_for(c, std::max(B.nnz, (i64)1), RK_TILE), OT, 0, form, B, d0, d1, reinterpret_cast<K*>(b.kA), b.pick,
                                         passes_of(bits), reinterpret_cast<SortHead*>(b.sort_tmp), b.pos, m, c.ctl);
    return e != cudaSuccess ? e : rw_reorder<K>(c, B.nnz, m, bits, true, b);
}

cudaError_t launch_rw_csf(const LaunchCtx& c, int form, const Csf3Dev& B, u64 d0, u64 d1, i64 m, int bits, const RowwiseBufs& b) {
    return bits <= 32 ? rw_csf_t<unsigned>(c, form, B, d0, d1, m, bits, b) : rw_csf_t<u64>(c, form, B, d0, d1, m, bits, b);
}

cudaError_t launch_rw_values(const LaunchCtx& c, const void* val, const int* src, i64 n, void* out) {
    if (n == 0) return cudaSuccess;
    if (c.is_f64) rw_values_kernel<double><<<grid_for(c, n, OT), OT, 0, c.stream>>>((const double*)val, src, n, (double*)out);
    else rw_values_kernel<float><<<grid_for(c, n, OT), OT, 0, c.stream>>>((const float*)val, src, n, (float*)out);
    ++c.launches;
    return cudaGetLastError();
}

cudaError_t launch_rw_fibre_rows(const LaunchCtx& c, bool values, const Csf3Dev& B, const Csr& C, const Csr& D, int* cnt, i64* fpos, int* fcrd,
                                 void* fval, i64* block_sums) {
    const int grid = grid_for(c, (i64)B.n1 * 32, OT);
    if (values) {
        if (B.n1 == 0) return cudaSuccess;
        if (c.is_f64) rw_fibre_rows_kernel<double, 2><<<grid, OT, 0, c.stream>>>(B, C, D, nullptr, fpos, nullptr, (double*)fval, c.ctl);
        else rw_fibre_rows_kernel<float, 2><<<grid, OT, 0, c.stream>>>(B, C, D, nullptr, fpos, nullptr, (float*)fval, c.ctl);
        ++c.launches;
        return cudaGetLastError();
    }
    if (B.n1 > 0) {
        rw_fibre_rows_kernel<float, 0><<<grid, OT, 0, c.stream>>>(B, C, D, cnt, nullptr, nullptr, nullptr, c.ctl);
        ++c.launches;
    }
    cudaError_t e = launch_scan_counts(c, cnt, B.n1, fpos, block_sums, nullptr);
    if (e != cudaSuccess || B.n1 == 0) return e;
    rw_fibre_rows_kernel<float, 1><<<grid, OT, 0, c.stream>>>(B, C, D, nullptr, fpos, fcrd, nullptr, c.ctl);
    ++c.launches;
    return cudaGetLastError();
}

cudaError_t launch_rw_coords(const LaunchCtx& c, int order, const i64* rowptr, const u64* row_key, i64 m, i64 nnz, u64 d, const int* cols, int* o0,
                             int* o1, int* o2, bool interleaved) {
    if (nnz == 0) return cudaSuccess;
    auto k = order == 3 ? (interleaved ? rw_coords_kernel<3, true> : rw_coords_kernel<3, false>)
                        : (interleaved ? rw_coords_kernel<2, true> : rw_coords_kernel<2, false>);
    int per_sm = 0;
    const cudaError_t e = resident_blocks((const void*)k, OT, 0, &per_sm);
    if (e != cudaSuccess) return e;
    const i64 grid = std::min((nnz + RC_TILE - 1) / RC_TILE, (i64)c.sm_count * std::max(per_sm, 1));
    k<<<(int)grid, OT, 0, c.stream>>>(rowptr, row_key, m, nnz, d, cols, o0, o1, o2);
    ++c.launches;
    return cudaGetLastError();
}

}  // namespace spws
