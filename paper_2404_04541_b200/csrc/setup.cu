// Symbolic-pass set-up kernels: input validation, per-row product upper bound and column
// span, routing of rows to workspaces (binning), exclusive scans, CSF level rebuild.
#include <algorithm>
#include "common.cuh"

namespace spws {

// ---------------------------------------------------------------------------------------
// Validation: pos non-decreasing with pos[0] = 0 and pos[rows] = nnz; coordinates in range
// and strictly increasing inside a row.
// ---------------------------------------------------------------------------------------
__global__ void validate_csr_kernel(Csr M, i64 nnz, int coord_limit, DevCtl* ctl) {
    const i64 stride = (i64)gridDim.x * blockDim.x;
    bool bad = false;
    for (i64 r = (i64)blockIdx.x * blockDim.x + threadIdx.x; r < M.nrows; r += stride) {
        const i64 s = M.pos[r], e = M.pos[r + 1];
        if (r == 0 && s != 0) bad = true;
        if (r == M.nrows - 1 && e != nnz) bad = true;
        if (s > e || s < 0 || e > nnz) { bad = true; continue; }
        int prev = -1;
        for (i64 p = s; p < e; ++p) {
            const int c = M.crd[p];
            if (c <= prev || c >= coord_limit) bad = true;
            prev = c;
        }
    }
    if (M.nrows == 0 && threadIdx.x == 0 && blockIdx.x == 0 && nnz != 0) bad = true;
    if (bad) raise_status(ctl, DEV_NONCANONICAL);
}

cudaError_t launch_validate(const LaunchCtx& c, const Csr& A, const Csr& B, i64 nnzA, i64 nnzB) {
    const int grid = c.sm_count * 8;
    validate_csr_kernel<<<grid, 256, 0, c.stream>>>(A, nnzA, B.nrows, c.ctl);
    validate_csr_kernel<<<grid, 256, 0, c.stream>>>(B, nnzB, B.ncols, c.ctl);
    c.launches += 2;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Per-row upper bound ub[i] = sum over A(i,:) of the picked B row's length, the exact span
// [jmin, jmax] of the candidate columns (first / last coordinate of the picked B rows, which
// are sorted), and the workspace class of the row.
// ---------------------------------------------------------------------------------------
// A span that ends before it begins comes from B rows that are not ascending: such a row has no bitmap whose words could be
// counted (the slots of all rows must lie inside the arena once their sum does).  The sparse workspaces read no span.
__device__ __forceinline__ int dense_class(i64 ub, i64 span_words, DevCtl* ctl) {
    if (span_words <= 0) { raise_status(ctl, DEV_NONCANONICAL); return CLS_EMPTY; }
    if (span_words <= DENSE_WARP_BM_WORDS && ub <= DENSE_WARP_MAX_UB) return CLS_DENSE_WARP;
    return ub >= DENSE_HUB_UB ? CLS_DENSE_HUB : CLS_DENSE_CTA;
}

// (a warp per row from 129 products on: 32 lanes of the group kernel took 41 + 51 us on 3e4 rows of 143 products, a warp 36 + 49)
__device__ __forceinline__ int small_ism_class(i64 ub) { return ub <= 64 ? CLS_ISM_GROUP8 : ub <= 128 ? CLS_ISM_GROUP16 : CLS_ISM_SMEM_S; }

__device__ __forceinline__ int classify_row(i64 ub, i64 entries, int jmin, int jmax, const ClassParams& prm, DevCtl* ctl) {
    if (ub == 0) return CLS_EMPTY;
    const i64 span = (i64)jmax - jmin + 1;
    const i64 span_words = (span + 31) >> 5;
    const bool dense_ok = span_words <= prm.max_span_words;
    const bool reg_ok = ub <= prm.reg_cap;      // (any span: 2.6e5 rows of 16 products over 2^28 columns, f32, by 8 lanes a row 100 + 111 us, by 4 28 + 41)
    if (prm.policy == 0) {                       // dense forced
        if (!dense_ok) { raise_status(ctl, DEV_WORKSPACE_TOO_LARGE); return CLS_EMPTY; }
        return dense_class(ub, span_words, ctl);
    }
    // a single entry: Insert, Sort and Merge are the identity and the output count is the B row's length,
    // known right here (up to COPY_MAX entries, which eight lanes copy; SpTTM with 41-entry rows, two
    // thirds of them from one entry: 1421 us through the warp dense workspace, 534 us with those copied and
    // most of the others through the register sort)
    if (entries == 1 && ub <= COPY_MAX && prm.policy != 3) return CLS_COPY;
    const int reg_cls = ub <= 8 ? CLS_ISM_REG8 : (ub <= 16 ? CLS_ISM_REG16 : CLS_ISM_REG);
    if (prm.policy == 1) {                       // sparse ISM forced
        if (reg_ok) return reg_cls;
        if (ub <= prm.smem_small_cap) return small_ism_class(ub);
        if (ub <= prm.smem_cap) return CLS_ISM_SMEM;
        return CLS_ISM_GLOBAL;
    }
    if (prm.policy == 3) {                       // hash forced
        if (ub <= HASH_SMALL_CAP) return CLS_HASH_S;
        if (ub <= HASH_CAP) return CLS_HASH;
        return CLS_ISM_GLOBAL;
    }
    // auto: few products -> sort them in registers; a bitmap that is small next to the work ->
    // dense; mid-size rows -> shared-memory ISM; long rows -> dense; otherwise global ISM.
    if (reg_ok) return reg_cls;
    // up to 128 products the register sort beats the bitmap whatever the span; up to 256 when the bitmap is wide
    // (6e6 products, f64, both passes, dense against ISM: 60 products a row 263 : 172 us, 117 a row 156 : 126
    // us, 240 a row on 94 words 119 : 113 us and on 626 words 160 : 110 us; 380 a row 98 : 168 us)
    if (ub <= prm.smem_small_cap && (ub <= 128 || span_words > 256)) return small_ism_class(ub);
    if (dense_ok && (float)span_words <= prm.span_words_per_product * (float)ub) return dense_class(ub, span_words, ctl);
    if (ub <= prm.smem_small_cap) return small_ism_class(ub);
    if (ub <= prm.smem_cap) return CLS_ISM_SMEM;
    if (dense_ok) return dense_class(ub, span_words, ctl);
    return CLS_ISM_GLOBAL;
}

// First column, last column and length of every B row, in one 16-byte record: when A has several
// times more entries than B has rows, the bounds kernel reads the record of the row an entry picks
// (one load, neighbouring rows share sectors) instead of two offsets and two coordinates.
// It is the first kernel of a pass and clears the control block on the way (ctl non-null).
__global__ void __launch_bounds__(256) brow_summary_kernel(Csr B, int4* __restrict__ brow, DevCtl* ctl) {
    const int tid = chained_start(threadIdx.x);
    if (ctl && blockIdx.x == 0)
        for (int w = threadIdx.x; w < (int)(sizeof(DevCtl) / 4); w += 256) reinterpret_cast<int*>(ctl)[w] = 0;
    for (i64 k = (i64)blockIdx.x * blockDim.x + tid; k < B.nrows; k += (i64)gridDim.x * blockDim.x) {
        const i64 qs = B.pos[k], qe = B.pos[k + 1];
        int4 s = make_int4(0x7fffffff, -1, 0, 0);
        if (qe > qs) {
            s.x = __ldg(B.crd + qs);
            s.y = __ldg(B.crd + qe - 1);
            s.z = (int)min(qe - qs, (i64)0x7fffffff);
        }
        brow[k] = s;
    }
}

// Arena words of a dense row: its bitmap, then the rank at the start of every 32-word chunk, 16-byte aligned.
__device__ __forceinline__ int slot_words(int lo, int hi) {
    const int nw = (hi - lo) / 32 + 1;
    return (nw + (nw + 31) / 32 + 3) & ~3;
}
__device__ __forceinline__ bool dense_cls(int cls) { return cls == CLS_DENSE_WARP || cls == CLS_DENSE_HUB || cls == CLS_DENSE_CTA; }

// Long and mid rows that a block lists for its threads and warps to take together; what does not fit is left to lane groups, as serial
// chains.  With four or five blocks an SM (1e5 rows of 60 entries among 1.9e6 of 2: lists of 32 and 64 rows 121 us, these 119; 2e4 rows of
// 1100 77 and 75; 5e4 147 and 146, where 16 blocks an SM with lists of 32 took 207).
constexpr int LONG_LIST = 128;
constexpr int MID_LIST = 256;

// Products and first / last column of the entries ps + at, ps + at + LANES, ..: four entries per step; the totals of
// a warp's lanes are returned in every lane.
template <bool SUMMARY, int LANES>
__device__ __forceinline__ void entry_totals(i64 ps, i64 pe, int at, const Csr& A, const Csr& B, const int4* __restrict__ brow, i64& u, int& lo,
                                             int& hi, int& bad) {
    u = 0;
    lo = 0x7fffffff, hi = -1, bad = 0;
    for (i64 p0 = ps + at; p0 < pe; p0 += 4 * LANES) {
        int k[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const i64 p = p0 + (i64)x * LANES;
            k[x] = p < pe ? __ldg(A.crd + p) : -1;
            if (p < pe && (unsigned)k[x] >= (unsigned)B.nrows) bad = 1;
        }
        if (SUMMARY) {
            int4 s[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) s[x] = (unsigned)k[x] < (unsigned)B.nrows ? __ldg(brow + k[x]) : make_int4(0x7fffffff, -1, 0, 0);
#pragma unroll
            for (int x = 0; x < 4; ++x) { u += s[x].z; lo = min(lo, s[x].x); hi = max(hi, s[x].y); }
        } else {
            i64 qs[4], qe[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                qs[x] = qe[x] = 0;
                if ((unsigned)k[x] < (unsigned)B.nrows) { qs[x] = __ldg(B.pos + k[x]); qe[x] = __ldg(B.pos + k[x] + 1); }
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (qe[x] > qs[x]) {
                    u += qe[x] - qs[x];
                    lo = min(lo, __ldg(B.crd + qs[x]));
                    hi = max(hi, __ldg(B.crd + qe[x] - 1));
                }
        }
    }
    for (int d = 16; d > 0; d >>= 1) {
        u += __shfl_xor_sync(0xffffffffu, u, d);
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, d));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, d));
        bad |= __shfl_xor_sync(0xffffffffu, bad, d);
    }
}

// Bounds and class of one long row by a whole block.
template <bool SUMMARY>
__device__ __forceinline__ void long_row_bounds(int row, const Csr& A, const Csr& B, const RowTables& tab, const ClassParams& prm, DevCtl* ctl,
                                                const int4* __restrict__ brow) {
    __shared__ i64 s_u[8];
    __shared__ int s_lo[8], s_hi[8], s_bad[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const i64 ps = A.pos[row], pe = A.pos[row + 1];
    i64 u;
    int lo, hi, bad;
    entry_totals<SUMMARY, 256>(ps, pe, tid, A, B, brow, u, lo, hi, bad);
    __syncthreads();                                   // the previous row's totals have been read
    if (lane == 0) { s_u[warp] = u; s_lo[warp] = lo; s_hi[warp] = hi; s_bad[warp] = bad; }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < 8; ++w) { u += s_u[w]; lo = min(lo, s_lo[w]); hi = max(hi, s_hi[w]); bad |= s_bad[w]; }
        if (bad) raise_status(ctl, DEV_NONCANONICAL);
        if (lo < 0 || hi >= B.ncols) { raise_status(ctl, DEV_NONCANONICAL); u = 0; }
        if (u > 0) lo &= ~31;
        const int cls = classify_row(u, pe - ps, lo, hi, prm, ctl);
        tab.ub[row] = u;
        tab.jmin[row] = lo;
        tab.jmax[row] = hi;
        tab.cnt[row] = cls == CLS_COPY ? (int)u : 0;
        tab.cls[row] = (unsigned char)cls;
        atomicAdd(&ctl->class_count[cls], 1);
        if (u) {
            atomicAdd((u64*)&ctl->class_products[cls], (u64)u);
            atomicAdd((u64*)&ctl->products, (u64)u);
            atomicMax(&ctl->max_ub, u);
            if (cls == CLS_ISM_GLOBAL) atomicMax(&ctl->max_ub_global, u);
            if (cls == CLS_ISM_SMEM) {
                atomicMax(&ctl->max_ub_smem, u);
                if (u <= ISM_WARP_MAX) atomicAdd(&ctl->order_words, (u64)order_words_of((int)u));
            }
            if (dense_cls(cls)) {
                atomicMax(&ctl->max_span_words, (hi - lo) / 32 + 1);
                atomicAdd(&ctl->bm_words, (u64)slot_words(lo, hi));
            }
        }
    }
}

// SUMMARY: brow holds the B-row summaries (the instantiation without them carries B's own arrays'
// two-level gathers and needs more registers).
template <int G, bool SUMMARY>
__global__ void __launch_bounds__(256, SUMMARY ? 5 : 4) row_bounds_kernel(Csr A, Csr B, RowTables tab, ClassParams prm, DevCtl* ctl,
                                                         const int4* __restrict__ brow) {
    // rows and products per class, one histogram per warp: 64-bit shared-memory adds are compare-and-swap loops,
    // which many threads on one address turn into a queue, so what fits is added in 32 bits (a thread's run of
    // products below 2^16; a warp adds fewer than 2^16 of those)
    __shared__ int s_hist[8][NCLASS];
    __shared__ unsigned s_clow[8][NCLASS];
    __shared__ i64 s_cprod[8][NCLASS];
    __shared__ i64 s_max_ub, s_max_ub_global, s_max_ub_smem, s_bm_words;
    __shared__ int s_max_span_words;
    __shared__ unsigned s_order_words;              // (at most 1024 a row: of 2^31 rows none of 592 blocks, four an SM, sees 2^22)
    // rows of more than LONG_A_ROW entries, which the block's threads take together at the end: left to
    // its lane group such a row is a serial chain that sets the kernel's time on power-law inputs
    __shared__ int s_long[LONG_LIST], s_nlong;
    // rows of more than two steps of a narrow lane group, which the block's warps take at the end
    __shared__ int s_mid[MID_LIST], s_nmid;
    chained_start();
    for (int x = threadIdx.x; x < 8 * NCLASS; x += blockDim.x) { (&s_hist[0][0])[x] = 0; (&s_clow[0][0])[x] = 0; (&s_cprod[0][0])[x] = 0; }
    if (threadIdx.x == 0) { s_max_ub = 0; s_max_ub_global = 0; s_max_ub_smem = 0; s_max_span_words = 0; s_bm_words = 0; s_order_words = 0; s_nlong = s_nmid = 0; }
    __syncthreads();
    int* const w_hist = s_hist[threadIdx.x >> 5];
    i64* const w_cprod = s_cprod[threadIdx.x >> 5];
    unsigned* const w_clow = s_clow[threadIdx.x >> 5];
    int low_adds = 0;                               // 32-bit additions of this thread
    auto flush = [&](int cls, int rows, i64 products) {
        if (rows) atomicAdd(&w_hist[cls], rows);
        if (products == 0) return;
        if (products < 65536 && low_adds < 2047) {  // 32 threads x 2047 additions x 65535 < 2^32
            atomicAdd(&w_clow[cls], (unsigned)products);
            ++low_adds;
        } else {
            atomicAdd((u64*)&w_cprod[cls], (u64)products);
        }
    };
    const int gl = threadIdx.x % G;
    const unsigned lane = threadIdx.x & 31;
    const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << (lane - gl));
    // eight lanes or more per row: neighbouring rows go to different blocks (the heaviest rows of a graph are often
    // neighbours); narrower groups take neighbouring rows for the sake of the row offsets they share
    const i64 ngroups = ((i64)gridDim.x * blockDim.x) / G;
    i64 group = G >= 8 ? (i64)(threadIdx.x / G) * gridDim.x + blockIdx.x : ((i64)blockIdx.x * blockDim.x + threadIdx.x) / G;
    not_before(group);
    unsigned my_max = 0;                            // most products of a row below 2^32
    // rows and products of the class of this group's last rows: neighbouring rows mostly share a
    // class, so the shared-memory histogram is touched only when the class changes
    int run_cls = -1, run_rows = 0;
    // (at most 2^14 + 2^9 words a row: 2^32 words are 2.5e5 rows of the widest bitmap in a group.  Groups of 8 lanes and fewer, 18944 of them
    // at least, do not see as many of 2^31 rows; those of 32, 4736, take rows of more than 32 entries on average when they are so
    // many, 3.8e10 entries in all, more than memory holds)
    unsigned my_bm_words = 0;
    i64 run_products = 0;
    auto classify = [&](int row, i64 entries, i64 u, int lo, int hi) {
        if (lo < 0 || hi >= B.ncols) { raise_status(ctl, DEV_NONCANONICAL); u = 0; }
        if (u > 0) lo &= ~31;               // bitmap words of every row start at a multiple of 32 columns
        const int cls = classify_row(u, entries, lo, hi, prm, ctl);
        tab.ub[row] = u;
        if (dense_cls(cls)) {                           // (nothing reads the span of the others)
            tab.jmin[row] = lo;
            tab.jmax[row] = hi;
        }
        tab.cnt[row] = cls == CLS_COPY ? (int)u : 0;
        tab.cls[row] = (unsigned char)cls;
        if (cls != run_cls) {
            if (run_rows) flush(run_cls, run_rows, run_products);
            run_cls = cls;
            run_rows = 0;
            run_products = 0;
        }
        ++run_rows;
        run_products += u;
        // (what is rare, or a maximum that seldom moves, goes straight to shared memory: in registers of every thread these
        // and the words of the bitmaps spilled, and the bounds of a 27-point stencil of 2^18 rows took 50 us, now 46.5)
        if (u >> 32) atomicMax(&s_max_ub, u);
        else my_max = max(my_max, (unsigned)u);
        if (cls == CLS_ISM_GLOBAL && u > s_max_ub_global) atomicMax(&s_max_ub_global, u);
        if (cls == CLS_ISM_SMEM) {
            if (u > s_max_ub_smem) atomicMax(&s_max_ub_smem, u);
            if (u <= ISM_WARP_MAX) atomicAdd(&s_order_words, (unsigned)order_words_of((int)u));
        }
        if (dense_cls(cls)) {
            const int span_words = (hi - lo) / 32 + 1;
            if (span_words > s_max_span_words) atomicMax(&s_max_span_words, span_words);
            my_bm_words += (unsigned)slot_words(lo, hi);
        }
    };
    // the next row's range and this lane's first entry of it are loaded while the current row is in hand: with
    // a few entries per row the kernel is a chain of dependent loads otherwise
    i64 ps_n = 0, pe_n = 0;
    int k_n = -1;
    if (group < A.nrows) {
        ps_n = A.pos[group];
        pe_n = A.pos[group + 1];
        if (ps_n + gl < pe_n) k_n = __ldg(A.crd + ps_n + gl);
    }
    for (i64 row = group; row < A.nrows; row += ngroups) {
        const i64 ps = ps_n, pe = pe_n;
        const int k_first = k_n;
        const bool more = row + ngroups < A.nrows;
        if (more) {
            ps_n = A.pos[row + ngroups];
            pe_n = A.pos[row + ngroups + 1];
        }
        if (pe - ps > (G < 32 ? 8 * G : LONG_A_ROW)) {
            const bool mid = G < 32 && pe - ps <= LONG_A_ROW;
            int at = 0;
            if (gl == 0) at = atomicAdd(mid ? &s_nmid : &s_nlong, 1);
            at = __shfl_sync(gmask, at, 0, G);
            if (at < (mid ? MID_LIST : LONG_LIST)) {
                if (gl == 0) (mid ? s_mid : s_long)[at] = (int)row;
                if (more && ps_n + gl < pe_n) k_n = __ldg(A.crd + ps_n + gl);
                continue;
            }
        }
        i64 u = 0;
        int lo = 0x7fffffff, hi = -1;
        bool bad = false;
        // four entries per lane and step, each level of loads issued for all four before the
        // next level needs it: a row with very many entries is a chain of dependent loads otherwise
        i64 p0 = ps + gl;
        if (pe - ps <= G) {                         // the common short row: one entry per lane
            if (p0 < pe) {
                const int k = k_first;
                if ((unsigned)k < (unsigned)B.nrows) {
                    if (SUMMARY) {
                        const int4 s = __ldg(brow + k);
                        u = s.z;
                        lo = s.x;
                        hi = s.y;
                    } else {
                        const i64 qs = __ldg(B.pos + k), qe = __ldg(B.pos + k + 1);
                        if (qe > qs) {
                            u = qe - qs;
                            lo = __ldg(B.crd + qs);
                            hi = __ldg(B.crd + qe - 1);
                        }
                    }
                } else {
                    bad = true;
                }
            }
            p0 = pe;
        }
        for (; p0 < pe; p0 += 4 * G) {
            int k[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const i64 p = p0 + (i64)x * G;
                k[x] = p < pe ? __ldg(A.crd + p) : -1;
                if (p < pe && (unsigned)k[x] >= (unsigned)B.nrows) bad = true;
            }
            if (SUMMARY) {
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    if ((unsigned)k[x] < (unsigned)B.nrows) {
                        const int4 s = __ldg(brow + k[x]);
                        u += s.z;
                        lo = min(lo, s.x);
                        hi = max(hi, s.y);
                    }
                continue;
            }
            i64 qs[4], qe[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                qs[x] = qe[x] = 0;
                if ((unsigned)k[x] < (unsigned)B.nrows) { qs[x] = __ldg(B.pos + k[x]); qe[x] = __ldg(B.pos + k[x] + 1); }
            }
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                if (qe[x] > qs[x]) {
                    u += qe[x] - qs[x];
                    lo = min(lo, __ldg(B.crd + qs[x]));
                    hi = max(hi, __ldg(B.crd + qe[x] - 1));
                }
            }
        }
        if (more && ps_n + gl < pe_n) k_n = __ldg(A.crd + ps_n + gl);
#pragma unroll
        for (int d = G / 2; d > 0; d >>= 1) {
            u += __shfl_xor_sync(gmask, u, d, G);
            lo = min(lo, __shfl_xor_sync(gmask, lo, d, G));
            hi = max(hi, __shfl_xor_sync(gmask, hi, d, G));
        }
        if (bad) raise_status(ctl, DEV_NONCANONICAL);
        if (gl == 0) classify((int)row, pe - ps, u, lo, hi);
    }
    if (G < 32) {
        __syncthreads();
        for (int r = threadIdx.x >> 5; r < min(s_nmid, MID_LIST); r += 8) {
            const int row = s_mid[r];
            const i64 ps = A.pos[row], pe = A.pos[row + 1];
            i64 u;
            int lo, hi, bad;
            entry_totals<SUMMARY, 32>(ps, pe, (int)lane, A, B, brow, u, lo, hi, bad);
            if (lane == 0) {
                if (bad) raise_status(ctl, DEV_NONCANONICAL);
                classify(row, pe - ps, u, lo, hi);
            }
        }
    }
    if (gl == 0 && run_rows) flush(run_cls, run_rows, run_products);
    __syncthreads();
    for (int r = 0; r < min(s_nlong, LONG_LIST); ++r) long_row_bounds<SUMMARY>(s_long[r], A, B, tab, prm, ctl, brow);
    // the totals: reduced over the warp first (lanes other than a group's first hold zeros)
    my_max = __reduce_max_sync(0xffffffffu, my_max);
    const unsigned bm_lo = __reduce_add_sync(0xffffffffu, my_bm_words & 0xffffu), bm_hi = __reduce_add_sync(0xffffffffu, my_bm_words >> 16);
    if (lane == 0) {
        if (bm_lo | bm_hi) atomicAdd((u64*)&s_bm_words, (u64)bm_lo + ((u64)bm_hi << 16));
        if (my_max) atomicMax(&s_max_ub, (i64)my_max);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        int rows = 0;
        i64 prods = 0;
        if (threadIdx.x < NCLASS) {
            for (int w = 0; w < 8; ++w) { rows += s_hist[w][threadIdx.x]; prods += s_cprod[w][threadIdx.x] + s_clow[w][threadIdx.x]; }
            if (rows) atomicAdd(&ctl->class_count[threadIdx.x], rows);
            if (prods) atomicAdd((u64*)&ctl->class_products[threadIdx.x], (u64)prods);
        }
        for (int d = 8; d > 0; d >>= 1) prods += __shfl_xor_sync(0xffffffffu, prods, d);
        if (threadIdx.x == 0 && prods) atomicAdd((u64*)&ctl->products, (u64)prods);
    }
    if (threadIdx.x == 0) {
        if (s_max_ub) atomicMax(&ctl->max_ub, s_max_ub);
        if (s_max_ub_global) atomicMax(&ctl->max_ub_global, s_max_ub_global);
        if (s_max_ub_smem) atomicMax(&ctl->max_ub_smem, s_max_ub_smem);
        if (s_order_words) atomicAdd(&ctl->order_words, (u64)s_order_words);
        if (s_max_span_words) atomicMax(&ctl->max_span_words, s_max_span_words);
        if (s_bm_words) atomicAdd(&ctl->bm_words, (u64)s_bm_words);
    }
}

cudaError_t launch_row_bounds(const LaunchCtx& c, const Csr& A, const Csr& B, i64 nnzA, bool clear_ctl) {
    if (A.nrows == 0) return clear_ctl ? cudaMemsetAsync(c.ctl, 0, sizeof(DevCtl), c.stream) : cudaSuccess;
    const double avg = (double)nnzA / (double)A.nrows;
    const int threads = 256;
    if (c.brow) {
        i64 want = ((i64)B.nrows + threads - 1) / threads;
        i64 cap = (i64)c.sm_count * 8;
        const cudaError_t e = launch_chained(c, brow_summary_kernel, want < cap ? want : cap, threads, 0, B, c.brow, clear_ctl ? c.ctl : nullptr);
        if (e != cudaSuccess) return e;
    } else if (clear_ctl) {
        cudaError_t e = cudaMemsetAsync(c.ctl, 0, sizeof(DevCtl), c.stream);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaSuccess;
    // as many blocks as are resident at once: a block's start and its totals cost as much as several of its rows (with 16 blocks an
    // SM, of which five are resident: 2e6 rows of one entry 35 -> 28 us, 1.6e5 of 9 33 -> 25, a stencil of 2^18 rows 48 -> 37,
    // of 8e4 25 -> 15, power law on 2^18 vertices 87 -> 72)
    auto launch = [&](auto kernel, int G) {
        int per_sm = 0;
        if ((e = resident_blocks((const void*)kernel, threads, 0, &per_sm)) != cudaSuccess) return;
        const i64 want = ((i64)A.nrows * G + threads - 1) / threads, cap = (i64)c.sm_count * std::max(per_sm, 1);
        e = launch_chained(c, kernel, std::min(want, cap), threads, 0, A, B, c.tab, c.prm, c.ctl, c.brow);
    };
    const bool sm = c.brow != nullptr;
    if (avg <= 1.5) sm ? launch(row_bounds_kernel<1, true>, 1) : launch(row_bounds_kernel<1, false>, 1);
    else if (avg <= 3.0) sm ? launch(row_bounds_kernel<2, true>, 2) : launch(row_bounds_kernel<2, false>, 2);
    else if (avg <= 6.0) sm ? launch(row_bounds_kernel<4, true>, 4) : launch(row_bounds_kernel<4, false>, 4);
    // (eight lanes take 32 entries in one step, four loads each, and the warps of a block take its longer rows at the
    // end: a 27-point stencil of 2^18 rows 90 -> 47 us, a power law of 2^18 rows 122 -> 89 us against a warp
    // per row; with so few rows that the longest sets the time a warp per row: power law of 16381 rows 28 -> 18 us.
    // Power laws of 14 .. 25 entries a row, eight lanes : a warp, us: 8000 rows 20 : 19, 16381 37 : 25, 32000 25 : 31,
    // 48000 37 : 42, 65000 41 : 50, 100000 61 : 67, 200000 97 : 114: they cross between 16381 and 32000 rows, so
    // the line, well on the side of many rows, gives up 6 us between 2^15 and 2^16)
    else if (avg <= (A.nrows >= (1 << 16) ? 32.0 : 12.0)) sm ? launch(row_bounds_kernel<8, true>, 8) : launch(row_bounds_kernel<8, false>, 8);
    else sm ? launch(row_bounds_kernel<32, true>, 32) : launch(row_bounds_kernel<32, false>, 32);
    return e;
}

// ---------------------------------------------------------------------------------------
// Word lists of long B rows.  The list of row k lives in `bw` at the positions of the row's own
// entries: bw[pos[k]] is a header (.x = number of pairs, 0 = no list), the pairs (.x = column / 32,
// .y = the bits of the row's entries in that word) follow.  A list is kept only when it has at
// most three quarters as many pairs as the row has entries.
// ---------------------------------------------------------------------------------------
// Rows of at least BW_BLOCK_ROW entries are listed from the end of bw_long and take a block each, the others from its start.
// Those take a warp each when they are more than BW_FEW, else a block each too: a block of 1024 threads spends 3.1 us on a row
// of 300 entries, a warp 13.5 us, of which 9472 run at once, and 27 us on one of 1000.  A block of 1024 for
// every row / a warp for all but those of 1024 entries / by the count, us: power law on 8000 vertices 9 / 25 / 9, 16381
// 24 / 33 / 24, 2^18 56 / 30 / 30; 2e4 rows of 256 207 / 31 / 31; 1e5 rows of 300 1078 / 142 / 140.  (256 threads for every row: 12,
// 20, 80, 54, 281; 3000 rows of 4000 60, with 1024 69, by a warp 150.)
constexpr int BW_BLOCK_ROW = 1024;
constexpr int BW_FEW = 2048;
// Also numbers the symbolic units of the CTA rows (`rows`, n of them), and clears the slots of those that are split, in which their
// blocks will unite their bitmaps.
constexpr int CP_THREADS = 256;
__global__ void __launch_bounds__(CP_THREADS) cta_prepare_kernel(Csr B, int* __restrict__ bw_long, int cap, const int* __restrict__ rows, int n, i64 part_products,
                                                                int unit_cap, RowTables tab, DevCtl* ctl) {
    __shared__ i64 s_slot[CP_THREADS];
    __shared__ int s_quads[CP_THREADS], s_n[3], s_base[2];          // shares of split rows, whole rows, split rows of the block
    if (ctl->status != 0) return;
    const int tid = threadIdx.x, lane = tid & 31;
    // (neighbours in perm go to different blocks: the rows to be split are often neighbours)
    for (i64 r0 = 0; r0 + blockIdx.x < n; r0 += (i64)gridDim.x * CP_THREADS) {
        const i64 r = r0 + (i64)tid * gridDim.x + blockIdx.x;
        const int row = r < n ? rows[r] : -1;
        const int parts = row >= 0 ? sym_parts_of_row(tab.ub[row], part_products) : 0;
        __syncthreads();
        if (tid < 3) s_n[tid] = 0;
        __syncthreads();
        // units reserved per block; whole rows: one addition a warp
        const unsigned whole = __ballot_sync(0xffffffffu, parts == 1);
        int at = 0;
        if (lane == 0 && whole) at = atomicAdd(&s_n[1], __popc(whole));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(whole & ((1u << lane) - 1u));
        if (parts > 1) {
            at = atomicAdd(&s_n[0], parts);
            const int x = atomicAdd(&s_n[2], 1);
            s_slot[x] = tab.bm_off[row];
            s_quads[x] = ((tab.jmax[row] - tab.jmin[row]) / 32 + 4) >> 2;
        }
        __syncthreads();
        if (tid < 2 && s_n[tid]) s_base[tid] = atomicAdd(&ctl->sym_units[tid], s_n[tid]);
        for (int x = tid >> 5; x < s_n[2]; x += CP_THREADS / 32) {
            uint4* const slot = reinterpret_cast<uint4*>(tab.bm_arena + s_slot[x]);
            for (int q = lane; q < s_quads[x]; q += 32) slot[q] = make_uint4(0u, 0u, 0u, 0u);
        }
        __syncthreads();
        // (the table holds a unit per row and 2^19 more; the shares of split rows are some 4096 and a share per such row)
        if (parts == 1) {
            tab.unit_row[unit_cap - 1 - (s_base[1] + at)] = row;
        } else if (parts > 1) {
            const int u0 = s_base[0] + at;
            tab.row_unit0[row] = u0;
            for (int t = 0; t < parts; ++t) tab.unit_row[u0 + t] = row;
        }
    }
    if (cap == 0) return;
    for (i64 k = (i64)blockIdx.x * CP_THREADS + tid; k < B.nrows; k += (i64)gridDim.x * CP_THREADS) {
        const i64 len = B.pos[k + 1] - B.pos[k];
        if (len >= BW_BLOCK_ROW) {
            const int at = atomicAdd(&ctl->n_longest, 1);
            if (at < cap) bw_long[cap - 1 - at] = (int)k;
        } else if (len >= BW_MIN_LEN) {
            const int at = atomicAdd(&ctl->n_long, 1);
            if (at < cap) bw_long[at] = (int)k;
        }
    }
}

constexpr int BWB_THREADS = 1024;
constexpr int BWB_ITEMS = 4;

// The list of row k by `THREADS` threads, of which this is thread `tid`.
template <int THREADS>
__device__ __forceinline__ void bw_build_row(int k, int tid, const Csr& B, uint2* __restrict__ bw, int* ws) {
    const i64 qs = B.pos[k], qe = B.pos[k + 1];
    const i64 len = qe - qs;
    const int* __restrict__ crd = B.crd;
    int carry = 0;                                       // pairs of the row before this tile
    for (i64 t0 = qs; t0 < qe; t0 += THREADS * BWB_ITEMS) {
        const i64 q0 = t0 + (i64)tid * BWB_ITEMS;
        unsigned word[BWB_ITEMS], bits[BWB_ITEMS];
        int nfirst = 0;
        unsigned prev = (q0 > qs && q0 < qe) ? ((unsigned)__ldg(crd + q0 - 1) >> 5) : 0xffffffffu;
#pragma unroll
        for (int x = 0; x < BWB_ITEMS; ++x) {
            const i64 q = q0 + x;
            word[x] = 0xffffffffu;                       // not the first entry of a word
            bits[x] = 0u;
            if (q < qe) {
                const unsigned c = (unsigned)__ldg(crd + q);
                if ((c >> 5) != prev) {
                    word[x] = c >> 5;
                    unsigned b = 1u << (c & 31);
                    for (i64 q2 = q + 1; q2 < qe; ++q2) {              // at most 31 more entries share the word
                        const unsigned c2 = (unsigned)__ldg(crd + q2);
                        if ((c2 >> 5) != word[x]) break;
                        b |= 1u << (c2 & 31);
                    }
                    bits[x] = b;
                    ++nfirst;
                }
                prev = c >> 5;
            }
        }
        int at = carry;
        if constexpr (THREADS == 32) {
            const int incl = warp_incl_scan(nfirst);
            at += incl - nfirst;
            carry += __shfl_sync(0xffffffffu, incl, 31);
        } else {
            int total;
            at += block_excl_scan<THREADS>(nfirst, ws, total);
            carry += total;
        }
#pragma unroll
        for (int x = 0; x < BWB_ITEMS; ++x)
            if (word[x] != 0xffffffffu) {
                if (at + 1 < len) bw[qs + 1 + at] = make_uint2(word[x], bits[x]);
                ++at;
            }
    }
    if (tid == 0) bw[qs] = make_uint2(4 * (i64)carry <= 3 * len ? (unsigned)carry : 0u, 0u);
}

__global__ void __launch_bounds__(BWB_THREADS, 2) bw_build_kernel(Csr B, const int* __restrict__ bw_long, int cap,
                                                                 uint2* __restrict__ bw, DevCtl* ctl) {
    __shared__ int ws[33];
    __shared__ int s_next;
    const int tid = threadIdx.x;
    const int n_longest = min(ctl->n_longest, cap), n_long = min(ctl->n_long, cap);
    const bool few = n_long <= BW_FEW;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_next = atomicAdd(&ctl->work_counter[BW_SLOT], 1);
        __syncthreads();
        const int r = s_next;
        if (r >= n_longest + (few ? n_long : 0)) break;
        bw_build_row<BWB_THREADS>(r < n_longest ? bw_long[cap - 1 - r] : bw_long[r - n_longest], tid, B, bw, ws);
    }
    while (!few) {
        int r = 0;
        if ((tid & 31) == 0) r = atomicAdd(&ctl->work_counter[BW_WARP_SLOT], 1);
        r = __shfl_sync(0xffffffffu, r, 0);
        if (r >= n_long) break;
        bw_build_row<32>(bw_long[r], tid & 31, B, bw, nullptr);
    }
}

cudaError_t launch_cta_prepare(const LaunchCtx& c, i64 products, const Csr& B) {
    const i64 rows = c.class_rows[CLS_DENSE_HUB] + c.class_rows[CLS_DENSE_CTA];
    const i64 want = std::max(((i64)B.nrows + CP_THREADS - 1) / CP_THREADS, std::min(rows, (i64)c.sm_count)), cap = (i64)c.sm_count * 8;
    i64 off = 0;
    for (int k = 0; k < CLS_DENSE_HUB; ++k) off += c.class_rows[k];
    cta_prepare_kernel<<<(int)(want < cap ? want : cap), CP_THREADS, 0, c.stream>>>(B, c.bw_long, c.bw ? c.bw_long_cap : 0, c.tab.perm + off, (int)rows,
                                                                                  sym_part_products(products), c.prm.unit_cap, c.tab, c.ctl);
    ++c.launches;
    if (!c.bw) return cudaGetLastError();
    bw_build_kernel<<<c.sm_count * 2, BWB_THREADS, 0, c.stream>>>(B, c.bw_long, c.bw_long_cap, c.bw, c.ctl);
    ++c.launches;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Binning: rows grouped by class into perm (class c occupies [off[c], off[c+1])); dense rows
// also reserve the slot of their occupancy bitmap in the arena.  Order inside a class follows
// block arrival.
// ---------------------------------------------------------------------------------------
// It also counts the units per bucket of rows and clears the words of the kernels that hand running sums
// from tile to tile.  A block of its own publishes the class sizes meanwhile, so that the host's next launch does not wait
// for the rows (2048 rows: 10 us and a gap of 10 us behind it when the last block published, 4 us without a gap now; published by
// the bounds kernel instead, the fences of its blocks cost 6 .. 14 us).
__global__ void __launch_bounds__(256, 4) bin_rows_kernel(int m, RowTables tab, ClassParams prm, DevCtl* ctl, HostBlock* host, int seq, u64* look, int n_look) {
    __shared__ int s_units[UNIT_BUCKETS];
    chained_start();
    const bool too_small = ctl->bm_words > prm.bm_arena_words;
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) {
            if (too_small) raise_status(ctl, DEV_SCRATCH_TOO_SMALL);
            *(volatile int*)&host->late = 0;            // (here and not by the host: the pass before may still raise one)
            ctl->host_status = &host->late;
        }
        __syncthreads();
        publish_ctl(ctl, host, seq);
        return;
    }
    if (too_small) return;
    const int block = blockIdx.x - 1, blocks = gridDim.x - 1;
    if (threadIdx.x < UNIT_BUCKETS) s_units[threadIdx.x] = 0;
    for (int w = block * 256 + threadIdx.x; w < n_look; w += blocks * 256) look[w] = 0;
    const i64 unit_products = dense_unit_products(ctl->products, prm.unit_products);
    __shared__ int s_hist[NCLASS], s_base[NCLASS], s_off[NCLASS];
    __shared__ int ws[33];
    __shared__ u64 s_bm_base;
    const int rows_per_block = blockDim.x * 4;
    if (threadIdx.x < 32) {                             // start of every class in perm
        const int n = threadIdx.x < NCLASS ? ctl->class_count[threadIdx.x] : 0;
        const int o = warp_incl_scan(n) - n;
        if (threadIdx.x < NCLASS) s_off[threadIdx.x] = o;
    }
    for (i64 r0 = (i64)block * rows_per_block; r0 < m; r0 += (i64)blocks * rows_per_block) {
        if (threadIdx.x < NCLASS) s_hist[threadIdx.x] = 0;
        int cls[4], rank[4], words[4], my_words = 0;
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const i64 row = r0 + x * blockDim.x + threadIdx.x;
            cls[x] = row < m ? (int)tab.cls[row] : -1;
        }
        __syncthreads();
        // bitmap words of this thread's dense rows
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const i64 row = r0 + x * blockDim.x + threadIdx.x;
            words[x] = 0;
            // one addition per class among the 32 rows (a block of like rows would queue at one counter otherwise)
            const unsigned peers = __match_any_sync(0xffffffffu, cls[x]);
            const int first = __ffs(peers) - 1;
            int at = 0;
            if (cls[x] >= 0 && (int)(threadIdx.x & 31) == first) at = atomicAdd(&s_hist[cls[x]], __popc(peers));
            rank[x] = __shfl_sync(0xffffffffu, at, first) + __popc(peers & ((1u << (threadIdx.x & 31)) - 1u));
            if (dense_cls(cls[x])) {
                words[x] = slot_words(tab.jmin[row], tab.jmax[row]);
                if (cls[x] != CLS_DENSE_WARP) {
                    const i64 u = tab.ub[row];
                    atomicAdd(&s_units[unit_bucket(u)], dense_units_of_row(u, unit_products));
                }
            }
            my_words += words[x];
        }
        // places in perm and in the arena: one reservation per class and one of the arena per block, side by side
        int block_words;
        int my_off = block_excl_scan<256>(my_words, ws, block_words);
        if (threadIdx.x < NCLASS && s_hist[threadIdx.x])
            s_base[threadIdx.x] = atomicAdd(&ctl->class_cursor[threadIdx.x], s_hist[threadIdx.x]);
        if (threadIdx.x == 32 && block_words) s_bm_base = atomicAdd(&ctl->bm_words_used, (u64)block_words);
        __syncthreads();
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const i64 row = r0 + x * blockDim.x + threadIdx.x;
            if (cls[x] < 0) continue;
            tab.perm[s_off[cls[x]] + s_base[cls[x]] + rank[x]] = (int)row;
            if (words[x]) {
                const u64 at = s_bm_base + (u64)my_off;
                my_off += words[x];
                tab.bm_off[row] = (i64)at;              // (inside the arena: the slots add up to the total compared above)
            }
        }
        __syncthreads();
    }
    if (threadIdx.x < UNIT_BUCKETS && s_units[threadIdx.x]) atomicAdd(&ctl->units_of[threadIdx.x], s_units[threadIdx.x]);
}

cudaError_t launch_bin_rows(const LaunchCtx& c, int m) {
    i64 want = ((i64)m + 1023) / 1024;
    i64 cap = (i64)c.sm_count * 8;
    if (want < 1) want = 1;
    return launch_chained(c, bin_rows_kernel, 1 + (want < cap ? want : cap), 256, 0, m, c.tab, c.prm, c.ctl, c.host, c.seq, c.look, c.n_look);
}

// ---------------------------------------------------------------------------------------
// Once the output counts are known, in ONE pass over the rows: the row pointer, the numeric routing of
// the dense rows, the outputs per class, and (TTM) C's fibre level.  A tile of FR_TILE rows per block;
// warp w owns the w-th run of 256 consecutive rows, a lane per row and step, so every load and store
// is contiguous.  Tiles hand the running sums on by a decoupled look-back.
//   Routing: a row the warp kernel counted and whose outputs fit a warp's accumulator stays with a warp;
//   every other dense row becomes one CTA unit, or several when it has many products: unit c of n takes
//   the c-th n-th of the row's A entries (all units of a row add into the same outputs).
//   TTM: a fibre (i,j) survives when it produced an output; survivors are packed (Cpos2, Ccrd1), and
//   sfp[s] receives the number of survivors before slice s.
// Replaces a three-launch scan, the routing and the per-class count (five launches; seven for the
// 3-tensor form).
// Bound by the chain of its steps (2048 rows: 6 us where the five launches took 13 and their gaps; 2e6 fibres: 27 us with five
// blocks an SM, 21 with seven, which hold all 963 tiles at once, for 24 bytes spilled).
// ---------------------------------------------------------------------------------------
constexpr int FR_THREADS = 256;
constexpr int FR_WARPS = FR_THREADS / 32;
constexpr int FR_ITEMS = 8;
constexpr int FR_TILE = FR_THREADS * FR_ITEMS;
constexpr int SL_TILE = FR_THREADS * 4;             // slices per block of the slice level

struct FibreArgs {
    const i64* Apos1;
    const int* Acrd1;
    int n_i;
    i64* sfp;
    int* Ccrd1;
    i64* Cpos2;
};

template <bool DENSE, bool TTM>
__global__ void __launch_bounds__(FR_THREADS, DENSE ? 3 : 7) finish_rows_kernel(int m, RowTables tab, ClassParams prm, DevCtl* ctl, HostBlock* host, int seq, u64* look,
                                                                 i64* __restrict__ rowptr, FibreArgs f) {
    __shared__ int s_tile, s_slice0;
    __shared__ i64 s_sum[FR_WARPS], s_before[2];
    __shared__ int s_part[1 + N_WARP_LISTS][FR_WARPS];     // survivors, warp rows on each list
    __shared__ int s_wbase[N_WARP_LISTS], s_units[UNIT_BUCKETS];           // places in the routing tables; units: the tile's count, then the running place
    __shared__ i64 s_cls[FR_WARPS][N_PUBLIC_CLASS];
    __shared__ i64 s_wp[FR_WARPS];
    __shared__ int s_wn[FR_WARPS], s_wm[N_WARP_LISTS][FR_WARPS];
    __shared__ int s_kept[TTM ? FR_TILE : 1];       // survivors of the tile before each fibre
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned all = 0xffffffffu, below = (1u << lane) - 1u;
    const int tiles = gridDim.x;
    chained_start();
    if (tid == 0) s_tile = atomicAdd(&ctl->rows_ticket, 1);
    for (int x = tid; x < FR_WARPS * N_PUBLIC_CLASS; x += FR_THREADS) (&s_cls[0][0])[x] = 0;
    if (tid >= 128 && tid < 128 + UNIT_BUCKETS) s_units[tid - 128] = 0;
    __syncthreads();
    const int tile = s_tile;
    const i64 tile0 = (i64)tile * FR_TILE;
    const i64 row0 = tile0 + warp * (FR_ITEMS * 32) + lane;
    const i64 unit_products = DENSE ? dense_unit_products(ctl->products, prm.unit_products) : 1;
    int unit_count = 0;                             // units of all rows but those that outgrow a warp
    if (DENSE)
        for (int k = 0; k < UNIT_BUCKETS; ++k) unit_count += ctl->units_of[k];
    const bool few = unit_count < UNIT_FEW;

    // ---- this warp's rows: counts, sums, routing
    int v[FR_ITEMS], cls[FR_ITEMS];
    i64 sum = 0, wp = 0;
    int kept = 0, wn = 0, to_warp[N_WARP_LISTS] = {}, wm[N_WARP_LISTS] = {};
    // all loads first: what the rows below need is a few registers, a load inside the loops is a wait each
    int q[DENSE ? FR_ITEMS : 1];                    // products of a warp-class row; bucket and units of another dense row
    int acrd[TTM ? FR_ITEMS : 1];
    {
        i64 ub[DENSE ? FR_ITEMS : 1];
#pragma unroll
        for (int x = 0; x < FR_ITEMS; ++x) {
            const i64 row = row0 + 32 * x;
            v[x] = row < m ? tab.cnt[row] : 0;
            cls[x] = row < m ? (int)tab.cls[row] : (int)CLS_EMPTY;
            if (DENSE) ub[x] = row < m ? tab.ub[row] : 0;
            if (TTM) acrd[x] = row < m ? f.Acrd1[row] : 0;
        }
        if (DENSE)
#pragma unroll
            for (int x = 0; x < FR_ITEMS; ++x)
                q[x] = cls[x] == CLS_DENSE_WARP ? (int)ub[x] : (unit_bucket(ub[x]) << 28) | dense_units_of_row(ub[x], unit_products);
    }
    // list of the warp numeric kernel a row goes to; -1: to CTA units or not dense
    auto list_of = [&](int x) -> int {
        if (!DENSE || cls[x] != CLS_DENSE_WARP || v[x] > prm.warp_outputs) return -1;
        return v[x] <= DENSE_WARP_ACC ? 0 : 1;
    };
    auto unit_row = [&](int x) { return DENSE && cls[x] >= CLS_DENSE_WARP && cls[x] <= CLS_DENSE_CTA && list_of(x) < 0; };
    // (a row that outgrew a warp has at most DENSE_WARP_MAX_UB products: one unit)
    auto units = [&](int x) { return cls[x] == CLS_DENSE_WARP ? 1 : q[x] & 0xfffffff; };
    auto bucket = [&](int x) { return !few ? 0 : cls[x] == CLS_DENSE_WARP ? UNIT_BUCKETS - 1 : q[x] >> 28; };
    bool one_class = true;
    // the (public) class of the warp's first row that is not empty in the first 32 rows (all empty: any)
    const unsigned some = __ballot_sync(all, cls[0] != CLS_EMPTY);
    const int cls0 = public_class(__shfl_sync(all, cls[0], some ? __ffs(some) - 1 : 0));
#pragma unroll
    for (int x = 0; x < FR_ITEMS; ++x) {
        sum += v[x];
        one_class &= public_class(cls[x]) == cls0 || cls[x] == CLS_EMPTY;
        if (TTM) kept += __popc(__ballot_sync(all, v[x] > 0));
        if (DENSE) {
            const int l = list_of(x);
#pragma unroll
            for (int t = 0; t < N_WARP_LISTS; ++t) {
                to_warp[t] += __popc(__ballot_sync(all, l == t));
                if (l == t) wm[t] = max(wm[t], v[x]);
            }
            if (l >= 0) { wp += q[x]; wn += v[x]; }
            if (unit_row(x)) atomicAdd(&s_units[bucket(x)], units(x));
        }
    }
    for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(all, sum, d);
    // outputs per class: this warp's sum when its 256 rows share a class, else one round per class and 32 rows
    if (__all_sync(all, one_class)) {
        if (lane == 0 && cls0 != CLS_EMPTY) s_cls[warp][cls0] = sum;
    } else {
#pragma unroll
        for (int x = 0; x < FR_ITEMS; ++x) {
            unsigned todo = __ballot_sync(all, cls[x] != CLS_EMPTY);
            while (todo) {
                const int k = public_class(__shfl_sync(all, cls[x], __ffs(todo) - 1));
                const bool mine = public_class(cls[x]) == k;
                const unsigned lo = __reduce_add_sync(all, mine ? (unsigned)v[x] & 0xffffu : 0u);
                const unsigned hi = __reduce_add_sync(all, mine ? (unsigned)v[x] >> 16 : 0u);
                if (lane == 0) s_cls[warp][k] += (i64)lo + ((i64)hi << 16);
                todo &= ~__ballot_sync(all, mine);
            }
        }
    }
    if (DENSE) {
        for (int d = 16; d > 0; d >>= 1) wp += __shfl_xor_sync(all, wp, d);
        wn = __reduce_add_sync(all, wn);                // at most 256 rows of 1024 outputs
#pragma unroll
        for (int t = 0; t < N_WARP_LISTS; ++t) wm[t] = __reduce_max_sync(all, wm[t]);
    }
    if (TTM && warp == FR_WARPS - 1) {              // first slice that starts in this tile or later: 32 probes per step
        int lo = 0, hi = f.n_i;                     // Apos1[lo - 1] < tile0 <= Apos1[hi]
        while (lo < hi) {
            const int step = (hi - lo + 31) >> 5, at = lo + lane * step;
            const int n = __popc(__ballot_sync(all, at < hi && f.Apos1[at] < tile0));     // probes that start earlier
            const int from = n ? lo + (n - 1) * step + 1 : lo;
            hi = min(hi, lo + n * step);
            lo = from;
        }
        if (lane == 0) s_slice0 = lo;
    }
    if (lane == 0) {
        s_sum[warp] = sum;
        s_part[0][warp] = kept;
        s_wp[warp] = wp;
        s_wn[warp] = wn;
#pragma unroll
        for (int t = 0; t < N_WARP_LISTS; ++t) {
            s_part[1 + t][warp] = to_warp[t];
            s_wm[t][warp] = wm[t];
        }
    }
    __syncthreads();
    i64 tile_sum = 0, warp_sum = 0;
    int total[1 + N_WARP_LISTS] = {}, mine[1 + N_WARP_LISTS] = {};
#pragma unroll
    for (int w = 0; w < FR_WARPS; ++w) {
        if (w == warp) warp_sum = tile_sum;
        tile_sum += s_sum[w];
#pragma unroll
        for (int t = 0; t < 1 + N_WARP_LISTS; ++t) {
            if (w == warp) mine[t] = total[t];
            total[t] += s_part[t][w];
        }
    }
    // ---- running sums from the tiles before; places in the routing tables
    if (warp == 0 || (TTM && warp == 1)) {
        u64* const words = look + (warp == 0 ? 0 : tiles);
        const i64 own = warp == 0 ? tile_sum : (i64)total[0];
        if (lane == 0) look_publish(words + tile, tile == 0 ? 2 : 1, own);
        i64 before = 0;
        if (tile > 0) {
            before = look_back_warp(words, tile, 0, ctl);
            if (lane == 0) look_publish(words + tile, 2, before + own);
        }
        if (lane == 0) s_before[warp] = before;
    }
    if (DENSE && warp >= 2 && warp < 2 + N_WARP_LISTS && lane == 0) {
        const int list = warp - 2;
        int n_rows = total[1];
#pragma unroll
        for (int t = 1; t < N_WARP_LISTS; ++t) n_rows = list == t ? total[1 + t] : n_rows;
        if (n_rows) s_wbase[list] = atomicAdd(&ctl->n_warp_rows[list], n_rows);
        i64 p = 0;
        int n = 0, most = 0;
        for (int w = 0; w < FR_WARPS; ++w) { p += s_wp[w]; n += s_wn[w]; most = max(most, s_wm[list][w]); }
        if (most) atomicMax(&ctl->max_warp_cnt[list], most);
        if (list == 0 && p) {
            atomicAdd((u64*)&ctl->dense_warp_products, (u64)p);
            atomicAdd((u64*)&ctl->dense_warp_nnz, (u64)n);
        }
    }
    if (DENSE && tid >= 160 && tid < 160 + UNIT_BUCKETS) {
        const int k = tid - 160, n = s_units[k];
        int at = 0;
        if (n) {
            if (few)
                for (int j = 0; j < k; ++j) at += ctl->units_of[j];
            at += atomicAdd(&ctl->unit_cursor[k], n);
        }
        s_units[k] = at;
    }
    if (tid >= 192 && tid < 192 + N_PUBLIC_CLASS) {
        i64 t = 0;
        for (int w = 0; w < FR_WARPS; ++w) t += s_cls[w][tid - 192];
        if (t) atomicAdd((u64*)&ctl->class_nnz[tid - 192], (u64)t);
    }
    __syncthreads();

    // ---- placement
    i64 run = s_before[0] + warp_sum;
    const i64 kbase = TTM ? s_before[1] : 0;
    int krun = mine[0];
    const bool small = tile_sum < (1ll << 31);      // (a tile of 2048 counts may total 2^31 or more)
#pragma unroll
    for (int x = 0; x < FR_ITEMS; ++x) {
        const i64 row = row0 + 32 * x;
        i64 excl;
        if (small) {
            const int incl = warp_incl_scan(v[x]);
            excl = incl - v[x];
            if (row < m) rowptr[row] = run + excl;
            excl += run;
            run += __shfl_sync(all, incl, 31);
        } else {
            i64 incl = v[x];
            for (int d = 1; d < 32; d <<= 1) {
                const i64 t = __shfl_up_sync(all, incl, d);
                if (lane >= d) incl += t;
            }
            excl = run + incl - v[x];
            if (row < m) rowptr[row] = excl;
            run += __shfl_sync(all, incl, 31);
        }
        if (TTM) {
            const unsigned live = __ballot_sync(all, v[x] > 0);
            const int k = krun + __popc(live & below);
            s_kept[warp * (FR_ITEMS * 32) + x * 32 + lane] = k;
            if (v[x] > 0) {
                f.Cpos2[kbase + k] = excl;
                f.Ccrd1[kbase + k] = acrd[x];
            }
            krun += __popc(live);
        }
        if (DENSE) {
            const int l = list_of(x);
#pragma unroll
            for (int t = 0; t < N_WARP_LISTS; ++t) {
                const unsigned on = __ballot_sync(all, l == t);
                if (l == t) {
                    const int k = s_wbase[t] + mine[1 + t] + __popc(on & below);
                    tab.warp_rows[t == 0 ? k : m - 1 - k] = (int)row;
                    tab.row_unit0[row] = -1;
                }
                mine[1 + t] += __popc(on);
            }
            if (unit_row(x)) {
                const int nu = units(x);
                const int u0 = atomicAdd(&s_units[bucket(x)], nu);
                if ((i64)u0 + nu > prm.unit_cap) {
                    raise_status(ctl, DEV_SCRATCH_TOO_SMALL);
                    tab.row_unit0[row] = -1;
                } else {
                    tab.row_unit0[row] = u0;
                    for (int t = 0; t < nu; ++t) tab.unit_row[u0 + t] = (int)row;
                }
            }
        }
    }
    if (tile == tiles - 1 && tid == 0) {
        const i64 nnz = s_before[0] + tile_sum;
        rowptr[m] = nnz;
        ctl->nnz = nnz;
        if (TTM) {
            const i64 k = kbase + total[0];
            f.Cpos2[k] = nnz;
            f.sfp[f.n_i] = k;
            ctl->kept[1] = k;
        }
    }
    if (TTM) {
        __syncthreads();
        for (int s = s_slice0 + tid; s < f.n_i; s += FR_THREADS) {
            const i64 at = f.Apos1[s] - tile0;
            if (at >= FR_TILE && tile != tiles - 1) break;
            f.sfp[s] = kbase + (at >= 0 && at < FR_TILE && tile0 + at < m ? s_kept[at] : total[0]);
        }
    }
    if (last_block(&ctl->rows_done, tiles)) {
        if (tid == 0) {
            int n = 0;
            for (int k = 0; k < UNIT_BUCKETS; ++k) n += ctl->unit_cursor[k];
            ctl->n_units = n;
        }
        __syncthreads();
        if (!TTM) publish_ctl(ctl, host, seq);           // (the slice level comes after the fibres)
    }
}

// A slice i survives when one of its fibres does: C's slice level from sfp.
__global__ void __launch_bounds__(FR_THREADS) finish_slices_kernel(int n_i, const i64* __restrict__ sfp, const int* __restrict__ Acrd0, DevCtl* ctl,
                                                                   HostBlock* host, int seq, u64* look, int* __restrict__ Ccrd0, i64* __restrict__ Cpos1,
                                                                   i64* __restrict__ Cpos0) {
    __shared__ int s_tile, s_part[FR_WARPS];
    __shared__ i64 s_before;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tiles = gridDim.x;
    chained_start();
    not_before(sfp);
    if (tid == 0) s_tile = atomicAdd(&ctl->slices_ticket, 1);
    __syncthreads();
    const int tile = s_tile;
    const i64 s0 = (i64)tile * SL_TILE + warp * 128 + lane;
    i64 first[4];
    unsigned live[4];
    int n = 0;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const i64 s = s0 + 32 * x;
        first[x] = s < n_i ? sfp[s] : 0;
        live[x] = __ballot_sync(0xffffffffu, s < n_i && sfp[s + 1] > first[x]);
        n += __popc(live[x]);
    }
    if (lane == 0) s_part[warp] = n;
    __syncthreads();
    int total = 0, mine = 0;
#pragma unroll
    for (int w = 0; w < FR_WARPS; ++w) {
        if (w == warp) mine = total;
        total += s_part[w];
    }
    if (warp == 0) {
        if (lane == 0) look_publish(look + tile, tile == 0 ? 2 : 1, total);
        i64 before = 0;
        if (tile > 0) {
            before = look_back_warp(look, tile, 0, ctl);
            if (lane == 0) look_publish(look + tile, 2, before + total);
        }
        if (lane == 0) s_before = before;
    }
    __syncthreads();
    i64 at = s_before + mine;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        if ((live[x] >> lane) & 1u) {
            const i64 o = at + __popc(live[x] & ((1u << lane) - 1u));
            Ccrd0[o] = Acrd0[s0 + 32 * x];
            Cpos1[o] = first[x];
        }
        at += __popc(live[x]);
    }
    if (tile == tiles - 1 && tid == 0) {
        const i64 k = s_before + total;
        Cpos1[k] = sfp[n_i];
        Cpos0[0] = 0;
        Cpos0[1] = k;
        ctl->kept[0] = k;
    }
    if (last_block(&ctl->slices_done, tiles)) publish_ctl(ctl, host, seq);
}

static int tiles_of(i64 n, int tile) { return n > 0 ? (int)((n + tile - 1) / tile) : 1; }

size_t look_words(i64 rows, i64 slices) { return (size_t)2 * tiles_of(rows, FR_TILE) + tiles_of(slices, SL_TILE); }

cudaError_t launch_finish_rows(const LaunchCtx& c, int m, bool any_dense, i64* rowptr) {
    const int tiles = tiles_of(m, FR_TILE);
    return launch_chained(c, any_dense ? finish_rows_kernel<true, false> : finish_rows_kernel<false, false>, tiles, FR_THREADS, 0, m, c.tab, c.prm, c.ctl,
                          c.host, c.seq + 1, c.look, rowptr, FibreArgs{});
}

cudaError_t launch_finish_fibres(const LaunchCtx& c, int n_i, int n_ij, bool any_dense, const i64* Apos1, const int* Acrd0, const int* Acrd1,
                                 i64* rowptr_raw, i64* sfp, i64* Cpos0, int* Ccrd0, i64* Cpos1, int* Ccrd1, i64* Cpos2) {
    const int tiles = tiles_of(n_ij, FR_TILE);
    const FibreArgs f{Apos1, Acrd1, n_i, sfp, Ccrd1, Cpos2};
    const cudaError_t e = launch_chained(c, any_dense ? finish_rows_kernel<true, true> : finish_rows_kernel<false, true>, tiles, FR_THREADS, 0, n_ij, c.tab,
                                         c.prm, c.ctl, c.host, c.seq + 1, c.look, rowptr_raw, f);
    if (e != cudaSuccess) return e;
    return launch_chained(c, finish_slices_kernel, tiles_of(n_i, SL_TILE), FR_THREADS, 0, n_i, sfp, Acrd0, c.ctl, c.host, c.seq + 1, c.look + 2 * tiles, Ccrd0,
                          Cpos1, Cpos0);
}

// ---------------------------------------------------------------------------------------
// Exclusive scan int32[n] -> int64[n+1] (reduce, scan of block sums, scan): no waits between
// blocks.  out[n] (and *total_out when given) receive the total.
// ---------------------------------------------------------------------------------------
constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

__global__ void __launch_bounds__(SCAN_THREADS) scan_reduce_kernel(const int* __restrict__ in, int n, i64* block_sums) {
    __shared__ i64 s_part[SCAN_THREADS / 32];
    const i64 base = (i64)blockIdx.x * SCAN_TILE;
    i64 s = 0;
    for (int x = 0; x < SCAN_ITEMS; ++x) {
        const i64 i = base + x * SCAN_THREADS + threadIdx.x;
        if (i < n) s += in[i];
    }
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        i64 t = 0;
        for (int w = 0; w < SCAN_THREADS / 32; ++w) t += s_part[w];
        block_sums[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(1024) scan_block_sums_kernel(i64* block_sums, int nblocks, i64* out_total, i64* total_out2) {
    __shared__ i64 s_warp[32];
    __shared__ i64 s_carry;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < nblocks; base += 1024) {
        const int i = base + threadIdx.x;
        const i64 v = (i < nblocks) ? block_sums[i] : 0;
        i64 incl = v;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        for (int d = 1; d < 32; d <<= 1) {
            const i64 t = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += t;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            i64 w = s_warp[lane];
            i64 wi = w;
            for (int d = 1; d < 32; d <<= 1) {
                const i64 t = __shfl_up_sync(0xffffffffu, wi, d);
                if (lane >= d) wi += t;
            }
            s_warp[lane] = wi - w;
        }
        __syncthreads();
        const i64 carry = s_carry;
        if (i < nblocks) block_sums[i] = carry + s_warp[warp] + incl - v;
        __syncthreads();
        if (threadIdx.x == 1023) s_carry = carry + s_warp[warp] + incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        *out_total = s_carry;
        if (total_out2) *total_out2 = s_carry;
    }
}

// The in-tile prefix is carried in 64 bits: a tile of 2048 counts may total 2^31 or more.
__global__ void __launch_bounds__(SCAN_THREADS) scan_apply_kernel(const int* __restrict__ in, int n, const i64* __restrict__ block_sums, i64* __restrict__ out) {
    __shared__ i64 s_warp[SCAN_THREADS / 32];
    const i64 base = (i64)blockIdx.x * SCAN_TILE + (i64)threadIdx.x * SCAN_ITEMS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int v[SCAN_ITEMS];
    i64 s = 0;
#pragma unroll
    for (int x = 0; x < SCAN_ITEMS; ++x) {
        v[x] = (base + x < n) ? in[base + x] : 0;
        s += v[x];
    }
    i64 incl = s;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const i64 t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    i64 before = 0;
#pragma unroll
    for (int w = 0; w < SCAN_THREADS / 32; ++w) before += (w < warp) ? s_warp[w] : 0;
    i64 run = block_sums[blockIdx.x] + before + incl - s;
#pragma unroll
    for (int x = 0; x < SCAN_ITEMS; ++x) {
        if (base + x < n) out[base + x] = run;
        run += v[x];
    }
}

cudaError_t launch_scan_counts(const LaunchCtx& c, const int* cnt, int n, i64* out, i64* block_sums, i64* total_out) {
    const int nblocks = (int)(((i64)n + SCAN_TILE - 1) / SCAN_TILE);
    if (nblocks > 0) scan_reduce_kernel<<<nblocks, SCAN_THREADS, 0, c.stream>>>(cnt, n, block_sums);
    scan_block_sums_kernel<<<1, 1024, 0, c.stream>>>(block_sums, nblocks, out + n, total_out);
    if (nblocks > 0) scan_apply_kernel<<<nblocks, SCAN_THREADS, 0, c.stream>>>(cnt, n, block_sums, out);
    c.launches += nblocks > 0 ? 3 : 1;
    return cudaGetLastError();
}

}  // namespace spws

// ---------------------------------------------------------------------------------------
// spws_row_pointer_static: the exclusive scan of the symbolic pass for callers that cannot
// allocate device memory.  The scan's block sums -- the one piece of scratch it needs -- live
// in a fixed array inside the library image instead of a caller-supplied buffer.
// ---------------------------------------------------------------------------------------
#include <mutex>

#include "../../include/spws.h"

namespace {

constexpr long long STATIC_BLOCK_SUMS = SPWS_STATIC_MAX_ROWS / spws::SCAN_TILE;   // 8192 partial sums
static_assert(SPWS_STATIC_MAX_ROWS % spws::SCAN_TILE == 0, "row limit must be a whole number of scan tiles");

// 64 KiB resident on every GPU that loads the library, until the process exits.
static __device__ __align__(256) long long g_static_block_sums[STATIC_BLOCK_SUMS + 2];

constexpr int MAX_DEVICES = 64;
std::mutex g_static_mutex;
void* g_static_addr[MAX_DEVICES] = {};

// The array's name is only a host-side handle; kernels need its device address, which differs
// per GPU and is looked up once per device with that device current.
spws_status_t static_scratch_address(spws::i64** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) {
        cudaGetLastError();
        return SPWS_CUDA_ERROR;
    }
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_addr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_block_sums) != cudaSuccess || !p) {
            cudaGetLastError();
            return SPWS_CUDA_ERROR;
        }
        g_static_addr[dev] = p;
    }
    *out = static_cast<spws::i64*>(g_static_addr[dev]);
    return SPWS_OK;
}

}  // namespace

extern "C" spws_status_t spws_row_pointer_static(const int32_t* counts, int64_t n, int64_t* pos, void* cuda_stream) {
    if (n < 0 || !pos || (n > 0 && !counts)) return SPWS_INVALID_ARGUMENT;
    if (n > SPWS_STATIC_MAX_ROWS) return SPWS_SCRATCH_TOO_SMALL;
    spws::i64* block_sums = nullptr;
    const spws_status_t st = static_scratch_address(&block_sums);
    if (st != SPWS_OK) return st;
    spws::LaunchCtx c{};
    c.stream = static_cast<cudaStream_t>(cuda_stream);
    // Every partial sum the scan reads is written earlier in the same call, so nothing left
    // behind by a previous call has to be cleared.
    if (spws::launch_scan_counts(c, counts, (int)n, reinterpret_cast<spws::i64*>(pos), block_sums, nullptr) != cudaSuccess) {
        cudaGetLastError();
        return SPWS_CUDA_ERROR;
    }
    return SPWS_OK;
}
