// Insert-sort-merge workspace held in registers: one group of G lanes per output row whose
// product count is at most G (Algorithm 1 with the accumulation array = the lanes of the group;
// coordinate-sort policy, Sec. 5.2: append without reduction, sort, reduce equal coordinates).
//   Insert : lane t takes the t-th product of the row in loop order (k, then j).
//   Sort   : bitonic network over the group on the packed word (j - jmin) << 5 | lane -- only
//            this integer moves (accumulation indexing, Sec. 5.1); values stay in their lane.
//   Merge  : equal coordinates are adjacent; the first lane of a run sums the run in product
//            order and writes it at row_ptr[i] + rank.
#include "common.cuh"

namespace spws {

template <typename T, int G, bool NUMERIC>
__device__ __forceinline__ void reg_rows(const int* __restrict__ rows, int n, int block, int blocks, const Csr& A, const Csr& B,
                                         const int* __restrict__ jmin, int* __restrict__ cnt, const i64* __restrict__ rowptr,
                                         int* __restrict__ Ccrd, T* __restrict__ Cval) {
    const unsigned lane = threadIdx.x & 31;
    const int gl = threadIdx.x % G;
    const unsigned gshift = lane - gl;
    const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << gshift);
    const i64 group = ((i64)block * blockDim.x + threadIdx.x) / G;
    const i64 ngroups = ((i64)blocks * blockDim.x) / G;
    const T* __restrict__ Aval = (const T*)A.val;
    const T* __restrict__ Bval = (const T*)B.val;

    // the row id and its A range are loaded one iteration ahead: with a handful of products per row
    // the kernel is a chain of dependent loads otherwise
    int row_n = 0;
    i64 ps_n = 0, pe_n = 0;
    if (group < n) {
        row_n = __ldg(rows + group);
        ps_n = __ldg(A.pos + row_n);
        pe_n = __ldg(A.pos + row_n + 1);
    }
    for (i64 r = group; r < n; r += ngroups) {
        const int row = row_n;
        const i64 ps = ps_n, pe = pe_n;
        if (r + ngroups < n) {
            row_n = __ldg(rows + r + ngroups);
            ps_n = __ldg(A.pos + row_n);
            pe_n = __ldg(A.pos + row_n + 1);
        }
        const int base = jmin[row];

        // ---- Insert: lane gl receives product number gl
        unsigned packed = 0xffffffffu;
        T val = 0;
        int done = 0;
        for (i64 p0 = ps; p0 < pe; p0 += G) {
            const i64 p = p0 + gl;
            int len = 0;
            i64 qs = 0;
            if (p < pe) {
                const int k = __ldg(A.crd + p);
                if ((unsigned)k < (unsigned)B.nrows) {
                    qs = __ldg(B.pos + k);
                    len = (int)(__ldg(B.pos + k + 1) - qs);
                }
            }
            int incl = len;
#pragma unroll
            for (int d = 1; d < G; d <<= 1) {
                const int t = __shfl_up_sync(gmask, incl, d, G);
                if (gl >= d) incl += t;
            }
            const int excl = incl - len + done;
            const int total = __shfl_sync(gmask, incl, G - 1, G);
            // entry that owns product gl: the last entry whose first product is <= gl
            int e = 0;
#pragma unroll
            for (int s = G / 2; s >= 1; s >>= 1) {
                const int v = __shfl_sync(gmask, excl, e + s, G);
                if (v <= gl) e += s;
            }
            const int e_excl = __shfl_sync(gmask, excl, e, G);
            const i64 e_qs = __shfl_sync(gmask, qs, e, G);
            if (gl >= done && gl < done + total) {
                const i64 q = e_qs + (gl - e_excl);
                const int j = __ldg(B.crd + q);
                packed = ((unsigned)(j - base) << 5) | (unsigned)gl;
                if (NUMERIC) val = mul_rn(__ldg(Aval + p0 + e), __ldg(Bval + q));
            }
            done += total;
        }

        // ---- Sort
#pragma unroll
        for (int k = 2; k <= G; k <<= 1) {
#pragma unroll
            for (int j = k >> 1; j > 0; j >>= 1) {
                const unsigned other = __shfl_xor_sync(gmask, packed, j, G);
                const bool up = (gl & k) == 0;
                const bool low = (gl & j) == 0;
                packed = (up == low) ? min(packed, other) : max(packed, other);
            }
        }

        // ---- Merge
        const bool valid = packed != 0xffffffffu;
        const unsigned key = packed >> 5;
        const unsigned prev = __shfl_up_sync(gmask, key, 1, G);
        const bool head = valid && (gl == 0 || key != prev);
        const unsigned heads = (__ballot_sync(gmask, head) >> gshift) & ((G == 32) ? 0xffffffffu : ((1u << G) - 1u));
        if (!NUMERIC) {
            if (gl == 0) cnt[row] = __popc(heads);
        } else {
            T v = __shfl_sync(gmask, val, packed & 31u, G);
            T sum = v;
            for (int d = 1; d < G; ++d) {
                const unsigned k2 = __shfl_down_sync(gmask, key, d, G);
                const T v2 = __shfl_down_sync(gmask, v, d, G);
                const bool more = valid && (gl + d < G) && (k2 == key);
                if (!__any_sync(gmask, more)) break;
                if (more) sum = add_rn(sum, v2);
            }
            if (head) {
                const int rank = __popc(heads & ((1u << gl) - 1u));
                const i64 out = rowptr[row] + rank;
                Ccrd[out] = (int)key + base;
                Cval[out] = sum;
            }
        }
    }
}

// Rows with ONE A entry (the commonest fibre of a hyper-sparse 3-tensor): the products are the picked B
// row itself, already sorted and free of duplicates, so Insert, Sort and Merge are the identity and the
// row is copied out scaled.  Every lane first walks one row's chain of dependent loads (row id, A
// range, A entry, B range, output offset), 32 chains per warp in flight; then the warp copies the 32
// rows together, eight lanes per row and four rows per step.  When at least half of all rows are of this
// class they are found by walking all rows in order (rows null, n = all rows): row offsets, entries and
// output offsets are then read, and the output written, as contiguous streams.
// 2e6 fibres of which 1.85e6 are copied (8 entries each, f64): 132 us for all four classes in four launches,
// 117 us in one with the copied rows in order.
template <typename T>
__device__ __forceinline__ void copy_rows(const int* __restrict__ rows, const unsigned char* __restrict__ cls, int n, int block, int blocks,
                                          const Csr& A, const Csr& B, const i64* __restrict__ rowptr, int* __restrict__ Ccrd,
                                          T* __restrict__ Cval) {
    const int lane = threadIdx.x & 31;
    const T* __restrict__ Aval = (const T*)A.val;
    const T* __restrict__ Bval = (const T*)B.val;
    const i64 stride = (i64)blocks * blockDim.x;
    for (i64 r0 = ((i64)block * blockDim.x + threadIdx.x) - lane; r0 < n; r0 += stride) {
        const i64 r = r0 + lane;
        i64 qs = 0, out = 0;
        int len = 0;
        T a = 0;
        if (r < n && (rows || cls[r] == CLS_COPY)) {
            const int row = rows ? __ldg(rows + r) : (int)r;
            const i64 p = __ldg(A.pos + row);
            const int k = __ldg(A.crd + p);
            a = __ldg(Aval + p);
            out = __ldg(rowptr + row);
            if ((unsigned)k < (unsigned)B.nrows) {
                qs = __ldg(B.pos + k);
                len = (int)min(__ldg(B.pos + k + 1) - qs, (i64)COPY_MAX);
            }
        }
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const int src = 4 * s + (lane >> 3);
            const i64 q = __shfl_sync(0xffffffffu, qs, src), o = __shfl_sync(0xffffffffu, out, src);
            const int l = __shfl_sync(0xffffffffu, len, src);
            const T av = __shfl_sync(0xffffffffu, a, src);
            for (int e = lane & 7; e < l; e += 8) {
                Ccrd[o + e] = __ldg(B.crd + q + e);
                Cval[o + e] = mul_rn(av, __ldg(Bval + q + e));
            }
        }
    }
}

// The copied class and the three register classes in one launch: consecutive ranges of blocks, so that the
// classes run side by side and no class waits for the last rows of another (four launches before).
struct RegBlocks { int end[4]; };       // blocks of the copied rows, of 8, 16 and 32 lanes per row: ends of the ranges

// (six blocks per SM, but five for double values, which spill at 40 registers: 2e6 fibres, count 25.5 -> 22.6 us; 65536
// rows of 16 products, f32, 19.3 + 27.2 -> 17.7 + 25.4 us)
template <typename T, bool NUMERIC>
__global__ void __launch_bounds__(256, NUMERIC && sizeof(T) == 8 ? 5 : 6) ism_reg_kernel(const int* __restrict__ perm, const unsigned char* __restrict__ cls, const DevCtl* __restrict__ ctl,
                                                      RegBlocks g, Csr A, Csr B,
                                                      const int* __restrict__ jmin, int* __restrict__ cnt, const i64* __restrict__ rowptr,
                                                      int* __restrict__ Ccrd, T* __restrict__ Cval) {
    if (ctl->status != 0) return;
    const int b = blockIdx.x;
    int off, n;
    if (b < g.end[0]) {
        if (NUMERIC) {
            class_range(ctl, CLS_COPY, off, n);
            const bool in_order = 2 * (i64)n >= A.nrows;
            copy_rows<T>(in_order ? nullptr : perm + off, cls, in_order ? A.nrows : n, b, g.end[0], A, B, rowptr, Ccrd, Cval);
        }
    } else if (b < g.end[1]) {
        class_range(ctl, CLS_ISM_REG8, off, n);
        reg_rows<T, 8, NUMERIC>(perm + off, n, b - g.end[0], g.end[1] - g.end[0], A, B, jmin, cnt, rowptr, Ccrd, Cval);
    } else if (b < g.end[2]) {
        class_range(ctl, CLS_ISM_REG16, off, n);
        reg_rows<T, 16, NUMERIC>(perm + off, n, b - g.end[1], g.end[2] - g.end[1], A, B, jmin, cnt, rowptr, Ccrd, Cval);
    } else {
        class_range(ctl, CLS_ISM_REG, off, n);
        reg_rows<T, 32, NUMERIC>(perm + off, n, b - g.end[2], g.end[3] - g.end[2], A, B, jmin, cnt, rowptr, Ccrd, Cval);
    }
}

cudaError_t launch_ism_reg(const LaunchCtx& c, bool numeric, const i64* rows, const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval) {
    const int threads = 256;
    const i64 cap = (i64)c.sm_count * 16;
    const i64 copied = numeric ? rows[CLS_COPY] : 0;
    const i64 groups[4] = {2 * copied >= A.nrows && copied > 0 ? (i64)A.nrows : copied, rows[CLS_ISM_REG8] * 8, rows[CLS_ISM_REG16] * 16, rows[CLS_ISM_REG] * 32};
    RegBlocks g;
    int end = 0;
    for (int k = 0; k < 4; ++k) {
        const i64 want = (groups[k] + threads - 1) / threads;
        end += (int)(want < cap ? want : cap);
        g.end[k] = end;
    }
    if (end == 0) return cudaSuccess;
    if (!numeric) ism_reg_kernel<float, false><<<end, threads, 0, c.stream>>>(c.tab.perm, c.tab.cls, c.ctl, g, A, B, c.tab.jmin, c.tab.cnt, rowptr, nullptr, nullptr);
    else if (c.is_f64)
        ism_reg_kernel<double, true><<<end, threads, 0, c.stream>>>(c.tab.perm, c.tab.cls, c.ctl, g, A, B, c.tab.jmin, c.tab.cnt, rowptr, Ccrd, (double*)Cval);
    else
        ism_reg_kernel<float, true><<<end, threads, 0, c.stream>>>(c.tab.perm, c.tab.cls, c.ctl, g, A, B, c.tab.jmin, c.tab.cnt, rowptr, Ccrd, (float*)Cval);
    ++c.launches;
    return cudaGetLastError();
}

}  // namespace spws
