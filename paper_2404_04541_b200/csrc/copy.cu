// Rows that are copied: one A entry, a B row of at most COPY_MAX entries.
#include "common.cuh"

namespace spws {

// Rows with ONE A entry (the commonest fibre of a hyper-sparse 3-tensor): the products are the picked B
// row itself, already sorted and free of duplicates, so Insert, Sort and Merge are the identity and the
// row is copied out scaled.  Every lane first walks one row's chain of dependent loads (row id, A
// range, A entry, B range, output offset), 32 chains per warp in flight; then the warp copies the 32
// rows together, eight lanes per row and four rows per step.  When at least half of all rows are of this
// class they are found by walking all rows in order (rows null, n = all rows): row offsets, entries and
// output offsets are then read, and the output written, as contiguous streams.
// 2e6 fibres of which 1.85e6 are copied (8 entries each, f64): 132 us with the other rows' classes in four launches, 117 us in one
// with the copied rows in order; 86 us by themselves, at six blocks per SM, beside 40 us of the others on another stream.
template <typename T>
__global__ void __launch_bounds__(256, 6) copy_rows_kernel(const int* __restrict__ rows, const unsigned char* __restrict__ cls, int n, const DevCtl* __restrict__ ctl,
                                                        Csr A, Csr B, const i64* __restrict__ rowptr, int* __restrict__ Ccrd, T* __restrict__ Cval) {
    if (ctl->status != 0) return;
    const int lane = threadIdx.x & 31;
    const T* __restrict__ Aval = (const T*)A.val;
    const T* __restrict__ Bval = (const T*)B.val;
    const i64 stride = (i64)gridDim.x * blockDim.x;
    for (i64 r0 = ((i64)blockIdx.x * blockDim.x + threadIdx.x) - lane; r0 < n; r0 += stride) {
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
#pragma unroll 1
        for (int s = 0; s < 8; ++s) {
            const int src = 4 * s + (lane >> 3);
            const i64 q = __shfl_sync(0xffffffffu, qs, src), o = __shfl_sync(0xffffffffu, out, src);
            const int l = __shfl_sync(0xffffffffu, len, src);
            const T av = __shfl_sync(0xffffffffu, a, src);
            for (int e = lane & 7; e < l; e += 16) {        // two elements a step, both loaded before either is stored
                const bool two = e + 8 < l;
                int c1 = 0;
                T v1 = 0;
                const int c0 = __ldg(B.crd + q + e);
                const T v0 = __ldg(Bval + q + e);
                if (two) { c1 = __ldg(B.crd + q + e + 8); v1 = __ldg(Bval + q + e + 8); }
                Ccrd[o + e] = c0;
                Cval[o + e] = mul_rn(av, v0);
                if (two) { Ccrd[o + e + 8] = c1; Cval[o + e + 8] = mul_rn(av, v1); }
            }
        }
    }
}

cudaError_t launch_copy_rows(const LaunchCtx& c, const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval) {
    const i64 copied = c.class_rows[CLS_COPY];
    const bool in_order = 2 * copied >= A.nrows;
    i64 off = 0;
    for (int k = 0; k < CLS_COPY; ++k) off += c.class_rows[k];
    const int* const rows = in_order ? nullptr : c.tab.perm + off;
    const int n = in_order ? A.nrows : (int)copied;
    const i64 want = ((i64)n + 255) / 256, cap = (i64)c.sm_count * 16;
    const int grid = (int)(want < cap ? want : cap);
    if (c.is_f64) copy_rows_kernel<double><<<grid, 256, 0, c.stream>>>(rows, c.tab.cls, n, c.ctl, A, B, rowptr, Ccrd, (double*)Cval);
    else copy_rows_kernel<float><<<grid, 256, 0, c.stream>>>(rows, c.tab.cls, n, c.ctl, A, B, rowptr, Ccrd, (float*)Cval);
    ++c.launches;
    return cudaGetLastError();
}

}  // namespace spws
