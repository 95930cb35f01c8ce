// Dense workspace: an occupancy bitmap along the last index plus a value array (Gustavson's
// workspace, Table 2: the flag marks positions that already hold a component, so a product
// deduplicates on insertion; position = coordinate, so the workspace is bucket-sorted; the
// flagged positions are copied out in order = boolean indexing).
//
// The bitmap covers the row's exact column span [jmin, jmax] and lives in shared memory.  The
// value array is NOT indexed by column but by the RANK of the column among the row's set bits
// (rank = prefix popcount), so it holds only as many entries as the row has outputs and is
// already in output order:
//   symbolic : gather the column indices of the row's products, set bits; cnt = popcount; the
//              bitmap is saved to the arena in scratch so the numeric pass need not rebuild it.
//   numeric  : reload the bitmap, prefix-sum its words, then acc[rank(j)] += a*b for every
//              product; acc is copied straight to the row's value segment and the set bits give
//              the column indices.
// Two granularities:
//   warp per row : bitmap <= 1024 words, <= 256 outputs (<= 1024 under `auto`, in a launch of their own, so
//              that the larger accumulators do not cost the others their occupancy).  A warp walks the A entries one at a
//              time with its lanes across the B row, so no two lanes ever hit the same slot and
//              the accumulator needs no atomics; sums are in loop order.
//   CTA units    : any span up to 2^19 columns.  A unit is a row, or an equal share of the A
//              entries of a row with very many products, so hub rows spread over many CTAs.
//              The first `unit_outputs` outputs of the row accumulate in shared memory
//              (atomics combine the CTA's warps), the rest in the row's value segment.  The
//              coordinates of these rows are written by a kernel of their own, which also clears
//              the value segments that several units add into.
#include <algorithm>
#include "common.cuh"

namespace spws {

constexpr int DW_THREADS = 256;            // warp-per-row kernels: 8 warps per CTA
constexpr int DW_WARPS = DW_THREADS / 32;
constexpr int DC_THREADS = 256;            // symbolic CTA kernel
constexpr int DC_WARPS = DC_THREADS / 32;
constexpr int DN_THREADS = 512;            // numeric CTA kernel: at most, and where four blocks of half of them fit an SM
constexpr int DN_THREADS_4 = 256;

// A warp-route row whose bitmap is mostly empty words saves only the non-empty ones; bm_off then
// carries a flag and the number of saved words above the slot offset.
constexpr i64 BM_COMPACT = 1ll << 62;
constexpr int BM_NZW_SHIFT = 44;
constexpr i64 BM_OFF_MASK = (1ll << BM_NZW_SHIFT) - 1;

// A dense row's slot in the arena: nw bitmap words, then for every chunk of 32 words the rank of
// the chunk's first bit (an exclusive prefix of the chunk popcounts).
__device__ __forceinline__ int chunks_of(int nw) { return (nw + 31) >> 5; }

// ---------------------------------------------------------------------------------------
// symbolic, warp per row
// ---------------------------------------------------------------------------------------
// Bound by instruction issue.  SCAN (spans of up to DW_SCAN_WORDS words): products only set their bit, and the words
// are counted afterwards, 32 per step; without it the lane that sets a bit first counts the output and
// keeps a summary of the non-empty words, so that nothing walks a wide span.  Fibres of 110 products on 94 words:
// 60 us without, 49 us with the scan; 729 products on 521 words: 408 us without, 457 us with it.
constexpr int DW_SCAN_WORDS = 256;

// Place of bitmap word w in shared memory.  The planes of a grid lie some multiple of 32 words apart when its sides are powers
// of two, its lines one or two words: bits 5 .. 8 of w move the words (and the two-byte ranks) of different planes to different
// banks.  For spans beyond DW_SCAN_WORDS only, where such planes fit and the two instructions pay: 64^3 stencil, f64, symbolic 410 ->
// 378 us, numeric 632 -> 611 us.
template <bool SPREAD>
__device__ __forceinline__ unsigned bank_spread(unsigned w) { return SPREAD ? w ^ ((w >> 4) & 30u) : w; }

template <bool SCAN>
__global__ void __launch_bounds__(DW_THREADS) dense_sym_warp_kernel(DevCtl* __restrict__ ctl, int warp_outputs, Csr A, Csr B, RowTables tab) {
    __shared__ unsigned s_bm[DW_WARPS][SCAN ? DW_SCAN_WORDS : DENSE_WARP_BM_WORDS];
    // bit w of the summary = bitmap word w is non-empty, so the copy-out walks only those words
    __shared__ unsigned s_sum[DW_WARPS][DENSE_WARP_BM_WORDS / 32];
    // descriptors of 32 A entries: (start of the B row << 16) | its length (a warp row has <= 4096 products)
    __shared__ __align__(16) u64 s_desc[DW_WARPS][32];
    if (ctl->status != 0) return;
    int off, n;
    class_range(ctl, CLS_DENSE_WARP, off, n);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned* bm = s_bm[warp];
    unsigned* sum = s_sum[warp];
    u64* desc = s_desc[warp];
    for (int w = lane; w < (SCAN ? DW_SCAN_WORDS : DENSE_WARP_BM_WORDS); w += 32) bm[w] = 0;     // every row leaves its bitmap clear
    sum[lane] = 0;
    __syncwarp();
    for (;;) {
        int r = 0;
        if (lane == 0) r = atomicAdd(&ctl->work_counter[CLS_DENSE_WARP], 1);
        r = __shfl_sync(0xffffffffu, r, 0);
        if (r >= n) break;
        const int row = tab.perm[off + r];
        const int base = tab.jmin[row];
        const int nw = min((tab.jmax[row] - base) / 32 + 1, SCAN ? DW_SCAN_WORDS : DENSE_WARP_BM_WORDS);
        const unsigned span = (unsigned)nw * 32u;
        const i64 ps = A.pos[row], pe = A.pos[row + 1];
        const int lg = pick_group_log(tab.ub[row], pe - ps), gs = 1 << lg;
        // the lane that sets a bit first counts the output; the lane that touches a word first
        // counts the word and flags it in the summary
        int cnt = 0, nzw = 0;
        auto mark = [&](unsigned rel) {
            if (rel < span) {
                const unsigned w = rel >> 5, bit = 1u << (rel & 31);
                if (SCAN) {
                    atomicOr(&bm[w], bit);
                    return;
                }
                const unsigned old = atomicOr(&bm[bank_spread<!SCAN>(w)], bit);
                if (!(old & bit)) {
                    ++cnt;
                    if (old == 0u) { ++nzw; atomicOr(&sum[w >> 5], 1u << (w & 31)); }
                }
            }
        };
        if (gs == 32) {
            // descriptors of 32 A entries at a time (one per lane, passed through shared memory), then
            // the first 32 elements of four B rows are loaded before any is consumed, to keep loads
            // in flight
            for (i64 p0 = ps; p0 < pe; p0 += 32) {
                u64 mine = 0;
                if (p0 + lane < pe) {
                    const int k = __ldg(A.crd + p0 + lane);
                    if ((unsigned)k < (unsigned)B.nrows) {
                        const i64 qs = __ldg(B.pos + k);
                        mine = ((u64)qs << 16) | (u64)(__ldg(B.pos + k + 1) - qs);
                    }
                }
                __syncwarp();
                desc[lane] = mine;
                __syncwarp();
                const int nE = (int)min((i64)32, pe - p0);
                for (int e = 0; e < nE; e += 4) {
                    const ulonglong2 d01 = *reinterpret_cast<const ulonglong2*>(desc + e);
                    const ulonglong2 d23 = *reinterpret_cast<const ulonglong2*>(desc + e + 2);
                    const u64 d[4] = {d01.x, d01.y, d23.x, d23.y};
                    i64 qs[4];
                    int len[4];
                    unsigned rel[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        qs[x] = (i64)(d[x] >> 16);
                        len[x] = (int)(d[x] & 0xffffu);                  // 0 past the last entry
                        rel[x] = (lane < len[x]) ? (unsigned)(__ldg(B.crd + qs[x] + lane) - base) : 0xffffffffu;
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        mark(rel[x]);
                        for (int t = lane + 32; t < len[x]; t += 32) mark((unsigned)(__ldg(B.crd + qs[x] + t) - base));
                    }
                }
            }
        } else {
            const int g = lane >> lg, gl = lane & (gs - 1), ng = 32 >> lg;
            for (i64 p = ps + g; p < pe; p += ng) {
                const int k = __ldg(A.crd + p);
                if ((unsigned)k >= (unsigned)B.nrows) continue;
                const i64 qs = __ldg(B.pos + k);
                const int len = (int)(__ldg(B.pos + k + 1) - qs);
                const int* __restrict__ ck = B.crd + qs;
                for (int t = gl; t < len; t += gs) mark((unsigned)(__ldg(ck + t) - base));
            }
        }
        __syncwarp();
        if (SCAN) {
            for (int w0 = 0; w0 < nw; w0 += 32) {
                const unsigned word = bm[w0 + lane];                    // (clear past the span)
                cnt += __popc(word);
                const unsigned m = __ballot_sync(0xffffffffu, word != 0u);
                if (lane == 0) sum[w0 >> 5] = m;
                nzw += __popc(m);
            }
            cnt = __reduce_add_sync(0xffffffffu, cnt);
        } else {
            cnt = __reduce_add_sync(0xffffffffu, cnt);
            nzw = __reduce_add_sync(0xffffffffu, nzw);
        }
        __syncwarp();
        const i64 slot = tab.bm_off[row];
        unsigned* out = tab.bm_arena + slot;
        if (cnt <= warp_outputs && 2 * nzw <= nw + chunks_of(nw)) {
            // compact form for the warp numeric kernel: only the non-empty words, as (bits, word
            // index) in column order; lane l owns the words its summary word flags
            uint2* out2 = reinterpret_cast<uint2*>(out);
            unsigned s = sum[lane];
            sum[lane] = 0;
            const int c = __popc(s);
            int at = warp_incl_scan(c) - c;
            while (s) {
                const int w = (lane << 5) + __ffs(s) - 1;
                s &= s - 1;
                out2[at++] = make_uint2(bm[bank_spread<!SCAN>(w)], (unsigned)w);
                bm[bank_spread<!SCAN>(w)] = 0;
            }
            if (lane == 0) tab.bm_off[row] = slot | ((i64)nzw << BM_NZW_SHIFT) | BM_COMPACT;
        } else {
            // full form: every word, then the rank at every 32-word chunk start
            sum[lane] = 0;
            int carry = 0;
            for (int w0 = 0; w0 < nw; w0 += 32) {
                const int w = w0 + lane;
                const unsigned word = (w < nw) ? bm[bank_spread<!SCAN>(w)] : 0u;
                if (w < nw) { out[w] = word; bm[bank_spread<!SCAN>(w)] = 0; }
                int c = __popc(word);
                for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
                if (lane == 0) out[nw + (w0 >> 5)] = (unsigned)carry;
                carry += c;
            }
        }
        if (lane == 0) tab.cnt[row] = cnt;
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------------------
// symbolic, CTA units.  A unit is a row, or an equal share of the A entries of a row with a large part of all products,
// whose blocks unite their bitmaps in the arena; the last of them counts.
// Bound by latency at few vertices, by the shared-memory atomics and instruction issue at many.  Warps that pulled batches of A
// entries of a row walked a chain of four loads per batch and had one B row's loads in flight; the entries of a round are
// now looked up by all threads at once and the warps pull tiles of the stream of their elements, each with 128 loads in flight
// whatever the length of the B rows.  Power law on 16381 / 60000 / 2^18 vertices: 201 / 622 / 2681 us by batches, one block a
// row, 80 / 418 / 2600 us now.
// ---------------------------------------------------------------------------------------
constexpr int DS_ENTRIES = DC_THREADS;      // A entries whose descriptors are staged per round
// elements a warp takes per fetch: a 64th of the round's, so that the warps finish together (at most 1024 / 2048 / 4096: power law on
// 2^18 vertices 2648 / 2621 / 2624 us)
constexpr int DS_TILE = 256, DS_TILE_MOST = 2048;

// What a block needs to know of a unit, fetched by one thread while the block is busy with the unit before.
struct SymUnit {
    i64 e_lo, e_hi, bm;
    int row, base, nw, parts;                  // row < 0: no more units
};

__global__ void __launch_bounds__(DC_THREADS, 6) dense_sym_cta_kernel(DevCtl* __restrict__ ctl, int smem_words, int unit_cap, i64 part_products, Csr A, Csr B, RowTables tab,
                                                                   const uint2* __restrict__ bw) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned* bm = reinterpret_cast<unsigned*>(smem_raw);                 // smem_words, clear between units
    int* chunk = reinterpret_cast<int*>(bm + smem_words);                  // smem_words / 32 + 1
    // staged descriptors: twice the start of the B row, or of its word list and one; elements of the entries before
    __shared__ i64 d_q[DS_ENTRIES];
    __shared__ int d_pre[DS_ENTRIES + 1], ws[DC_WARPS];
    __shared__ SymUnit s_unit[2];
    __shared__ int s_tile, s_last;
    if (ctl->status != 0) return;
    const int n_split = ctl->sym_units[0], n = n_split + ctl->sym_units[1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto fetch_unit = [&](SymUnit& U) {                 // one thread
        const int t = atomicAdd(&ctl->work_counter[CLS_DENSE_CTA], 1);
        U.row = -1;
        if (t >= n) return;
        const int u = t < n_split ? t : unit_cap - 1 - (t - n_split);
        const int row = tab.unit_row[u], base = tab.jmin[row];
        const i64 ps = A.pos[row], entries = A.pos[row + 1] - ps;
        int part = 0, parts = 1;
        if (t < n_split) {
            part = u - tab.row_unit0[row];
            parts = sym_parts_of_row(tab.ub[row], part_products);
        }
        U.bm = tab.bm_off[row];
        U.nw = min((tab.jmax[row] - base) / 32 + 1, smem_words);
        U.e_lo = ps + entries * part / parts;
        U.e_hi = ps + entries * (part + 1) / parts;
        U.parts = parts;
        U.base = base;
        U.row = row;
    };
    if (tid == 0) fetch_unit(s_unit[0]);
    for (int w = tid; w < smem_words; w += DC_THREADS) bm[w] = 0;
    __syncthreads();
    for (int cur = 0;; cur ^= 1) {
        const SymUnit& U = s_unit[cur];
        if (U.row < 0) break;
        const int base = U.base, nw = U.nw;
        const unsigned base_w = (unsigned)base >> 5;                     // base is a multiple of 32
        const i64 e_hi = U.e_hi;
        bool next_known = false;
        // Rounds of DS_ENTRIES A entries, one per thread: a block scan turns the lengths of the B rows (or of their word
        // lists) into a running count, and warps pull tiles of that stream.
        for (i64 e0 = U.e_lo; e0 < e_hi; e0 += DS_ENTRIES) {
            const int nE = (int)min((i64)DS_ENTRIES, e_hi - e0);
            int len = 0;
            if (tid < nE) {
                const int k = __ldg(A.crd + e0 + tid);
                i64 q = 0;
                if ((unsigned)k < (unsigned)B.nrows) {
                    const i64 qs = __ldg(B.pos + k);
                    len = (int)(__ldg(B.pos + k + 1) - qs);
                    q = 2 * qs;
                    if (bw && len >= BW_MIN_LEN) {
                        const int np = (int)__ldg(&bw[qs].x);
                        if (np > 0) { len = np; q = 2 * (qs + 1) + 1; }
                    }
                }
                d_q[tid] = q;
            }
            const int incl = warp_incl_scan(len);
            if (lane == 31) ws[warp] = incl;
            __syncthreads();
            const int wt = lane < DC_WARPS ? ws[lane] : 0;
            const int wi = warp_incl_scan(wt);
            const int total = __shfl_sync(0xffffffffu, wi, 31);
            const int excl = __shfl_sync(0xffffffffu, wi - wt, warp) + incl - len;
            if (tid < nE) d_pre[tid] = excl;
            if (tid == 0) { d_pre[nE] = total; s_tile = 0; }
            __syncthreads();
            if (!next_known && tid == DC_THREADS - 1) fetch_unit(s_unit[cur ^ 1]);
            next_known = true;
            __syncwarp();
            const bool long_rows = total >= 64 * nE;
            const int tile = min(max((total >> 6) & ~127, DS_TILE), DS_TILE_MOST);
            for (;;) {
                int t0 = 0;
                if (lane == 0) t0 = atomicAdd(&s_tile, tile);
                t0 = __shfl_sync(0xffffffffu, t0, 0);
                if (t0 >= total) break;
                const int t1 = min(total, t0 + tile);
                // the last entry whose running count is <= t0: among 32 spread entries, then among those in between
                constexpr int STRIDE = DS_ENTRIES / 32;
                const int i1 = lane * STRIDE;
                const int lo = (__popc(__ballot_sync(0xffffffffu, i1 < nE && d_pre[i1] <= t0)) - 1) * STRIDE;
                const int i2 = lo + lane;
                int e = lo + __popc(__ballot_sync(0xffffffffu, lane < STRIDE && i2 < nE && d_pre[i2] <= t0)) - 1;
                if (long_rows) {
                    // the tile's part of one B row after the other, 128 elements a step, four per lane, all loads first
                    while (t0 < t1) {
                        int next = d_pre[e + 1];
                        while (next <= t0) next = d_pre[++e + 1];
                        int m = min(t1, next) - t0;
                        const i64 d = d_q[e];
                        const i64 q = (d >> 1) + (t0 - d_pre[e]) + lane;
                        t0 += m;
                        if (d & 1) {
                            auto set = [&](uint2 v) {
                                const unsigned w = v.x - base_w;
                                if (w < (unsigned)nw) atomicOr(&bm[w], v.y);
                            };
                            const uint2* __restrict__ pk = bw + q;
                            for (; m >= 128; m -= 128, pk += 128) {
                                const uint2 v0 = __ldg(pk), v1 = __ldg(pk + 32), v2 = __ldg(pk + 64), v3 = __ldg(pk + 96);
                                set(v0); set(v1); set(v2); set(v3);
                            }
                            if (m > 0) {
                                uint2 v[4];
#pragma unroll
                                for (int x = 0; x < 4; ++x) v[x] = lane + 32 * x < m ? __ldg(pk + 32 * x) : make_uint2(base_w - 1u, 0u);
#pragma unroll
                                for (int x = 0; x < 4; ++x) set(v[x]);
                            }
                        } else {
                            auto set = [&](int c) {
                                const unsigned rel = (unsigned)(c - base);
                                if (rel < (unsigned)nw * 32u) atomicOr(&bm[rel >> 5], 1u << (rel & 31));
                            };
                            const int* __restrict__ ck = B.crd + q;
                            for (; m >= 128; m -= 128, ck += 128) {
                                const int c0 = __ldg(ck), c1 = __ldg(ck + 32), c2 = __ldg(ck + 64), c3 = __ldg(ck + 96);
                                set(c0); set(c1); set(c2); set(c3);
                            }
                            if (m > 0) {
                                int c[4];
#pragma unroll
                                for (int x = 0; x < 4; ++x) c[x] = lane + 32 * x < m ? __ldg(ck + 32 * x) : base - 1;
#pragma unroll
                                for (int x = 0; x < 4; ++x) set(c[x]);
                            }
                        }
                    }
                } else {
                    // short B rows: a step = 128 consecutive elements of the stream, four per lane; every lane advances its
                    // own entry index across row boundaries
                    for (; t0 < t1; t0 += 128) {
                        unsigned w[4], bits[4];
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int t = t0 + lane + 32 * x;
                            w[x] = 0xffffffffu;
                            bits[x] = 0u;
                            if (t < t1) {
                                while (d_pre[e + 1] <= t) ++e;
                                const i64 d = d_q[e];
                                const i64 q = (d >> 1) + (t - d_pre[e]);
                                if (d & 1) {
                                    const uint2 v = __ldg(bw + q);
                                    w[x] = v.x - base_w;
                                    bits[x] = v.y;
                                } else {
                                    const unsigned rel = (unsigned)(__ldg(B.crd + q) - base);
                                    w[x] = rel >> 5;
                                    bits[x] = 1u << (rel & 31);
                                }
                            }
                        }
#pragma unroll
                        for (int x = 0; x < 4; ++x)
                            if (w[x] < (unsigned)nw) atomicOr(&bm[w[x]], bits[x]);
                    }
                }
            }
            __syncthreads();
        }
        if (!next_known) {                              // a share without entries
            __syncthreads();
            if (tid == 0) fetch_unit(s_unit[cur ^ 1]);
            __syncthreads();
        }
        // save the bitmap, then the rank at every chunk start
        unsigned* out = tab.bm_arena + U.bm;
        const int nch = chunks_of(nw), row = U.row, parts = U.parts;
        uint4* const bm4 = reinterpret_cast<uint4*>(bm);
        uint4* const out4 = reinterpret_cast<uint4*>(out);
        if (parts > 1) {
            for (int q = tid; 4 * q < nw; q += DC_THREADS) {
                const uint4 v = bm4[q];
                if (v.x) atomicOr(out + 4 * q, v.x);
                if (v.y) atomicOr(out + 4 * q + 1, v.y);
                if (v.z) atomicOr(out + 4 * q + 2, v.z);
                if (v.w) atomicOr(out + 4 * q + 3, v.w);
                bm4[q] = make_uint4(0u, 0u, 0u, 0u);
            }
            __threadfence();
            __syncthreads();
            if (tid == 0) s_last = atomicAdd(&tab.cnt[row], 1) == parts - 1;       // (the bounds kernel left a zero)
            __syncthreads();
            if (!s_last) continue;
            __threadfence();
        }
        // four words a lane, eight lanes a chunk (words past the span are clear; a slot holds a multiple of four words); a word a
        // lane: power law on 2^18 vertices 2820 us, 2740 like this
        for (int q0 = warp * 32; q0 < nch * 8; q0 += DC_WARPS * 32) {
            const int q = q0 + lane;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (4 * q < nw) {
                if (parts > 1) {
                    v = __ldcg(out4 + q);
                } else {
                    v = bm4[q];
                    out4[q] = v;
                    bm4[q] = make_uint4(0u, 0u, 0u, 0u);
                }
            }
            int pc = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
            pc += __shfl_xor_sync(0xffffffffu, pc, 1);
            pc += __shfl_xor_sync(0xffffffffu, pc, 2);
            pc += __shfl_xor_sync(0xffffffffu, pc, 4);
            if ((lane & 7) == 0 && (q >> 3) < nch) chunk[q >> 3] = pc;
        }
        __syncthreads();
        if (warp == 0) {                                // the others go on with the next unit
            int carry = 0;
            for (int c0 = 0; c0 < nch; c0 += 32) {
                const int v = c0 + lane < nch ? chunk[c0 + lane] : 0;
                const int incl = warp_incl_scan(v);
                if (c0 + lane < nch) out[nw + c0 + lane] = (unsigned)(carry + incl - v);
                carry += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) tab.cnt[row] = carry;
        }
    }
}

// ---------------------------------------------------------------------------------------
// numeric, warp per row
// ---------------------------------------------------------------------------------------
// CEIL = true: the same walk over rows, entries and B rows with the workspace stripped (Sec. 7.2,
// iteration-only lower bound); the gathered indices and products go into two checksums.
template <typename T, bool CEIL, bool SPREAD>
__global__ void __launch_bounds__(DW_THREADS) dense_num_warp_kernel(DevCtl* __restrict__ ctl, const int* __restrict__ rows, int step, int n, int slot_,
                                                                    int bmw, int accw, Csr A, Csr B, RowTables tab,
                                                                    const i64* __restrict__ rowptr, int* __restrict__ Ccrd,
                                                                    T* __restrict__ Cval, u64* __restrict__ chk_idx,
                                                                    double* __restrict__ chk_val) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (ctl->status != 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    // per warp: bmw bitmap words, the number of outputs before each (16 bits: 629 us against 643 with both in
    // eight bytes, which keep fewer warps on an SM), and accw values (sized from the widest / largest row of this launch)
    unsigned* bits = reinterpret_cast<unsigned*>(smem_raw) + warp * bmw;
    unsigned short* rank = reinterpret_cast<unsigned short*>(reinterpret_cast<unsigned*>(smem_raw) + warps * bmw) + warp * bmw;
    T* acc = reinterpret_cast<T*>(smem_raw + 6 * warps * bmw) + warp * accw;
    // descriptors of 32 A entries: (start of the B row << 16) | its length, and the A value; one broadcast load
    // per entry where shuffles took five slots of the same pipe (bmw and accw are multiples of 32: aligned)
    struct __align__(16) Desc { u64 row; T a; };
    Desc* desc = reinterpret_cast<Desc*>(reinterpret_cast<T*>(smem_raw + 6 * warps * bmw) + warps * accw) + warp * 32;
    const T* __restrict__ Aval = (const T*)A.val;
    const T* __restrict__ Bval = (const T*)B.val;
    if (!CEIL)
        for (int w = lane; w < bmw; w += 32) bits[w] = 0u;              // every row leaves its bitmap clear
    __syncwarp();
    u64 my_idx = 0;
    double my_val = 0.0;
    for (;;) {
        int r = 0;
        if (lane == 0) r = atomicAdd(&ctl->work_counter[slot_], 1);
        r = __shfl_sync(0xffffffffu, r, 0);
        if (r >= n) break;
        const int row = __ldg(rows + (i64)r * step);
        const int base = tab.jmin[row];
        const int nw = min((tab.jmax[row] - base) / 32 + 1, bmw);
        const unsigned span = (unsigned)nw * 32u;
        const i64 ps = A.pos[row], pe = A.pos[row + 1];
        const i64 out0 = rowptr[row];
        const int cnt = min((int)(rowptr[row + 1] - out0), accw);
        const i64 slot = tab.bm_off[row];
        const bool compact = (slot & BM_COMPACT) != 0;
        const int nzw = (int)((slot & ~BM_COMPACT) >> BM_NZW_SHIFT);
        const unsigned* src = tab.bm_arena + (slot & BM_OFF_MASK);
        const uint2* src2 = reinterpret_cast<const uint2*>(src);
        if (CEIL) {
            // no workspace to set up
        } else if (compact) {
            // the saved non-empty words in column order: ranks by a running prefix of their bit counts
            int carry = 0;
            for (int i0 = 0; i0 < nzw; i0 += 32) {
                const int i = i0 + lane;
                const uint2 e = (i < nzw) ? src2[i] : make_uint2(0u, 0u);
                const int c = __popc(e.x);
                const int incl = warp_incl_scan(c);
                if (i < nzw && e.y < (unsigned)nw) { const unsigned at = bank_spread<SPREAD>(e.y); bits[at] = e.x; rank[at] = (unsigned short)(carry + incl - c); }
                carry += __shfl_sync(0xffffffffu, incl, 31);
            }
        } else {
            // the whole bitmap; rank of each word's first bit = chunk rank + prefix inside the chunk
            for (int w0 = 0; w0 < nw; w0 += 32) {
                const int w = w0 + lane;
                const unsigned word = (w < nw) ? src[w] : 0u;
                const int c = __popc(word);
                const int incl = warp_incl_scan(c);
                if (w < nw) { const unsigned at = bank_spread<SPREAD>(w); bits[at] = word; rank[at] = (unsigned short)(src[nw + (w0 >> 5)] + (unsigned)(incl - c)); }
            }
        }
        if (!CEIL)
            for (int x = lane; x < cnt; x += 32) acc[x] = 0;
        __syncwarp();
        // one product into the workspace: rank of its column, then add (plain when no other lane can
        // hold the same column, atomic otherwise); stripped to the checksums when CEIL
        auto put = [&](unsigned rel, T prod, bool shared_slot) {
            if (CEIL) {
                if (rel != 0xffffffffu) { my_idx += (u64)(rel + (unsigned)base); my_val += (double)prod; }
            } else if (rel < span) {
                const unsigned w = bank_spread<SPREAD>(rel >> 5);
                const int at_ = (int)rank[w] + __popc(bits[w] & ((1u << (rel & 31)) - 1u));
                if (at_ < accw) {
                    if (shared_slot) atomicAdd(&acc[at_], prod);
                    else acc[at_] = add_rn(acc[at_], prod);
                }
            }
        };
        const int lg = pick_group_log(tab.ub[row], pe - ps), gs = 1 << lg;
        if (gs == 32) {
            // one A entry at a time, lanes across its B row: distinct columns, no atomics,
            // every output summed in loop order
            // (the entries' descriptors are fetched 32 at a time, one per lane, and the first 32
            // elements of two B rows are loaded before either is consumed, to keep loads in flight)
            for (i64 p0 = ps; p0 < pe; p0 += 32) {
                Desc mine;
                mine.row = 0;
                mine.a = 0;
                if (p0 + lane < pe) {
                    const int k = __ldg(A.crd + p0 + lane);
                    if ((unsigned)k < (unsigned)B.nrows) {
                        const i64 qs = __ldg(B.pos + k);
                        mine.row = ((u64)qs << 16) | (u64)(__ldg(B.pos + k + 1) - qs);
                    }
                    mine.a = __ldg(Aval + p0 + lane);
                }
                desc[lane] = mine;
                __syncwarp();
                const int nE = (int)min((i64)32, pe - p0);
                for (int e = 0; e < nE; e += 2) {
                    const Desc d0 = desc[e], d1 = desc[e + 1];           // (length 0 past the last entry)
                    const i64 qs0 = (i64)(d0.row >> 16), qs1 = (i64)(d1.row >> 16);
                    const int len0 = (int)(d0.row & 0xffffu), len1 = (int)(d1.row & 0xffffu);
                    const T a0 = d0.a, a1 = d1.a;
                    unsigned rel0 = 0xffffffffu, rel1 = 0xffffffffu;
                    T v0 = 0, v1 = 0;
                    if (lane < len0) { rel0 = (unsigned)(__ldg(B.crd + qs0 + lane) - base); v0 = __ldg(Bval + qs0 + lane); }
                    if (lane < len1) { rel1 = (unsigned)(__ldg(B.crd + qs1 + lane) - base); v1 = __ldg(Bval + qs1 + lane); }
                    // entry e
                    put(rel0, mul_rn(a0, v0), false);
                    for (int t = lane + 32; t < len0; t += 32)
                        put((unsigned)(__ldg(B.crd + qs0 + t) - base), mul_rn(a0, __ldg(Bval + qs0 + t)), false);
                    __syncwarp();
                    // entry e + 1
                    put(rel1, mul_rn(a1, v1), false);
                    for (int t = lane + 32; t < len1; t += 32)
                        put((unsigned)(__ldg(B.crd + qs1 + t) - base), mul_rn(a1, __ldg(Bval + qs1 + t)), false);
                    __syncwarp();
                }
            }
        } else {
            // short B rows: several A entries in flight, so slots can collide -> atomics
            const int g = lane >> lg, gl = lane & (gs - 1), ng = 32 >> lg;
            for (i64 p = ps + g; p < pe; p += ng) {
                const int k = __ldg(A.crd + p);
                if ((unsigned)k >= (unsigned)B.nrows) continue;
                const i64 qs = __ldg(B.pos + k);
                const int len = (int)(__ldg(B.pos + k + 1) - qs);
                const T a = __ldg(Aval + p);
                for (int t = gl; t < len; t += gs)
                    put((unsigned)(__ldg(B.crd + qs + t) - base), mul_rn(a, __ldg(Bval + qs + t)), true);
            }
            __syncwarp();
        }
        if (CEIL) continue;
        // copy out: values are already in output order; set bits give the coordinates; the table
        // words the row used are cleared on the way
        for (int x = lane; x < cnt; x += 32) Cval[out0 + x] = acc[x];
        if (compact) {
            for (int i = lane; i < nzw; i += 32) {
                const uint2 e = src2[i];
                if (e.y >= (unsigned)nw) continue;
                unsigned word = e.x;
                const unsigned at = bank_spread<SPREAD>(e.y);
                i64 o = out0 + rank[at];
                bits[at] = 0u;
                while (word) {
                    const int b = __ffs(word) - 1;
                    word &= word - 1;
                    Ccrd[o++] = base + (int)(e.y << 5) + b;
                }
            }
        } else {
            for (int w = lane; w < nw; w += 32) {
                const unsigned at = bank_spread<SPREAD>(w);
                unsigned word = bits[at];
                i64 o = out0 + rank[at];
                bits[at] = 0u;
                while (word) {
                    const int b = __ffs(word) - 1;
                    word &= word - 1;
                    Ccrd[o++] = base + (w << 5) + b;
                }
            }
        }
        __syncwarp();
    }
    if (CEIL) {
        for (int d = 16; d > 0; d >>= 1) {
            my_idx += __shfl_xor_sync(0xffffffffu, my_idx, d);
            my_val += __shfl_xor_sync(0xffffffffu, my_val, d);
        }
        if (lane == 0) { atomicAdd(chk_idx, my_idx); atomicAdd(chk_val, my_val); }
    }
}

// ---------------------------------------------------------------------------------------
// numeric, CTA units.  A unit is a row, or an equal share of the A entries of a row with very
// many products.  Every unit streams its B rows once, whole.  Outputs with rank < CAP accumulate
// in shared memory; outputs beyond accumulate straight into the row's value segment in global
// memory (zeroed beforehand), which keeps any row to a single pass whatever its output count.
// Bound by latency: the ranks and the compare-and-swap loops of the shared-memory additions form chains, at 32 warps
// per SM (64 registers; two blocks of 512 threads, or four of 256, see the launch).  By blocks of 512, power law on 2^18 / 16381 vertices, f64 / f32: with nine barriers per unit,
// metadata fetched between them and loads one step ahead 14050 / 309 us; without the prefetch (its register copies
// cost more than the other warps' work hides) and with two steps to find a tile's entry 13590 / 287 us; with three barriers and the next unit
// fetched meanwhile 12770 / 252 us.  Every output in shared memory, by segments of a row's ranks: 28000 / 339 us.
// ---------------------------------------------------------------------------------------
template <int THREADS> __host__ __device__ constexpr int dn_entries() { return THREADS * 3 / 2; }      // A entries whose descriptors are staged per round
constexpr int DN_TILE = 256;         // products a warp takes per fetch
constexpr int DN_CAP_LEAST = 1024;   // outputs in shared memory at least, for the sake of more blocks

// What a block needs to know of a unit, fetched by one thread while the block is busy with the unit before.
struct CtaUnit {
    i64 e_lo, e_hi, out0, bm;           // A entries, first output, bitmap
    int base, nw, cnt, nun, mean, valid;    // mean: products per entry
};

// CEIL = true is the same traversal with the workspace stripped (the iteration-only lower bound of
// Sec. 7.2): units, descriptor rounds, product tiles and gathers as below, but no bitmap, no rank
// and no accumulation; every gathered column index and product is folded into two checksums.
template <typename T, bool CEIL, int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) dense_num_cta_kernel(DevCtl* __restrict__ ctl, int smem_words, int CAP, i64 unit_products,
                                                                   Csr A, Csr B, RowTables tab, const i64* __restrict__ rowptr,
                                                                   int* __restrict__ Ccrd, T* __restrict__ Cval,
                                                                   u64* __restrict__ chk_idx, double* __restrict__ chk_val) {
    constexpr int WARPS = THREADS / 32, ENTRIES = dn_entries<THREADS>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* acc = reinterpret_cast<T*>(smem_raw);                                        // CAP
    // per bitmap word: .x = the word, .y = outputs of the row before it, less one (one load gives a rank)
    uint2* bmr = reinterpret_cast<uint2*>(acc + CAP);                                // smem_words
    // staged descriptors of up to ENTRIES A entries: B-row start, A value, running product count
    i64* d_qs = reinterpret_cast<i64*>(smem_raw + ((sizeof(T) * (size_t)CAP + 8 * (size_t)smem_words + 15) & ~(size_t)15));
    T* d_a = reinterpret_cast<T*>(d_qs + ENTRIES);
    int* d_pre = reinterpret_cast<int*>(d_a + ENTRIES);                           // ENTRIES + 1
    __shared__ CtaUnit s_unit[2];
    __shared__ int s_tile, ws[WARPS];
    if (ctl->status != 0) return;
    const int n_units = ctl->n_units;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const T* __restrict__ Aval = (const T*)A.val;
    const T* __restrict__ Bval = (const T*)B.val;
    if (!CEIL)
        for (int x = tid; x < CAP; x += THREADS) acc[x] = 0;
    u64 my_idx = 0;
    double my_val = 0.0;

    auto fetch_unit = [&](CtaUnit& U) {                 // one thread
        const int t = atomicAdd(&ctl->work_counter[(CEIL ? CEIL_SLOT : NUM_SLOT) + CLS_DENSE_CTA], 1);
        U.valid = t < n_units;
        if (t >= n_units) return;
        const int u = unit_at(t, n_units);
        const int row = tab.unit_row[u];
        const int uidx = u - tab.row_unit0[row];
        const i64 ub = tab.ub[row], ps = A.pos[row], n = A.pos[row + 1] - ps, out0 = rowptr[row];
        const int nun = dense_units_of_row(ub, unit_products), base = tab.jmin[row];
        U.nw = min((tab.jmax[row] - base) / 32 + 1, smem_words);
        U.bm = tab.bm_off[row];
        U.cnt = (int)(rowptr[row + 1] - out0);
        U.e_lo = ps + n * uidx / nun;
        U.e_hi = ps + n * (uidx + 1) / nun;
        U.mean = (int)min(ub / max(n, (i64)1), (i64)0x7fffffff);
        U.out0 = out0;
        U.base = base;
        U.nun = nun;
    };
    if (tid == 0) fetch_unit(s_unit[0]);
    __syncthreads();

    // Three barriers per round of descriptors and none besides: whatever a unit writes before its first tile is
    // next read behind two of them, and the unit before has left its tiles behind one.
    for (int cur = 0;; cur ^= 1) {
        const CtaUnit& U = s_unit[cur];
        if (!U.valid) break;
        if (!CEIL) {
            if (U.nun == 1)                             // outputs beyond the shared-memory part start at zero
                for (int x = CAP + tid; x < U.cnt; x += THREADS) Cval[U.out0 + x] = 0;
            // the row's bitmap with the rank of every word's first bit (the symbolic pass saved the
            // rank at every chunk start).  A warp takes two groups of 128 words at a time, all loads first: one scan
            // per group.  Power law on 2^18 / 16381 vertices: a scan per chunk of 32 words 12850 / 249 us; four groups at a
            // time, which spill registers that the accumulation needs, 12650 / 238; two 12380 / 230 (spans of 16384 words and
            // few outputs pay for the more steps: 10^4 rows of 8192 products 1041, 886, 932 us).
            const unsigned* src = tab.bm_arena + U.bm;
            const int nw = U.nw, nch = chunks_of(nw), ng = (nch + 3) >> 2;
            const uint4* src4 = reinterpret_cast<const uint4*>(src);         // slots are 16-byte aligned
            for (int g0 = warp; g0 < ng; g0 += WARPS * 2) {
                uint4 word[2];
                unsigned rank_g[2];
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const int g = g0 + x * WARPS, w0 = (g << 7) + (lane << 2);
                    word[x] = make_uint4(0u, 0u, 0u, 0u);
                    if (w0 < nw) {
                        word[x] = src4[(g << 5) + lane];
                        if (w0 + 1 >= nw) word[x].y = 0u;
                        if (w0 + 2 >= nw) word[x].z = 0u;
                        if (w0 + 3 >= nw) word[x].w = 0u;
                    }
                    rank_g[x] = (g < ng) ? src[nw + (g << 2)] : 0u;
                }
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const int g = g0 + x * WARPS, w0 = (g << 7) + (lane << 2);
                    const int p0 = __popc(word[x].x), p1 = p0 + __popc(word[x].y), p2 = p1 + __popc(word[x].z), p3 = p2 + __popc(word[x].w);
                    const unsigned r = rank_g[x] + (unsigned)(warp_incl_scan(p3) - p3) - 1u;
                    const uint4 lo = make_uint4(word[x].x, r, word[x].y, r + (unsigned)p0);
                    const uint4 hi = make_uint4(word[x].z, r + (unsigned)p1, word[x].w, r + (unsigned)p2);
                    // (lanes 4 .. 7 of eight store their second half first: no bank conflict)
                    if (w0 < smem_words) {
                        uint4* to = reinterpret_cast<uint4*>(bmr + w0);
                        const bool second = lane & 4;
                        to[second] = second ? hi : lo;
                        to[!second] = second ? lo : hi;
                    }
                }
            }
        }

        const int base = U.base, cnt = U.cnt;
        const unsigned span_bits = (unsigned)U.nw * 32u;
        T* const gacc = Cval + U.out0;
        auto add = [&](unsigned rel, T v) {
            if (CEIL) {
                if (rel != 0xffffffffu) { my_idx += (u64)(rel + (unsigned)base); my_val += (double)v; }
            } else if (rel < span_bits) {
                const uint2 br = bmr[rel >> 5];
                // the column's bit is set: bits up to and including it, one less in the table
                const unsigned r = br.y + (unsigned)__popc(__funnelshift_l(0u, br.x, ~rel));
                if (r < (unsigned)CAP) atomicAdd(&acc[r], v);
                else if (r < (unsigned)cnt) atomicAdd(gacc + r, v);
            }
        };

        bool next_known = false;
        // Rounds of up to ENTRIES A entries.  Step 1: every thread fetches the descriptors
        // of two entries; a block scan turns the B-row lengths into a running product count.
        // Step 2: warps pull tiles of DN_TILE consecutive products of that stream, so the
        // work is shared evenly however long the individual B rows are.
        const i64 e_hi = U.e_hi;
        for (i64 e0 = U.e_lo; e0 < e_hi; e0 += ENTRIES) {
            const int nE = (int)min((i64)ENTRIES, e_hi - e0);
            int len2[2] = {0, 0};
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const int i = 2 * tid + x;
                if (i < nE) {
                    const int k = __ldg(A.crd + e0 + i);
                    i64 qs = 0;
                    if ((unsigned)k < (unsigned)B.nrows) {
                        qs = __ldg(B.pos + k);
                        len2[x] = (int)(__ldg(B.pos + k + 1) - qs);
                    }
                    d_qs[i] = qs;
                    d_a[i] = __ldg(Aval + e0 + i);
                }
            }
            const int incl = warp_incl_scan(len2[0] + len2[1]);
            if (lane == 31) ws[warp] = incl;
            if (tid == 0) s_tile = 0;
            __syncthreads();
            const int wt = lane < WARPS ? ws[lane] : 0;
            const int wi = warp_incl_scan(wt);
            const int total = __shfl_sync(0xffffffffu, wi, 31);
            const int excl = __shfl_sync(0xffffffffu, wi - wt, warp) + incl - len2[0] - len2[1];
            if (2 * tid < nE) d_pre[2 * tid] = excl;
            if (2 * tid + 1 < nE) d_pre[2 * tid + 1] = excl + len2[0];
            if (tid == 0) d_pre[nE] = total;
            __syncthreads();
            if (!next_known && tid == THREADS - 1) fetch_unit(s_unit[cur ^ 1]);
            next_known = true;
            __syncwarp();

            int t0 = 0, t1 = 0, e = 0;              // stream position, end of the tile in hand, entry at t0
            auto next_tile = [&]() -> bool {
                int s = 0;
                if (lane == 0) s = atomicAdd(&s_tile, DN_TILE);
                t0 = __shfl_sync(0xffffffffu, s, 0);
                if (t0 >= total) return false;
                t1 = min(total, t0 + DN_TILE);
                // the last entry whose running count is <= t0: among 32 spread entries, then among those in between
                constexpr int STRIDE = ENTRIES / 32;
                static_assert(STRIDE <= 32, "two steps");
                const int i1 = lane * STRIDE;
                const int lo = (__popc(__ballot_sync(0xffffffffu, i1 < nE && d_pre[i1] <= t0)) - 1) * STRIDE;
                const int i2 = lo + lane;
                e = lo + __popc(__ballot_sync(0xffffffffu, lane < STRIDE && i2 < nE && d_pre[i2] <= t0)) - 1;
                return true;
            };
            if (U.mean >= 64) {
                // a step = up to 128 consecutive products of one B row, four per lane, all loads first
                while (t0 < t1 || next_tile()) {
                    int next = d_pre[e + 1];
                    while (next <= t0) next = d_pre[++e + 1];
                    const int n = min(min(t1, next) - t0, 128);
                    const i64 q = d_qs[e] + (t0 - d_pre[e]) + lane;
                    const int* __restrict__ ck = B.crd + q;
                    const T* __restrict__ vk = Bval + q;
                    const T a = d_a[e];
                    unsigned rel[4];
                    T b[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        rel[x] = 0xffffffffu;
                        if (lane + 32 * x < n) { rel[x] = (unsigned)(__ldg(ck + 32 * x) - base); b[x] = __ldg(vk + 32 * x); }
                    }
                    t0 += n;
#pragma unroll
                    for (int x = 0; x < 4; ++x) add(rel[x], a * b[x]);
                }
            } else {
                // short B rows: a step = 128 consecutive products of the stream, four per lane; every lane advances
                // its own entry index across row boundaries
                while (next_tile()) {
                    int my_e = e;
                    for (; t0 < t1; t0 += 128) {
                        unsigned rel[4];
                        T b[4];
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int t = t0 + lane + 32 * x;
                            rel[x] = 0xffffffffu;
                            if (t < t1) {
                                while (d_pre[my_e + 1] <= t) ++my_e;
                                const i64 q = d_qs[my_e] + (t - d_pre[my_e]);
                                rel[x] = (unsigned)(__ldg(B.crd + q) - base);
                                b[x] = d_a[my_e] * __ldg(Bval + q);
                            }
                        }
#pragma unroll
                        for (int x = 0; x < 4; ++x) add(rel[x], b[x]);
                    }
                }
            }
            __syncthreads();
        }
        if (!next_known) {                              // a share without entries
            __syncthreads();
            if (tid == 0) fetch_unit(s_unit[cur ^ 1]);
            __syncthreads();
        }

        // copy out the shared-memory part of the values (the coordinates are written by
        // dense_emit_crd_kernel)
        const int n_smem = CEIL ? 0 : min(cnt, CAP);
        if (U.nun == 1) {
            for (int x = tid; x < n_smem; x += THREADS) { gacc[x] = acc[x]; acc[x] = 0; }
        } else {
            for (int x = tid; x < n_smem; x += THREADS) {
                const T v = acc[x];
                acc[x] = 0;
                if (v != (T)0) atomicAdd(gacc + x, v);
            }
        }
    }
    if (CEIL) {
        for (int d = 16; d > 0; d >>= 1) {
            my_idx += __shfl_xor_sync(0xffffffffu, my_idx, d);
            my_val += __shfl_xor_sync(0xffffffffu, my_val, d);
        }
        if (lane == 0) { atomicAdd(chk_idx, my_idx); atomicAdd(chk_val, my_val); }
    }
}

// Coordinates of the CTA-unit rows, and the clearing of the value segments that several units
// add into.  Runs before the accumulation kernel.  The saved bitmap carries the rank at every
// 32-word chunk, so any stretch of a row can be expanded on its own: unit c of a row's n units
// takes the c-th n-th of the row's 128-word groups, which spreads a hub row over as many warps as
// it has units.  A warp takes one group at a time, four consecutive words per lane (one 16-byte
// load); the lanes' bit counts are scanned once per group.  Unless the non-empty words of a group
// are half full on average, every lane expands its own words into a small shared-memory stage at
// their ranks and the stage goes out with contiguous stores; otherwise the warp takes one word
// per step with a lane per bit.  Bound by instruction issue, most of it the expansion: 1.25e9 coordinates, 2.3
// to a word, 3760 us taking a word's bits from the lowest, 3640 us from the highest, 3510 us with one reduction for the four
// ballots (a lane per output, which finds its word among flagged first outputs, 3656 us).
constexpr int DE_THREADS = 256;
constexpr int DE_WARPS = DE_THREADS / 32;
constexpr int DE_STAGE = 2048;       // coordinates a warp stages at once (128 words, 16 bits each on average)

template <typename T>
__global__ void __launch_bounds__(DE_THREADS) dense_emit_crd_kernel(DevCtl* __restrict__ ctl, i64 unit_products, RowTables tab,
                                                                    const i64* __restrict__ rowptr, int* __restrict__ Ccrd,
                                                                    T* __restrict__ Cval) {
    __shared__ __align__(16) unsigned short s_stage[DE_WARPS][DE_STAGE];
    if (ctl->status != 0) return;
    const int n_units = ctl->n_units;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned short* const stage = s_stage[warp];
    uint2* const list = reinterpret_cast<uint2*>(stage);                 // (a group uses one or the other)
    for (;;) {
        int u = 0;
        if (lane == 0) u = atomicAdd(&ctl->work_counter[EMIT_SLOT], 1);
        u = __shfl_sync(0xffffffffu, u, 0);
        if (u >= n_units) break;
        u = unit_at(u, n_units);
        const int row = tab.unit_row[u];
        const int uidx = u - tab.row_unit0[row];
        const int nun = dense_units_of_row(tab.ub[row], unit_products);
        const int base = tab.jmin[row];
        const int nw = (tab.jmax[row] - base) / 32 + 1;
        const int nch = chunks_of(nw);
        const int ng = (nch + 3) >> 2;                                  // groups of four chunks = 128 words
        const int g_lo = (int)((i64)ng * uidx / nun), g_hi = (int)((i64)ng * (uidx + 1) / nun);
        const unsigned* src = tab.bm_arena + tab.bm_off[row];
        const uint4* src4 = reinterpret_cast<const uint4*>(src);         // slots are 16-byte aligned
        const i64 out0 = rowptr[row];
        const int cnt_row = (int)(rowptr[row + 1] - out0);
        const bool clear = nun > 1;                                      // several units add into this row's values

        // words 128 g + 4 lane .. + 3 (zero past the end of the bitmap) and the ranks at both ends of group g
        auto load_group = [&](int g, uint4& w, int& r0, int& r1) {
            w = make_uint4(0u, 0u, 0u, 0u);
            r0 = r1 = cnt_row;
            if (g >= g_hi) return;
            const int w0 = (g << 7) + (lane << 2);
            if (w0 < nw) {
                w = src4[(g << 5) + lane];
                if (w0 + 1 >= nw) w.y = 0u;
                if (w0 + 2 >= nw) w.z = 0u;
                if (w0 + 3 >= nw) w.w = 0u;
            }
            r0 = (int)src[nw + (g << 2)];
            if ((g << 2) + 4 < nch) r1 = (int)src[nw + (g << 2) + 4];
        };
        uint4 w, wn;
        int r0, r1, r0n, r1n;
        load_group(g_lo, w, r0, r1);
        for (int g = g_lo; g < g_hi; ++g) {
            load_group(g + 1, wn, r0n, r1n);                             // next group's loads fly during this expansion
            const int n = r1 - r0;
            if (n > 0) {
                const int p = __popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w);
                const int e = warp_incl_scan(p) - p;
                const i64 o = out0 + r0;
                const int nzw = (int)__reduce_add_sync(0xffffffffu, (unsigned)((w.x != 0u) + (w.y != 0u) + (w.z != 0u) + (w.w != 0u)));
                if (n <= DE_STAGE && n < 16 * nzw) {
                    // every lane expands its own four words into the stage at their ranks (as 16-bit
                    // offsets from the group's first column), then the stage goes out with
                    // contiguous stores
                    int slot = e;
                    auto expand = [&](unsigned word, int off0) {
                        slot += __popc(word);
                        int at = slot;                                   // (the highest bit takes one instruction to find)
                        while (word) {
                            const int b = 31 - __clz(word);
                            word ^= 1u << b;
                            stage[--at] = (unsigned short)(off0 + b);
                        }
                    };
                    const int off = lane << 7;
                    expand(w.x, off); expand(w.y, off + 32); expand(w.z, off + 64); expand(w.w, off + 96);
                    __syncwarp();
                    const int gcol0 = base + (g << 12);
                    for (int y = lane; y < n; y += 32) Ccrd[o + y] = gcol0 + (int)stage[y];
                    __syncwarp();
                } else {
                    // half-full words or fuller: the warp expands a word per step, lane b testing bit b, so the
                    // word's outputs leave as one contiguous store.  The words and their ranks go through shared memory: one
                    // broadcast load a word, where taking turns among the lanes with words cost two shuffles and a search.
                    // Lanes without words are passed over: a step for every word costs a group of one full word 128 of them.
                    // 10^4 rows, us by turns / every word / this: 6500 outputs on 313 words 162 / 70 / 71; 128 blocks of 64 columns
                    // on 16384 words 292 / 888 / 289.  (A list of the non-empty words alone: 78 and 291 us, and more
                    // registers or spills, for which the rows of few bits a word pay: power law on 2^18 vertices 3590 us.)
                    const unsigned e1 = (unsigned)(e + __popc(w.x)), e2 = e1 + (unsigned)__popc(w.y), e3 = e2 + (unsigned)__popc(w.z);
                    uint4* const mine = reinterpret_cast<uint4*>(list + (lane << 2));
                    mine[0] = make_uint4(w.x, (unsigned)e, w.y, e1);
                    mine[1] = make_uint4(w.z, e2, w.w, e3);
                    const unsigned some = __ballot_sync(0xffffffffu, p != 0);
                    __syncwarp();
                    const unsigned below = (1u << lane) - 1u;
                    const int col = base + (g << 12) + lane;
                    for (unsigned m = some; m; m &= m - 1) {
                        const int at = (__ffs(m) - 1) << 2;
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const uint2 d = list[at + x];
                            if ((d.x >> lane) & 1u) Ccrd[o + d.y + __popc(d.x & below)] = col + ((at + x) << 5);
                        }
                    }
                    __syncwarp();
                }
                if (clear)
                    for (int y = lane; y < n; y += 32) Cval[o + y] = (T)0;
            }
            w = wn; r0 = r0n; r1 = r1n;
        }
    }
}

// ---------------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------------
static int persistent_grid(const LaunchCtx& c, int per_sm, i64 work) {
    i64 grid = (i64)c.sm_count * (per_sm > 0 ? per_sm : 1);
    if (work >= 0 && work < grid) grid = work > 0 ? work : 1;
    return (int)grid;
}

cudaError_t launch_dense_sym_warp(const LaunchCtx& c, int max_span_words, const Csr& A, const Csr& B) {
    auto k = max_span_words <= DW_SCAN_WORDS ? dense_sym_warp_kernel<true> : dense_sym_warp_kernel<false>;
    int per_sm = 0;
    cudaError_t e = resident_blocks((const void*)k, DW_THREADS, 0, &per_sm);
    if (e != cudaSuccess) return e;
    k<<<persistent_grid(c, per_sm, -1), DW_THREADS, 0, c.stream>>>(c.ctl, c.prm.warp_outputs, A, B, c.tab);
    ++c.launches;
    return cudaGetLastError();
}

cudaError_t launch_dense_sym_cta(const LaunchCtx& c, i64 products, const Csr& A, const Csr& B) {
    const size_t smem = (size_t)c.dense_smem_words * 4 + (size_t)(c.dense_smem_words / 32 + 1) * 4;
    cudaError_t e;
    int per_sm = 0;
    if ((e = resident_blocks((const void*)dense_sym_cta_kernel, DC_THREADS, smem, &per_sm)) != cudaSuccess) return e;
    dense_sym_cta_kernel<<<persistent_grid(c, per_sm, -1), DC_THREADS, smem, c.stream>>>(c.ctl, c.dense_smem_words, c.prm.unit_cap, sym_part_products(products), A, B,
                                                                                                c.tab, c.bw);
    ++c.launches;
    return cudaGetLastError();
}

template <typename T, bool CEIL, bool SPREAD>
static cudaError_t num_warp_t(const LaunchCtx& c, const int* n, const int* max_cnt, int m, int bmw, const Csr& A, const Csr& B, const i64* rowptr,
                              int* Ccrd, void* Cval, u64* chk_idx, double* chk_val) {
    auto k = dense_num_warp_kernel<T, CEIL, SPREAD>;
    const int* const rows[N_WARP_LISTS] = {c.tab.warp_rows, c.tab.warp_rows + m - 1};
    for (int list = N_WARP_LISTS - 1; list >= 0; --list) {          // the longest rows first
        if (n[list] == 0) continue;
        // values reserved per warp; of 256, 128 and 64 threads the CTA size that keeps most warps on an SM, since
        // whole CTAs must fit its shared memory (64^3 stencil, f64, 6 KB a warp: 32 warps in CTAs of 256, 36 in CTAs
        // of 128: 690 -> 643 us)
        const int accw = (max_cnt[list] + 31) & ~31;
        const size_t per_warp = sizeof(T) * (size_t)accw + 6 * (size_t)bmw + 16 * 32;
        int threads = 0, per_sm = 0;
        for (int t = DW_THREADS; t >= 64; t >>= 1) {
            int fit = 0;
            const cudaError_t e = resident_blocks((const void*)k, t, per_warp * (t / 32), &fit);
            if (e != cudaSuccess) return e;
            if (fit * t > per_sm * threads) { threads = t; per_sm = fit; }
        }
        if (threads == 0) return cudaErrorInvalidConfiguration;
        const int warps = threads / 32;
        const size_t smem = per_warp * warps;
        k<<<persistent_grid(c, per_sm, ((i64)n[list] + warps - 1) / warps), threads, smem, c.stream>>>(
            c.ctl, rows[list], list == 0 ? 1 : -1, n[list], (CEIL ? CEIL_WARP_SLOT : WARP_SLOT) + list, bmw, accw, A, B, c.tab, rowptr, Ccrd, (T*)Cval,
            chk_idx, chk_val);
        ++c.launches;
    }
    return cudaGetLastError();
}

cudaError_t launch_dense_num_warp(const LaunchCtx& c, const int* n, const int* max_cnt, int m, int max_span_words, const Csr& A, const Csr& B,
                                  const i64* rowptr, int* Ccrd, void* Cval, u64* chk_idx, double* chk_val) {
    // bitmap words reserved per warp: the widest dense row of this pass, at most the class limit
    int bmw = max_span_words > 0 ? ((max_span_words + 31) & ~31) : DENSE_WARP_BM_WORDS;
    if (bmw > DENSE_WARP_BM_WORDS) bmw = DENSE_WARP_BM_WORDS;
    if (chk_idx)      // same launch shape (shared memory reserved, hence occupancy) as the full kernel
        return c.is_f64 ? num_warp_t<double, true, false>(c, n, max_cnt, m, bmw, A, B, rowptr, Ccrd, Cval, chk_idx, chk_val)
                        : num_warp_t<float, true, false>(c, n, max_cnt, m, bmw, A, B, rowptr, Ccrd, Cval, chk_idx, chk_val);
    const bool spread = bmw > DW_SCAN_WORDS;
    auto go = c.is_f64 ? (spread ? num_warp_t<double, false, true> : num_warp_t<double, false, false>)
                       : (spread ? num_warp_t<float, false, true> : num_warp_t<float, false, false>);
    return go(c, n, max_cnt, m, bmw, A, B, rowptr, Ccrd, Cval, nullptr, nullptr);
}

template <typename T, bool CEIL>
static cudaError_t num_cta_t(const LaunchCtx& c, int phase, int n_units_host, int words, i64 total_products, const Csr& A,
                             const Csr& B, const i64* rowptr, int* Ccrd, void* Cval, u64* chk_idx, double* chk_val) {
    const i64 unit_products = dense_unit_products(total_products, c.prm.unit_products);
    cudaError_t e;
    if (phase == 0) {
        // units are dealt out dynamically, so the grid is what is resident at once
        int emit_per_sm = 0;
        if ((e = resident_blocks((const void*)dense_emit_crd_kernel<T>, DE_THREADS, 0, &emit_per_sm)) != cudaSuccess) return e;
        const i64 work = n_units_host >= 0 ? ((i64)n_units_host + DE_WARPS - 1) / DE_WARPS : -1;
        dense_emit_crd_kernel<T><<<persistent_grid(c, emit_per_sm, work), DE_THREADS, 0, c.stream>>>(c.ctl, unit_products, c.tab, rowptr, Ccrd, (T*)Cval);
        ++c.launches;
        return cudaGetLastError();
    }
    auto smem_of = [&](int cap, int entries) {
        return ((sizeof(T) * (size_t)cap + (size_t)words * 8 + 15) & ~(size_t)15) + (size_t)entries * (8 + sizeof(T)) + (size_t)(entries + 1) * 4 + 16;
    };
    // A block waits at its barriers for its slowest warp and, between units, for chains of loads: four blocks of 256 threads do
    // so less than two of 512, where four find room (with fewer outputs in shared memory if need be: a reduction in global memory
    // costs about the same) and the units are enough for all of them.  Accumulation, 512 / 256 threads: power law on 16381
    // (f32) / 60000 (f64) / 100003 (f32) vertices 229 / 191, 1780 / 1580, 1795 / 1540 us; 10^4 rows of 10^4 products, f64, 419 / 356.
    // With few units 512: power law on 1500 / 4001 vertices, f32, units of 2^13, 18 / 23 and 33 / 38.  Nor where the values that the
    // blocks of a full grid add into and B together outgrow what a half of L2 keeps, which they read and write back from memory
    // then (the second column: MB of both): f64, degree 16, 8e4 vertices 46: 3270 / 3145 us, 1e5 52: 4001 / 4211, 131072 55: 4589 / 5761 (DRAM
    // traffic 6.4 / 13.7 GB); 150000, degree 8, 47: 3187 / 3034, degree 12 63: 5564 / 7548; f32, 180000 48: 8074 / 7715.
    constexpr i64 LIVE_BYTES = 49ll << 20;
    const i64 live = 4ll * c.sm_count * c.unit_nnz * (i64)sizeof(T) + c.b_bytes;
    int CAP = c.prm.unit_outputs, per_sm = 0;
    auto quarter = dense_num_cta_kernel<T, CEIL, DN_THREADS_4>;
    if (n_units_host > 8 * c.sm_count && live <= LIVE_BYTES)
        for (int cap = CAP; cap >= std::min(CAP, DN_CAP_LEAST); cap >>= 1) {
            const size_t smem = smem_of(cap, dn_entries<DN_THREADS_4>());
            if (4 * (smem + 2048) > 228 * 1024) continue;
            if ((e = resident_blocks((const void*)quarter, DN_THREADS_4, smem, &per_sm)) != cudaSuccess) return e;
            if (per_sm < 4) continue;
            quarter<<<persistent_grid(c, per_sm, n_units_host), DN_THREADS_4, smem, c.stream>>>(c.ctl, words, cap, unit_products, A, B, c.tab, rowptr, Ccrd,
                                                                                           (T*)Cval, chk_idx, chk_val);
            ++c.launches;
            return cudaGetLastError();
        }
    auto half = dense_num_cta_kernel<T, CEIL, DN_THREADS>;
    const size_t smem = smem_of(CAP, dn_entries<DN_THREADS>());
    if ((e = resident_blocks((const void*)half, DN_THREADS, smem, &per_sm)) != cudaSuccess) return e;
    half<<<persistent_grid(c, per_sm, n_units_host), DN_THREADS, smem, c.stream>>>(c.ctl, words, CAP, unit_products, A, B, c.tab, rowptr, Ccrd, (T*)Cval, chk_idx,
                                                                               chk_val);
    ++c.launches;
    return cudaGetLastError();
}

cudaError_t launch_dense_num_cta(const LaunchCtx& c, int phase, int n_units_host, int max_span_words, i64 total_products,
                                 const Csr& A, const Csr& B, const i64* rowptr, int* Ccrd, void* Cval, u64* chk_idx, double* chk_val) {
    int words = max_span_words > 0 ? max_span_words : c.dense_smem_words;
    words = (words + 31) & ~31;
    if (chk_idx)      // same launch shape as the full kernel
        return c.is_f64 ? num_cta_t<double, true>(c, 1, n_units_host, words, total_products, A, B, rowptr, Ccrd, Cval, chk_idx, chk_val)
                        : num_cta_t<float, true>(c, 1, n_units_host, words, total_products, A, B, rowptr, Ccrd, Cval, chk_idx, chk_val);
    return c.is_f64 ? num_cta_t<double, false>(c, phase, n_units_host, words, total_products, A, B, rowptr, Ccrd, Cval, nullptr, nullptr)
                    : num_cta_t<float, false>(c, phase, n_units_host, words, total_products, A, B, rowptr, Ccrd, Cval, nullptr, nullptr);
}

}  // namespace spws
