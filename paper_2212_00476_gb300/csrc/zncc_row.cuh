// zncc_row.cuh -- ZNCC cost of one image row for a range of disparities, optionally fused
// with the first horizontal DT pass pair (Sec. V-C fuses the cost with L2R the same way) or
// with WTA (no aggregation). Instantiated once per window radius R in zncc_row.cu.
#pragma once

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace zncc {

// Block (row y, a run of spb disparity slices of 4*tq disparities): thread (chunk k, dq)
// computes the costs of pixels x in [16k, 16k+16) for the four disparities d0 + 4dq ..
// d0 + 4dq + 3 of each slice. The chunk count is padded to whole warps; pixels x >= W are
// computed from clamped reads and dropped.
//
// Bound by the latency of its phases (window sums, normalisation, the pass pair and its two
// barriers a slice) and by shared-memory wavefronts, not by its store of the volume (38 us at
// 1280x384x128 F32): the 96-register variant with two blocks per SM (20 warps) takes 104-106 us
// there at 48% of the issue slots, one block with 128 registers 117-119 us at 42%.
//
// Cost (Eq. (1) through Eq. (2)): with P = sum over the window of I_R(x+i, y+j) *
// I_T(x-d+i, y+j), n = (2R+1)^2 and the window sums S of each image,
//   C = (n P - S_R(x) S_T(x-d)) * inv_sigma_R(x) * inv_sigma_T(x-d),
// inv_sigma = 1/sqrt(n Q - S^2) (0 for a flat window, which makes C = 0). The integer
// numerator is exact: its true value is bounded by sqrt((nQ_R - S_R^2)(nQ_T - S_T^2)) <
// 2^31, so it is computed modulo 2^32 in unsigned arithmetic.
//
// P is built from column sums over the window's rows: the block packs, for every column
// of the band of rows y-R..y+R, up to 16 pixels into four 32-bit words, so that a column
// dot product is at most four __dp4a. A thread walks x' from 16k-R to 16k+15+R keeping
// the target columns of its four disparities in a sliding register window (one new
// shared-memory load per step serves all four, since column x'-d at step x' is column
// (x'-1)-(d-1) of the previous step), and turns the running prefix of column sums into the
// window sums P(x) = prefix(x+R) - prefix(x-R-1). The packed bands are staged once per
// block and serve all of its disparity slices; the window statistics of both images
// (Sec. IV-B-1, Eq. (sum1)) come from the same packed columns: a column's pixel sum is
// __dp4a(word, 0x01010101) and its sum of squares __dp4a(word, word), slid like P.
// Four packed columns xs .. xs+3 (all inside the row) of a band of l raw rows in shared memory
// (row j at raw + j * Wr, Wr a multiple of 16), xs = S (mod 4): per row one 32-bit word of the
// four pixels (two aligned words funnel-shifted when S > 0), then a 4 x 4 byte transpose per
// packed word.
template <int l, int S>
__device__ __forceinline__ void pack4_raw(const uint8_t* raw, int Wr, int xs, uint4 (&col)[4]) {
    constexpr int NW = (l + 3) / 4;
    const unsigned* r32 = reinterpret_cast<const unsigned*>(raw);
    const int a4 = (xs - S) >> 2, wr4 = Wr >> 2;
    unsigned w[4 * NW];
#pragma unroll
    for (int j = 0; j < 4 * NW; ++j) {
        if (j < l) {
            const unsigned lo = r32[j * wr4 + a4];
            w[j] = S ? __funnelshift_r(lo, r32[j * wr4 + a4 + 1], 8 * S) : lo;
        } else {
            w[j] = 0u;
        }
    }
    unsigned o[4][4] = {{0u, 0u, 0u, 0u}, {0u, 0u, 0u, 0u}, {0u, 0u, 0u, 0u}, {0u, 0u, 0u, 0u}};
#pragma unroll
    for (int k = 0; k < NW; ++k) {
        const unsigned t0 = __byte_perm(w[4 * k], w[4 * k + 1], 0x5140), t1 = __byte_perm(w[4 * k + 2], w[4 * k + 3], 0x5140);
        const unsigned t2 = __byte_perm(w[4 * k], w[4 * k + 1], 0x7362), t3 = __byte_perm(w[4 * k + 2], w[4 * k + 3], 0x7362);
        o[0][k] = __byte_perm(t0, t1, 0x5410);
        o[1][k] = __byte_perm(t0, t1, 0x7632);
        o[2][k] = __byte_perm(t2, t3, 0x5410);
        o[3][k] = __byte_perm(t2, t3, 0x7632);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) col[c] = make_uint4(o[c][0], o[c][1], o[c][2], o[c][3]);
}

// Centres per run of the right window statistics. A run's column walk reads up to kStatsItem - 1
// columns past the last centre of the band, so the packed right band holds kStatsItem spare
// entries.
constexpr int kStatsItem = 12;

// Bytes of the rows a visit stages by bulk copies: l rows of each image, Wr = W + 16 apart.
__host__ __device__ inline int bulk_row_stride(int W) { return W + 16; }

// One visit of the cost kernel: row y of one pair, disparity slices [s_begin, s_end).
// The block has the pair's nch * tq threads. Returns
// false when a bulk copy of the image rows timed out (the fault is recorded; the block stops).
template <int R, typename T, int MODE, bool PAD>
__device__ __forceinline__ bool zncc_row_item(const RowArgs& a, int y, int s_begin, int s_end,
                                              uint4* smem_u4, unsigned long long* bar, unsigned& phase,
                                              unsigned* fault) {
    constexpr int l = 2 * R + 1;
    constexpr int NW = (l + 3) / 4;     // packed words per column
    const int tq = a.tq, ds = kG * tq, nch = a.nch, span = nch * kL;
    const int W = a.W, H = a.H;
    const int tid = threadIdx.x;
    const int nthr = nch * tq;
    // FastDT codes are against d_arb = 0: a visit that starts past slice 0 computes that slice
    // first, for its references alone
    constexpr bool kFast = std::is_same<T, uint8_t>::value;
    const int s_first = kFast ? 0 : s_begin;
    // every lane's disparities lie in [blk_lo, blk_hi)
    const int blk_lo = a.d_lo + s_first * ds, blk_hi = a.d_lo + s_end * ds;

    // ---- shared memory carve (zncc_row_layout) ----
    const int NLP = span + 2 * R;                      // left columns x' in [-R, span+R)
    const int NRP = span + 2 * R + (blk_hi - blk_lo) - 1;
    const int xr0 = -R - (blk_hi - 1);                 // right columns x'' in [xr0, xr0+NRP)
    const int NSR = span + (blk_hi - blk_lo) - 1;      // right centres c in [c0, c0+NSR)
    const int c0 = -(blk_hi - 1);
    unsigned char* const sm = reinterpret_cast<unsigned char*>(smem_u4);
    // The left columns and statistics are chunk-major (entry 0 = column -R resp. x = 0): the
    // lanes of a chunk read the same entry and the eight chunks of a warp distinct banks, one
    // shared-memory wavefront a load where a layout with two chunks to a bank group takes four.
    // (lpad: the spare entry per chunk, left out where the row would not fit with it.)
    uint4* const LP = smem_u4;
    const int lpad = PAD ? 1 : a.lpad;
    auto lpos = [&](int idx) { return idx + (idx >> 4) * lpad; };
    const CostArray<PAD, uint4> RP{reinterpret_cast<uint4*>(sm + a.rp_off), a.rp_plane};
    // (S, 1/sigma bits) per x, and per right centre
    int2* const SL = reinterpret_cast<int2*>(sm + a.sl_off);
    const CostArray<PAD, int2> SR{reinterpret_cast<int2*>(sm + a.sr_off), a.sr_plane};
    float4* const co = reinterpret_cast<float4*>(sm + a.co_off);     // HPair, chunk-major
    // FastDT codes (HPair): the row's output scales and the reference values v(d_arb = 0)
    float* const mrow = reinterpret_cast<float*>(sm + a.mrow_off);   // chunk-major (kCS)
    float* const ref = reinterpret_cast<float*>(sm + a.ref_off);
    // (bulk) the guide row y for the coefficients
    uint8_t* const grow = sm + a.grow_off;

    // ---- stage the packed bands (and the DT coefficients) ----
    const bool bulk = MODE == kModeHPair && a.bulk;
    if (bulk) {
        // Bulk copies (the TMA unit) of the clamped rows y-R .. y+R of both images into the
        // region that the statistics and coefficients take once the bands are packed, and of
        // the guide row y; one thread issues them, every thread waits on the mbarrier.
        const int Wr = bulk_row_stride(W);
        uint8_t* rawL = sm + a.sl_off;
        uint8_t* rawR = rawL + l * Wr;
        fence_proxy_async_smem();                       // earlier accesses of the region, then the copies
        __syncthreads();
        if (tid == 0) {
            mbar_expect_tx(bar, (unsigned)((2 * l + 1) * W));
#pragma unroll
            for (int j = 0; j < l; ++j) {
                const size_t ro = (size_t)min(max(y - R + j, 0), H - 1) * a.pitch;
                bulk_copy_g2s(rawL + j * Wr, a.left + ro, (unsigned)W, bar);
                bulk_copy_g2s(rawR + j * Wr, a.right + ro, (unsigned)W, bar);
            }
            bulk_copy_g2s(grow, a.left + (size_t)y * a.pitch, (unsigned)W, bar);
        }
        bool ok = mbar_wait(bar, phase, kBulkWaitPolls);
        if (__syncthreads_or(!ok)) {                     // a copy did not land in time: record it,
            if (tid == 0) atomicOr(fault, kFaultBulkWait);
            ok = mbar_wait(bar, phase, kBulkWaitPolls);  // wait for the copies still in flight
            if (__syncthreads_or(!ok) && tid == 0) atomicOr(fault, kFaultBulkDrain);
            return false;
        }
        phase ^= 1u;
        // pack four columns per thread where they lie inside the row, single columns (clamped)
        // at the ends
        auto pack1 = [&](const uint8_t* raw, int xc) {
            unsigned w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int j = 0; j < l; ++j) w[j >> 2] |= (unsigned)raw[j * Wr + xc] << (8 * (j & 3));
            return make_uint4(w[0], w[1], w[2], w[3]);
        };
        constexpr int SLS = ((-R) % 4 + 4) % 4, SRS = ((1 - R) % 4 + 4) % 4;   // (-R) & 3, xr0 & 3
        const int ngl = (NLP + 3) >> 2, ngr = (NRP + 3) >> 2;
        for (int g = tid; g < ngl + ngr; g += blockDim.x) {
            const bool left = g < ngl;
            const int g4 = left ? g : g - ngl;
            const int xs = left ? 4 * g4 - R : xr0 + 4 * g4;   // image column of entry 4 g4
            const int nent = left ? NLP : NRP;
            const CostArray<PAD, uint4> rdst = RP.from(4 * g4);
            uint4* const ldst = LP + lpos(4 * g4);
            auto put = [&](int c, const uint4& col) {
                if (left) ldst[c] = col;
                else rdst.at(c) = col;
            };
            const uint8_t* raw = left ? rawL : rawR;
            if (xs >= 0 && xs + 3 < W && 4 * g4 + 3 < nent) {
                uint4 col[4];
                if (left) pack4_raw<l, SLS>(raw, Wr, xs, col);
                else pack4_raw<l, SRS>(raw, Wr, xs, col);
#pragma unroll
                for (int c = 0; c < 4; ++c) put(c, col[c]);
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (4 * g4 + c < nent) put(c, pack1(raw, min(max(xs + c, 0), W - 1)));
            }
        }
        __syncthreads();                                 // the raw rows are consumed
    } else {
        size_t roff[l];                                 // the band's clamped rows
#pragma unroll
        for (int j = 0; j < l; ++j) roff[j] = (size_t)min(max(y - R + j, 0), H - 1) * a.pitch;
        auto pack = [&](const uint8_t* img, int xc) {
            unsigned w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int j = 0; j < l; ++j) w[j >> 2] |= (unsigned)img[roff[j] + xc] << (8 * (j & 3));
            return make_uint4(w[0], w[1], w[2], w[3]);
        };
        for (int t = tid; t < NLP; t += blockDim.x) LP[lpos(t)] = pack(a.left, min(max(t - R, 0), W - 1));
        for (int t = tid; t < NRP; t += blockDim.x) RP[t] = pack(a.right, min(max(xr0 + t, 0), W - 1));
    }
    if constexpr (MODE == kModeHPair) {
        // the row's DT coefficients (w, chunk prefix product, next w, chunk suffix product),
        // computed here from the guide (the left image) as k_dt_coef computes them: 16
        // consecutive lanes hold one chunk (span and the block are whole warps)
        const uint8_t* g = bulk ? grow : a.left + (size_t)y * a.pitch;
        auto weight = [&](int q) -> float {      // the step q-1 -> q
            return (q >= 1 && q < W) ? a.K * expf(-fabsf((float)(g[q] - g[q - 1])) * a.inv_sr255) : 0.0f;
        };
        for (int t = tid; t < span; t += blockDim.x) {
            const int i = t & (kL - 1);
            const float w = weight(t);
            float wn = __shfl_down_sync(kFull, w, 1, kL);
            if (i == kL - 1) wn = weight(t + 1);
            float A = w, B = wn;
#pragma unroll
            for (int off = 1; off < kL; off <<= 1) {
                const float a2 = __shfl_up_sync(kFull, A, off, kL);
                const float b2 = __shfl_down_sync(kFull, B, off, kL);
                if (i >= off) A *= a2;
                if (i + off < kL) B *= b2;
            }
            co[cpos(t)] = t < W ? make_float4(w, A, wn, B) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (a.coefH_out && s_begin == 0 && t < W) a.coefH_out[(size_t)y * W + t] = make_float4(w, A, wn, B);
            if constexpr (kFast)
                mrow[cpos(t)] = t < W ? __ldg(a.mulmap + (size_t)y * W + t).y : 0.0f;
        }
    }
    __syncthreads();

    // ---- window statistics: runs of consecutive centres per thread, left then right ----
    // Left runs are chunks; right runs start 12 columns apart, so that the 16-byte column loads of
    // the eight lanes of a quarter warp fall in distinct bank groups (16 apart, they would share
    // two).
    const unsigned n = (unsigned)(l * l);
    // A fused horizontal pair (F32, F16) in the scaled form multiplies its result by
    // s2 = (1-K)^2; the pair is linear, so the factor rides on the left 1/sigma instead
    // (FastDT codes take per-position scales in the pair).
    const float lscale = (MODE == kModeHPair && !kFast) ? a.s2 : 1.0f;
    // the statistics of COUNT centres whose first window starts at column 0 of the walk
    auto stats = [&](auto count, auto column, auto store) {
        constexpr int COUNT = decltype(count)::value;
        int Sx[COUNT], Qx[COUNT];           // (an entry lives from its first touch to its centre's store)
        unsigned ps = 0u, pq = 0u;
#pragma unroll
        for (int u = 0; u < COUNT + 2 * R; ++u) {
            const uint4 w = column(u);
            ps = __dp4a(w.x, 0x01010101u, ps);
            pq = __dp4a(w.x, w.x, pq);
            if (NW > 1) { ps = __dp4a(w.y, 0x01010101u, ps); pq = __dp4a(w.y, w.y, pq); }
            if (NW > 2) { ps = __dp4a(w.z, 0x01010101u, ps); pq = __dp4a(w.z, w.z, pq); }
            if (NW > 3) { ps = __dp4a(w.w, 0x01010101u, ps); pq = __dp4a(w.w, w.w, pq); }
            if (u + 1 < COUNT) { Sx[u + 1] = (int)ps; Qx[u + 1] = (int)pq; }
            const int i = u - 2 * R;                                    // the centre completed
            if (i >= 0 && i < COUNT) {
                const int S = (int)ps - (i > 0 ? Sx[i] : 0), Q = (int)pq - (i > 0 ? Qx[i] : 0);
                const int var = (int)(n * (unsigned)Q - (unsigned)S * (unsigned)S);
                store(i, S, var > 0 ? rsqrtf((float)var) : 0.0f);          // as k_window_stats
            }
        }
    };
    // (the right runs start at a whole warp, so that no warp walks both kinds one after the other)
    const int nrc = (NSR + kStatsItem - 1) / kStatsItem, right0 = (nch + 31) & ~31;
    for (int t = tid; t < right0 + nrc; t += blockDim.x) {
        if (t < right0) {
            if (t >= nch) continue;
            const uint4* const col = LP + lpos(t * kL);
            int2* const out = SL + lpos(t * kL);
            stats(std::integral_constant<int, kL>(), [&](int u) { return col[u + (u >> 4) * lpad]; },
                  [&](int i, int S, float is) { out[i] = make_int2(S, __float_as_int(is * lscale)); });
        } else {
            const int c = (t - right0) * kStatsItem;                       // first centre, from c0
            const CostArray<PAD, uint4> col = RP.from(c);               // (its first column is c0 + c - R = xr0 + c)
            const CostArray<PAD, int2> out = SR.from(c);
            stats(std::integral_constant<int, kStatsItem>(), [&](int u) { return col.at(u); },
                  [&](int i, int S, float is) { if (c + i < NSR) out.at(i) = make_int2(S, __float_as_int(is)); });
        }
    }
    __syncthreads();

    WtaRegs wr;
    if constexpr (MODE == kModeWta) wr.reset();

    for (int sl = s_first; sl < s_end; sl = kFast && sl < s_begin ? s_begin : sl + 1) {
        float v[kL][4];
        // A thread's place (chunk, lane of the chunk) is taken from its index anew in each phase:
        // the tile of sums leaves few registers for what would be kept across it.
        {
            const int t1 = thread_index(), x0 = (t1 >> a.tq_shift) * kL;
            const int d_first = a.d_lo + sl * ds + (t1 & (tq - 1)) * kG;
            // ---- window sums of products, times n, for 16 pixels x 4 disparities ----
            // n P[i] = n prefix(i + 2R) - n prefix(i - 1): each entry is set at its first touch
            // (-n prefix(i - 1) at step i - 1; n P[0] at step 2R) and completed at step i + 2R;
            // the factor n of Eq. (2)'s numerator rides on those multiply-adds (mod 2^32)
            unsigned P[kL][4];
            // RP index of column x' - d_first - j at step t (x' = x0 - R + t) is rbase + t - j,
            // rbase = x0 - R - d_first - xr0 >= 3 (d_first + 3 < blk_hi); rbase + 1 = x0 - d_first +
            // blk_hi is a multiple of 4 (as are x0, d_first and blk_hi, d_lo being one), so the
            // columns are at constant offsets from the pointer to entry rbase + 1 - 4
            const uint4* const lpp = LP + lpos(x0);
            const CostArray<PAD, uint4> rpp = RP.from(x0 - d_first + blk_hi - 4);
            uint4 rp[4];
            rp[1] = rpp.at(2);
            rp[2] = rpp.at(1);
            rp[3] = rpp.at(0);
            unsigned pre[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int t = 0; t < kL + 2 * R; ++t) {
                const uint4 lp = lpp[t + (t >> 4) * lpad];
                rp[0] = rpp.at(t + 3);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    pre[j] = __dp4a(lp.x, rp[j].x, pre[j]);
                    if (NW > 1) pre[j] = __dp4a(lp.y, rp[j].y, pre[j]);
                    if (NW > 2) pre[j] = __dp4a(lp.z, rp[j].z, pre[j]);
                    if (NW > 3) pre[j] = __dp4a(lp.w, rp[j].w, pre[j]);
                    if (t == 2 * R) P[0][j] = n * pre[j];
                    else if (t - 2 * R > 0 && t - 2 * R < kL) P[t - 2 * R][j] += n * pre[j];
                    if (t + 1 < kL) P[t + 1][j] = (0u - n) * pre[j];
                }
                rp[3] = rp[2];
                rp[2] = rp[1];
                rp[1] = rp[0];
            }

            // ---- normalization, Eq. (2); the target statistics slide like the columns ----
            // (SR index of (i, j) is x0 - d_first - c0 + i - j >= 3, one less than a multiple of 4)
            const int t2 = thread_index(), xn = (t2 >> a.tq_shift) * kL;
            const int dn = a.d_lo + sl * ds + (t2 & (tq - 1)) * kG;
            const int2* const slp = SL + lpos(xn);
            const CostArray<PAD, int2> srp = SR.from(xn - dn + blk_hi - 4);
            int2 sr[4];
            sr[1] = srp.at(2);
            sr[2] = srp.at(1);
            sr[3] = srp.at(0);
            // Pixels past the row and disparities past the range are computed like the others (their
            // columns and statistics are staged) and never stored or compared; the zero weights
            // past the row keep them out of the pass pair.
#pragma unroll
            for (int i = 0; i < kL; ++i) {
                const int2 st = slp[i];
                sr[0] = srp.at(i + 3);
                const float isl = __int_as_float(st.y);      // (times the pair's scale)
                const unsigned nsl = 0u - (unsigned)st.x;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const unsigned num = nsl * (unsigned)sr[j].x + P[i][j];       // n P - S_R S_T
                    v[i][j] = (float)(int)num * isl * __int_as_float(sr[j].y);
                }
                sr[3] = sr[2];
                sr[2] = sr[1];
                sr[1] = sr[0];
            }
        }

        if constexpr (MODE == kModeWta) {
            const int t3 = thread_index(), dn = a.d_lo + sl * ds + (t3 & (tq - 1)) * kG;
            wr.fold(v, max(0, min(4, a.d_hi - dn)), dn);
            continue;
        }
        const int t3 = thread_index(), k = t3 >> a.tq_shift, dq = t3 & (tq - 1);
        if constexpr (MODE == kModeHPair) {
            float4* const sb = reinterpret_cast<float4*>(sm + a.sb_off);
            float* const sa = reinterpret_cast<float*>(sm + a.sa_off);
            const int shift = 5 - a.tq_shift, nvg = nthr >> 5;      // scan groups: the warps
            dt_group_pair<kFast, PAD, 0>(v, co + k * kCS, tq, shift, t3 & 31, k, nvg, false, sa + dq, sb + dq, kFast ? a.s2 : 1.0f,
                                          kFast ? mrow + k * kCS : (const float*)nullptr, 0, nthr, NoHook());
        }
        const int x0 = k * kL, d_first = a.d_lo + sl * ds + dq * kG;
        const int nvalid = max(0, min(4, a.d_hi - d_first));
        T* q = reinterpret_cast<T*>(a.vol) + (size_t)(d_first >> a.sd_shift) * a.slab_stride +
               ((size_t)y * W + x0) * a.dstride + (d_first & ((1 << a.sd_shift) - 1));    // [slab][H][W][dstride]
        if constexpr (kFast) {
            // near-zero-mean codes against d_arb = 0, held by lane dq 0 in slice 0, the visit's first
            if (sl == 0) {
                if (dq == 0)
#pragma unroll
                    for (int i = 0; i < kL; ++i) ref[k * kCS + i] = v[i][0];
                __syncthreads();
            }
            if (sl < s_begin) {                              // (stored by the visit that owns slice 0)
            } else if (nvalid == 4 && x0 + kL <= W) {        // a whole chunk of whole groups
#pragma unroll
                for (int i = 0; i < kL; ++i)
                    *reinterpret_cast<unsigned*>(q + (size_t)i * a.dstride) = fastdt_pack(v[i], ref[k * kCS + i], 4);
            } else if (nvalid > 0) {
#pragma unroll
                for (int i = 0; i < kL; ++i) {
                    if (x0 + i < W) *reinterpret_cast<unsigned*>(q) = fastdt_pack(v[i], ref[k * kCS + i], nvalid);
                    q += a.dstride;
                }
            }
        } else if constexpr (MODE == kModeRawAny) {
            // Pixels off the alignment of whole groups are stored one entry at a time. Four lanes (the
            // two of a chunk with tq = 2) first trade their 4 x 4 (2 x 4) entries, so that a store
            // instruction writes four (two) adjacent entries of each chunk instead of every fourth one
            // and a 32-byte sector is written in fewer pieces (us a call, every fourth entry and this:
            // 1280x384x127 F32 276 and 186, 1296x315x246 F16 414 and 258, 2500x700x61 F32 672 and 568).
            // (A block is whole warps, all of them here.)
            // Small volumes (a.trade) are written from registers as they are: there the kernel is a matter of
            // latency and of fetching its instructions (160x64x17 F32 6.7 and 5.4 us, 59x76x1 F16 7.6 and
            // 6.3, 200x100x19 6.5 and 5.5; level at 160x100x33, 320x96x21 F16 6.7 and 7.6).
            if (!PAD && !a.trade) {
                if (nvalid > 0)
#pragma unroll
                    for (int i = 0; i < kL; ++i) {
                        if (x0 + i < W) st4(q, nvalid, false, v[i]);
                        q += a.dstride;
                    }
            } else {
                const bool quad = tq >= 4;
                const int l = dq & (quad ? 3 : 1);
                const int left = a.d_hi - (d_first - 3 * l);     // entries from the first that this lane stores
                T* p = q - 3 * l;
                const int o2 = quad ? 8 : 2, o3 = o2 + 4;
#pragma unroll
                for (int i = 0; i < kL; ++i) {
                    float e[4] = {v[i][0], v[i][1], v[i][2], v[i][3]};
                    const float r0 = __shfl_xor_sync(kFull, l & 1 ? e[0] : e[1], 1);
                    const float r1 = __shfl_xor_sync(kFull, l & 1 ? e[2] : e[3], 1);
                    if (l & 1) { e[0] = r0; e[2] = r1; } else { e[1] = r0; e[3] = r1; }
                    if (quad) {
                        const float r2 = __shfl_xor_sync(kFull, l & 2 ? e[0] : e[2], 2);
                        const float r3 = __shfl_xor_sync(kFull, l & 2 ? e[1] : e[3], 2);
                        if (l & 2) { e[0] = r2; e[1] = r3; } else { e[2] = r2; e[3] = r3; }
                    }
                    if (x0 + i < W) {
                        if (0 < left) st1(p, e[0]);
                        if (4 < left) st1(p + 4, e[1]);
                        if (o2 < left) st1(p + o2, e[2]);
                        if (o3 < left) st1(p + o3, e[3]);
                    }
                    p += a.dstride;
                }
            }
        } else if (nvalid > 0) {
            // (Raw: the costs are finished before the first store; interleaved, the addresses would
            // not fit in 96 registers beside the tile)
            if constexpr (MODE == kModeRaw && PAD) asm volatile("" ::: "memory");
            if (nvalid == 4 && x0 + kL <= W) {               // a whole chunk of whole groups
#pragma unroll
                for (int i = 0; i < kL; ++i) st4(q + (size_t)i * a.dstride, 4, true, v[i]);
            } else {
#pragma unroll
                for (int i = 0; i < kL; ++i) {
                    if (x0 + i < W) st4(q, nvalid, true, v[i]);
                    q += a.dstride;
                }
            }
        }
    }

    if constexpr (MODE == kModeWta) {
        {
            // the chunk's lanes merge their running bests; each lane writes its share of positions
            wr.merge(tq, tid & 31, [&](int i, float best, int bd) {
                const int x = (tid >> a.tq_shift) * kL + i;
                if (x < W) {
                    const size_t o = (size_t)y * W + x;
                    if (!a.wta.first) {                                // earlier launches: smaller d
                        const float pb = a.wta.bestv[o];
                        if (!(best > pb)) { best = pb; bd = a.wta.bestd[o]; }
                    }
                    if (a.wta.last) a.wta.disp[o] = (uint16_t)bd;
                    else {
                        a.wta.bestv[o] = best;
                        a.wta.bestd[o] = bd;
                    }
                }
            });
        }
    }
    return true;
}

// SINGLE: the launch holds one pair, whose arguments are then read at constant offsets of
// the parameter block instead of through a dynamic index.
// Work units: (row, disparity slice) in row-major order, pair by pair (Wta: whole rows, since
// a row's running best stays in registers). Block b takes the units [b*total/G, (b+1)*total/G)
// and visits them row by row, at most spb slices per visit, so that the band of a row is
// staged once per visit and every block gets the same work within one unit.
template <int R, typename T, int MODE, int MINB, bool SINGLE>
__global__ void __launch_bounds__(MINB == 2 ? 320 : 512, MINB) 
k_zncc_row(const __grid_constant__ RowBatchOf<SINGLE ? 1 : kMaxBatch> b) {
    extern __shared__ uint4 smem_u4[];
    __shared__ unsigned long long bar;                  // bulk copies of the image rows (HPair)
    unsigned phase = 0;
    if (MODE == kModeHPair && threadIdx.x == 0) mbar_init(&bar, 1);
    __syncthreads();
    griddep_wait();
    const int i0 = (int)((long long)blockIdx.x * b.total_items / b.grid);
    const int i1 = (int)((long long)(blockIdx.x + 1) * b.total_items / b.grid);
    int pi = 0;
    for (int u = i0; u < i1;) {
        if (!SINGLE)
            while (u >= b.p[pi].item0 + b.p[pi].nitems) ++pi;
        const RowArgs& a = b.p[SINGLE ? 0 : pi];
        const int ds = kG * a.tq;
        const int nslices = (a.d_hi - a.d_lo + ds - 1) / ds;
        const int local = u - a.item0;
        int y, s_begin, s_end;
        if constexpr (MODE == kModeWta) {       // whole rows
            y = local;
            s_begin = 0;
            s_end = nslices;
            u += 1;
        } else {
            y = local / nslices;
            s_begin = local - y * nslices;
            const int last = min(i1, a.item0 + (y + 1) * nslices);      // this block, this row
            s_end = min(s_begin + a.spb, s_begin + (last - u));
            u += s_end - s_begin;
        }
        if (u >= i1) griddep_launch_dependents();       // this block's last visit
        if (!zncc_row_item<R, T, MODE, MINB == 2>(a, y, s_begin, s_end, smem_u4, &bar, phase, b.fault)) return;
        __syncthreads();                                 // the next visit restages shared memory
    }
}

// The shared memory of a visit of k_zncc_row: offsets into a, bytes returned. pad: for the
// two-blocks-per-SM variant (CostArray).
inline size_t zncc_row_fill_layout(int R, int mode, int dtype, RowArgs& a, int nthreads, bool pad) {
    const int ds = kG * a.tq, span = a.nch * kL;
    const int nslices = (a.d_hi - a.d_lo + ds - 1) / ds;
    const int drange = std::min(a.spb, nslices) * ds;
    a.tq_shift = 0;
    while ((1 << a.tq_shift) < a.tq) ++a.tq_shift;
    auto len = [&](int n) { return pad ? cost_array_len<true>(n) : cost_array_len<false>(n); };
    const int nlp = span + 2 * R, nrp = nlp + drange - 1 + kStatsItem, nsr = span + drange - 1;
    a.rp_plane = plane_of(nrp);
    a.sr_plane = plane_of(nsr);
    int b = 16 * (kL + a.lpad) * ((nlp + kL - 1) / kL);
    auto take = [&](int& off, int bytes) {
        off = b = (b + 15) & ~15;
        b += bytes;
    };
    const bool pair = mode == kModeHPair, fast = pair && dtype == 2;
    take(a.rp_off, 16 * len(nrp));
    take(a.sl_off, 8 * (kL + a.lpad) * a.nch);
    take(a.sr_off, 8 * len(nsr));
    take(a.co_off, pair ? 16 * a.nch * kCS : 0);
    take(a.sb_off, pair ? 2 * (nthreads / 32) * a.tq * 16 : 0);
    take(a.sa_off, pair ? 2 * (nthreads / 32) * a.tq * 4 : 0);
    take(a.mrow_off, fast ? 4 * a.nch * kCS : 0);
    take(a.ref_off, fast ? 4 * a.nch * kCS : 0);
    take(a.grow_off, pair && a.bulk ? (a.W + 15) / 16 * 16 : 0);
    return (size_t)b;
}

// Whether a visit's raw rows (both images, bulk_row_stride apart) fit in the shared memory that
// the statistics and the later per-visit arrays take (HPair): the region after the packed bands.
inline bool zncc_row_bulk_fits(int R, const RowArgs& a) {
    return 2 * (2 * R + 1) * bulk_row_stride(a.W) <= a.grow_off - a.sl_off;
}

template <int R, int MINB, bool SINGLE>
static const void* row_fn_t(int mode, int dtype) {
    if constexpr (SINGLE) {
        if (mode == kModeRaw)
            return dtype == 0 ? (const void*)k_zncc_row<R, float, kModeRaw, MINB, true>
                              : (const void*)k_zncc_row<R, __half, kModeRaw, MINB, true>;
        if (mode == kModeRawAny)
            return dtype == 0 ? (const void*)k_zncc_row<R, float, kModeRawAny, MINB, true>
                              : (const void*)k_zncc_row<R, __half, kModeRawAny, MINB, true>;
    }
    if (mode == kModeHPair)
        return dtype == 0   ? (const void*)k_zncc_row<R, float, kModeHPair, MINB, SINGLE>
               : dtype == 1 ? (const void*)k_zncc_row<R, __half, kModeHPair, MINB, SINGLE>
                            : (const void*)k_zncc_row<R, uint8_t, kModeHPair, MINB, SINGLE>;
    return (const void*)k_zncc_row<R, float, kModeWta, MINB, SINGLE>;
}

// Batched launches come from the fused path only (HPair, Wta); a batched Raw launch would
// use the single-pair variant's arguments and is never made.
template <int R>
static const void* row_fn(int mode, int dtype, bool minb2, bool single) {
    if (single) return minb2 ? row_fn_t<R, 2, true>(mode, dtype) : row_fn_t<R, 1, true>(mode, dtype);
    if (mode == kModeRaw || mode == kModeRawAny) return nullptr;
    return minb2 ? row_fn_t<R, 2, false>(mode, dtype) : row_fn_t<R, 1, false>(mode, dtype);
}

// The variant limited to 96 registers (two resident blocks per SM) serves blocks of up to
// 320 threads when minb2 is set; larger blocks use the 128-register one.
template <int R>
cudaError_t zncc_row_occupancy_impl(int mode, int dtype, int threads, size_t smem, bool minb2, bool single,
                                    int* bps) {
    const void* fn = row_fn<R>(mode, dtype, minb2, single);
    if (!fn) return cudaErrorInvalidValue;
    cudaError_t e = set_max_smem(fn, smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, fn, threads, smem);
}

template <int R>
cudaError_t launch_zncc_row_impl(const RowBatch& b, int threads, size_t smem, int mode, int dtype,
                                 cudaStream_t st) {
    const void* fn = row_fn<R>(mode, dtype, b.p[0].minb2 != 0, b.npairs == 1);
    if (!fn) return cudaErrorInvalidValue;
    cudaError_t e = set_max_smem(fn, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    launch_config(cfg, attr, dim3(b.grid), dim3(threads), smem, st, 1);
    return b.npairs == 1 ? launch_batch(cfg, fn, first_pair<RowHead>(b)) : launch_batch(cfg, fn, b);
}

}  // namespace zncc
