// dt_lines.cu -- the DT pass pair along rows or columns (Sec. III-B, Eqs. (3)-(6)) over a volume
// in disparity slabs, F32 or F16 storage, with the WTA fused into the last pair (Sec. V-C).
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace zncc {

// ---------------------------------------------------------------------------------------
// A thread holds 16 consecutive positions (a chunk) x 4 disparities in registers; `lanes`
// lanes share a chunk, so a step is 4 * lanes disparities of `lines` adjacent lines. The block
// takes the steps [s0, s1) of all (line group, disparity slice) in order, slices innermost.
//
// The result of a pass depends, in its last bits, on how the chunks' affine maps are composed:
// in scan groups of `scan` consecutive chunks by doubling rounds, then group by group. The scan
// group is given by the caller and does not depend on the lanes per chunk, so a shape can be
// chosen for speed alone.
//
// Bound by HBM for F32 store passes: a pass moves the volume once in and once out, and an
// in-place pass of a plain kernel over the same bytes takes 78-82 us at 1280x384x128. Measured
// there (k_line_pair -> this kernel, us): columns 94 -> 87, rows 95 -> 86, last columns with WTA
// 75 -> 58; F16 at 1242x375x128: columns 77 -> 60, rows 110 -> 64, WTA 84 -> 53; F32 at
// 1920x1080x256: columns 1188 -> 735, rows 888 -> 636, WTA 790 -> 510.
//
// Staging: one lane per chunk copies the box of the next step's chunk (all lines of the group)
// into shared memory by TMA as soon as the lines' warps have read the last one into registers,
// so that the copy is in flight during the whole step. A warp waits for its own chunks only
// (an mbarrier per warp of a line), and the two barriers of the pass pair are per line: the
// lines of a block share nothing but their boxes.
// The WTA of a step (Eq. (WTA1)): each thread takes the best of its four disparities at each
// of its 16 positions, the chunk's lanes merge theirs by halving rounds (WtaRegs::merge), and
// a lane keeps the running best of the 16 / lanes positions that it ends up with: a few
// registers where a running best of all 16 positions took 24 (which spilled).
template <int lanes>
struct StepWta {
    static constexpr int kHeld = kL / lanes;
    float rv[kHeld];
    int rd[kHeld];
    __device__ __forceinline__ void reset() {
#pragma unroll
        for (int k = 0; k < kHeld; ++k) {
            rv[k] = -INFINITY;
            rd[k] = 0x7FFFFFFF;
        }
    }
    // slices arrive in increasing d, so that a later equal value does not replace an earlier one
    __device__ __forceinline__ void fold(float (&v)[kL][4], int nvalid, int d_first, int dq) {
        if (nvalid < 4) {
#pragma unroll
            for (int i = 0; i < kL; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j >= nvalid) v[i][j] = -INFINITY;
        }
        float bv[kL];
        int bd[kL];
#pragma unroll
        for (int i = 0; i < kL; ++i) {
            const float m01 = fmaxf(v[i][0], v[i][1]), m23 = fmaxf(v[i][2], v[i][3]);
            const bool lo = m01 >= m23;
            bv[i] = lo ? m01 : m23;
            bd[i] = d_first + (lo ? (v[i][0] >= v[i][1] ? 0 : 1) : (v[i][2] >= v[i][3] ? 2 : 3));
        }
        wta_halve<16>(bv, bd, (dq & 1) != 0, 1);
        if constexpr (lanes > 2) wta_halve<8>(bv, bd, (dq & 2) != 0, 2);
        if constexpr (lanes > 4) wta_halve<4>(bv, bd, (dq & 4) != 0, 4);
#pragma unroll
        for (int k = 0; k < kHeld; ++k)
            if (bv[k] > rv[k]) {
                rv[k] = bv[k];
                rd[k] = bd[k];
            }
    }
    // the first of the positions that lane dq holds
    __device__ __forceinline__ static int first(int dq) {
        return ((dq & 1) ? 8 : 0) + ((dq & 2) ? 4 : 0) + ((dq & 4) ? 2 : 0);
    }
};

// COLS = 2: the lanes of a chunk in shuffles are those of two adjacent columns (lane bits: dq,
// column, chunk), so that a quarter warp reads 128 contiguous bytes of a box of 64-byte pixels
// (with eight chunks of one column per warp two chunks share each bank group) and chunks pad
// to four per line instead of eight. "Line" below then stands for the pair of columns that share a
// barrier and scan buffers.
template <typename T, int MODE, int lanes, int COLS, int NP, int MAXT>
__global__ void __launch_bounds__(MAXT) k_dt_lines(const __grid_constant__ DtBatch<NP> b) {
    constexpr bool SINGLE = NP == 1;
    constexpr int ds = kG * lanes;                       // disparities per step
    constexpr int LC = lanes * COLS, cpw = 32 / LC;      // lanes per chunk in shuffles, chunks per warp
    constexpr bool kChain = MODE == kLineStore && MAXT <= 512;      // (the 96-register variants would spill)
    extern __shared__ __align__(128) unsigned char dt_smem[];
    __shared__ unsigned long long full[kDtThreads / 32], empty[kDtThreads / 32], drill_bar;
    if (threadIdx.x < b.s.nwl) {            // per warp of a line: its chunks' boxes, their readers
        mbar_init(&full[threadIdx.x], (unsigned)cpw);
        mbar_init(&empty[threadIdx.x], (unsigned)(b.s.lines / COLS));
    }
    // (tests) the wait drill, as in k_line_pair
    if (b.drill && threadIdx.x == 0) mbar_init(&drill_bar, 1);
    __syncthreads();
    if (b.drill && threadIdx.x == 0 && !mbar_wait(&drill_bar, 0, kDrillWaitPolls)) atomicOr(b.fault, kFaultTmaWait);
    griddep_wait();

    auto P = [&](int pi) -> const DtArgs& { return b.p[SINGLE ? 0 : pi]; };
    // A step: the pair, the line group and the slice. Of one pair's groups the blocks take whole
    // ones in turn (block i the groups i, i + grid, ...), so that the blocks are at adjacent
    // lines at any time and their short runs of a pixel row fall together in DRAM; the groups
    // that do not fill a round, and the groups of several pairs, go by equal ranges of steps.
    struct Cursor {
        int pi, g, sl;
    };
    const int full_rounds = SINGLE ? b.p[0].ngroups / b.grid * b.grid : 0;        // groups taken in turn
    Cursor rest;                            // the block's first step among the others
    int left;                               // steps from the cursor to the end of the block's
    {
        const int first = full_rounds * (SINGLE ? b.p[0].nsl : 0), others = b.total_steps - first;
        const int s0 = first + (int)((long long)blockIdx.x * others / b.grid);
        left = first + (int)((long long)(blockIdx.x + 1) * others / b.grid) - s0;
        rest.pi = 0;
        if (!SINGLE)
            while (rest.pi + 1 < b.npairs && s0 >= b.p[rest.pi + 1].step0) ++rest.pi;
        rest.g = (s0 - P(rest.pi).step0) / P(rest.pi).nsl;
        rest.sl = s0 - P(rest.pi).step0 - rest.g * P(rest.pi).nsl;
        left += first / b.grid;
    }
    auto next_group = [&](Cursor& q) {
        q.sl = 0;
        if (SINGLE && q.g < full_rounds) {
            q.g += b.grid;
            if (q.g >= full_rounds) q = rest;
        } else if (++q.g == P(q.pi).ngroups && !SINGLE && q.pi + 1 < b.npairs) {
            q.g = 0;
            ++q.pi;
        }
    };
    auto advance = [&](Cursor& q) {
        if (++q.sl == P(q.pi).nsl) next_group(q);
    };
    Cursor o = rest;
    if (SINGLE && full_rounds > 0) o = Cursor{0, (int)blockIdx.x, 0};

    // this thread's place: line li of the group (column col of the pair), warp w of the line, chunk k,
    // lane dq of the chunk
    const int li = threadIdx.x / b.s.per_line;
    const int w = (threadIdx.x - li * b.s.per_line) >> 5;
    const int lane = threadIdx.x & 31;
    const int dq = lane & (lanes - 1), k = w * cpw + lane / LC;
    const int col = COLS > 1 ? lane / lanes & (COLS - 1) : 0, lc = li * COLS + col;      // column of the group
    // shared memory: [staging][coefficients: nco per line][multipliers: nco][scan buffers]
    unsigned char* const base = dt_smem + (-smem_addr(dt_smem) & 127u);      // (a tensor copy's alignment)
    const T* const mine = reinterpret_cast<T*>(base) + k * b.s.slot + lc * b.s.line_off + dq * kG;
    float4* const co_mine = reinterpret_cast<float4*>(base + b.s.co_off) + lc * b.s.nco * b.s.arr;     // this column's
    float2* const mul_mine = reinterpret_cast<float2*>(base + b.s.mul_off) + lc * b.s.nco * b.s.arr;
    float4* const sb = reinterpret_cast<float4*>(base + b.s.scan_off) + li * 3 * b.s.nvg * LC + (lane & (LC - 1));
    float* const sa = reinterpret_cast<float*>(base + b.s.scan_off + b.s.lines * 3 * b.s.nvg * lanes * 16) +
                      li * 2 * b.s.nvg * LC + (lane & (LC - 1));

    auto prefetch_coef = [&](const Cursor& q, int cbuf) {
        const DtArgs& a = P(q.pi);
        const int ln = q.g * b.s.lines + lc;
        // (each column's own lanes copy its coefficients)
        for (int t = COLS > 1 ? k * lanes + dq : w * 32 + lane; t < b.s.nch * kL; t += b.s.per_line / COLS) {
            const bool in = ln < a.nlines && t < a.n;
            const size_t at = (size_t)ln * a.n + t;
            cp_async<16>(co_mine + cbuf * b.s.arr + cpos(t), in ? a.coef + at : a.coef, in);
            if (b.s.mul) cp_async<8>(mul_mine + cbuf * b.s.arr + cpos(t), in ? a.mulmap + at : a.mulmap, in);
        }
        cp_async_commit();
    };
    // the box of this chunk at the step of cursor q (lines past the pass, positions past the
    // line and disparities past the volume read as zero)
    auto load_box = [&](const Cursor& q) {
        const int d0 = q.sl * ds, sd_shift = P(q.pi).sd_shift;
        const int slab = d0 >> sd_shift, dd = d0 & ((1 << sd_shift) - 1);
        unsigned long long* bar = &full[w];
        T* dst = reinterpret_cast<T*>(base) + k * b.s.slot;
        fence_proxy_async_smem();
        mbar_expect_tx(bar, (unsigned)(b.s.slot * sizeof(T)));
        const CUtensorMap* m = &b.tmap[SINGLE ? 0 : q.pi];
        const int at = k * kL, line0 = q.g * b.s.lines;
        tma_load_4d(dst, m, dd, b.s.horiz ? at : line0, b.s.horiz ? line0 : at, slab, bar);
    };
    if (lc == 0 && dq == 0 && left > 0) load_box(o);
    if (b.s.nco == 2) prefetch_coef(o, 0);

    StepWta<lanes> wr;
    int cbuf = b.s.nco - 1;
    bool fresh = true;
    for (unsigned par = 0; left > 0; par ^= 1u, --left) {
        const DtArgs& a = P(o.pi);
        if (left == 1) griddep_launch_dependents();
        if (fresh) {                            // a new line group: its coefficients
            if (b.s.nco == 1) {                 // one buffer: filled once its readers are done
                named_barrier(1 + li, b.s.per_line);
                prefetch_coef(o, 0);
            }
            cp_async_wait<0>();
            named_barrier(1 + li, b.s.per_line);
            if (b.s.nco == 2) {                 // two: the next group's arrive during this one
                cbuf ^= 1;
                if (left > a.nsl - o.sl) {
                    Cursor nx = o;
                    next_group(nx);
                    prefetch_coef(nx, cbuf ^ 1);
                }
            }
            if constexpr (MODE == kLineWta) wr.reset();
        }
        const float4* co = co_mine + cbuf * b.s.arr + k * kCS;
        const float2* mul = b.s.mul ? mul_mine + cbuf * b.s.arr + k * kCS : nullptr;
        if (!mbar_wait(&full[w], par, kBulkWaitPolls)) {       // (a timeout is recorded, then waited
            atomicOr(b.fault, kFaultTmaWait);                   // for once more)
            mbar_wait(&full[w], par, kBulkWaitPolls);
        }
        float v[kL][4];
#pragma unroll
        for (int i = 0; i < kL; ++i) lds4(mine + i * b.s.ps, v[i]);
        if (b.s.mul) {
#pragma unroll
            for (int i = 0; i < kL; ++i) mul4<true>(mul[i].x, v[i]);
        }
        dt_group_pair<MODE != kLineWta, true, LC, kChain>(v, co, LC, b.s.scan_shift, lane, k, b.s.nvg, b.s.chain != 0, sa, sb, b.s2, mul, 1 + li, b.s.per_line,
            [&]() {
                // the box has been read: the lines' warps say so, and its loader refills it
                __syncwarp();
                if (b.s.lines > COLS && lane == 0) mbar_arrive(&empty[w]);
                if (lc == 0 && dq == 0 && left > 1) {
                    if (b.s.lines > COLS && !mbar_wait(&empty[w], par, kBulkWaitPolls)) {
                        atomicOr(b.fault, kFaultTmaWait);
                        mbar_wait(&empty[w], par, kBulkWaitPolls);
                    }
                    Cursor q = o;
                    advance(q);
                    load_box(q);
                }
            });
        const int dl = o.sl * ds + dq * kG;
        const int nvalid = max(0, min(4, a.dcount - dl));
        const int line = o.g * b.s.lines + lc;
        if constexpr (MODE == kLineWta) {
            wr.fold(v, nvalid, dl, dq);
            if (o.sl == a.nsl - 1 || left == 1) {
#pragma unroll
                for (int i = 0; i < wr.kHeld; ++i) {
                    const int pos = k * kL + wr.first(dq) + i;
                    if (line < a.nlines && pos < a.n)
                        atomicMax(a.keys + (size_t)line * a.pix_line + (size_t)pos * a.pix_pos, wta_key(wr.rv[i], wr.rd[i]));
                }
            }
        } else if (line < a.nlines && nvalid > 0) {
            const int slab = dl >> a.sd_shift, dd = dl & ((1 << a.sd_shift) - 1), npos = a.n - k * kL;
            T* q = reinterpret_cast<T*>(a.vol) + slab * a.slab_stride + line * a.line_stride + (k * kL) * a.pos_stride + dd;
            const long long es = a.pos_stride;
            if (npos >= kL) {
#pragma unroll
                for (int i = 0; i < kL; ++i) st4(q + i * es, 4, true, v[i]);
            } else {
#pragma unroll
                for (int i = 0; i < kL; ++i)
                    if (i < npos) st4(q + i * es, 4, true, v[i]);
            }
        }
        fresh = o.sl + 1 == a.nsl;
        advance(o);
    }
    cp_async_wait<0>();
}

#if !defined(DT_LINES_F16)
size_t dt_lines_layout(int dtype, bool mul, DtShape& s) {
    const int elem = dtype == 0 ? 4 : 2, ds = kG * s.lanes;
    s.mul = mul;
    s.chain = 0;
    s.per_line = s.nch * s.lanes * s.cols;
    s.nwl = s.per_line / 32;
    s.nvg = s.nch / s.scan;
    s.scan_shift = 0;
    while ((1 << s.scan_shift) < s.scan) ++s.scan_shift;
    s.slot = s.lines * kL * ds;
    s.ps = s.horiz ? ds : s.lines * ds;
    s.line_off = s.horiz ? kL * ds : ds;
    s.arr = s.nch * kCS;
    s.co_off = s.nch * s.slot * elem;
    s.mul_off = s.co_off + s.lines * s.nco * s.arr * 16;
    s.scan_off = s.mul_off + (mul ? s.lines * s.nco * s.arr * 8 : 0);
    return 128 + (size_t)s.scan_off + (size_t)s.lines * s.nvg * s.lanes * (3 * 16 + 2 * 4);   // (lines / cols sets of lanes * cols)
}
#define DT_NAME(f) f##_f32
using DtElem = float;
#else
#define DT_NAME(f) f##_f16
using DtElem = __half;
#endif

template <int MODE, int NP, int MAXT>
static const void* dt_lines_fn_t(int lanes, int cols) {
    if constexpr (std::is_same<DtElem, float>::value)
        if (cols == 2) return lanes == 4 ? (const void*)k_dt_lines<DtElem, MODE, 4, 2, NP, MAXT> : nullptr;
    return lanes == 8   ? (const void*)k_dt_lines<DtElem, MODE, 8, 1, NP, MAXT>
           : lanes == 4 ? (const void*)k_dt_lines<DtElem, MODE, 4, 1, NP, MAXT>
                        : (const void*)k_dt_lines<DtElem, MODE, 2, 1, NP, MAXT>;
}
template <int NP>
static const void* dt_lines_fn(int mode, int lanes, int cols, int threads) {
    if (mode == kLineStore) {
        if (threads <= 512) return dt_lines_fn_t<kLineStore, NP, 512>(lanes, cols);
        // (F32 store passes take blocks of at most 512 threads: a larger one has no kernel)
        if constexpr (std::is_same<DtElem, float>::value) return nullptr;
        else return dt_lines_fn_t<kLineStore, NP, kDtThreads>(lanes, cols);
    }
    return threads <= 512 ? dt_lines_fn_t<kLineWta, NP, 512>(lanes, cols) : dt_lines_fn_t<kLineWta, NP, kDtThreads>(lanes, cols);
}

cudaError_t DT_NAME(dt_lines_occupancy)(int mode, const DtShape& s, int threads, size_t smem, bool single,
                                        int* blocks_per_sm) {
    const void* fn = single ? dt_lines_fn<1>(mode, s.lanes, s.cols, threads)
                            : dt_lines_fn<kMaxBatch>(mode, s.lanes, s.cols, threads);
    if (!fn) return cudaErrorInvalidValue;
    cudaError_t e = set_max_smem(fn, smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, threads, smem);
}

cudaError_t DT_NAME(launch_dt_lines)(const DtBatch<kMaxBatch>& b, size_t smem, int mode, cudaStream_t st) {
    const int threads = b.s.lines / b.s.cols * b.s.per_line;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    launch_config(cfg, attr, dim3(b.grid), dim3(threads), smem, st, 1);
    const bool single = b.npairs == 1;
    const void* fn = single ? dt_lines_fn<1>(mode, b.s.lanes, b.s.cols, threads)
                            : dt_lines_fn<kMaxBatch>(mode, b.s.lanes, b.s.cols, threads);
    if (!fn) return cudaErrorInvalidValue;
    cudaError_t e = set_max_smem(fn, smem);
    if (e != cudaSuccess) return e;
    if (!single) return launch_batch(cfg, fn, b);
    DtBatch<1> o = first_pair<DtHead>(b);
    o.tmap[0] = b.tmap[0];
    return launch_batch(cfg, fn, o);
}

}  // namespace zncc
