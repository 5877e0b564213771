// Traceback kernels: the CIGAR of each extension, after the score path has
// found its end cell.
//
// Two forms.  tbf16_kernel aligns and traces in one launch (below: "Fused").
// The others run after the score path: one warp takes one pair from a device
// queue (longest first, like the score kernels).  It recomputes anti-diagonals
// 0..r_end of the pair's band with a DIR variant of a score step, which writes one
// direction byte per band slot: lane L stores its C bytes of anti-diagonal r
// at table[r * 32C + L*C] with one vector store, so a warp writes a 32C-byte
// row per step, coalesced.  Two such kernels share the walk:
//   tb16_kernel  the 16-bit packed-lane step (kernel_warp16.cuh): two cells
//                per instruction, its slot frame B(r) = floor((r-w)/2), bytes
//                2p and 2p+1 of a lane from the halves of register p; a pair
//                whose scores leave the 16-bit range is marked (n = -1) and
//                the host hands it to
//   tb_kernel    the int32 step (kernel_warp.cuh): frame ceil((r-w)/2),
//                bytes in slot order.
// The table lives in HBM (a batch's tables take tens to hundreds of GB; the
// host runs the batch in waves that fit).
//
// Then the warp walks back from the end cell.  Each step moves to anti-
// diagonal r-1 or r-2 and its slot changes by at most one per anti-diagonal
// (see agatha_dev.cuh for the slot frame), so the cells of the next 32
// anti-diagonals that the path can reach lie within +-31 slots of the
// current one.  The warp loads that window (80 or 144 bytes of each of 32
// rows, one row per lane, 16-byte loads; TbLayout) into shared memory with
// one round trip to memory, and lane 0 follows the path through it; a path
// of n steps costs about n/24 memory round trips instead of n.
//
// Walk rule (the reading of the oracle's traceback): in state H the cell's
// byte says which input H took (diagonal, E, F, E2, F2; the int32 kernel
// stores the index, the 16-bit kernel one "differs" bit per input).  A diagonal step
// emits M and moves to (t-1, q-1); E/E2 emit D and move to (t-1, q); F/F2
// emit I and move to (t, q-1).  Whether the gap continues is stored at the
// cell it moves to (the Eo/Fo bits of that cell), so the state is resolved
// there before anything else: continue the gap, or take that cell's H.
// Reaching the virtual row (t = -1) adds q+1 leading insertions, the virtual
// column (q = -1) t+1 leading deletions.
//
// Runs are written end first into the pair's scratch (one uint32 per run,
// (length << 4) | op, op M=0 I=1 D=2); the gather kernel reverses them into
// the caller's order.
#pragma once

#include "kernel_warp16.cuh"

namespace agatha {

constexpr int TB_WIN_ROWS = 32;     // rows (anti-diagonals) per window

// Where a slot's byte sits and which bytes of a row the walk window holds.
// The window covers slots [ws, ws + WB) of 32 rows: every slot the path can
// reach within 31 anti-diagonals of slot jc (|slot change| <= 1 per
// anti-diagonal) when ws <= jc - 31 and ws + WB > jc + 31.  With the 16-bit
// kernel's byte order it must cover whole lanes, so ws is a multiple of WA,
// itself a multiple of C and of 16 (16-byte loads).
template <int C, bool PACKED>
struct TbLayout {
    static constexpr int32_t ROW = 32 * C;
    static constexpr int32_t P = C / 2;
    static constexpr int32_t WA = (PACKED && C > 16) ? 48 : 16;
    static constexpr int32_t WB = (PACKED && C > 16) ? 144 : 80;
    static_assert(WA % 16 == 0 && (!PACKED || WA % C == 0) && WB % WA == 0 && WB >= 62 + WA &&
                      ROW >= WB && (ROW - WB) % WA == 0,
                  "window geometry");
    __device__ __forceinline__ static int32_t frame(int32_t r, int32_t w) {
        return PACKED ? floor_div2(r - w) : ceil_div2(r - w);
    }
    __device__ __forceinline__ static int32_t byte_of(int32_t j) {
        if constexpr (!PACKED) {
            return j;
        } else {
            const int32_t lb = (j / C) * C, jl = j - lb;
            return lb + (jl < P ? 2 * jl : 2 * (jl - P) + 1);
        }
    }
    // H source (0 diagonal, 1 E, 2 F, 3 E2, 4 F2) from a byte
    __device__ __forceinline__ static int32_t source(uint32_t b) {
        if constexpr (!PACKED) {
            const int32_t s = (int32_t)(b & 7u);
            return s > 4 ? 0 : s;           // never written; keeps the walk moving
        } else {
            return (int32_t)(__ffs(~b & 0xfu) ? __ffs(~b & 0xfu) - 1 : 4);
        }
    }
    // whether the gap state k (1 E, 2 F, 3 E2, 4 F2) leaving this cell extended
    __device__ __forceinline__ static bool extended(uint32_t b, int32_t k) {
        return (b >> ((PACKED ? 3 : 2) + k)) & 1u;
    }
};

enum : uint32_t { TB_OP_M = 0, TB_OP_I = 1, TB_OP_D = 2 };

// Walk states: 0..4 = the H source being followed (diagonal, E, F, E2, F2),
// TB_H = decode H at this cell, TB_PEND + k = the gap state k (1..4) arrived
// here and its continuation bit must be read at this cell.
enum : int32_t { TB_DIAG = 0, TB_H = 5, TB_PEND = 5 };

struct TbRuns {
    uint32_t *ops;
    int32_t cap, n;
    uint32_t op, len;
    __device__ __forceinline__ void push(uint32_t o, uint32_t l, int32_t lane = 0) {
        if (len > 0 && op == o) { len += l; return; }
        if (len > 0 && n < cap && lane == 0) ops[n] = (len << 4) | op;
        if (len > 0) ++n;
        op = o;
        len = l;
    }
};

// Walk back from (t, q) through the direction table dt of a pair with band
// half-width w.  Returns the number of runs (on every lane).
template <int C, bool PACKED>
__device__ __forceinline__ int32_t tb_walk(uint8_t *__restrict__ win, const uint8_t *dt,
                                           uint32_t *ops, int32_t cap, int32_t t, int32_t q,
                                           int32_t w, int32_t lane) {
    using Lay = TbLayout<C, PACKED>;
    constexpr int32_t ROW = Lay::ROW, WB = Lay::WB, WA = Lay::WA;
    TbRuns runs{ops, cap, 0, 0u, 0u};
    int32_t st = TB_H;
    int32_t done = (t < 0 || q < 0);
    for (;;) {
        t = __shfl_sync(FULL, t, 0);
        q = __shfl_sync(FULL, q, 0);
        done = __shfl_sync(FULL, done, 0);
        if (done) break;
        // window: rows r0 - lane, slots [ws, ws + WB) around the current slot
        const int32_t r0 = t + q;
        const int32_t jc = t - Lay::frame(r0, w);
        int32_t ws = jc - (TB_WIN_ROWS - 1);
        ws = ws < 0 ? 0 : (ws / WA) * WA;
        ws = min(ws, ROW - WB);
        const int32_t rk = r0 - lane;
        if (rk >= 0) {
            const uint4 *src = reinterpret_cast<const uint4 *>(dt + (int64_t)rk * ROW + ws);
            uint4 *dst = reinterpret_cast<uint4 *>(win + lane * WB);
#pragma unroll
            for (int i = 0; i < WB / 16; ++i) dst[i] = __ldcg(src + i);
        }
        __syncwarp();
        if (lane == 0) {
            for (;;) {
                if (t < 0 || q < 0) {
                    if (t < 0 && q >= 0) runs.push(TB_OP_I, (uint32_t)(q + 1));
                    if (q < 0 && t >= 0) runs.push(TB_OP_D, (uint32_t)(t + 1));
                    done = 1;
                    break;
                }
                const int32_t r = t + q;
                if (r < r0 - (TB_WIN_ROWS - 1)) break;          // next window
                const int32_t j = Lay::byte_of(t - Lay::frame(r, w)) - ws;   // in [0, WB)
                const uint32_t b = win[(r0 - r) * WB + j];
                if (st > TB_PEND)                                 // a gap arrived here
                    st = Lay::extended(b, st - TB_PEND) ? st - TB_PEND : TB_H;
                if (st == TB_H) st = Lay::source(b);
                if (st == TB_DIAG) {
                    runs.push(TB_OP_M, 1u); --t; --q; st = TB_H;
                } else if (st & 1) {                              // E, E2: a step in t
                    runs.push(TB_OP_D, 1u); --t; st += TB_PEND;
                } else {                                          // F, F2: a step in q
                    runs.push(TB_OP_I, 1u); --q; st += TB_PEND;
                }
            }
        }
        __syncwarp();
    }
    if (lane == 0) runs.push(0xfu, 1u);                           // flush the last run
    return __shfl_sync(FULL, runs.n, 0);
}

template <int C>
__global__ void __launch_bounds__(WARP_BLOCK_THREADS)
tb_kernel(const DevBatch *__restrict__ d_batch, const TbItem *__restrict__ items, int32_t n_items,
          int32_t *head, uint8_t *dir, uint32_t *ops, int32_t *n_cigar) {
    __shared__ __align__(16) uint8_t win[WARP_BLOCK_THREADS / 32][TB_WIN_ROWS * TbLayout<C, false>::WB];
    const DevBatch B = *d_batch;
    const int lane = threadIdx.x & 31;
    uint8_t *my_win = win[threadIdx.x >> 5];
    for (;;) {
        int32_t k = 0;
        if (lane == 0) k = atomicAdd(head, 1);
        k = __shfl_sync(FULL, k, 0);
        if (k >= n_items) break;
        const TbItem it = items[k];
        uint8_t *dt = dir + it.dir_off;
        {
            WarpPair<C, true> wp;
            wp.run_dir(B, it.pair, lane, it.end_t + it.end_q, dt);
        }
        __syncwarp();   // the table rows this warp wrote are read by other lanes
        const int32_t w = effective_w(B.params.w, B.t_len[it.pair], B.q_len[it.pair]);
        const int32_t n = tb_walk<C, false>(my_win, dt, ops + it.ops_off, it.end_t + it.end_q + 2,
                                            it.end_t, it.end_q, w, lane);
        if (lane == 0) n_cigar[it.pair] = n;
    }
}

// The same on 16-bit lanes; MINB resident blocks per SM as for the score kernel.
template <int C, int MINB>
__global__ void __launch_bounds__(WARP_BLOCK_THREADS, MINB)
tb16_kernel(const DevBatch *__restrict__ d_batch, const TbItem *__restrict__ items, int32_t n_items,
            int32_t *head, uint8_t *dir, uint32_t *ops, int32_t *n_cigar) {
    __shared__ Cold16 cold[WARP_BLOCK_THREADS / 32];
    __shared__ __align__(16) uint8_t win[WARP_BLOCK_THREADS / 32][TB_WIN_ROWS * TbLayout<C, true>::WB];
    const DevBatch B = *d_batch;
    const int lane = threadIdx.x & 31;
    uint8_t *my_win = win[threadIdx.x >> 5];
    for (;;) {
        int32_t k = 0;
        if (lane == 0) k = atomicAdd(head, 1);
        k = __shfl_sync(FULL, k, 0);
        if (k >= n_items) break;
        const TbItem it = items[k];
        uint8_t *dt = dir + it.dir_off;
        bool ok;
        {
            WarpPair16<C, (MINB < 4 && C <= 16) || MINB < 3, false, true> wp(cold[threadIdx.x >> 5]);
            ok = wp.run_dir(B, it.pair, lane, it.end_t + it.end_q, dt);
        }
        if (!ok) {                                  // scores left the 16-bit range
            if (lane == 0) n_cigar[it.pair] = -1;
            continue;
        }
        __syncwarp();
        const int32_t w = effective_w(B.params.w, B.t_len[it.pair], B.q_len[it.pair]);
        const int32_t n = tb_walk<C, true>(my_win, dt, ops + it.ops_off, it.end_t + it.end_q + 2,
                                           it.end_t, it.end_q, w, lane);
        if (lane == 0) n_cigar[it.pair] = n;
    }
}

// Fused score path and traceback on 16-bit lanes, with direction bytes: for the
// scorings of kernel_step.cuh, and for steps too steep for the kept states below
// (TRACE_STEP_MAX).  Each warp aligns a pair as warp16_step_kernel does, writing
// the direction bytes of every anti-diagonal, then walks back from the end cell
// it found.  The table of an item has room for every anti-diagonal of the pair
// and its run scratch for tlen + qlen runs; a pair that leaves the 16-bit range
// goes to the int32 score kernel's list and gets n = -1.  Against kept states
// whose score path finds no room for lazy blocks: 2,666 pairs of 600 bp at w =
// 100, ONT scoring at a threshold of 30, 1.31 ms a call and 2.74.
template <int C, int MINB>
__global__ void __launch_bounds__(WARP_BLOCK_THREADS, MINB)
tbs16_kernel(const DevBatch *__restrict__ d_batch, const TbItem *__restrict__ items, int32_t n_items,
             int32_t *head, uint8_t *dir, uint32_t *ops, int32_t *n_cigar) {
    __shared__ Cold16 cold[WARP_BLOCK_THREADS / 32];
    __shared__ __align__(16) uint8_t win[WARP_BLOCK_THREADS / 32][TB_WIN_ROWS * TbLayout<C, true>::WB];
    const DevBatch B = *d_batch;
    const int lane = threadIdx.x & 31;
    uint8_t *my_win = win[threadIdx.x >> 5];
    for (;;) {
        int32_t k = 0;
        if (lane == 0) k = atomicAdd(head, 1);
        k = __shfl_sync(FULL, k, 0);
        if (k >= n_items) break;
        const TbItem it = items[k];
        uint8_t *dt = dir + it.dir_off;
        bool ok;
        int32_t et, eq;
        {
            // without the deferred arg-max (DEFER): its saved registers cost
            // more here, beside the direction bits, than the searches they save
            // (20,000 ONT-like pairs: 171 against 179 ms)
            WarpPair16<C, (MINB < 4 && C <= 16) || MINB < 3, false, true, true> wp(cold[threadIdx.x >> 5]);
            ok = wp.run(B, it.pair, lane, true, dt);
            et = wp.end_t;
            eq = wp.end_q;
        }
        if (!ok) {                                  // the int32 score kernel takes it
            if (lane == 0) {
                const int32_t slot = atomicAdd(&B.counters[CTR_NOVF], 1);
                B.ovf_list[slot] = it.pair;
                n_cigar[it.pair] = -1;
            }
            continue;
        }
        if (et < 0 || eq < 0) {                     // the maximum is the origin
            if (lane == 0) n_cigar[it.pair] = 0;
            continue;
        }
        __syncwarp();   // the table rows this warp wrote are read by other lanes
        const int32_t w = effective_w(B.params.w, B.t_len[it.pair], B.q_len[it.pair]);
        const int32_t n = tb_walk<C, true>(my_win, dt, ops + it.ops_off, et + eq + 2, et, eq, w, lane);
        if (lane == 0) n_cigar[it.pair] = n;
    }
}

template <int C, int MINB>
cudaError_t launch_tbs16_c(const DevBatch *d_batch, const TbItem *items, int32_t n_items, int32_t *head,
                           uint8_t *dir, uint32_t *ops, int32_t *n_cigar, int n_blocks, cudaStream_t s) {
    tbs16_kernel<C, MINB><<<n_blocks, WARP_BLOCK_THREADS, 0, s>>>(d_batch, items, n_items, head, dir, ops,
                                                                  n_cigar);
    return cudaGetLastError();
}

template <int C, int MINB>
int occupancy_tbs16_c() {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, tbs16_kernel<C, MINB>, WARP_BLOCK_THREADS, 0) !=
        cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

// Fused score path and traceback on 16-bit lanes, from kept states.
//
// Each warp aligns a pair exactly as warp16_align_kernel does, on lazy blocks,
// and keeps the band's state of every 32nd anti-diagonal in memory (TRACE).
// Then it goes back over the segments between those states: it recomputes the
// 64 slots of a segment that the path can depend on by the same lazy step, two
// slots per lane, holds their scores in shared memory and follows the path
// through them.  No direction byte is computed or stored.
//
// What bounds it: the score path's integer ALU pipe, and for a few thousand
// pairs the longest one, whose 32 anti-diagonals of a segment take 4,500 clocks
// (a chain of a shuffle and seven operations each) and the walk through them
// 750 to 1,300.  The first form wrote a direction byte per cell from a step of
// 36 lane-instructions per cell (against 8 to 9 of the lazy step) and walked
// back through the table one cell at a time; the second kept states but took
// every segment on the whole frame.  One GB300, kernel time of the three:
// 20,000 ONT-like pairs 155, 95, 65 ms, 2,000 56, 29.6, 21.8, 20,000 of Pareto
// lengths at w = 750 -, 94, 56, 20,000 reads of 150 bp 2.4, 1.11, 1.14.
//
// The path from scores alone (the rules at the top of this file): a diagonal
// step is taken wherever H equals the diagonal's H plus the substitution, so
// the lanes test the coming diagonal cells at once and the run is as long as
// the first that fails.  There, H came from E iff some cell l steps back in t
// has H - (q + e l) equal to it, from F iff one l steps back in q, from E2, F2
// the same with the second piece; the gap's length is the smallest such l
// (opening is preferred to extending on ties), found by the lanes at once.
// Past the segment's start the state E (F, E2, F2) kept there stands for all
// longer gaps: a gap that equals only that one continues in the segment
// before, where the smallest l is looked for that opens it.
// The scores of a segment's anti-diagonals on 64 slots around the path: a path
// and the gaps from it move at most one slot per two anti-diagonals (39 slots
// would hold them), and what the window's ends get wrong comes in as slowly.
template <class S>
struct TraceWin {
    static constexpr int C = S::P * 2, P = S::P;
    static constexpr int ROWS = 38;               // the first segment starts at -2
    static constexpr int WORDS = 32 * (ROWS + 4) + ROWS;
    uint32_t *rows;                               // [row][32], two slots per word
    uint32_t *st;                                 // [E, F, E2, F2][32] leaving row rk
    int32_t *off;                                 // from a row's stored value to the score
    int32_t jb, rk, st_off;                       // the window's first slot, even; the segment's start
    __device__ __forceinline__ explicit TraceWin(uint4 *mem)
        : rows(reinterpret_cast<uint32_t *>(mem)), st(rows + 32 * ROWS), off(reinterpret_cast<int32_t *>(st + 4 * 32)) {}
    __device__ __forceinline__ static int32_t at(const uint32_t *row, int32_t j) {
        return reinterpret_cast<const uint16_t *>(row)[j];
    }
    __device__ __forceinline__ int32_t score(const S &s, int32_t t, int32_t r) const {
        const int32_t i = r - rk + 1;
        return at(rows + 32 * i, t - s.frame(r) - jb) + off[i];
    }
    // the gap state k (0 E, 1 F, 2 E2, 3 F2) leaving cell (t, rk - t)
    __device__ __forceinline__ int32_t state(const S &s, int k, int32_t t) const {
        return at(st + 32 * k, t - s.frame(rk) - jb) + st_off;
    }
    // the window's slots of a whole frame's registers
    __device__ __forceinline__ void put(const S &s, uint32_t *row, const uint32_t (&x)[P]) const {
        uint16_t *d = reinterpret_cast<uint16_t *>(row);
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int32_t lo = s.j0 + p - jb, hi = lo + P;
            if ((uint32_t)lo < 64u) d[lo] = (uint16_t)x[p];
            if ((uint32_t)hi < 64u) d[hi] = (uint16_t)(x[p] >> 16);
        }
    }
    __device__ __forceinline__ void keep(const S &s, int32_t r, const uint32_t (&H)[P], int32_t o) const {
        put(s, rows + 32 * (r - rk + 1), H);
        if (s.lane == 0) off[r - rk + 1] = o;
    }
};

// This lane's two slots of the six arrays of state `entry`: neighbouring
// registers p, p + 1 of lane a / C, the same half of both.
template <class S>
__device__ __forceinline__ void trace_gather(const S &s, const TraceWin<S> &W, const uint4 *entry, uint32_t (&x)[6]) {
    constexpr int P = S::P, C = S::P * 2;
    const int32_t a = W.jb + 2 * s.lane, local = a % C, p = local % P;
    const uint32_t sel = local < P ? 0x5410u : 0x7632u;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const int32_t word = i * P + p;
        const uint2 v = *reinterpret_cast<const uint2 *>(
            reinterpret_cast<const uint32_t *>(entry + (word >> 2) * 32 + a / C) + (word & 3));
        x[i] = prmt(v.x, v.y, sel);
    }
}
// n pairs of anti-diagonals after rk on the window alone, from the arrays x
// (H of rk - 1 and rk, E, F, E2, F2; drifting since rs): the lazy step
// (WarpPair16::lazy_step) with two slots per lane.  The cuts at slots 0 and
// w + 1 act where the window holds them; at its other ends garbage enters, one
// slot per two anti-diagonals.  Cells past the table's last row and column
// come out wrong and feed none of the table's.
template <class S, bool TWO>
__device__ __forceinline__ void trace_narrow(const S &s, TraceWin<S> &W, const uint32_t (&x)[6], int32_t rk, int32_t rs,
                                             int32_t n, const typename S::LazyConst &k) {
    const int32_t a = W.jb + 2 * s.lane, w1 = s.w + 1 - a, lane = s.lane;
    uint32_t Hev = x[0], Hod = x[1], Eo = x[2], Fo = x[3], E2o = x[4], F2o = x[5];
    const uint32_t NEG = s.NEGp;
    const uint32_t low = a == 0 ? 0x0000ffffu : 0u;                      // slot 0
    const uint32_t top = w1 == 0 ? 0x0000ffffu : (w1 == 1 ? 0xffff0000u : 0u);   // slot w + 1
    const uint32_t past = lane == 31 && w1 == 2 ? 0xffff0000u : 0u;      // it would come in next
    const int32_t B = s.frame(rk), tb = B + a + s.tph, qb = rk - B - a + s.qph + 1;    // (see lazy_windows)
    uint32_t t0 = load_rel(s.tp, s.tspan, tb), t1 = load_rel(s.tp, s.tspan, tb + 16);
    uint32_t q0 = rev2_32(load_rel(s.qp, s.qspan, qb)), q1 = rev2_32(load_rel(s.qp, s.qspan, qb - 16));
    uint32_t *row = W.rows + 32 * (rk - W.rk) + lane;
    const int32_t d = s.lazy_drift();
    if (rk == W.rk) {
        row[0] = Hev;
        row[32] = Hod;
        W.st[lane] = Eo;
        W.st[32 + lane] = Fo;
        W.st[64 + lane] = TWO ? E2o : Eo;
        W.st[96 + lane] = TWO ? __vmaxu2(F2o, Hod) : Fo;
        W.st_off = s.base - s.OFF - d * (rk + 1 - rs);
        if (lane < 2) W.off[lane] = s.lazy_off() - d * (rk - 1 + lane - rs);
    }
    if (lane < 2 * n) W.off[rk - W.rk + 2 + lane] = s.lazy_off() - d * (rk + 1 + lane - rs);
    const auto score = [&](uint32_t Hd, uint32_t E, uint32_t F, uint32_t E2, uint32_t F2, uint32_t &hoe) {
        const uint32_t m = t0 ^ q1, mb = (((m | (m >> 1)) & 5u) * 0x4001u) & 0x10001u;
        const uint32_t X = __viaddmax_u16x2(mb * s.NABs + Hd, k.A, E);
        const uint32_t H = TWO ? __vmaxu2(__vimax3_u16x2(X, F, E2), F2) : __vmaxu2(X, F);
        hoe = H - k.OE;
        return H - k.H2;
    };
#pragma unroll 1
    for (; n > 0; --n) {
        row += 64;
        t0 = __funnelshift_r(t0, t1, 2);
        t1 >>= 2;
        uint32_t F = mux(past, NEG, prmt(Fo, __shfl_down_sync(FULL, Fo, 1), 0x5432)), F2 = 0, hoe;
        if constexpr (TWO) {
            const uint32_t y = __vmaxu2(F2o, Hod);
            F2 = mux(past, NEG, prmt(y, __shfl_down_sync(FULL, y, 1), 0x5432));
        }
        Hev = score(Hev, Eo, F, E2o, F2, hoe);
        Eo = TWO ? __viaddmax_u16x2(Eo, k.NE, hoe) : __vmaxu2(Eo, Hev);
        Fo = TWO ? __viaddmax_u16x2(F, k.NE, hoe) : __vmaxu2(F, Hev);
        if constexpr (TWO) F2o = __vmaxu2(F2, Hev);
        row[0] = Hev;
        q1 = __funnelshift_l(q0, q1, 2);
        q0 <<= 2;
        uint32_t E = prmt(__shfl_up_sync(FULL, Eo, 1), Eo, 0x5432), E2 = 0;
        if constexpr (TWO) {
            const uint32_t y = __vmaxu2(E2o, Hev);
            E2 = prmt(__shfl_up_sync(FULL, y, 1), y, 0x5432);
        }
        Hod = score(Hod, E, Fo, E2, F2o, hoe);
        Eo = mux(low, NEG, TWO ? __viaddmax_u16x2(E, k.NE, hoe) : __vmaxu2(E, Hod));
        Fo = mux(top, NEG, TWO ? __viaddmax_u16x2(Fo, k.NE, hoe) : __vmaxu2(Fo, Hod));
        if constexpr (TWO) {
            E2o = mux(low, NEG, __vmaxu2(E2, Hod));
            F2o = mux(top, NEG, F2o);
            Hod = mux(top, NEG, Hod);
        }
        row[32] = Hod;
    }
}

// Recompute anti-diagonals rk + 1 .. target (or one more) from state seg into
// the window: on its own slots, after the masked step on the whole frame at
// the table's corner and where the virtual cells leave the band.
template <class S>
__device__ __forceinline__ void trace_segment(S &s, TraceWin<S> &W, int32_t seg, int32_t target,
                                              const typename S::LazyConst &k, bool two, bool head) {
    constexpr int P = S::P;
    const int32_t w = s.w, turn = !head ? 0 : (s.cover ? INT_MAX : w - 3);
    const auto runs_lazy = [&](int32_t r) { return r > w || ((target - r + 1) & ~1) <= turn - r; };
    int32_t r = -3, rs = 0;
    uint32_t x[6];
    bool drifting = false, narrow = false;
    if (seg == 0) {
#pragma unroll
        for (int p = 0; p < P; ++p)
            s.Hev[p] = s.Hod[p] = s.Eo[p] = s.E2o[p] = s.Fo[p] = s.F2o[p] = s.NEGp;
        s.base = 0;
    } else {
        r = W.rk;
        drifting = s.trace_meta(seg, rs);
        narrow = __any_sync(FULL, runs_lazy(r));
        if (narrow) {
            trace_gather(s, W, s.trace_entry(seg), x);
        } else {
            s.trace_load(seg);
            if (drifting) s.lazy_leave(k, two, r - rs);
            drifting = false;
            W.keep(s, r - 1, s.Hev, s.base - s.OFF);
            W.keep(s, r, s.Hod, s.base - s.OFF);
            W.put(s, W.st, s.Eo);
            W.put(s, W.st + 32, s.Fo);
            W.put(s, W.st + 64, s.E2o);
            W.put(s, W.st + 96, s.F2o);
            W.st_off = s.base - s.OFF;
        }
    }
    if (!narrow) {
        while (r < target) {
            if (r >= s.first_r() && ((r - w) & 1) && r + 6 <= target && runs_lazy(r)) {
                uint32_t *tmp = W.rows + 32 * (r - W.rk + 2);      // six of the rows to come
                __syncwarp();
                W.put(s, tmp, s.Hev);
                W.put(s, tmp + 32, s.Hod);
                W.put(s, tmp + 64, s.Eo);
                W.put(s, tmp + 96, s.Fo);
                W.put(s, tmp + 128, s.E2o);
                W.put(s, tmp + 160, s.F2o);
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 6; ++i) x[i] = tmp[32 * i + s.lane];
                __syncwarp();
                narrow = true;
                break;
            }
            ++r;
            s.masked_step(r);
            W.keep(s, r, ((r - w) & 1) ? s.Hod : s.Hev, s.base - s.OFF);
        }
    }
    if (__any_sync(FULL, narrow)) {
        if (!drifting) {                             // as lazy_enter
            x[0] -= k.H2 + k.D;
            x[1] -= k.H2;
#pragma unroll
            for (int i = 2; i < 6; ++i) x[i] += k.D;
            rs = r;
        }
        const int32_t n = (target - r + 1) >> 1;
        if (two) trace_narrow<S, true>(s, W, x, r, rs, n, k);
        else trace_narrow<S, false>(s, W, x, r, rs, n, k);
    }
    __syncwarp();
}

// Walk back from (s.end_t, s.end_q).  Returns the number of runs, or -1 if no
// move explains a score: the pair is then traced on int32 lanes like one that left
// the 16-bit range, rather than by a path that is not its own.
template <class S>
__device__ __forceinline__ int32_t tb_trace(S &s, uint32_t *ops, int32_t cap) {
    using TW = TraceWin<S>;
    TW W(s.ck);
    TbRuns runs{ops, cap, 0, 0u, 0u};
    const DevParams &prm = s.prm;
    const int32_t w = s.w, g0 = s.first_r(), lane = s.lane;
    const bool two = prm.q2 != prm.q || prm.e2 != prm.e;
    const bool head = __any_sync(FULL, w >= 8 && s.lazy_head_ok());
    const auto k = s.lazy_consts(two);
    s.blind = true;
    s.ovf = false;
    int32_t t = s.end_t, q = s.end_q;
    int32_t kind = -1, tau = 0;               // a gap of this kind under way (-1: none): see below
    while (t >= 0 && q >= 0) {
        const int32_t rc = t + q;
        const int32_t seg = rc <= g0 + 32 ? 0 : (rc - g0 - 1) >> 5;
        W.rk = seg ? g0 + 32 * seg : -2;
        W.jb = min(max(t - s.frame(rc) - 32, 0) & ~1, S::NS - 64);
        trace_segment(s, W, seg, rc, k, two, head);
        while (t >= 0 && q >= 0 && t + q > W.rk) {
            int32_t r = t + q;
            if (kind < 0) {
                // lane i: whether cell (t - i, q - i) took the diagonal
                const int32_t ti = t - lane, qi = q - lane, ri = r - 2 * lane;
                bool ok = false;
                if (ti >= 0 && qi >= 0 && ri > W.rk) {
                    const int32_t tb = ti + s.tph, qb = qi + s.qph;
                    const uint32_t x = (__ldg(s.tp + (tb >> 4)) >> (2 * (tb & 15))) ^
                                       (__ldg(s.qp + (qb >> 4)) >> (2 * (qb & 15)));
                    const int32_t m = max(ti, qi);
                    const int32_t from = ti && qi ? W.score(s, ti - 1, ri - 2) : (m ? -gap_cost(prm, m) : 0);
                    ok = W.score(s, ti, ri) == from + ((x & 3u) ? -prm.b : prm.a);
                }
                const uint32_t miss = ~__ballot_sync(FULL, ok);
                const int32_t n = miss ? __ffs(miss) - 1 : 32;
                if (n > 0) {
                    runs.push(TB_OP_M, (uint32_t)n, lane);
                    t -= n;
                    q -= n;
                    r -= 2 * n;
                    if (t < 0 || q < 0 || r <= W.rk) break;
                }
            }
            // a gap: H (or, under way, its state one step on) equals the score
            // l steps back less the gap's cost
            const int32_t want = kind < 0 ? W.score(s, t, r) : tau;
            const int32_t D = r - W.rk;
            uint64_t hit[4] = {0, 0, 0, 0};       // bit l - 1: the gap of length l
            for (int32_t l = lane + 1;; l += 32) {
                // (only the first segment has more than 32 anti-diagonals)
                constexpr int32_t OUT = -(1 << 29);
                const int32_t rl = r - l, te = t - l, qf = q - l;
                int32_t he = OUT, hf = OUT;
                if (rl >= W.rk) {
                    if (te >= 0) { if (te - q >= -w) he = W.score(s, te, rl); }
                    else if (te == -1 && q <= w) he = -gap_cost(prm, q + 1);
                    if (qf >= 0) { if (t - qf <= w) hf = W.score(s, t, rl); }
                    else if (qf == -1 && t <= w) hf = -gap_cost(prm, t + 1);
                }
                const int32_t c1 = want + prm.q + prm.e * l, c2 = want + prm.q2 + prm.e2 * l;
                const int sh = l > 32 ? 32 : 0;
                hit[0] |= (uint64_t)__ballot_sync(FULL, he == c1) << sh;
                hit[1] |= (uint64_t)__ballot_sync(FULL, hf == c1) << sh;
                hit[2] |= (uint64_t)__ballot_sync(FULL, he == c2) << sh;
                hit[3] |= (uint64_t)__ballot_sync(FULL, hf == c2) << sh;
                if (sh || D <= 32) break;
            }
            int32_t at = 0, pick = -1, value = 0;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (pick >= 0 || (kind >= 0 && kind != c)) continue;
                if (hit[c]) {
                    pick = c;
                    at = __ffsll((long long)hit[c]);
                } else if (W.rk > 0) {
                    // the state leaving the segment's first anti-diagonal, if
                    // the gap reaches it inside the table and the band
                    const int32_t ts = (c & 1) ? t : t - D, qs = W.rk - ts;
                    if (ts >= 0 && qs >= 0 && ts - qs <= w && qs - ts <= w) {
                        value = W.state(s, c, ts);
                        if (__any_sync(FULL, value - (c < 2 ? prm.e : prm.e2) * (D - 1) == want)) pick = c;
                    }
                }
            }
            const int32_t n = at ? at : D;
            if (pick < 0) return -1;              // (cannot be)
            runs.push((pick & 1) ? TB_OP_I : TB_OP_D, (uint32_t)n, lane);
            if (pick & 1) q -= n;
            else t -= n;
            kind = at ? -1 : pick;
            tau = value + (pick < 2 ? prm.e : prm.e2);
        }
        __syncwarp();                             // the window is written again
    }
    if (t < 0 && q >= 0) runs.push(TB_OP_I, (uint32_t)(q + 1), lane);
    if (q < 0 && t >= 0) runs.push(TB_OP_D, (uint32_t)(t + 1), lane);
    runs.push(0xfu, 1u, lane);                    // flush the last run
    return runs.n;
}

// The memory of an item has room for the states of every anti-diagonal of the pair
// (trace_bytes), and its run scratch for tlen + qlen runs.  A pair that leaves the
// 16-bit range goes to the int32 score kernel's list and gets n = -1.
template <int C>
using TracePair = WarpPair16<C, false, false, false, true, 1, true, false, 32, true, true>;
template <int C>
__host__ __device__ constexpr int tbf16_warp_smem() {                 // 16-byte words of a warp
    using S = TracePair<C>;
    constexpr int a = 2 * S::CKV * 32 + S::RING / 4, b = (TraceWin<S>::WORDS + 3) / 4;
    return a > b ? a : b;
}

// One block per SM of MINB warps per scheduler; TierQueue hands out the items,
// with the slot's counters as its heads.
template <int C, int MINB>
__global__ void __launch_bounds__(WARP_BLOCK_THREADS * MINB, 1)
tbf16_kernel(const DevBatch *__restrict__ d_batch, const TbItem *__restrict__ items, int32_t n_items,
             uint8_t *states, uint32_t *ops, int32_t *n_cigar) {
    __shared__ Cold16 cold[WARP_BLOCK_THREADS * MINB / 32];
    __shared__ TierQueue q;
    __shared__ int32_t first[4], place[WARP_BLOCK_THREADS * MINB / 32];
    extern __shared__ uint4 lazy_smem[];
    const DevBatch B = *d_batch;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tier = warp >> 2;
    const int32_t units = 4 * (int32_t)gridDim.x;
    if (threadIdx.x == 0) q.open(&B.counters[CTR_HEAD], 0, n_items, units);
    if (lane == 0) place[warp] = q.first_place(tier);
    __syncthreads();
    int32_t k = INT_MAX;
    if (tier == 0 && lane == 0) first[warp] = k = q.next(place[warp]);
    __syncthreads();
    if (tier > 0) {
        const auto steps = [&](int32_t i) { return items[i].end_t + items[i].end_q + 1; };
        if (tier_crowded(q, first[warp & 3], tier, units, warp16_lone(C), steps)) k = n_items;
        else if (lane == 0) k = q.next(place[warp]);
    }
    for (;;) {
        k = __reduce_min_sync(FULL, k);
        if (k >= n_items) break;
        const TbItem it = items[k];
        k = INT_MAX;
        TracePair<C> wp(cold[warp]);
        wp.ck = lazy_smem + warp * tbf16_warp_smem<C>();
        int32_t n = -1;
        if (!wp.run(B, it.pair, lane, true, states + it.dir_off)) {    // the int32 score kernel takes it
            if (lane == 0) {
                const int32_t slot = atomicAdd(&B.counters[CTR_NOVF], 1);
                B.ovf_list[slot] = it.pair;
            }
        } else {
            __syncwarp();
            n = wp.end_t < 0 || wp.end_q < 0 ? 0      // the maximum is the origin
                                             : tb_trace(wp, ops + it.ops_off, wp.end_t + wp.end_q + 2);
        }
        if (lane == 0) {
            n_cigar[it.pair] = n;
            k = q.next(place[warp]);
        }
    }
}

template <int C, int MINB>
cudaError_t launch_tbf16_c(const DevBatch *d_batch, const TbItem *items, int32_t n_items,
                           uint8_t *dir, uint32_t *ops, int32_t *n_cigar, int n_blocks, cudaStream_t s) {
    tbf16_kernel<C, MINB><<<n_blocks, WARP_BLOCK_THREADS * MINB,
                            (WARP_BLOCK_THREADS * MINB / 32) * 16 * tbf16_warp_smem<C>(), s>>>(
        d_batch, items, n_items, dir, ops, n_cigar);
    return cudaGetLastError();
}

template <int C, int MINB>
int occupancy_tbf16_c() {
    int nb = 0;
    constexpr int smem = (WARP_BLOCK_THREADS * MINB / 32) * 16 * tbf16_warp_smem<C>();
    if (cudaFuncSetAttribute(tbf16_kernel<C, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, tbf16_kernel<C, MINB>, WARP_BLOCK_THREADS * MINB, smem) !=
            cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

template <int C>
cudaError_t launch_tb_c(const DevBatch *d_batch, const TbItem *items, int32_t n_items, int32_t *head,
                        uint8_t *dir, uint32_t *ops, int32_t *n_cigar, int n_blocks, cudaStream_t s) {
    tb_kernel<C><<<n_blocks, WARP_BLOCK_THREADS, 0, s>>>(d_batch, items, n_items, head, dir, ops, n_cigar);
    return cudaGetLastError();
}

template <int C>
int occupancy_tb_c() {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, tb_kernel<C>, WARP_BLOCK_THREADS, 0) !=
        cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

template <int C, int MINB>
cudaError_t launch_tb16_c(const DevBatch *d_batch, const TbItem *items, int32_t n_items, int32_t *head,
                          uint8_t *dir, uint32_t *ops, int32_t *n_cigar, int n_blocks, cudaStream_t s) {
    tb16_kernel<C, MINB><<<n_blocks, WARP_BLOCK_THREADS, 0, s>>>(d_batch, items, n_items, head, dir, ops,
                                                                 n_cigar);
    return cudaGetLastError();
}

template <int C, int MINB>
int occupancy_tb16_c() {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, tb16_kernel<C, MINB>, WARP_BLOCK_THREADS, 0) !=
        cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

}  // namespace agatha
