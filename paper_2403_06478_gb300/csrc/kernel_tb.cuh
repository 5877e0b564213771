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
            WarpPair<C> wp;
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

// Fused score path and traceback on 16-bit lanes.
//
// Each warp aligns a pair exactly as warp16_align_kernel does, on lazy blocks,
// and keeps the band's state of every 32nd anti-diagonal in memory (TRACE).
// Then it goes back over the segments between those states: it recomputes a
// segment on the same lazy step, holds the scores of the 34 to 36 anti-diagonals
// of the few lanes the path can reach in it in shared memory, and follows the
// path through them.  No direction byte is computed or stored.
//
// What bounds it: the integer ALU pipe, twice the score kernel's work (and for
// a few thousand pairs the longest one).  The form before wrote a direction
// byte per cell from a step of 36 lane-instructions per cell (against 8 to 9 of
// the lazy step, twice) and walked back through the table one cell at a time.
// One GB300, kernel time: 20,000 ONT-like pairs 155 -> 95 ms, 2,000 56 -> 36
// ms, 20,000 reads of 150 bp 2.4 -> 1.6 ms.
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
template <class S>
struct TraceWin {
    static constexpr int C = S::P * 2, P = S::P;
    // lanes that hold 39 neighbouring slots wherever they start: a path and
    // the gaps from it move at most one slot per two anti-diagonals
    static constexpr int NL = (39 + C - 1 + C - 1) / C;
    static constexpr int ROWS = 38;               // the first segment starts at -2
    static constexpr int WORDS = NL * (ROWS + 4) * P + ROWS;
    uint32_t *rows;                               // [lane - la][row][register]
    uint32_t *st;                                 // [E, F, E2, F2][lane - la][register] leaving row rk
    int32_t *off;                                 // from a row's stored value to the score
    int32_t la, rk, st_off;
    __device__ __forceinline__ explicit TraceWin(uint4 *mem)
        : rows(reinterpret_cast<uint32_t *>(mem)), st(rows + NL * ROWS * P),
          off(reinterpret_cast<int32_t *>(st + 4 * NL * P)) {}
    __device__ __forceinline__ int32_t score(const S &s, int32_t t, int32_t r) const {
        const int32_t j = t - s.frame(r), local = j % C, i = r - rk + 1;
        return S::half_of(rows[((j / C - la) * ROWS + i) * P + local % P], local) + off[i];
    }
    // the gap state k (0 E, 1 F, 2 E2, 3 F2) leaving cell (t, rk - t)
    __device__ __forceinline__ int32_t state(const S &s, int k, int32_t t) const {
        const int32_t j = t - s.frame(rk), local = j % C;
        return S::half_of(st[k * (NL * P) + (j / C - la) * P + local % P], local) + st_off;
    }
    __device__ __forceinline__ void keep(const S &s, int32_t r, const uint32_t (&H)[P], int32_t o) {
        const int32_t l = s.lane - la;
        if (l >= 0 && l < NL) {
#pragma unroll
            for (int p = 0; p < P; ++p) rows[(l * ROWS + r - rk + 1) * P + p] = H[p];
        }
        if (s.lane == 0) off[r - rk + 1] = o;
    }
};

// Recompute anti-diagonals rk + 1 .. target (or one more) from state seg into
// the window.
template <class S>
__device__ __forceinline__ void trace_segment(S &s, TraceWin<S> &W, int32_t seg, int32_t target,
                                              const typename S::LazyConst &k, bool two, bool head, int32_t end) {
    using TW = TraceWin<S>;
    constexpr int P = S::P;
    const int32_t w = s.w, d = s.lazy_drift();
    const int32_t turn = s.cover ? INT_MAX : w - 3;
    int32_t r, rs = 0;
    bool drifting = false;
    if (seg == 0) {
#pragma unroll
        for (int p = 0; p < P; ++p)
            s.Hev[p] = s.Hod[p] = s.Eo[p] = s.E2o[p] = s.Fo[p] = s.F2o[p] = s.NEGp;
        s.base = 0;
        r = -3;
    } else {
        r = W.rk;
        drifting = s.trace_load(seg, rs);
        if (!drifting) {
            s.lazy_enter(k, two);
            rs = r;
            drifting = true;
        }
        W.keep(s, r - 1, s.Hev, s.lazy_off() - d * (r - 1 - rs));
        W.keep(s, r, s.Hod, s.lazy_off() - d * (r - rs));
        W.st_off = s.base - s.OFF - d * (r + 1 - rs);
        const int32_t l = s.lane - W.la;
        if (l >= 0 && l < TW::NL) {
#pragma unroll
            for (int p = 0; p < P; ++p) {
                W.st[l * P + p] = s.Eo[p];
                W.st[TW::NL * P + l * P + p] = s.Fo[p];
                W.st[2 * TW::NL * P + l * P + p] = two ? s.E2o[p] : s.Eo[p];
                W.st[3 * TW::NL * P + l * P + p] = two ? __vmaxu2(s.F2o[p], s.Hod[p]) : s.Fo[p];
            }
        }
    }
    while (r < target) {
        // the lazy step wherever it holds (lazy_drive), else the masked one
        const int32_t limit = r <= w ? (head ? min(turn, end) : INT_MIN) : end;
        if (r >= s.first_r() && ((r - w) & 1) && limit >= r + 2) {
            if (!drifting) {
                s.lazy_enter(k, two);
                rs = r;
                drifting = true;
            }
            const int32_t n = min((min(target + 1, limit) - r) >> 1, LAZY_PAIRS);
            typename S::LazyWin B;
            s.lazy_windows(B, r);
            const int32_t l = s.lane - W.la;
            const bool in = l >= 0 && l < TW::NL;
            const uint32_t *first = W.rows + ((in ? l : 0) * TW::ROWS + r + 1 - W.rk + 1) * P;
            LazyEdge g{__reduce_max_sync(FULL, 1), in ? 0 : -1, -(1 << 20),
                       (uint32_t)__cvta_generic_to_shared(first), 0};
            if (two) s.template lazy_block<true>(n, B, k, g);
            else s.template lazy_block<false>(n, B, k, g);
            if (s.lane < 2 * n) W.off[r + 1 + s.lane - W.rk + 1] = s.lazy_off() - d * (r + 1 + s.lane - rs);
            r += 2 * n;
        } else {
            if (drifting) {
                s.lazy_leave(k, two, r - rs);
                drifting = false;
            }
            ++r;
            s.masked_step(r);
            W.keep(s, r, ((r - w) & 1) ? s.Hod : s.Hev, s.base - s.OFF);
        }
    }
    __syncwarp();
}

// Walk back from (s.end_t, s.end_q).  Returns the number of runs.
template <class S>
__device__ __forceinline__ int32_t tb_trace(S &s, uint32_t *ops, int32_t cap) {
    using TW = TraceWin<S>;
    TW W(s.ck);
    TbRuns runs{ops, cap, 0, 0u, 0u};
    const DevParams &prm = s.prm;
    const int32_t w = s.w, g0 = s.first_r(), lane = s.lane;
    const bool two = prm.q2 != prm.q || prm.e2 != prm.e;
    const bool head = __any_sync(FULL, w >= 8 && s.lazy_head_ok());
    const int32_t L = min(s.tlen, s.qlen);
    const int32_t end = abs(s.tlen - s.qlen) <= w ? s.last_r - 1 : max(L - 2, 2 * L - 3 - w);
    const auto k = s.lazy_consts(two);
    s.blind = true;
    s.ovf = false;
    int32_t t = s.end_t, q = s.end_q;
    int32_t kind = -1, tau = 0;               // a gap of this kind under way (-1: none): see below
    while (t >= 0 && q >= 0) {
        const int32_t rc = t + q;
        const int32_t seg = rc <= g0 + 32 ? 0 : (rc - g0 - 1) >> 5;
        W.rk = seg ? g0 + 32 * seg : -2;
        W.la = min(max(t - s.frame(rc) - 19, 0) / TW::C, 32 - TW::NL);
        trace_segment(s, W, seg, rc, k, two, head, end);
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
            if (pick < 0) {                       // (cannot be; keeps the walk moving)
                runs.push(TB_OP_M, 1u, lane);
                --t;
                --q;
                kind = -1;
                continue;
            }
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

// The memory of an item has room for the direction table of every
// anti-diagonal of the pair (tlen + qlen - 1 rows of 32 C bytes), of which the
// states take three eighths, and its run scratch for tlen + qlen runs.  A pair
// that leaves the 16-bit range goes to the int32 score kernel's list and gets
// n = -1.
template <int C>
using TracePair = WarpPair16<C, false, false, false, 1, true, false, 32, true, true>;
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
