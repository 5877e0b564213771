// The course of a pair on lazy blocks: which anti-diagonals run without a
// maximum and a termination test, and how the exact global maximum and its
// cell are found all the same.  Shared by the 16-bit kernel (kernel_warp16.cuh)
// and the int32 kernel (kernel_lazy32.cuh), which supply the lanes: the masked
// step, the lazy step, checkpoints and maxima.
#pragma once

#include <climits>

#include "kernel_warp.cuh"

namespace agatha {

constexpr int LAZY_PAIRS = 16;      // anti-diagonal pairs of one word of each sequence

struct Cold16 {
    int32_t mqe, mqe_t, mte, mte_q, gscore;
    int32_t gt, gq;               // cell of the global maximum
    int32_t Dp, LOWCHK, kint;     // step bound, lowest allowed score, rebase interval
    // the two checkpoints of the lazy blocks: anti-diagonal, start of its
    // drift, base, and the steps then left to the next rebase
    int32_t ck_r[2], ck_rs[2], ck_base[2], ck_u0[2];
};

// Where the last row's and column's cells sit, as slots of this lane (on: the
// block may hold such cells; uniform), and the ring's shared address.
struct LazyEdge { int32_t on, dt, dq; uint32_t ring; };

// Pairs of anti-diagonals the next block may hold: n, 16, 8, 4 or 2 (0: none) such
// that no anti-diagonal of it can fire the Z-drop test.  g, m, mu: an upper
// bound of the global maximum, the maximum of the last two anti-diagonals,
// and that maximum with the virtual cells.  k anti-diagonals on, no score is
// above mu + a ceil(k/2), and the maximum is at least m - o - c ceil(k/2):
// away from the last row and column (c = b, o = min(q+e, q2+e2)) the cell
// of m continues along its diagonal, after one gap step if the parity asks
// for it; near them (c = max(b, 2e), o = q+e + q + c) it may have to go on
// along the edge by a gap, towards the corner, which lies in the band.
__device__ __forceinline__ int32_t lazy_span(const DevParams &prm, int32_t n, int32_t g, int32_t m, int32_t mu,
                                             int32_t o, int32_t c) {
    if (prm.zdrop < 0) return n;
#pragma unroll 1
    while (n > 0 && max(g - m, mu - m + prm.a * n) + o + c * n > prm.zdrop)
        n = n > 16 ? 16 : (n > 8 ? 8 : (n > 4 ? 4 : (n > 2 ? 2 : 0)));
    return n;
}

// The best score on the last row and column of anti-diagonals r0 + 1 ..
// r0 + 2n (lane i takes the i-th of them) from the ring.  off: from a
// drifting h of anti-diagonal r0 to its true score.
template <class S>
__device__ __forceinline__ void lazy_edges(S &s, int32_t r0, int32_t n, int32_t off, int32_t d) {
    __syncwarp();
    s.group_sync();
    const int32_t r = r0 + 1 + s.lane, B = floor_div2(r - s.w);
    off -= d * (1 + s.lane);
    const int32_t lo = max(max(0, r - s.qlen + 1), ceil_div2(r - s.w));
    const int32_t hi = min(min(s.tlen - 1, r), floor_div2(r + s.w));
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int32_t t = c == 0 ? s.tlen - 1 : r - s.qlen + 1;
        int32_t v = INT_MIN;
        if (s.lane < 2 * n && lo <= t && t <= hi) v = s.ring_value(c, s.lane, t - B) + off;
        const int32_t m = __reduce_max_sync(FULL, v);
        if (m > (c == 0 ? s.cold.mte : s.cold.mqe)) {
            const int32_t at = r0 + 1 + __ffs(__ballot_sync(FULL, v == m)) - 1;
            if (s.leader()) {
                if (c == 0) { s.cold.mte = m; s.cold.mte_q = at - (s.tlen - 1); }
                else { s.cold.mqe = m; s.cold.mqe_t = at - (s.qlen - 1); }
            }
        }
    }
    __syncwarp();
}

// The pair on lazy blocks and, where they may not run, the masked step.
// At the end of each block the maximum of its last two anti-diagonals is
// taken; a score inside the block is at most U, from that maximum and the
// one at the block's start (a up, c down per two anti-diagonals: U weighs
// the two bounds so that its place drops out).  A block whose U does not
// exceed the largest maximum seen before it cannot hold the global maximum;
// one whose U stays below a later maximum does not hold it for good either.
// So only the blocks since the last checkpoint that this rules in can hold
// it, and when the exact maximum and its cell are wanted (the Z-drop bound
// no longer holds, the score has passed a peak, or the table ends) the pair
// goes back to that checkpoint and takes the lazy step again from there, with
// the maximum of every pair of anti-diagonals (the masked step, up to
// exact_until, where a rebase lies between).  If the head's end lies between,
// it goes on from there as if for the first time, with the exact maximum up to
// there: a read that diverges soon after took its masked steps all the way
// from the checkpoint before (16 reads with one such 112 -> 69 us).  Blocks
// start and end on odd anti-diagonals ((r - w) odd).
// The head's last four anti-diagonals (w - 2 .. w + 1), where the virtual
// cells leave the band, run the masked step without its test (blind), as a
// block of their own; a band that covers the table (cover) has no such
// place.  Returns the last anti-diagonal processed.
template <class S>
__device__ __forceinline__ int32_t lazy_drive(S &s, bool use_fast) {
    constexpr int32_t NONE = INT_MIN;
    constexpr int32_t LOW_UNTIL = S::TRACE ? 40 : 16;  // rebase when fewer anti-diagonals are left to it
    const DevParams &prm = s.prm;
    const int32_t w = s.w, tlen = s.tlen, qlen = s.qlen, last_r = s.last_r;
    // lazy blocks in the head too (by a vote: shared memory's values are not
    // uniform for the compiler, see WarpPair16::run)
    const bool head = __any_sync(FULL, use_fast && w >= 8 && s.lazy_head_ok());
    const int32_t L = min(tlen, qlen);
    const int32_t r_in = max(L - 2, 2 * L - 3 - w);    // no cell of the last row or column up to here
    // lazy blocks end here at the latest; past r_in only if the corner is in the band
    const int32_t end = abs(tlen - qlen) <= w ? last_r - 1 : r_in;
    const int32_t turn = s.cover ? INT_MAX : w - 3;    // the crossing of the head's end starts after it
    const int32_t c0 = prm.b, c1 = max(prm.b, 2 * prm.e);
    const int32_t o0 = min(s.oe, s.oe2), o1 = s.oe + prm.q + c1;
    const bool two = prm.q2 != prm.q || prm.e2 != prm.e;
    const auto k = s.lazy_consts(two);
    const int32_t d = s.lazy_drift();
    const float inv0 = 1.0f / (float)max(prm.a + c0, 1), inv1 = 1.0f / (float)max(prm.a + c1, 1);
    const uint32_t ring = s.ring_address();

    int32_t r = -3;
    // the masked step runs up to exact_until, first the first r >= 1 with (r - w) odd
    int32_t exact_until = !use_fast ? INT_MAX : (head ? 1 + (w & 1) : w + 1);
    // blocks under way: the largest maximum seen, the bound of the blocks not
    // ruled out (NONE: there are none, the global maximum is best), its value
    // at the checkpoint, the checkpoint, the one at the block's start
    bool open = false;
    int32_t best = 0, upper = NONE, gval = 0, old = 0, last = 0;
    int32_t m0 = 0, mu = 0, n = 0;                     // the current block: see lazy_span
    bool block = false, edge = false;
    for (;;) {
        if constexpr (S::REBASES) {
            // (one place for it: a second copy costs the instruction cache)
            if (s.until_rebase < LOW_UNTIL && r >= 0) {
                s.lazy_rebase(open ? m0 : s.last_max(), r);
                if (s.ovf) return r;
            }
        }
        if (r < exact_until || !((r - w) & 1)) {
            if (r >= last_r) return r;
            ++r;
            if (s.masked_step(r)) return r;
            if constexpr (S::TRACE) {
                if (s.trace_mark(r)) s.trace_save(r, r, false);
            }
            continue;
        }
        if (!open) {
            if (r <= w && r > turn) { exact_until = w + 1; continue; }
            if (r + 8 > (r <= w && w + 1 > end ? min(turn, end) : end)) { exact_until = INT_MAX; continue; }
            const int32_t m = s.last_max();
            if (lazy_span(prm, 4, s.gmax, m, m, o1, c1) != 4) { exact_until = r + 8; continue; }
        }
        s.blind = false;
        int32_t rs = r, u0 = s.until_rebase;
        s.lazy_enter(k, two);
        int32_t target = NONE, seen = NONE, fresh = 0;     // taking blocks again: see below
        typename S::LazyWin W;
        for (;;) {
            const int32_t m1 = s.lazy_max(k, r, r > w && r <= r_in) + s.lazy_off() - d * (r - rs);
            if (target != NONE) {
                // the blocks since the checkpoint once more, pair by pair: the
                // state of the pair with the highest maximum is kept, which
                // holds the cell
                if (m1 > s.gmax) {
                    s.gmax = m1;
                    s.lazy_save(old ^ 1, r, rs, u0);
                    seen = r;
                }
                if (r >= target) {
                    if (seen != NONE) s.lazy_locate(k, old ^ 1, seen, s.gmax - s.lazy_off() + d * (seen - rs));
                    target = NONE;
                    best = gval = s.gmax;
                    upper = NONE;
                    old = 1;
                }
            } else if (!open) {
                open = true;
                best = gval = s.gmax;
                upper = NONE;
                old = 1;
            } else if (block) {
                // (the float's error is well below what is added)
                const float x = (float)prm.a * (float)(m1 - mu + (edge ? prm.q + c1 * n : c0 * n)) *
                                (edge ? inv1 : inv0);
                const int32_t U = mu + (int32_t)(x + fabsf(x) * 1e-6f) + 1;
                if (m1 > best && m1 > upper) {
                    // the blocks before this one are ruled out
                    gval = upper == NONE ? best : -(1 << 29);
                    old = last;
                    upper = U;
                } else if (U > best) {
                    if (upper == NONE) { gval = best; old = last; }
                    upper = max(upper, U);
                }
                best = max(best, m1);
            }
            block = false;
            m0 = m1;
            if (target == NONE) {
                if constexpr (S::TRACE) {
                    if (s.trace_mark(r)) {
                        if (u0 - (r - rs) < 36) break; // a rebase first: none within 32 anti-diagonals of it
                        s.trace_save(r, rs, true);
                    }
                }
                const bool cross = r == turn;
                bool close = false;                    // the Z-drop bound leaves no block
                // the end, or past a peak
                bool stop = r + 2 > end || (cross && w + 1 > end) ||
                            (upper != NONE && m0 + prm.a * LAZY_PAIRS <= best);
                if (!stop) {
                    int32_t left = S::BLOCK_PAIRS;
                    if constexpr (S::REBASES) {
                        // a rebase is due: no block, and so no checkpoint, lies
                        // closer before one, because the pair may come back to
                        // it with another place's maximum, to which it must not
                        // rebase before the next masked step has taken its own
                        left = (u0 - (r - rs) - 4) >> 1;
                        if (left < (LOW_UNTIL - 4) / 2) break;
                    }
                    edge = cross || r + 2 > r_in;
                    n = (min(edge ? end : r_in, r < turn ? min(turn, end) : end) - r) >> 1;
                    if (edge && n < 2 * LAZY_PAIRS) n = min(n, max(4, (n + 1) >> 1));   // shorter towards the end
                    n = cross ? 2 : min(min(n, left), edge ? S::EDGE_PAIRS : S::BLOCK_PAIRS);
                    if constexpr (S::TRACE) {
                        if (!cross) n = min(n, s.trace_room(r));
                    }
                    mu = r < w ? max(m0, -gap_cost(prm, r + 1)) : m0;
                    const int32_t fit =
                        lazy_span(prm, n, max(best, upper), m0, mu, edge ? o1 : o0, edge ? c1 : c0);
                    close = fit == 0 || (cross && fit < n);
                    stop = close;
                    n = fit;
                }
                if (stop) {
                    const int32_t to = r;
                    int32_t goal = to, exact = to + (close ? 8 : 0);
                    bool again = upper != NONE;
                    if (again) {                       // back to the checkpoint
                        s.lazy_load(old);
                        r = __reduce_max_sync(FULL, s.cold.ck_r[old]);
                        rs = __reduce_max_sync(FULL, s.cold.ck_rs[old]);
                        if (r <= turn && to > turn) {
                            // up to the head's end, exact from there on or on
                            // the masked step behind it
                            goal = turn;
                            again = r < turn;
                            if (!again) exact = w + 1;
                        }
                        if constexpr (S::REBASES) {
                            s.base = __reduce_max_sync(FULL, s.cold.ck_base[old]);
                            u0 = __reduce_max_sync(FULL, s.cold.ck_u0[old]);
                            again = again && goal - rs <= u0 - 4;
                        }
                        s.gmax = gval;
                    }
                    if (!again) {                      // on the masked step, if at all
                        exact_until = exact;
                        open = false;
                        break;
                    }
                    target = goal;
                    exact_until = goal;                // (a crossing done before is undone)
                    seen = NONE;
                    fresh = 0;
                } else {
                    last = old ^ 1;
                    s.lazy_save(last, r, rs, u0);
                    block = true;
                    fresh = 0;                         // (the bases are read again)
                    if (cross) {
                        s.blind = true;
                        exact_until = r + 4;
                        break;
                    }
                }
            }
            int32_t run = n;
            if (target != NONE) {
                if (r >= target) continue;             // (a checkpoint at the place itself)
                run = 1;
            }
            const bool rim = edge && target == NONE;
            const int32_t B = floor_div2(r - w);
            LazyEdge g{__reduce_max_sync(FULL, rim ? 1 : 0), tlen - 1 - B - s.j0, r - qlen + 1 - B - s.j0, ring};
            if (!s.owns()) g.dt = g.dq = -(1 << 20);
#pragma unroll 1
            for (int32_t done = 0;;) {
                if (fresh == 0) {
                    s.lazy_windows(W, r + 2 * done);
                    fresh = LAZY_PAIRS;
                }
                const int32_t m = min(run - done, fresh);
                if (two) s.template lazy_block<true>(m, W, k, g);
                else s.template lazy_block<false>(m, W, k, g);
                fresh -= m;
                done += m;
                if (S::BLOCK_PAIRS <= LAZY_PAIRS || done >= run) break;
            }
            if (rim) lazy_edges(s, r, run, s.lazy_off() - d * (r - rs), d);
            r += 2 * run;
        }
        s.lazy_leave(k, two, r - rs);
        if constexpr (S::REBASES) s.until_rebase = u0 - (r - rs);
        s.set_last_max(m0);
    }
}

}  // namespace agatha
