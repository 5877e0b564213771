// Batched persistent kernel on int32 lanes: one warp aligns one pair, lane L
// owning band slots L*C .. L*C + C - 1 of the 16-bit kernel's frame
// (kernel_warp16.cuh: B(r) = floor((r - w) / 2); when (r - w) is even E comes
// from slot j and F from slot j + 1, when odd E from slot j - 1, F from slot j).
// Used where 16-bit lanes do not apply: scorings beyond them, bands of 768 to
// 1023, the pairs they hand back, and callers that ask for int32 lanes.
//
// Nearly all anti-diagonals run in lazy blocks (lazy_drive.cuh; scorings that
// leave them no room take the kernel of kernel_step.cuh).  What bounds
// it: the integer ALU pipe when the chip is full (add-max and 3-input max
// issue at half rate on 32 bits too, so a cell costs twice what it does on
// 16-bit lanes), and for batches of a few thousand long pairs the longest
// pair's own chain of anti-diagonals, where a shorter step counts directly.
// The lazy step has about 13 instructions per cell; the step it replaced,
// which took the maximum with its position, the test and the band's mask on
// every anti-diagonal, had about 30.  The substitution is a predicated add of
// the mismatch bit (one lop3 into a predicate): as a shift, mask and
// multiply-add, the form of the 16-bit kernel, 2,500 ONT-like pairs took 41
// ms, so 23.7 (64.6 before lazy blocks, 20.4 with the longest pairs alone on
// their schedulers; 20,000 pairs 232 -> 72.6 ms).
#pragma once

#include "lazy_drive.cuh"

namespace agatha {

// K warps share one pair's band: warp k holds
// lanes 30k .. 30k + 31 of the frame, so that neighbouring warps have two lanes
// in common.  Lane 0 of every warp but the first and lane 31 of every one but
// the last are halos, copies of the neighbour's lanes 30 and 1: whatever enters
// at a warp's outer end reaches one slot further with every pair of
// anti-diagonals, so after C pairs the halo's C slots are used up and the warps'
// own lanes are still exact.  Only then is the halo refreshed through shared
// memory (refresh): one barrier per 2C anti-diagonals instead of one or more
// on each.
template <int C, int K = 1>
struct LazyPair32 {
    static_assert(C % 4 == 0 && C <= 32, "4 to 32 slots per lane");
    static constexpr int32_t NS = K == 1 ? 32 * C : (30 * K + 2) * C;
    static constexpr int HALO = 2 * K * 2 * 6 * C;        // words of the halo exchange (double-buffered)
    static constexpr bool REBASES = false, TRACE = false;
    static constexpr int TW = C <= 16 ? 2 : 3;            // window words: C bases and 16 to come
    static constexpr int V = C / 4;                       // 16-byte words of a lane's array
    static constexpr int BLOCK_PAIRS = C <= 4 ? 16 : 32;  // most pairs of a block (see WarpPair16)
    static constexpr int EDGE_PAIRS = 8;                  // pairs of a block with the last row or column
    static constexpr int RING = 2 * 2 * EDGE_PAIRS * C;   // words of the edge ring (row | column)
    static constexpr int CKV = 6 * V;                     // 16-byte words of a checkpoint per lane

    struct LazyWin { uint32_t t[TW], q[TW]; };
    struct LazyConst { int32_t A, NE, OE, H2, D, pr; bool l0, top, last; };

    const uint32_t *tp, *qp;
    int32_t tspan, qspan, tph, qph;
    int32_t tlen, qlen, w, last_r, lane, j0;
    DevParams prm;
    int32_t oe, oe2;
    // H(r) overwrites H(r-2) in the array of its parity; gap states leaving the
    // last anti-diagonal (on lazy blocks: see lazy_step)
    int32_t Hev[C], Hod[C], Eo[C], Fo[C], E2o[C], F2o[C];
    int32_t gmax, zdropped, lastm, until_rebase;
    bool cover, blind;
    Cold16 &cold;
    int32_t *ring;
    int32_t wk;                   // this warp's place in the group
    int32_t *xch0;                // K > 1: of group 0, the halo exchange, then two maxima and one place per
                                  // warp, and the next pair
    int32_t age, flip, mflip;     // anti-diagonals since the halo was fresh; buffer halves
    int4 *ck;                     // this lane's words of the warp's two checkpoints

    __device__ explicit LazyPair32(Cold16 &c, int32_t *rg, int4 *ck_, int32_t wk_, int32_t *x)
        : cold(c), ring(rg), wk(wk_), xch0(x), flip(0), mflip(0), ck(ck_) {}

    static constexpr int XCH = K > 1 ? (HALO + 3 * K + 4) / 4 * 4 : 4;
    // the group's exchange and barrier, from the thread's place each time: no
    // registers to keep them in
    __device__ __forceinline__ static int32_t group() { return (int32_t)(threadIdx.x / (32 * K)); }
    __device__ __forceinline__ int32_t *xch() const { return xch0 + group() * XCH; }
    __device__ __forceinline__ static void group_sync() {
        if constexpr (K > 1) asm volatile("bar.sync %0, %1;" :: "r"(1 + group()), "n"(32 * K) : "memory");
    }
    __device__ __forceinline__ bool leader() const { return lane == 0 && wk == 0; }
    // not a halo lane
    __device__ __forceinline__ bool owns() const {
        return K == 1 || (lane >= (wk > 0 ? 1 : 0) && lane <= (wk < K - 1 ? 30 : 31));
    }
    __device__ __forceinline__ int32_t group_max(int32_t v) {
        int32_t m = __reduce_max_sync(FULL, v);
        if constexpr (K > 1) {
            int32_t *x = xch() + HALO + mflip * K;
            mflip ^= 1;
            if (lane == 0) x[wk] = m;
            group_sync();
#pragma unroll
            for (int i = 0; i < K; ++i) m = max(m, x[i]);
            m = __reduce_max_sync(FULL, m);
        }
        return m;
    }
    // The halo lanes from the neighbours' own lanes.
    __device__ __forceinline__ void refresh() {
        if constexpr (K > 1) {
            int4 *x = reinterpret_cast<int4 *>(xch()) + flip * (K * 2 * CKV);
            flip ^= 1;
            if (lane == 1 || lane == 30) put(x + (wk * 2 + (lane == 30 ? 1 : 0)) * CKV, 1);
            group_sync();
            if (!owns()) get(x + (lane == 0 ? (wk - 1) * 2 + 1 : (wk + 1) * 2) * CKV, 1);
            __syncwarp();
            age = 0;
        }
    }

    // t field i: T[B + j0 + i]; q: the bases in falling order, field 16 + jl of
    // the 16 * TW being Q[r - B - j0 - jl].
    __device__ __forceinline__ void lazy_windows(LazyWin &W, int32_t r) const {
        const int32_t B = floor_div2(r - w);
        const int32_t tb = B + j0 + tph, qb = r - B - j0 + qph + 1;
#pragma unroll
        for (int i = 0; i < TW; ++i) {
            W.t[i] = load_rel(tp, tspan, tb + 16 * i);
            W.q[i] = rev2_32(load_rel(qp, qspan, qb - 16 * i));
        }
    }
    // bit 2 (p mod 16) of word p / 16: slot p's bases differ
    __device__ __forceinline__ static uint2 mismatch(const LazyWin &W) {
        const uint32_t x0 = W.t[0] ^ W.q[1];
        uint2 n = make_uint2((x0 | (x0 >> 1)) & 0x55555555u, 0u);
        if constexpr (C > 16) {
            const uint32_t x1 = W.t[1] ^ W.q[2];
            n.y = (x1 | (x1 >> 1)) & 0x55555555u;
        }
        return n;
    }
    __device__ __forceinline__ static bool mismatch_of(const uint2 &n, int p) {
        return (p < 16 ? n.x : n.y) & (1u << (2 * (p & 15)));
    }
    __device__ __forceinline__ static int32_t pick(const int32_t (&H)[C], int32_t local) {
        int32_t v = H[0];
#pragma unroll
        for (int p = 1; p < C; ++p) v = local == p ? H[p] : v;
        return v;
    }

    // ------------------------------------------------------- masked step
    // One anti-diagonal with every case handled per slot: a band cell of the
    // table keeps its value, a virtual row or column cell (in the head) gets
    // its own, anything else is minus infinity.  Then the last row and column,
    // the maximum and the termination test (Eq. 4-7).
    // (One copy for both parities: it runs on few anti-diagonals, and the
    // instruction cache is what the pair's other steps need.)
    __device__ __forceinline__ bool masked_step(int32_t r) {
        const bool odd = ((r - w) & 1) != 0;
        const int32_t B = floor_div2(r - w);
        int32_t st = 0, en = -1;
        if constexpr (K > 1) {
            if (age >= 2 * C) refresh();
            ++age;
        }
        if (r >= 0) {
            st = max(max(0, r - qlen + 1), ceil_div2(r - w));
            en = min(min(tlen - 1, r), floor_div2(r + w));
            if (st > en) { zdropped = 1; return true; }    // the band left the table
        }
        const int32_t lo = st - B - j0, hi = en - B - j0;
        int32_t v1 = -1, v2 = -1;                          // local slots of virtual cells
        if (r < w) {                                       // (see WarpPair16::virtual_bits)
            if (r + 1 < qlen) v1 = -1 - B - j0;                // (-1, r + 1)
            if (r >= -1 && r + 1 < tlen) v2 = r + 1 - B - j0;  // (r + 1, -1)
        }
        const int32_t vv = r == -2 ? 0 : -gap_cost(prm, r + 2);
        int32_t eL = __shfl_up_sync(FULL, Eo[C - 1], 1), e2L = __shfl_up_sync(FULL, E2o[C - 1], 1);
        int32_t fR = __shfl_down_sync(FULL, Fo[0], 1), f2R = __shfl_down_sync(FULL, F2o[0], 1);
        if (lane == 0 && wk == 0) eL = e2L = K_NEG;
        if (lane == 31 && wk == K - 1) {
            // slot NS of r - 1: the virtual column cell (t, -1) when q == -1 there
            fR = f2R = K_NEG;
            const int32_t ts = floor_div2(r - 1 - w) + NS, qs = r - 1 - ts;
            if (qs == -1 && ts >= 0 && ts < tlen && ts <= w) {
                const int32_t v = -gap_cost(prm, ts + 1);
                fR = v - oe;
                f2R = v - oe2;
            }
        }
        LazyWin Wx;
        lazy_windows(Wx, r);
        const uint2 nm = mismatch(Wx);
        int32_t lm = INT_MIN;
        int32_t nE[C], nE2[C], nF[C], nF2[C], Hd[C];
#pragma unroll
        for (int p = 0; p < C; ++p) {
            const int32_t Ein = odd ? (p ? Eo[p - 1] : eL) : Eo[p];
            const int32_t E2in = odd ? (p ? E2o[p - 1] : e2L) : E2o[p];
            const int32_t Fin = odd ? Fo[p] : (p < C - 1 ? Fo[p + 1] : fR);
            const int32_t F2in = odd ? F2o[p] : (p < C - 1 ? F2o[p + 1] : f2R);
            const int32_t s = mismatch_of(nm, p) ? -prm.b : prm.a;
            const int32_t H = max(max((odd ? Hod[p] : Hev[p]) + s, Ein), max(max(Fin, E2in), F2in));
            const bool real = p >= lo && p <= hi;
            const int32_t Hm = real ? H : (p == v1 || p == v2 ? vv : K_NEG);
            nE[p] = max(Ein - prm.e, Hm - oe);
            nF[p] = max(Fin - prm.e, Hm - oe);
            nE2[p] = max(E2in - prm.e2, Hm - oe2);
            nF2[p] = max(F2in - prm.e2, Hm - oe2);
            Hd[p] = Hm;
            lm = real ? max(lm, Hm) : lm;
        }
#pragma unroll
        for (int p = 0; p < C; ++p) {
            Eo[p] = nE[p];
            Fo[p] = nF[p];
            E2o[p] = nE2[p];
            F2o[p] = nF2[p];
            Hod[p] = odd ? Hd[p] : Hod[p];
            Hev[p] = odd ? Hev[p] : Hd[p];
        }
        if (r < 0) return false;
        // the lane that owns the last row's (column's) cell looks at it
        bool set_gs = false;
        int32_t gs = K_NEG_OUT;
        const int32_t jt = tlen - 1 - B - j0, jq = r - qlen + 1 - B - j0;
        if (st <= tlen - 1 && tlen - 1 <= en && (uint32_t)jt < (uint32_t)C && owns()) {
            const int32_t v = pick(Hd, jt);
            if (v > cold.mte) { cold.mte = v; cold.mte_q = r - (tlen - 1); }
            if (r == last_r) { gs = v; set_gs = true; }    // kept unless Z-drop stops r
        }
        if (st <= r - qlen + 1 && r - qlen + 1 <= en && (uint32_t)jq < (uint32_t)C && owns()) {
            const int32_t v = pick(Hd, jq);
            if (v > cold.mqe) { cold.mqe = v; cold.mqe_t = r - (qlen - 1); }
        }
        __syncwarp();
        if (blind) {
            group_sync();
            return false;
        }
        const int32_t m = group_max(owns() ? lm : INT_MIN);
        lastm = m;
        if (m > gmax || (prm.zdrop >= 0 && gmax - m > prm.zdrop)) {
            // its lowest slot
            int32_t li = 0;
#pragma unroll
            for (int p = C - 1; p >= 0; --p) li = p >= lo && p <= hi && Hd[p] == m ? p : li;
            const uint32_t ball = __ballot_sync(FULL, lm == m && owns());
            int32_t tstar = __shfl_sync(FULL, B + j0 + li, ball ? __ffs(ball) - 1 : 0);
            if constexpr (K > 1) {
                // of the first warp that has it
                int32_t *x = xch() + HALO + 2 * K;
                if (lane == 0) x[wk] = ball ? tstar : INT_MAX;
                group_sync();
                tstar = x[0];
#pragma unroll
                for (int i = 1; i < K; ++i) tstar = min(tstar, x[i]);
                group_sync();
            }
            const int32_t qstar = r - tstar;
            if (m > gmax) {
                gmax = m;
                if (leader()) { cold.gt = tstar; cold.gq = qstar; }
                __syncwarp();
                group_sync();
            } else {
                const int32_t gt = cold.gt, gq = cold.gq;
                const bool drop = tstar >= gt && qstar >= gq &&
                                  gmax - m > prm.zdrop + abs((tstar - gt) - (qstar - gq)) * prm.e2;
                if (__any_sync(FULL, drop)) { zdropped = 1; return true; }
            }
        }
        if (set_gs) cold.gscore = gs;
        return false;
    }

    // --------------------------------------------------------- lazy blocks
    // The step of the 16-bit kernel's lazy blocks (kernel_warp16.cuh tells why
    // it is exact) on int32: scores drift by d = e2 (e with one gap piece) per
    // anti-diagonal, Hev/Hod hold h = H - q2, E2 is brought up to date on odd
    // anti-diagonals and F2 on even ones, and only the flows across the band's
    // ends are cut, after each pair of anti-diagonals (cut).
    template <bool ODD, bool TWO>
    __device__ __forceinline__ void lazy_step(LazyWin &W, const LazyConst &k) {
        int32_t (&Hd)[C] = ODD ? Hod : Hev;
        const int32_t (&Hx)[C] = ODD ? Hev : Hod;
        if constexpr (!ODD) {
#pragma unroll
            for (int i = 0; i + 1 < TW; ++i) W.t[i] = __funnelshift_r(W.t[i], W.t[i + 1], 2);
            W.t[TW - 1] >>= 2;
        } else {
#pragma unroll
            for (int i = TW - 1; i > 0; --i) W.q[i] = __funnelshift_l(W.q[i - 1], W.q[i], 2);
            W.q[0] <<= 2;
        }
        const uint2 nm = mismatch(W);
        int32_t edge, edge2 = 0;
        if constexpr (ODD) {
            edge = __shfl_up_sync(FULL, Eo[C - 1], 1);
            if constexpr (TWO) edge2 = __shfl_up_sync(FULL, max(E2o[C - 1], Hev[C - 1]), 1);
        } else {
            edge = __shfl_down_sync(FULL, Fo[0], 1);
            edge = k.last ? K_NEG : edge;
            if constexpr (TWO) {
                edge2 = __shfl_down_sync(FULL, max(F2o[0], Hod[0]), 1);
                edge2 = k.last ? K_NEG : edge2;
            }
        }
        const int32_t nab = -(prm.a + prm.b);
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const int p = ODD ? C - 1 - i : i;
            const int n = ODD ? (p > 0 ? p - 1 : 0) : (p < C - 1 ? p + 1 : 0);
            const bool own = ODD ? p > 0 : p < C - 1;
            const int32_t Ein = ODD ? (own ? Eo[n] : edge) : Eo[p];
            const int32_t Fin = ODD ? Fo[p] : (own ? Fo[n] : edge);
            const int32_t X = __viaddmax_s32(mismatch_of(nm, p) ? Hd[p] + nab : Hd[p], k.A, Ein);
            if constexpr (TWO) {
                const int32_t E2in = ODD ? (own ? E2o[n] : edge2) : E2o[p];
                const int32_t F2in = ODD ? F2o[p] : (own ? F2o[n] : edge2);
                const int32_t H = max(__vimax3_s32(X, Fin, E2in), F2in);
                const int32_t h = H - k.H2, hoe = H - k.OE;
                Eo[p] = __viaddmax_s32(Ein, k.NE, hoe);
                Fo[p] = __viaddmax_s32(Fin, k.NE, hoe);
                if constexpr (ODD) E2o[p] = own ? __vimax3_s32(E2in, Hx[n], h) : max(E2in, h);
                else F2o[p] = own ? __vimax3_s32(F2in, Hx[n], h) : max(F2in, h);
                Hd[p] = h;
            } else {
                const int32_t h = max(X, Fin) - k.H2;
                Eo[p] = max(Ein, h);
                Fo[p] = max(Fin, h);
                Hd[p] = h;
            }
        }
    }
    // After an odd anti-diagonal: nothing flows into the band from slot 0 (of
    // lane 0) or from slot w + 1, register k.pr of the lane with k.top.
    template <bool TWO, int LO = 0, int HI = C>
    __device__ __forceinline__ void cut_top(const LazyConst &k) {
        if constexpr (HI - LO == 1) {
            Fo[LO] = k.top ? K_NEG : Fo[LO];
            if constexpr (TWO) {
                F2o[LO] = k.top ? K_NEG : F2o[LO];
                Hod[LO] = k.top ? K_NEG : Hod[LO];
            }
        } else {
            constexpr int MID = (LO + HI) / 2;
            if (k.pr < MID) cut_top<TWO, LO, MID>(k);
            else cut_top<TWO, MID, HI>(k);
        }
    }
    __device__ __forceinline__ static void ring_store(uint32_t d, int32_t j, const int32_t (&H)[C]) {
#pragma unroll
        for (int p = 0; p < C; p += 4)
            asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %0, %1;\n\t"
                         "@q st.shared.v4.b32 [%2], {%3, %4, %5, %6};\n\t}"
                         :: "r"(j), "n"(C), "r"(d + 4 * p), "r"(H[p]), "r"(H[p + 1]), "r"(H[p + 2]), "r"(H[p + 3])
                         : "memory");
    }
    template <bool TWO>
    __device__ __forceinline__ void lazy_block(int32_t n, LazyWin &W, const LazyConst &k, LazyEdge &g) {
#pragma unroll 1
        for (; n > 0; --n) {
            if constexpr (K > 1) {
                if (age > 2 * C - 2) refresh();
                age += 2;
            }
            lazy_step<false, TWO>(W, k);
            lazy_step<true, TWO>(W, k);
            Eo[0] = k.l0 ? K_NEG : Eo[0];
            if constexpr (TWO) E2o[0] = k.l0 ? K_NEG : E2o[0];
            cut_top<TWO>(k);
            if (g.on) {
                // the last row's slot moved down before the first
                // anti-diagonal, the column's moves up before the second
                --g.dt;
                ring_store(g.ring, g.dt, Hev);
                ring_store(g.ring + 2 * RING, g.dq, Hev);
                ++g.dq;
                ring_store(g.ring + 4 * C, g.dt, Hod);
                ring_store(g.ring + 4 * C + 2 * RING, g.dq, Hod);
                g.ring += 8 * C;
            }
        }
    }

    // ------------------------------------------- what lazy_drive asks for
    __device__ __forceinline__ LazyConst lazy_consts(bool) const {
        LazyConst k;
        k.D = prm.e2;
        k.H2 = prm.q2;
        k.A = prm.a + prm.q2 + 2 * prm.e2;
        k.NE = prm.e2 - prm.e;
        k.OE = oe - prm.e2;
        k.pr = (w + 1) % C;
        k.l0 = lane == 0 && wk == 0;
        k.last = w + 1 == NS && lane == 31 && wk == K - 1;
        k.top = w + 1 < NS && (uint32_t)(w + 1 - j0) < (uint32_t)C;
        return k;
    }
    __device__ __forceinline__ int32_t lazy_drift() const { return prm.e2; }
    __device__ __forceinline__ int32_t lazy_off() const { return prm.q2; }
    // minus infinity stays far below every score (within +-2^28), drift included
    __device__ __forceinline__ bool lazy_head_ok() const { return true; }
    __device__ __forceinline__ int32_t last_max() const { return lastm; }
    __device__ __forceinline__ void set_last_max(int32_t m) { lastm = m; }
    __device__ __forceinline__ uint32_t ring_address() const { return (uint32_t)__cvta_generic_to_shared(ring); }
    __device__ __forceinline__ int32_t ring_value(int c, int32_t i, int32_t j) const {
        return ring[c * (RING / 2) + i * C + j % C];
    }
    // Into the drifting form after anti-diagonal r ((r - w) odd), and back
    // (steps anti-diagonals later; slots off the band to minus infinity).
    __device__ __forceinline__ void lazy_enter(const LazyConst &k, bool) {
#pragma unroll
        for (int p = 0; p < C; ++p) {
            Hod[p] -= k.H2;
            Hev[p] -= k.H2 + k.D;
            Eo[p] += k.D;
            Fo[p] += k.D;
            E2o[p] += k.D;
            F2o[p] += k.D;
        }
    }
    __device__ __forceinline__ void lazy_leave(const LazyConst &k, bool two, int32_t steps) {
        const int32_t c = k.D * (steps + 1), lo = K_NEG + c;
#pragma unroll
        for (int p = 0; p < C; ++p) {
            const bool de = j0 + p > w, dodd = de || j0 + p == 0;
            const int32_t f2 = max(F2o[p], Hod[p]);
            Eo[p] = dodd ? K_NEG : max(Eo[p], lo) - c;
            Fo[p] = dodd ? K_NEG : max(Fo[p], lo) - c;
            E2o[p] = two ? (dodd ? K_NEG : max(E2o[p], lo) - c) : Eo[p];
            F2o[p] = two ? (dodd ? K_NEG : max(f2, lo) - c) : Fo[p];
            Hod[p] = dodd ? K_NEG : max(Hod[p] + k.H2 + k.D, lo) - c;
            Hev[p] = de ? K_NEG : max(Hev[p] + k.H2 + 2 * k.D, lo) - c;
        }
    }
    // The maximum over the band cells of anti-diagonals r and r - 1, drifting.
    __device__ __forceinline__ int32_t lazy_max(const LazyConst &k, int32_t r, bool) {
        const int32_t B1 = floor_div2(r - w), B0 = floor_div2(r - 1 - w);
        const int32_t lo1 = max(max(0, r - qlen + 1), ceil_div2(r - w)) - B1 - j0;
        const int32_t hi1 = min(min(tlen - 1, r), floor_div2(r + w)) - B1 - j0;
        const int32_t lo0 = max(max(0, r - qlen), ceil_div2(r - 1 - w)) - B0 - j0;
        const int32_t hi0 = min(min(tlen - 1, r - 1), floor_div2(r - 1 + w)) - B0 - j0;
        int32_t m = INT_MIN;
#pragma unroll
        for (int p = 0; p < C; ++p) {
            const int32_t a = p >= lo1 && p <= hi1 ? Hod[p] : INT_MIN;
            const int32_t b = p >= lo0 && p <= hi0 ? Hev[p] + k.D : INT_MIN;
            m = __vimax3_s32(m, a, b);
        }
        return group_max(owns() ? m : INT_MIN);
    }
    __device__ __forceinline__ static int4 four(const int32_t (&x)[C], int i) {
        return make_int4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
    }
    __device__ __forceinline__ static void four(int32_t (&x)[C], int i, const int4 &v) {
        x[4 * i] = v.x;
        x[4 * i + 1] = v.y;
        x[4 * i + 2] = v.z;
        x[4 * i + 3] = v.w;
    }
    // The cell of the maximum m (drifting form of r) of the pair r - 1, r whose
    // state checkpoint buf holds: the first anti-diagonal's first.
    __device__ __forceinline__ void lazy_locate(const LazyConst &k, int buf, int32_t r, int32_t m) {
        const int4 *d = ck + buf * (CKV * 32);
        int32_t t[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int32_t rr = r - 1 + c, B = floor_div2(rr - w);
            const int32_t lo = max(max(0, rr - qlen + 1), ceil_div2(rr - w)) - B - j0;
            const int32_t hi = min(min(tlen - 1, rr), floor_div2(rr + w)) - B - j0;
            int32_t at = INT_MAX;
#pragma unroll
            for (int i = V - 1; i >= 0; --i) {
                const int4 v = d[(c * V + i) * 32];
                const int32_t h[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int x = 3; x >= 0; --x) {
                    const int p = 4 * i + x;
                    if (p >= lo && p <= hi && h[x] + (c ? 0 : k.D) == m) at = B + j0 + p;
                }
            }
            t[c] = __reduce_min_sync(FULL, owns() ? at : INT_MAX);
        }
        if constexpr (K > 1) {
            int32_t *x = xch() + HALO;                  // 2 K words: both halves of the maxima
            group_sync();
            if (lane == 0) { x[2 * wk] = t[0]; x[2 * wk + 1] = t[1]; }
            group_sync();
#pragma unroll
            for (int i = 0; i < K; ++i) {
                t[0] = min(t[0], x[2 * i]);
                t[1] = min(t[1], x[2 * i + 1]);
            }
            group_sync();
        }
        if (leader()) {
            const bool first = t[0] != INT_MAX;
            cold.gt = first ? t[0] : t[1];
            cold.gq = (first ? r - 1 : r) - cold.gt;
        }
        __syncwarp();
        group_sync();
    }
    // A lane's state as 16-byte words, at d[0], d[stride] ...
    __device__ __forceinline__ void put(int4 *d, int stride) const {
#pragma unroll
        for (int i = 0; i < V; ++i) {
            d[i * stride] = four(Hev, i);
            d[(V + i) * stride] = four(Hod, i);
            d[(2 * V + i) * stride] = four(Eo, i);
            d[(3 * V + i) * stride] = four(Fo, i);
            d[(4 * V + i) * stride] = four(E2o, i);
            d[(5 * V + i) * stride] = four(F2o, i);
        }
    }
    __device__ __forceinline__ void get(const int4 *d, int stride) {
#pragma unroll
        for (int i = 0; i < V; ++i) {
            four(Hev, i, d[i * stride]);
            four(Hod, i, d[(V + i) * stride]);
            four(Eo, i, d[(2 * V + i) * stride]);
            four(Fo, i, d[(3 * V + i) * stride]);
            four(E2o, i, d[(4 * V + i) * stride]);
            four(F2o, i, d[(5 * V + i) * stride]);
        }
    }
    __device__ __forceinline__ void lazy_save(int buf, int32_t r, int32_t rs, int32_t) {
        put(ck + buf * (CKV * 32), 32);
        if (leader()) {
            cold.ck_r[buf] = r;
            cold.ck_rs[buf] = rs;
        }
        __syncwarp();
    }
    __device__ __forceinline__ void lazy_load(int buf) {
        get(ck + buf * (CKV * 32), 32);
        age = 2 * C;                  // (the halo's age then is not kept)
    }

    __device__ __forceinline__ void run(const DevBatch &Bt, int32_t pair, int32_t lane_, bool use_fast) {
        prm = Bt.params;
        lane = lane_;
        // the values that steer the pair, uniform for the compiler too (see
        // WarpPair16::run)
        tlen = __reduce_max_sync(FULL, Bt.t_len[pair]);
        qlen = __reduce_max_sync(FULL, Bt.q_len[pair]);
        int32_t *v = &prm.a;
#pragma unroll
        for (int i = 0; i < (int)(sizeof(DevParams) / 4); ++i) v[i] = __reduce_max_sync(FULL, v[i]);
        agatha_result *out = Bt.out + pair;
        if (tlen <= 0 || qlen <= 0) {
            if (leader()) write_empty_result(out);
            return;
        }
        const int64_t toff = Bt.t_off[pair], qoff = Bt.q_off[pair];
        const int64_t tw0 = toff >> 4, qw0 = qoff >> 4;
        tp = Bt.t_packed + tw0;
        qp = Bt.q_packed + qw0;
        tph = (int32_t)(toff & 15);
        qph = (int32_t)(qoff & 15);
        // the words the pair's bases occupy (inside the stream: checked by prep)
        tspan = (int32_t)min(Bt.t_words - tw0, (int64_t)((tph + tlen + 15) >> 4));
        qspan = (int32_t)min(Bt.q_words - qw0, (int64_t)((qph + qlen + 15) >> 4));
        w = effective_w(prm.w, tlen, qlen);
        const int32_t len = max(tlen, qlen);
        cover = w >= len && len < NS - 1;             // as in WarpPair16::run
        if (cover) w = NS - 1;
        if (prm.q + prm.e > prm.q2 + prm.e2) { prm.q = prm.q2; prm.e = prm.e2; }
        oe = prm.q + prm.e;
        oe2 = prm.q2 + prm.e2;
        j0 = (wk * 30 + lane) * C;
        age = 0;
        last_r = tlen + qlen - 2;
        until_rebase = INT_MAX;
        blind = false;
#pragma unroll
        for (int p = 0; p < C; ++p) Hev[p] = Hod[p] = Eo[p] = Fo[p] = E2o[p] = F2o[p] = K_NEG;
        gmax = 0;
        lastm = 0;
        zdropped = 0;
        if (leader()) {
            cold.mqe = K_NEG_OUT; cold.mqe_t = -1; cold.mte = K_NEG_OUT; cold.mte_q = -1;
            cold.gscore = K_NEG_OUT;
            cold.gt = -1; cold.gq = -1;
        }
        __syncwarp();
        group_sync();
        const int32_t r = lazy_drive(*this, use_fast);
        __syncwarp();
        group_sync();                 // every warp's last writes to cold are in
        if (leader()) {
            agatha_result o;
            const int32_t mqe = cold.mqe;
            o.max = gmax; o.te = cold.gt; o.qe = cold.gq;
            o.gscore = cold.gscore; o.mqe = mqe; o.mqe_t = cold.mqe_t; o.mte = cold.mte;
            o.mte_q = cold.mte_q;
            // band cells of anti-diagonals 0 .. r (none on r when the band
            // left the table there)
            const int32_t st_r = max(max(0, r - qlen + 1), ceil_div2(r - w));
            const int32_t en_r = min(min(tlen - 1, r), floor_div2(r + w));
            o.cells = band_cells_through(tlen, qlen, w, st_r > en_r ? r - 1 : r);
            o.zdropped = (uint8_t)zdropped;
            o.reach_end = (uint8_t)(!zdropped && mqe != K_NEG_OUT && mqe + prm.end_bonus > gmax);
            o.lane16 = 0;
            for (int i = 0; i < 5; ++i) o.pad[i] = 0;
            *out = o;
        }
        __syncwarp();
    }
};

// Warps per scheduler (K > 1: groups per SM) the registers are cut for: the faster
// count on the workloads, within what the checkpoints' shared memory admits.  Not
// all of it fits: <4, 1> spills 8 bytes, <8, 1> 74, <8, 3> 152, <12, 3> 206 (whose 9
// warps leave 168 registers a thread, since one scheduler holds three), <16, 1> none.
template <int C, int K>
__host__ __device__ constexpr int warp32_blocks() {
    return K > 1 ? (C <= 8 ? 5 : 3) : (C <= 4 ? 5 : (C <= 8 ? 4 : 2));
}
template <int C, int K>
__host__ __device__ constexpr int warp32_threads() { return (K == 1 ? WARP_BLOCK_THREADS : 32 * K) * warp32_blocks<C, K>(); }
// Dynamic shared memory of a block: two checkpoints of every warp.
template <int C, int K>
constexpr int warp32_smem() {
    return warp32_threads<C, K>() / 32 * 2 * LazyPair32<C, K>::CKV * 32 * 16;
}

// What a lone warp (group) takes per anti-diagonal of what one costs on a full SM.
template <int C, int K>
__host__ __device__ constexpr float warp32_lone() {
    return K > 1 ? (C <= 8 ? 1.8f : 1.5f) : (C <= 4 ? 1.6f : (C <= 8 ? 1.4f : 1.15f));
}

// One block per SM; see TierQueue.
template <int C, int K>
__global__ void __launch_bounds__(warp32_threads<C, K>(), 1)
warp_align_kernel(const DevBatch *__restrict__ d_batch, int32_t use_fast, int32_t list) {
    constexpr int G = warp32_threads<C, K>() / (32 * K);         // pairs at a time
    constexpr int U = K == 1 ? 4 : 1;                            // of the first tier
    using Pair = LazyPair32<C, K>;
    __shared__ Cold16 cold[G];
    __shared__ __align__(16) int32_t ring[G][Pair::RING];
    __shared__ __align__(16) int32_t xch[K > 1 ? G : 1][Pair::XCH];
    __shared__ TierQueue q;
    __shared__ int32_t first[U], place[G];
    extern __shared__ int4 lazy32_smem[];
    const DevBatch B = *d_batch;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = warp / K, wk = warp - g * K, tier = g / U;
    const bool asks = lane == 0 && wk == 0;
    const WorkList L = work_list(B, list);
    const int32_t l_end = __reduce_max_sync(FULL, L.end);
    if (list == WARP_LIST_OVERFLOW && l_end == 0) return;        // nearly always
    if (threadIdx.x == 0) q.open(L.head, L.begin, l_end, U * (int32_t)gridDim.x);
    if (asks) place[g] = q.first_place(tier);
    __syncthreads();
    int32_t k = INT_MAX;
    if (tier == 0 && asks) first[g] = k = q.next(place[g]);
    __syncthreads();
    if (tier > 0) {
        if (list_sorted(L, list) &&
            tier_crowded(q, first[g % U], tier, U * (int32_t)gridDim.x, warp32_lone<C, K>(),
                         ListSteps{L.items, B.t_len, B.q_len}))
            k = l_end;
        else if (asks) k = q.next(place[g]);
    }
    for (;;) {
        if constexpr (K > 1) {
            int32_t &next = xch[g][Pair::HALO + 3 * K];
            if (asks) next = k;
            Pair::group_sync();
            k = next;
            Pair::group_sync();
        }
        k = __reduce_min_sync(FULL, k);
        if (k >= l_end) break;
        const int32_t pair = L.items ? L.items[k] : k;
        k = INT_MAX;
        if (__any_sync(FULL, L.items || (pair_valid(B, pair) && warp_takes(B, pair)))) {
            Pair wp(cold[g], ring[g], lazy32_smem + warp * (2 * Pair::CKV * 32) + lane, wk, xch[0]);
            wp.run(B, pair, lane, use_fast != 0);
        }
        if (asks) k = q.next(place[g]);
    }
    if (asks && (q.had(place[g]) || blockIdx.x == 0)) mark_step_end(B.counters);
}

template <int C, int K>
cudaError_t launch_warp_c(const DevBatch *d_batch, int n_blocks, cudaStream_t s, int use_fast,
                          int list) {
    warp_align_kernel<C, K><<<n_blocks, warp32_threads<C, K>(), warp32_smem<C, K>(), s>>>(d_batch, use_fast, list);
    return cudaGetLastError();
}

// Resident blocks per SM; also lets the kernel have its shared memory, so a
// plan is made before the first launch on a device.
template <int C, int K>
int occupancy_warp_c() {
    int nb = 0;
    if (cudaFuncSetAttribute(warp_align_kernel<C, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             warp32_smem<C, K>()) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, warp_align_kernel<C, K>,
                                                      warp32_threads<C, K>(),
                                                      warp32_smem<C, K>()) != cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

}  // namespace agatha
