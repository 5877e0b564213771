// Local extension from an initial score: the BWA-MEM variant of the
// extension (the paper applies its kernel to BWA-MEM's guided alignment,
// Section 5.9).  The rules are this library's reading of BWA-MEM's published
// extension, stated in include/agatha.h beside agatha_align_batch_local:
//   - the origin holds the seed's score h0 > 0 and the virtual row and column
//     h0 - gap(l), kept only while positive;
//   - a path is kept only while its score stays positive: every state is
//     floored at 0 and a diagonal step out of an empty cell (H = 0) stays
//     empty;
//   - the termination test runs one query row at a time: the row's best cell
//     (lowest t on ties) becomes the best so far when strictly higher, else
//     the Z-drop test may stop the extension; a row without a positive cell
//     ends it.
//
// One warp aligns one pair on int32 lanes, in the same anti-diagonal frame as
// the int32 score kernel (lane L owns slots L*C .. L*C + C - 1 of the band,
// slot j being cell t = B(r) + j with B(r) = ceil((r - w) / 2)), every
// anti-diagonal through one per-cell step that classifies each slot as a band
// cell, a virtual cell or nothing.  The rows are handled without leaving the
// frame: a row q is the cells (t, q) for increasing t, which is exactly the
// way the E state travels (from (t-1, q) to (t, q)), so two more states ride
// along with E: the row's best score so far (RM) and its lowest t (RT).  A
// row is complete on the anti-diagonal of its last band cell,
// t = min(tlen - 1, q + w); at most one row completes per anti-diagonal, in
// increasing q, and its best is then read from the slot of that cell.  The
// cells past the completing row that the frame has already computed (up to w
// anti-diagonals ahead) are dropped with it when the extension stops there.
#include <climits>

#include "lazy_drive.cuh"

namespace agatha {

template <int C>
struct LocalPair {
    using W = typename WarpWin<C>::T;
    const uint32_t *tp, *qp;
    int64_t tw, qw, toff, qoff;
    int32_t tlen, qlen, w, lane, j0, h0;
    DevParams P;
    int32_t oe, oe2;
    // band state: H of r-1 and r-2, the gap states leaving r-1 (floored at
    // 0: 0 is "no live path"), and the row accumulators leaving r-1 (RM = -1:
    // no cell of the row yet)
    int32_t H1[C], H2[C], Eo[C], E2o[C], Fo[C], F2o[C], RM[C], RT[C];
    W Tw, Qw;
    uint32_t Tpf, Qpf;
    int32_t tcnt, qcnt;
    int64_t tpos, qpos;
    // rows (uniform across the warp)
    int32_t gmax, gt, gq, mqe, mqe_t, mte, mte_q, gscore;
    int64_t cells;
    int32_t zdropped;

    __device__ __forceinline__ static int32_t pos(int32_t x) { return x > 0 ? x : 0; }

    __device__ __forceinline__ void init_windows(int32_t r) {
        const int32_t B = ceil_div2(r - w);
        const int64_t tb = (int64_t)B + j0;
        const int64_t qb = (int64_t)r - B - j0;
        if constexpr (C <= 16) {
            Tw = load16(tp, tw, toff + tb) & WarpWin<C>::MASK;
            const uint32_t nat = load16(qp, qw, qoff + qb - C + 1);
            Qw = rev2_32(nat) >> (2 * (16 - C));
        } else {
            Tw = load32(tp, tw, toff + tb) & WarpWin<C>::MASK;
            const uint64_t nat = load32(qp, qw, qoff + qb - C + 1);
            Qw = rev2_64(nat) >> (2 * (32 - C));
        }
        tpos = tb + C;
        qpos = qb + 1;
        Tpf = load16(tp, tw, toff + tpos);
        Qpf = load16(qp, qw, qoff + qpos);
        tpos += 16;
        qpos += 16;
        tcnt = 16;
        qcnt = 16;
    }
    __device__ __forceinline__ void shift_t() {
        Tw = (Tw >> 2) | ((W)(Tpf & 3u) << (2 * C - 2));
        Tpf >>= 2;
        if (--tcnt == 0) {
            Tpf = load16(tp, tw, toff + tpos);
            tpos += 16;
            tcnt = 16;
        }
    }
    __device__ __forceinline__ void shift_q() {
        Qw = ((Qw << 2) | (W)(Qpf & 3u)) & WarpWin<C>::MASK;
        Qpf >>= 2;
        if (--qcnt == 0) {
            Qpf = load16(qp, qw, qoff + qpos);
            qpos += 16;
            qcnt = 16;
        }
    }

    // value of the virtual cell (t, q) (t == -1 or q == -1), 0 when no path
    // with a positive score reaches it
    __device__ __forceinline__ int32_t virtual_H(int32_t t, int32_t q) const {
        if (t == -1 && q == -1) return h0;
        return pos(h0 - gap_cost(P, (t == -1 ? q : t) + 1));
    }

    // One anti-diagonal; then, if a row completes on it, that row's rules.
    // Returns true when the extension ends (stop or last row done).
    __device__ __forceinline__ bool step(int32_t r) {
        const int32_t B = ceil_div2(r - w);
        const int32_t d = (r - w) & 1;
        // the slot below lane 0 (cell (B-1, r-B) of r-1): a virtual row cell
        // only when B == 0; its E states and an empty row accumulator
        int32_t eL = __shfl_up_sync(FULL, Eo[C - 1], 1);
        int32_t e2L = __shfl_up_sync(FULL, E2o[C - 1], 1);
        int32_t rmL = __shfl_up_sync(FULL, RM[C - 1], 1);
        int32_t rtL = __shfl_up_sync(FULL, RT[C - 1], 1);
        int32_t fR = __shfl_down_sync(FULL, Fo[0], 1);
        int32_t f2R = __shfl_down_sync(FULL, F2o[0], 1);
        if (lane == 0) {
            const int32_t ts = B - 1, qs = r - B;
            if (ts == -1 && qs >= -1 && qs < qlen) {
                const int32_t v = virtual_H(ts, qs);
                eL = pos(v - oe);
                e2L = pos(v - oe2);
            } else {
                eL = 0;
                e2L = 0;
            }
            rmL = -1;
            rtL = -1;
        }
        if (lane == 31) { fR = 0; f2R = 0; }
        const W x = Tw ^ Qw;
        const W nm = (x | (x >> 1)) & WarpWin<C>::LOW;     // bit 2*jl: mismatch
        int32_t nH[C], nE[C], nE2[C], nF[C], nF2[C], nRM[C], nRT[C];
#pragma unroll
        for (int jl = 0; jl < C; ++jl) {
            const int32_t t = B + j0 + jl;
            const int32_t q = r - t;
            const int32_t Ein = d ? Eo[jl] : (jl ? Eo[jl - 1] : eL);
            const int32_t E2in = d ? E2o[jl] : (jl ? E2o[jl - 1] : e2L);
            const int32_t RMin = d ? RM[jl] : (jl ? RM[jl - 1] : rmL);
            const int32_t RTin = d ? RT[jl] : (jl ? RT[jl - 1] : rtL);
            const int32_t Fin = d ? (jl < C - 1 ? Fo[jl + 1] : fR) : Fo[jl];
            const int32_t F2in = d ? (jl < C - 1 ? F2o[jl + 1] : f2R) : F2o[jl];
            const int32_t s = ((nm >> (2 * jl)) & 1) ? -P.b : P.a;
            const int32_t k = t - q;
            const bool real = t >= 0 && q >= 0 && t < tlen && q < qlen && k <= w && -k <= w;
            int32_t H, ne, ne2, nf, nf2, rm = -1, rt = -1;
            if (real) {
                const int32_t Hd = H2[jl];               // H(t-1, q-1)
                H = Hd > 0 ? pos(Hd + s) : 0;
                H = max(max(H, Ein), max(max(Fin, E2in), F2in));
                ne = pos(max(H - oe, Ein - P.e));
                nf = pos(max(H - oe, Fin - P.e));
                ne2 = pos(max(H - oe2, E2in - P.e2));
                nf2 = pos(max(H - oe2, F2in - P.e2));
                // the row's best so far: strictly higher keeps the lowest t
                if (H > RMin) { rm = H; rt = t; } else { rm = RMin; rt = RTin; }
            } else if ((t == -1 && q >= -1 && q < qlen) || (q == -1 && t >= 0 && t < tlen)) {
                H = virtual_H(t, q);
                ne = nf = pos(H - oe);
                ne2 = nf2 = pos(H - oe2);
            } else {
                H = 0;
                ne = nf = ne2 = nf2 = 0;
            }
            nH[jl] = H; nE[jl] = ne; nE2[jl] = ne2; nF[jl] = nf; nF2[jl] = nf2; nRM[jl] = rm; nRT[jl] = rt;
        }
#pragma unroll
        for (int jl = 0; jl < C; ++jl) {
            H2[jl] = H1[jl]; H1[jl] = nH[jl];
            Eo[jl] = nE[jl]; E2o[jl] = nE2[jl]; Fo[jl] = nF[jl]; F2o[jl] = nF2[jl];
            RM[jl] = nRM[jl]; RT[jl] = nRT[jl];
        }
        if (r < 0) return false;
        // the row completing on r: its last band cell t = min(tlen-1, q+w) has
        // t + q = r (2q + w = r while q + w < tlen, then q = r - tlen + 1)
        int32_t qc = -1;
        if (((r - w) & 1) == 0) {
            const int32_t qa = (r - w) >> 1;
            if (qa >= 0 && qa < qlen && qa + w < tlen - 1) qc = qa;
        }
        {
            const int32_t qb = r - tlen + 1;
            if (qb >= 0 && qb < qlen && qb + w >= tlen - 1) qc = qb;
        }
        if (qc < 0) return false;
        const int32_t tl = min(tlen - 1, qc + w);
        const int32_t tf = max(0, qc - w);
        // read its row accumulator and H at the slot of (tl, qc)
        const int32_t j = tl - B, owner = j / C, loc = j - owner * C;
        int32_t v_rm = RM[0], v_rt = RT[0], v_h = H1[0];
#pragma unroll
        for (int jl = 1; jl < C; ++jl) {
            if (loc == jl) { v_rm = RM[jl]; v_rt = RT[jl]; v_h = H1[jl]; }
        }
        const int32_t row = __shfl_sync(FULL, v_rm, owner);
        const int32_t row_t = __shfl_sync(FULL, v_rt, owner);
        const int32_t h_end = __shfl_sync(FULL, v_h, owner);
        cells += tl - tf + 1;
        if (tl == tlen - 1 && h_end > 0 && h_end > mte) { mte = h_end; mte_q = qc; }
        if (qc == qlen - 1 && row > 0) { mqe = row; mqe_t = row_t; }
        if (row <= 0) { zdropped = 1; return true; }          // no live cell left
        if (row > gmax) {
            gmax = row; gt = row_t; gq = qc;
        } else if (P.zdrop >= 0) {
            int32_t l = (qc - gq) - (row_t - gt);
            l = l < 0 ? -l : l;
            if (gmax - row > P.zdrop + l * P.e2) { zdropped = 1; return true; }
        }
        if (qc == qlen - 1) {
            if (tl == tlen - 1 && h_end > 0) gscore = h_end;
            return true;                                      // every row done
        }
        if (qc + 1 - w > tlen - 1) { zdropped = 1; return true; }   // the next row has no band cell
        return false;
    }

    __device__ __forceinline__ void run(const DevBatch &Bt, int32_t pair, int32_t lane_) {
        P = Bt.params;
        lane = lane_;
        tp = Bt.t_packed; qp = Bt.q_packed; tw = Bt.t_words; qw = Bt.q_words;
        tlen = Bt.t_len[pair]; qlen = Bt.q_len[pair];
        toff = Bt.t_off[pair]; qoff = Bt.q_off[pair];
        h0 = Bt.h0[pair];
        agatha_result *out = Bt.out + pair;
        gmax = h0; gt = -1; gq = -1;
        mqe = K_NEG_OUT; mqe_t = -1; mte = K_NEG_OUT; mte_q = -1; gscore = K_NEG_OUT;
        cells = 0; zdropped = 0;
        if (tlen > 0 && qlen > 0) {
            w = effective_w(P.w, tlen, qlen);
            oe = P.q + P.e; oe2 = P.q2 + P.e2;
            j0 = lane * C;
#pragma unroll
            for (int i = 0; i < C; ++i) {
                H1[i] = H2[i] = Eo[i] = E2o[i] = Fo[i] = F2o[i] = 0;
                RM[i] = RT[i] = -1;
            }
            // the last row completes on anti-diagonal tlen + qlen - 2 at the latest
            const int32_t last_r = tlen + qlen - 2;
            int32_t r = -2;
            init_windows(r);
            bool stop = step(r);
            while (!stop && r < last_r) {
                ++r;
                if ((r - w) & 1) shift_t(); else shift_q();
                stop = step(r);
            }
        }
        if (lane == 0) {
            agatha_result o;
            o.max = gmax; o.te = gt; o.qe = gq;
            o.gscore = gscore; o.mqe = mqe; o.mqe_t = mqe_t; o.mte = mte; o.mte_q = mte_q;
            o.cells = cells;
            o.zdropped = (uint8_t)zdropped;
            o.reach_end = (uint8_t)(!zdropped && mqe != K_NEG_OUT && mqe + P.end_bonus > gmax);
            o.lane16 = 0;
            for (int i = 0; i < 5; ++i) o.pad[i] = 0;
            *out = o;
        }
    }
};

// The same extension without per-cell cases, for nearly every pair (fits):
// the frame, the windows and the lazy step of the int32 score kernel
// (kernel_lazy32.cuh: scores drift by d per anti-diagonal, h = H - q2 kept, E2
// and F2 brought up to date on every second anti-diagonal, only the flows
// across the band's ends cut), with what the local rules add:
//  - Gap states need no floor: gap moves never raise a score, so a state at or
//    below zero stays there.  Only a diagonal step could revive an empty cell:
//    it is taken where the cell's H is above the drifting zero (z), and H is
//    floored there in the spare input of its last 3-input max.
//  - A row's best score and its lowest t ride along with E as one key,
//    1024 H + age: each step in t adds one to the age and takes the maximum
//    with 1024 H of the new cell, one add-max per cell.  Ages stay below 1024
//    (2w <= 1022), so they only break ties, for the older cell.
//  - The rows that complete in a block of up to 32 anti-diagonals are read at
//    its end, one per lane, from a ring the owning lanes have filled, and a
//    warp scan applies the rows' rules in order.  A block computed past the row
//    that stops the extension is dropped with it.
//  - The virtual row and column come out of the recurrence from the origin;
//    the virtual row's cells are kept out of the keys as long as they are live
//    (MASK).  Where they would still be live when they leave the band (w - 6
//    and on; never when the band covers the table) the pair takes the per-cell
//    step above.
// What bounds it: the integer ALU pipe (about 8 of its instructions per cell,
// and per step the exchange of two or three edge words).  100,000 reads of 150
// bp (w = 100, BWA-MEM's scoring) on one GB300: 12.7 ms a call on the per-cell
// step, whose every slot is told apart and which reads the completing row on
// each anti-diagonal, 3.7 ms on this one.
template <int C>
struct LocalRows {
    static constexpr int32_t NS = 32 * C;
    static constexpr int TW = 2;
    static constexpr int RING = 2 * 2 * LAZY_PAIRS * C;   // words: keys, then h, of a block's anti-diagonals
    static constexpr int32_t LOW = -(1 << 30);            // no cell yet
    static constexpr int32_t NEG = -(1 << 28);

    struct Win { uint32_t t[TW], q[TW]; };

    const uint32_t *tp, *qp;
    int32_t tspan, qspan, tph, qph;
    int32_t tlen, qlen, w, lane, j0, h0;
    DevParams prm;
    int32_t oe, oe2;
    int32_t Hev[C], Hod[C], Eo[C], Fo[C], E2o[C], F2o[C], RM[C];
    int32_t *ring;
    // constants of the step (see LazyPair32), and the drifting zero of the
    // next anti-diagonal
    int32_t A, NE, OE, pr, z;
    bool l0, top, last;

    // Whether the pair runs here: keys fit 32 bits, and live virtual cells
    // never leave the band inside the table.
    __device__ __forceinline__ static bool fits(const DevParams &p, int32_t tlen, int32_t qlen, int32_t h0) {
        if (tlen <= 0 || qlen <= 0) return true;
        if ((int64_t)h0 + (int64_t)p.a * min(tlen, qlen) >= (1 << 20)) return false;
        const int32_t len = max(tlen, qlen), w = effective_w(p.w, tlen, qlen);
        return (w >= len && len < NS - 1) || (w >= 8 && h0 <= gap_cost(p, w - 6));
    }

    __device__ __forceinline__ void windows(Win &W, int32_t r) const {
        const int32_t B = floor_div2(r - w);
        const int32_t tb = B + j0 + tph, qb = r - B - j0 + qph + 1;
#pragma unroll
        for (int i = 0; i < TW; ++i) {
            W.t[i] = load_rel(tp, tspan, tb + 16 * i);
            W.q[i] = rev2_32(load_rel(qp, qspan, qb - 16 * i));
        }
    }

    // One anti-diagonal.  lo (MASK): the lane's first slot with t >= 0.
    template <bool ODD, bool TWO, bool MASK>
    __device__ __forceinline__ void step(Win &W, int32_t lo) {
        int32_t (&Hd)[C] = ODD ? Hod : Hev;
        const int32_t (&Hx)[C] = ODD ? Hev : Hod;
        if constexpr (!ODD) {
            W.t[0] = __funnelshift_r(W.t[0], W.t[1], 2);
            W.t[1] >>= 2;
        } else {
            W.q[1] = __funnelshift_l(W.q[0], W.q[1], 2);
            W.q[0] <<= 2;
        }
        const uint32_t x = W.t[0] ^ W.q[1];
        const uint32_t nm = x | (x >> 1);              // even bits: the bases differ
        int32_t edge, edge2 = 0, edger = 0;
        if constexpr (ODD) {
            edge = __shfl_up_sync(FULL, Eo[C - 1], 1);
            edger = __shfl_up_sync(FULL, RM[C - 1], 1);
            if constexpr (TWO) edge2 = __shfl_up_sync(FULL, max(E2o[C - 1], Hev[C - 1]), 1);
        } else {
            edge = __shfl_down_sync(FULL, Fo[0], 1);
            edge = last ? NEG : edge;
            if constexpr (TWO) {
                edge2 = __shfl_down_sync(FULL, max(F2o[0], Hod[0]), 1);
                edge2 = last ? NEG : edge2;
            }
        }
        const int32_t nab = -(prm.a + prm.b);
        const int32_t live = z - 2 * prm.e2 - prm.q2;  // h of r - 2 above this: a live cell
        const uint32_t zk = 0u - (uint32_t)z * 1024u;
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const int p = ODD ? C - 1 - i : i;
            const int n = ODD ? (p > 0 ? p - 1 : 0) : (p < C - 1 ? p + 1 : 0);
            const bool own = ODD ? p > 0 : p < C - 1;
            const int32_t Ein = ODD ? (own ? Eo[n] : edge) : Eo[p];
            const int32_t Fin = ODD ? Fo[p] : (own ? Fo[n] : edge);
            const int32_t RMin = ODD ? (own ? RM[n] : edger) : RM[p];
            const int32_t Hs = (nm & (1u << (2 * p))) ? Hd[p] + nab : Hd[p];
            const int32_t D = __viaddmax_s32(Hs, A, Ein);
            const int32_t X = Hd[p] > live ? D : Ein;
            int32_t H;
            if constexpr (TWO) {
                const int32_t E2in = ODD ? (own ? E2o[n] : edge2) : E2o[p];
                const int32_t F2in = ODD ? F2o[p] : (own ? F2o[n] : edge2);
                H = __vimax3_s32(__vimax3_s32(X, Fin, E2in), F2in, z);
                const int32_t h = H - prm.q2, hoe = H - OE;
                Eo[p] = __viaddmax_s32(Ein, NE, hoe);
                Fo[p] = __viaddmax_s32(Fin, NE, hoe);
                if constexpr (ODD) E2o[p] = own ? __vimax3_s32(E2in, Hx[n], h) : max(E2in, h);
                else F2o[p] = own ? __vimax3_s32(F2in, Hx[n], h) : max(F2in, h);
                Hd[p] = h;
            } else {
                H = __vimax3_s32(X, Fin, z);
                const int32_t h = H - prm.q2;
                Eo[p] = max(Ein, h);
                Fo[p] = max(Fin, h);
                Hd[p] = h;
            }
            int32_t key = row_key(H, zk);
            if constexpr (MASK) key = p >= lo ? key : LOW;
            RM[p] = __viaddmax_s32(RMin, 1, key);
        }
        z += prm.e2;
    }
    // After an odd anti-diagonal (see LazyPair32::cut_top).
    template <bool TWO, int LO = 0, int HI = C>
    __device__ __forceinline__ void cut_top() {
        if constexpr (HI - LO == 1) {
            Fo[LO] = top ? NEG : Fo[LO];
            if constexpr (TWO) {
                F2o[LO] = top ? NEG : F2o[LO];
                Hod[LO] = top ? NEG : Hod[LO];
            }
        } else {
            constexpr int MID = (LO + HI) / 2;
            if (pr < MID) cut_top<TWO, LO, MID>();
            else cut_top<TWO, MID, HI>();
        }
    }
    template <bool TWO>
    __device__ __forceinline__ void cut() {
        Eo[0] = l0 ? NEG : Eo[0];
        RM[0] = l0 ? LOW : RM[0];
        if constexpr (TWO) E2o[0] = l0 ? NEG : E2o[0];
        cut_top<TWO>();
    }
    __device__ __forceinline__ static void ring_store(uint32_t d, int32_t j, const int32_t (&v)[C]) {
#pragma unroll
        for (int p = 0; p < C; p += 4)
            asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %0, %1;\n\t"
                         "@q st.shared.v4.b32 [%2], {%3, %4, %5, %6};\n\t}"
                         :: "r"(j), "n"(C), "r"(d + 4 * p), "r"(v[p]), "r"(v[p + 1]), "r"(v[p + 2]), "r"(v[p + 3])
                         : "memory");
    }
    // n pairs of anti-diagonals from the odd anti-diagonal r on; slot offset j
    // of the completing rows' cells falls by fall per pair.
    template <bool TWO, bool MASK>
    __device__ __forceinline__ void block(int32_t r, int32_t n, int32_t j, int32_t fall) {
        Win W;
        windows(W, r);
        int32_t lo = -floor_div2(r - w) - j0;
        uint32_t d = (uint32_t)__cvta_generic_to_shared(ring);
#pragma unroll 1
        for (; n > 0; --n) {
            --lo;
            j -= fall;
            step<false, TWO, MASK>(W, lo);
            ring_store(d, j, RM);
            ring_store(d + 2 * RING, j, Hev);
            step<true, TWO, MASK>(W, lo);
            ring_store(d + 4 * C, j, RM);
            ring_store(d + 4 * C + 2 * RING, j, Hod);
            cut<TWO>();
            d += 8 * C;
        }
    }

    __device__ __forceinline__ void run(const DevBatch &Bt, int32_t pair, int32_t lane_) {
        prm = Bt.params;
        lane = lane_;
        tlen = __reduce_max_sync(FULL, Bt.t_len[pair]);
        qlen = __reduce_max_sync(FULL, Bt.q_len[pair]);
        h0 = __reduce_max_sync(FULL, Bt.h0[pair]);
        int32_t *v = &prm.a;
#pragma unroll
        for (int i = 0; i < (int)(sizeof(DevParams) / 4); ++i) v[i] = __reduce_max_sync(FULL, v[i]);
        agatha_result *out = Bt.out + pair;
        int32_t gmax = h0, gt = -1, gq = -1;
        int32_t mqe = K_NEG_OUT, mqe_t = -1, mte = K_NEG_OUT, mte_q = -1, gscore = K_NEG_OUT;
        int32_t rows = 0, zdropped = 0;                     // rows processed
        w = 0;
        if (tlen > 0 && qlen > 0) {
            const int64_t toff = Bt.t_off[pair], qoff = Bt.q_off[pair];
            const int64_t tw0 = toff >> 4, qw0 = qoff >> 4;
            tp = Bt.t_packed + tw0;
            qp = Bt.q_packed + qw0;
            tph = (int32_t)(toff & 15);
            qph = (int32_t)(qoff & 15);
            tspan = (int32_t)min(Bt.t_words - tw0, (int64_t)((tph + tlen + 15) >> 4));
            qspan = (int32_t)min(Bt.q_words - qw0, (int64_t)((qph + qlen + 15) >> 4));
            w = effective_w(prm.w, tlen, qlen);
            const int32_t len = max(tlen, qlen);
            if (w >= len && len < NS - 1) w = NS - 1;       // the band covers the table: as the whole frame
            if (prm.q + prm.e > prm.q2 + prm.e2) { prm.q = prm.q2; prm.e = prm.e2; }
            const bool two = prm.q2 != prm.q || prm.e2 != prm.e;
            const int32_t d = prm.e2;
            oe = prm.q + prm.e;
            oe2 = prm.q2 + prm.e2;
            j0 = lane * C;
            A = prm.a + prm.q2 + 2 * d;
            NE = d - prm.e;
            OE = oe - d;
            pr = (w + 1) % C;
            l0 = lane == 0;
            top = w + 1 < NS && lane == (w + 1) / C;
            last = w + 1 == NS && lane == 31;
            // the origin, on anti-diagonal -2 (drift 0 there)
            const int32_t s0 = -1 - floor_div2(-2 - w) - j0;
            const bool odd0 = (w & 1) != 0;                 // (-2 - w) odd
#pragma unroll
            for (int p = 0; p < C; ++p) {
                const bool o = p == s0;
                Hev[p] = o && !odd0 ? h0 - prm.q2 : NEG;
                Hod[p] = o && odd0 ? h0 - prm.q2 : NEG;
                Eo[p] = Fo[p] = o ? h0 - oe + d : NEG;
                E2o[p] = F2o[p] = o ? h0 - oe2 + d : NEG;
                RM[p] = LOW;
            }
            z = d;
            int32_t r = -2;
            if (!odd0) {                                    // anti-diagonal -1, to start after an odd one
                Win W;
                windows(W, r);
                const int32_t lo = -floor_div2(-1 - w) - j0;
                if (two) { step<true, true, true>(W, lo); cut<true>(); }
                else { step<true, false, true>(W, lo); cut<false>(); }
                r = -1;
            }
            // virtual row cells are live up to this anti-diagonal
            const int32_t g1 = prm.e > 0 ? (h0 - 1 - prm.q) / prm.e : (h0 > prm.q ? 1 << 26 : 0);
            const int32_t g2 = prm.e2 > 0 ? (h0 - 1 - prm.q2) / prm.e2 : (h0 > prm.q2 ? 1 << 26 : 0);
            const int32_t vend = max(g1, g2) - 2;
            const int32_t r2 = 2 * (tlen - 1) - w;          // from here on a row ends with the table
            const int32_t last_r = tlen + qlen - 2;
            bool stop = false;
            while (!stop && r < last_r) {
                const bool second = r + 1 >= r2;
                int32_t n = min((last_r - r + 1) >> 1, LAZY_PAIRS);
                if (!second) n = min(n, (r2 - 1 - r) >> 1);
                const bool mask = r + 1 <= vend;
                if (mask) n = min(n, max(1, (vend - r + 1) >> 1));
                const int32_t j = (second ? tlen - 1 - floor_div2(r - w) : w) - j0, fall = second ? 1 : 0;
                if (mask) {
                    if (two) block<true, true>(r, n, j, fall);
                    else block<false, true>(r, n, j, fall);
                } else {
                    if (two) block<true, false>(r, n, j, fall);
                    else block<false, false>(r, n, j, fall);
                }
                __syncwarp();
                // lane i: the row that completes on anti-diagonal r + 1 + i
                const int32_t ri = r + 1 + lane, zi = z - d * (2 * n - lane);
                int32_t q = -1, te = 0;
                if (second) { q = ri - tlen + 1; te = tlen - 1; }
                else if (((ri - w) & 1) == 0) { q = (ri - w) >> 1; te = q + w; }
                const bool has = lane < 2 * n && q >= 0 && q < qlen && te - q <= w;
                int32_t score = INT_MIN, rt = -1, he = 0;
                if (has) {
                    const int32_t loc = (te - floor_div2(ri - w)) % C;
                    const int32_t key = ring[lane * C + loc];
                    score = key >> 10;
                    rt = te - (key & 1023);
                    he = ring[RING / 2 + lane * C + loc] + prm.q2 - zi;
                }
                // the best row up to each lane's (the first of the highest)
                int32_t bs = score, bi = lane;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int32_t os = __shfl_up_sync(FULL, bs, o), oi = __shfl_up_sync(FULL, bi, o);
                    if (lane >= o && os >= bs) { bs = os; bi = oi; }
                }
                // before this lane's row
                int32_t ps = __shfl_up_sync(FULL, bs, 1), pi = __shfl_up_sync(FULL, bi, 1);
                if (lane == 0) { ps = INT_MIN; pi = 0; }
                const int32_t pt = __shfl_sync(FULL, rt, pi), pq = __shfl_sync(FULL, q, pi);
                const bool in_block = ps > gmax;
                const int32_t g = in_block ? ps : gmax, ct = in_block ? pt : gt, cq = in_block ? pq : gq;
                bool drop = false;
                if (has) {
                    if (score <= 0) drop = true;            // no live cell left
                    else if (score <= g && prm.zdrop >= 0)
                        drop = g - score > prm.zdrop + abs((q - cq) - (rt - ct)) * prm.e2;
                }
                const bool fin = has && (q == qlen - 1 || q + 1 - w > tlen - 1);
                const uint32_t ends = __ballot_sync(FULL, drop || fin);
                const int32_t f = ends ? __ffs(ends) - 1 : 31;         // rows of lanes 0 .. f count
                const uint32_t with = __ballot_sync(FULL, has) & (f == 31 ? FULL : (2u << f) - 1u);
                if (with) {
                    const int32_t li = 31 - __clz(with);
                    rows = __shfl_sync(FULL, q, li) + 1;
                    const int32_t fs = __shfl_sync(FULL, bs, li), fi = __shfl_sync(FULL, bi, li);
                    if (fs > gmax) {
                        gmax = fs;
                        gt = __shfl_sync(FULL, rt, fi);
                        gq = __shfl_sync(FULL, q, fi);
                    }
                    // the best cell of the last target base, the first of the highest
                    const bool mine = (with >> lane) & 1u;
                    const int32_t hv = mine && second && he > 0 ? he : INT_MIN;
                    const int32_t hm = __reduce_max_sync(FULL, hv);
                    if (hm > mte) {
                        mte = hm;
                        mte_q = __shfl_sync(FULL, q, __ffs(__ballot_sync(FULL, hv == hm)) - 1);
                    }
                    if (rows == qlen) {                     // the last query row is done
                        const int32_t s = __shfl_sync(FULL, score, li);
                        if (s > 0) { mqe = s; mqe_t = __shfl_sync(FULL, rt, li); }
                    }
                }
                if (__any_sync(FULL, ends != 0)) {
                    stop = true;
                    const bool dropped = (__ballot_sync(FULL, drop) >> f) & 1u;
                    zdropped = dropped || rows < qlen;
                    if (!dropped && rows == qlen) {
                        const int32_t hl = __shfl_sync(FULL, he, f);
                        if (__shfl_sync(FULL, te, f) == tlen - 1 && hl > 0) gscore = hl;
                    }
                }
                __syncwarp();
                r += 2 * n;
            }
        }
        if (lane == 0) {
            agatha_result o;
            o.max = gmax; o.te = gt; o.qe = gq;
            o.gscore = gscore; o.mqe = mqe; o.mqe_t = mqe_t; o.mte = mte; o.mte_q = mte_q;
            // band cells of rows 0 .. rows - 1: sums of min(tlen - 1, q + w)
            // and of max(0, q - w)
            const int64_t R = rows, k1 = max((int64_t)0, min(R, (int64_t)tlen - 1 - w));
            const int64_t hi = k1 * (k1 - 1) / 2 + k1 * w + (R - k1) * (tlen - 1);
            const int64_t m = R - 1 - w, lo = m > 0 ? m * (m + 1) / 2 : 0;
            o.cells = rows ? hi - lo + R : 0;
            o.zdropped = (uint8_t)zdropped;
            o.reach_end = (uint8_t)(!zdropped && mqe != K_NEG_OUT && mqe + prm.end_bonus > gmax);
            o.lane16 = 0;
            for (int i = 0; i < 5; ++i) o.pad[i] = 0;
            *out = o;
        }
    }
};

// Warps per scheduler the registers are cut for.
template <int C>
__host__ __device__ constexpr int local_tiers() { return C == 4 ? 5 : (C == 8 ? 4 : 3); }
template <int C>
constexpr int local_smem() { return 4 * local_tiers<C>() * LocalRows<C>::RING * 4; }

// The pairs of the queue, handed out by TierQueue to one block per SM; those
// that do not fit go to the hand-back list.  Whole calls against one queue for
// all warps: 600 reads of 150 bp 170 -> 129 us, of 300 bp 251 -> 163, 100,000 of
// 150 bp 3.70 -> 3.64 ms.
template <int C>
__global__ void __launch_bounds__(WARP_BLOCK_THREADS * local_tiers<C>(), 1)
local_rows_kernel(const DevBatch *__restrict__ d_batch) {
    extern __shared__ __align__(16) int32_t local_ring[];
    __shared__ TierQueue q;
    __shared__ int32_t first[4], place[4 * local_tiers<C>()];
    const DevBatch B = *d_batch;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tier = warp >> 2;
    const int32_t units = 4 * (int32_t)gridDim.x;
    const WorkList L = work_list(B, WARP_LIST_MAIN);
    const int32_t l_end = __reduce_max_sync(FULL, L.end);
    if (threadIdx.x == 0) q.open(L.head, L.begin, l_end, units);
    if (lane == 0) place[warp] = q.first_place(tier);
    __syncthreads();
    int32_t k = INT_MAX;
    if (tier == 0 && lane == 0) first[warp] = k = q.next(place[warp]);
    __syncthreads();
    if (tier > 0) {
        if (list_sorted(L, WARP_LIST_MAIN) &&
            tier_crowded(q, first[warp & 3], tier, units, 1.5f, ListSteps{L.items, B.t_len, B.q_len}))
            k = l_end;
        else if (lane == 0) k = q.next(place[warp]);
    }
    for (;;) {
        k = __reduce_min_sync(FULL, k);
        if (k >= l_end) break;
        const int32_t pair = L.items ? L.items[k] : k;
        k = INT_MAX;
        if (__any_sync(FULL, L.items || (pair_valid(B, pair) && warp_takes(B, pair)))) {
            const int32_t h0 = B.h0[pair];
            if (__any_sync(FULL, h0 < 1 || h0 > LOCAL_H0_MAX)) {    // an initial score outside the supported range
                if (lane == 0) {
                    atomicExch(&B.counters[CTR_ERR], DEV_ERR_BAD_PAIR);
                    write_empty_result(B.out + pair);
                }
            } else if (!__any_sync(FULL, LocalRows<C>::fits(B.params, B.t_len[pair], B.q_len[pair], h0))) {
                if (lane == 0) B.ovf_list[atomicAdd(&B.counters[CTR_NOVF], 1)] = pair;
            } else {
                LocalRows<C> lp;
                lp.ring = local_ring + warp * LocalRows<C>::RING;
                lp.run(B, pair, lane);
            }
        }
        if (lane == 0) k = q.next(place[warp]);
    }
    if (lane == 0 && (q.had(place[warp]) || blockIdx.x == 0)) mark_step_end(B.counters);
}

// The pairs handed back, on the per-cell step.  The loop checks its pairs as if the
// list might hold any: without that (they need no check) the compiler's code for the
// 4-slot step is slower (all pairs of a batch handed back, whole calls: 50,000 reads
// of 150 bp 7.33 ms, so 6.50; 200 reads 0.34 and 0.31).
template <int C>
__global__ void __launch_bounds__(WARP_BLOCK_THREADS)
local_align_kernel(const DevBatch *__restrict__ d_batch) {
    const DevBatch B = *d_batch;
    const int lane = threadIdx.x & 31;
    const WorkList L = work_list(B, WARP_LIST_OVERFLOW);
    if (L.end == 0) return;                                         // nearly always
    for (;;) {
        int32_t k = 0;
        if (lane == 0) k = L.begin + atomicAdd(L.head, 1);
        k = __shfl_sync(FULL, k, 0);
        if (k >= L.end) break;
        const int32_t pair = L.items ? L.items[k] : k;
        if (!L.items && (!pair_valid(B, pair) || !warp_takes(B, pair))) continue;
        const int32_t h0 = B.h0[pair];
        if (h0 < 1 || h0 > LOCAL_H0_MAX) {
            if (lane == 0) {
                atomicExch(&B.counters[CTR_ERR], DEV_ERR_BAD_PAIR);
                write_empty_result(B.out + pair);
            }
            continue;
        }
        LocalPair<C> lp;
        lp.run(B, pair, lane);
    }
    if (lane == 0) mark_step_end(B.counters);
}

template <int C>
static cudaError_t launch_local_c(const DevBatch *d_batch, int n_sm, cudaStream_t s) {
    int cells = 0;
    cudaError_t e = cudaFuncSetAttribute(local_rows_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         local_smem<C>());
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&cells, local_align_kernel<C>, WARP_BLOCK_THREADS, 0);
    if (e != cudaSuccess) return e;
    local_rows_kernel<C><<<n_sm, WARP_BLOCK_THREADS * local_tiers<C>(), local_smem<C>(), s>>>(d_batch);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    local_align_kernel<C><<<n_sm * (cells > 0 ? cells : 1), WARP_BLOCK_THREADS, 0, s>>>(d_batch);
    return cudaGetLastError();
}

// C = 4, 8 or 16 slots per lane (bands up to 511; the state of wider ones
// would not fit the registers)
cudaError_t launch_local(int C, const DevBatch *d_batch, int n_sm, cudaStream_t s) {
    switch (C) {
        case 4: return launch_local_c<4>(d_batch, n_sm, s);
        case 8: return launch_local_c<8>(d_batch, n_sm, s);
        case 16: return launch_local_c<16>(d_batch, n_sm, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace agatha
