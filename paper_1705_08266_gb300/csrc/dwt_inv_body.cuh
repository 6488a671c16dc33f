#pragma once
// Inverse transform: the warp body of the TMA-fed warp-streaming kernels (one
// image per launch, batched, and persistent queue), 1 or 2 levels per work
// item.
//
// Coarse to fine.  A warp owns a strip of output columns and a segment of
// output rows.  Each slot of its shared-memory ring holds, for four level-1
// quadruple rows, the three level-1 detail bands and (two fused levels) the
// LL and three detail bands of the two level-2 rows that produce those
// level-1 rows' LL values.  Every box is 2-D TMA; a box starts at the column
// rounded down to 16 bytes and the lane reads from the remainder on.  The
// level-2 engine runs LAG + RHO rows ahead of level 1 (its first slots of a
// work item load and push level 2 only), so the LL rows it hands down are
// exact from the first level-1 row of the item on.
#include <type_traits>

#include "dwt_engine.cuh"
#include "dwt_internal.h"
#include "dwt_tma.cuh"

namespace dwt {

constexpr int kInvWarps = kInvTmaWarps;  // warps per CTA (independent)
constexpr int kInvSlots = 3;  // ring depth per warp

// Level-1 quadruple rows per slot: 4, or 2 with 4 columns per lane (the same
// 8 quadruples per lane per lifting step as 2 columns in 4 rows).
template <int Q1>
__host__ __device__ constexpr int inv_slot_quads() { return Q1 >= 4 ? 2 : 4; }

// Box widths carry A extra elements (16 bytes) so a box can start at the
// column rounded down to 16 bytes.
template <class S, int NL, int Q1>
struct InvLayout {
    static constexpr int SR = inv_slot_quads<Q1>();  // level-1 rows per slot
    static constexpr int SR2 = SR / 2;               // level-2 rows per slot
    static constexpr int A = 16 / (int)sizeof(S);
    static constexpr int Q2 = Q1 / 2;
    static constexpr int W1 = 32 * Q1 + A;     // level-1 box width (elements)
    static constexpr int W2 = 32 * Q2 + A;     // level-2 box width
    static constexpr int E128 = 128 / (int)sizeof(S);
    static constexpr int R1 = (SR * W1 + E128 - 1) / E128 * E128;   // one level-1 box region, 128-B multiple
    static constexpr int R2 = (SR2 * W2 + E128 - 1) / E128 * E128;  // one level-2 box region
    // NL == 1: LL1 HL1 LH1 HH1; NL == 2: HL1 LH1 HH1, LL2 HL2 LH2 HH2
    static constexpr int SLOT = NL == 1 ? 4 * R1 : 3 * R1 + 4 * R2;
    static constexpr uint32_t BYTES1 = SR * W1 * sizeof(S);  // bytes one level-1 box brings
    static constexpr uint32_t BYTES2 = SR2 * W2 * sizeof(S);
};

// Lane's Q values of one band row held in shared memory at p (+ lane * Q).
// A box starts at a multiple of 16 bytes, so its offset in the box is any;
// EVEN: it is even, and the values are read in pairs.
template <class S, class T, int Q, bool EVEN = false>
__device__ __forceinline__ void lds_cols(T (&v)[Q], const S* p) {
    if constexpr (EVEN && Q % 2 == 0) {
#pragma unroll
        for (int j = 0; j < Q; j += 2) {
            S w[2];
            ld_vec<S, 2>(w, p + j);
            v[j] = Storage<S>::ld(w[0]);
            v[j + 1] = Storage<S>::ld(w[1]);
        }
    } else {
#pragma unroll
        for (int j = 0; j < Q; ++j) v[j] = Storage<S>::ld(p[j]);
    }
}

template <class S, int SCH, int NL, int Q1>
struct InvWarpT {
    using T = typename Storage<S>::T;
    using Lay = InvLayout<S, NL, Q1>;
    static constexpr int LAG = std::is_same<T, float>::value ? 2 : 1;
    static constexpr int Q2 = Lay::Q2;
    Engine<T, Q1, SCH, false, NL == 1 || sizeof(S) == 4> e1;
    Engine<T, (Q2 > 0 ? Q2 : 1), SCH, false> e2;
    LevelCtx x1, x2;
    // column offsets of lane 0 inside each box (elements)
    int o1h, o1l, o2h, o2l;
    S* out;
    long long opitch;
    int out_h, lane, A0, A1;
    int x0l;        // first output column of this lane
    int n_out;      // output columns this lane stores
    bool whole;     // warp-uniform: every lane stores whole vectors or nothing
    bool even;      // warp-uniform: the level-1 box offsets are even
    // border strips: per level and band parity (even columns: LL, LH; odd: HL,
    // HH) the column outside the band that this lane fills with the mirrored
    // one (offsets from the lane-0 column, destination in the low half; -1: none)
    int fix1e, fix1o, fix2e, fix2o;
    bool fix;        // warp-uniform: this strip has such columns
    int ref1;        // width of level 1 if its LL rows are mirrored again past it (0: no)

    static constexpr int SR = Lay::SR;
    static constexpr int SR2 = Lay::SR2;

    // ROWS rows of NB bands, band i at p + i REGION with its lane-0 column at
    // off[i] and this lane's column f[i].  Every load comes before the first store, or the loads
    // would wait for the stores they might alias.
    template <int NB, int ROWS, int PITCH, int REGION>
    __device__ __forceinline__ static void fix_bands(S* p, const int (&off)[NB], const int (&f)[NB]) {
        S v[NB][ROWS];
#pragma unroll
        for (int i = 0; i < NB; ++i)
#pragma unroll
            for (int r = 0; r < ROWS; ++r)
                v[i][r] = p[i * REGION + off[i] + r * PITCH + max(f[i] >> 16, 0)];
#pragma unroll
        for (int i = 0; i < NB; ++i)
#pragma unroll
            for (int r = 0; r < ROWS; ++r)
                if (f[i] >= 0) p[i * REGION + off[i] + r * PITCH + (f[i] & 0xffff)] = v[i][r];
    }

    // Columns outside the bands take the mirrored ones, in shared memory,
    // before any lane reads them (a band's box holds its neighbour bands there).
    __device__ __forceinline__ void extend_columns(S* sm, bool level1) {
        if constexpr (NL == 1) {
            fix_bands<4, SR, Lay::W1, Lay::R1>(sm, {o1l, o1h, o1l, o1h}, {fix1e, fix1o, fix1e, fix1o});
        } else {
            if (level1) fix_bands<3, SR, Lay::W1, Lay::R1>(sm, {o1h, o1l, o1h}, {fix1o, fix1e, fix1o});
            fix_bands<4, SR2, Lay::W2, Lay::R2>(sm + 3 * Lay::R1, {o2l, o2h, o2l, o2h},
                                                {fix2e, fix2o, fix2e, fix2o});
        }
        __syncwarp();
    }

    // The level-2 output becomes level 1's LL.  Past the last column it is
    // mirrored about that column; an even width wants it repeated instead (the
    // border of level 1 lies between two samples), so those columns are
    // rewritten.  Scratch: the level-2 boxes, which have been read.
    __device__ __forceinline__ void extend_ll(S* sm2, Block<T, Q1, SR>& b) {
        static_assert(NL == 1 || 4 * Lay::R2 * sizeof(S) >= SR * 32 * Q1 * sizeof(T), "scratch");
        T* scratch = reinterpret_cast<T*>(sm2);
        const int g0 = x0l >> 1, gw = g0 - Q1 * lane, n = (ref1 + 1) >> 1;
        __syncwarp();
#pragma unroll
        for (int k = 0; k < SR; ++k) st_vec<T, Q1>(scratch + k * 32 * Q1 + Q1 * lane, b.r[k].c[0]);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < Q1; ++j) {
            const int g = g0 + j;
            if (g < 0 || g >= n) {
                const int src = min(max((reflect(2 * min(g, n + 15), ref1) >> 1) - gw, 0), 32 * Q1 - 1);
#pragma unroll
                for (int k = 0; k < SR; ++k) b.r[k].c[0][j] = scratch[k * 32 * Q1 + src];
            }
        }
        __syncwarp();
    }

    // The level-1 bands of the slot (the detail bands, and the LL of one level).
    template <bool EVEN>
    __device__ __forceinline__ void load_level1(Block<T, Q1, SR>& b, const S* sm) {
        constexpr int D = NL == 1 ? 1 : 0;  // first detail band
#pragma unroll
        for (int k = 0; k < SR; ++k) {
            const S* row = sm + k * Lay::W1 + Q1 * lane;
            if constexpr (NL == 1) lds_cols<S, T, Q1, EVEN>(b.r[k].c[0], row + o1l);
            lds_cols<S, T, Q1, EVEN>(b.r[k].c[1], row + (D + 0) * Lay::R1 + o1h);
            lds_cols<S, T, Q1, EVEN>(b.r[k].c[2], row + (D + 1) * Lay::R1 + o1l);
            lds_cols<S, T, Q1, EVEN>(b.r[k].c[3], row + (D + 2) * Lay::R1 + o1h);
        }
    }

    template <int E>
    __device__ __forceinline__ void slot(S* sm, int q0, bool level1) {
        if (__builtin_expect(fix, 0)) extend_columns(sm, level1);
        Block<T, Q1, SR> b1;
        if constexpr (NL == 2) {
            constexpr int QQ = Q2;
            Block<T, QQ, SR2> b2;
            S* base2 = sm + 3 * Lay::R1;
#pragma unroll
            for (int k = 0; k < SR2; ++k) {
                lds_cols<S, T, QQ>(b2.r[k].c[0], base2 + 0 * Lay::R2 + k * Lay::W2 + o2l + QQ * lane);
                lds_cols<S, T, QQ>(b2.r[k].c[1], base2 + 1 * Lay::R2 + k * Lay::W2 + o2h + QQ * lane);
                lds_cols<S, T, QQ>(b2.r[k].c[2], base2 + 2 * Lay::R2 + k * Lay::W2 + o2l + QQ * lane);
                lds_cols<S, T, QQ>(b2.r[k].c[3], base2 + 3 * Lay::R2 + k * Lay::W2 + o2h + QQ * lane);
            }
            e2.template push<E, SR2>(b2, q0 / 2 + LAG, x2);
            if (!level1) return;
            // level-2 rows q0/2 .. q0/2 + SR2 - 1 -> LL rows q0 .. q0 + SR - 1 of level 1
#pragma unroll
            for (int k = 0; k < SR2; ++k) {
#pragma unroll
                for (int j = 0; j < QQ; ++j) {
                    b1.r[2 * k].c[0][2 * j] = b2.r[k].c[0][j];
                    b1.r[2 * k].c[0][2 * j + 1] = b2.r[k].c[1][j];
                    b1.r[2 * k + 1].c[0][2 * j] = b2.r[k].c[2][j];
                    b1.r[2 * k + 1].c[0][2 * j + 1] = b2.r[k].c[3][j];
                }
            }
            if (__builtin_expect(ref1 != 0, 0)) extend_ll(base2, b1);
        }
        if (__builtin_expect(even, 1)) load_level1<true>(b1, sm);
        else load_level1<false>(b1, sm);
        e1.template push<E, SR>(b1, q0, x1);
        const int r1 = q0 - LAG;
        // quadruple row r -> output rows 2r (c0 c1 interleaved) and 2r + 1
        // (c2 c3); one row address per slot, advanced by the pitch
        S* p = out + (long long)(2 * r1) * opitch + x0l;
#pragma unroll
        for (int k = 0; k < SR; ++k) {
            const int r = r1 + k;
            const bool ok = r >= A0 && r < A1;
            T ev[2 * Q1], od[2 * Q1];
#pragma unroll
            for (int j = 0; j < Q1; ++j) {
                ev[2 * j] = b1.r[k].c[0][j];
                ev[2 * j + 1] = b1.r[k].c[1][j];
                od[2 * j] = b1.r[k].c[2][j];
                od[2 * j + 1] = b1.r[k].c[3][j];
            }
            if (__builtin_expect(whole, 1)) {
                st_px<true>(ev, p, ok);
                st_px<true>(od, p + opitch, ok && (E == kInner || 2 * r + 1 < out_h));
            } else {
                st_px<false>(ev, p, ok);
                st_px<false>(od, p + opitch, ok && (E == kInner || 2 * r + 1 < out_h));
            }
            p += 2 * opitch;
        }
    }

    // One output row of this lane at p: a whole aligned vector (output rows
    // start on 16 bytes, lanes on whole vectors of them), or the columns left
    // at the right border.
    template <bool WHOLE>
    __device__ __forceinline__ void st_px(const T (&v)[2 * Q1], S* p, bool ok) {
        S w[2 * Q1];
#pragma unroll
        for (int j = 0; j < 2 * Q1; ++j) w[j] = Storage<S>::st(v[j]);
        if (WHOLE || n_out == 2 * Q1) {
            if (ok && n_out > 0 && store_ok(p, 2 * Q1 * (int)sizeof(S))) st_vec<S, 2 * Q1>(p, w);
        } else if (ok && store_ok(p, n_out * (int)sizeof(S))) {
#pragma unroll
            for (int j = 0; j < 2 * Q1; ++j)
                if (j < n_out) p[j] = w[j];
        }
    }
};

__device__ __forceinline__ bool inv_rows_interior(int q0, int sr, int nl, int lag, const int* no_r) {
    // level 1: rows [q0, q0 + sr - 1]; level 2: rows [q0/2 + lag, q0/2 + lag + sr/2 - 1]
    if (q0 - lag - 1 < 0 || q0 + sr >= no_r[0]) return false;
    if (nl >= 2) {
        const int lo = q0 / 2 + lag;
        if (lo - lag - 1 < 0 || lo + sr / 2 >= no_r[1]) return false;
    }
    return true;
}

// Returns false if a bounded wait gave up (the status word is set).
template <class S, int SCH, int NL, int Q1>
__device__ __forceinline__ bool inv_body(const CUtensorMap* m1p, const CUtensorMap* m2p,
                                         const CUtensorMap* mlp, const FusedArgs& a, int wid,
                                         unsigned char* smem_raw) {
    using W = InvWarpT<S, SCH, NL, Q1>;
    using Lay = InvLayout<S, NL, Q1>;
    constexpr int LAG = W::LAG;
    constexpr int RHO = LAG;
    constexpr int SR = Lay::SR;
    constexpr int PRO = NL == 2 ? 2 * LAG : 0;  // level-2 rows pushed ahead (LAG + RHO)
    constexpr int PRO_SLOTS = PRO / (SR / 2);    // slots that feed level 2 only

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;

    static_assert(kInvWarps * kInvSlots * (Lay::SLOT * sizeof(S) + 8) <= kSmemBytes, "rings need an opt-in");
    S* ring = reinterpret_cast<S*>(smem_raw) + (size_t)warp * kInvSlots * Lay::SLOT;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw + (size_t)kInvWarps * kInvSlots *
                                                              Lay::SLOT * sizeof(S)) +
                     warp * kInvSlots;

    const int strip = wid % a.nstrips;
    W w;
    w.lane = lane;
    const int xb = strip * a.valid_px - a.xoff;
    const bool lane_ok = lane >= a.lane_lo && lane < a.lane_hi;
    w.out = reinterpret_cast<S*>(a.out);
    w.opitch = a.out_pitch;
    w.out_h = a.lv[0].h;
    w.x0l = xb + 2 * Q1 * lane;
    w.n_out = lane_ok ? min(max(a.lv[0].w - w.x0l, 0), 2 * Q1) : 0;
    w.whole = __all_sync(kFull, w.n_out == 0 || w.n_out == 2 * Q1);
    set_store_windows(a.out, a.out_elems * (long long)sizeof(S), nullptr, 0, a.err);
    const int ne1 = (a.lv[0].h + 1) >> 1;
    seg_rows(a, wid / a.nstrips, ne1, w.A0, w.A1);

    int no_r[2] = {a.lv[0].h >> 1, NL >= 2 ? (a.lv[1].h >> 1) : 0};
    const int g1w = xb >> 1;
    const int ne_c1 = (a.lv[0].w + 1) >> 1, ne_r1 = ne1;
    w.x1 = make_ctx(g1w + Q1 * lane, Q1, a.lv[0].h, a.lv[0].w, a.lv[0].s);
    const int xh1 = ne_c1 + g1w, xl1 = g1w;
    constexpr int AM = Lay::A - 1;
    w.o1h = xh1 & AM;
    w.o1l = xl1 & AM;
    // A level one column wide has no HL and HH.  Their boxes would hold another
    // level's coefficients, whose infinities and NaNs the steps' zero
    // coefficients do not stop, so they start left of the array and come as
    // zeros (clearing the columns in the ring made every border strip 3 % longer).
    constexpr int kOutside = -4096;
    static_assert(kOutside % Lay::A == 0 && kOutside + Lay::W1 < 0, "aligned and all of it outside");
    const int bx1h = a.lv[0].w > 1 ? xh1 - w.o1h : kOutside, bx1l = xl1 - w.o1l;
    w.even = !((w.o1h | w.o1l) & 1);
    bool active = a.lv[0].w > 1 && a.lv[0].h > 1;  // both axes of every fused level
    // the column of a band (parity par of a level of width n) outside it that
    // this lane fills: lanes 0-15 left of it, 16-31 right of it (the halo of
    // two fused levels takes 8)
    auto fix_of = [&](int gw, int n, int par, int Q) {
        const int nb = (n + 1 - par) >> 1;
        const int g = lane < 16 ? gw + lane : nb + lane - 16;
        if (nb <= 0 || (lane < 16 ? g >= 0 : g < gw || g >= gw + 32 * Q)) return -1;
        const int src = (reflect(2 * g + par, n) - par) >> 1;
        return (g - gw) | (min(max(src - gw, 0), 32 * Q - 1) << 16);
    };
    w.fix = xb < 0 || xb + 64 * Q1 > a.lv[0].w;
    w.fix1e = w.fix1o = w.fix2e = w.fix2o = -1;
    if (w.fix) {
        w.fix1e = fix_of(g1w, a.lv[0].w, 0, Q1);
        w.fix1o = fix_of(g1w, a.lv[0].w, 1, Q1);
    }
    w.ref1 = 0;
    int bx2h = 0, bx2l = 0, ne_r2 = 0;
    if constexpr (NL >= 2) {
        const int g2w = xb >> 2;
        const int ne_c2 = (a.lv[1].w + 1) >> 1;
        ne_r2 = (a.lv[1].h + 1) >> 1;
        w.x2 = make_ctx(g2w + W::Q2 * lane, W::Q2, a.lv[1].h, a.lv[1].w, a.lv[1].s);
        const int xh2 = ne_c2 + g2w, xl2 = g2w;
        w.o2h = xh2 & AM;
        w.o2l = xl2 & AM;
        bx2h = a.lv[1].w > 1 ? xh2 - w.o2h : kOutside;
        bx2l = xl2 - w.o2l;
        active = active && a.lv[1].w > 1 && a.lv[1].h > 1;
        if (w.fix) {
            w.fix2e = fix_of(g2w, a.lv[1].w, 0, W::Q2);
            w.fix2o = fix_of(g2w, a.lv[1].w, 1, W::Q2);
        }
        if (!(a.lv[0].w & 1) && xb + 64 * Q1 > a.lv[0].w) w.ref1 = a.lv[0].w;
    }
    w.e1.init();
    if constexpr (NL >= 2) w.e2.init();

    // level-1 input rows of this item: outputs [A0, A1) need [A0 - RHO, A1 - 1 + LAG]
    const int qstart = max(w.A0 - RHO, 0) & ~(inv_row_align(NL) - 1);
    const int nmain = (w.A1 + LAG - qstart + SR - 1) / SR;
    const int nslots = nmain + PRO_SLOTS;
    const int qbase = qstart - SR * PRO_SLOTS;

    // everything above came from the parameters: wait for the previous grid
    // (its output is this launch's input) only now
    grid_dependency_wait();

    const uint32_t ring_s = smem_u32(ring);
    const uint32_t bar_s = smem_u32(bars);
    // Lane k issues box k of a slot, all with one instruction: 2 fused levels
    // HL1 LH1 HH1, LL2 HL2 LH2 HH2; one level LL1 HL1 LH1 HH1.
    constexpr int NB = NL == 1 ? 4 : 7;  // boxes per slot
    constexpr int N1 = NL == 1 ? 4 : 3;  // of level 1
    const bool fine = lane < N1;
    const int band = fine ? lane + (4 - N1) : lane - N1;  // 0 LL, 1 HL, 2 LH, 3 HH
    const CUtensorMap* map = band == 0 ? mlp : (fine ? m1p : m2p);
    const int box_x = fine ? ((band & 1) ? bx1h : bx1l) : ((band & 1) ? bx2h : bx2l);
    int box_y = fine ? (band >= 2 ? ne_r1 : 0) + qbase : (band >= 2 ? ne_r2 : 0) + qbase / 2 + LAG;
    const uint32_t box_dst = (uint32_t)((fine ? lane * Lay::R1 : N1 * Lay::R1 + band * Lay::R2) * sizeof(S));
    // slots are issued in order, one after the other
    auto issue = [&](int s) {
        const int b = s % kInvSlots;
        const uint32_t bar = bar_s + 8 * b;
        const bool l1 = s >= PRO_SLOTS;
        if (lane == 0)
            mbar_arrive_expect_tx(bar, (l1 ? N1 * Lay::BYTES1 : 0) + (NL == 2 ? 4 * Lay::BYTES2 : 0));
        __syncwarp();
        if (lane < NB && (l1 || !fine))
            tma_load_2d(ring_s + (uint32_t)(b * Lay::SLOT * sizeof(S)) + box_dst, map, box_x, box_y, bar);
        box_y += fine ? SR : SR / 2;
    };
    if (lane == 0) {
        for (int b = 0; b < kInvSlots; ++b) mbar_init(bar_s + 8 * b, 1);
        fence_mbar_init();
    }
    __syncwarp();
    for (int s = 0; s < kInvSlots && s < nslots; ++s) issue(s);

    // the border-free slots form one run [si0, si1) (see the forward body)
    int si0 = nslots, si1 = nslots;
    if (active) {
        si0 = 0;
        while (si0 < nslots && !inv_rows_interior(qbase + SR * si0, SR, NL, LAG, no_r)) ++si0;
        si1 = nslots;
        while (si1 > si0 && !inv_rows_interior(qbase + SR * (si1 - 1), SR, NL, LAG, no_r)) --si1;
    }

    bool failed = false;
    int s = 0;
    for (; s < nslots; ++s) {
        const int b = s % kInvSlots;
        const bool ok = mbar_wait_bounded(bar_s + 8 * b, (s / kInvSlots) & 1, kWaitBudget);
        if (!__all_sync(kFull, ok)) {
            failed = true;
            break;
        }
        const int q0 = qbase + SR * s;
        const bool l1 = s >= PRO_SLOTS;
        if (s >= si0 && s < si1)
            w.template slot<kInner>(ring + b * Lay::SLOT, q0, l1);
        else
            w.template slot<kEdgeRows>(ring + b * Lay::SLOT, q0, l1);
        __syncwarp();
        if (s + kInvSlots < nslots) {
            fence_proxy_async_smem();  // every lane: its reads and writes before the refill
            issue(s + kInvSlots);
        }
    }
    if (failed) {
        if (lane == 0) atomicExch(a.err, -6);
        for (int t = s; t < nslots && t < s + kInvSlots; ++t)
            mbar_wait_bounded(bar_s + 8 * (t % kInvSlots), (t / kInvSlots) & 1, kWaitBudget);
        return false;
    }
    // every copy has landed: the barriers may be initialised again.  The last
    // kInvSlots slots were not refilled, so no fence has ordered this lane's
    // accesses to them (mirrored columns are stored there) before the copies
    // that the warp's next work item issues into the same ring.
    fence_proxy_async_smem();
    if (lane == 0)
        for (int b = 0; b < kInvSlots; ++b) mbar_inval(bar_s + 8 * b);
    __syncwarp();
    return true;
}

}  // namespace dwt
