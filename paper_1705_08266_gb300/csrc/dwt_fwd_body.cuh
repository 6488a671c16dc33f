#pragma once
// Forward transform: the warp body of the TMA-fed warp-streaming kernels
// (one image per launch, batched, and persistent queue), 1..3 levels per
// work item.
//
// Each warp takes one work item (a strip of 64 Q1 input pixels, including a
// halo, and a segment of rows) and streams its rows through a private ring of
// shared-memory slots that the warp's lane 0 fills with 2-D TMA boxes.  The
// level-1 engine (Q1 quadruple columns per lane) emits finished rows; their
// detail bands are stored and their LL values are paired into level-2
// quadruple rows (Q1/2 columns per lane), and so on to level 3.  Values are
// stored as S (float, int, half or bfloat16) and lifted as float or int.
// Only the LL of the last fused level leaves the chip besides the detail
// bands, so a launch that fuses k levels reads the input once and
// writes every coefficient once.
#include <type_traits>

#include "dwt_engine.cuh"
#include "dwt_internal.h"
#include "dwt_tma.cuh"

namespace dwt {

// A whole vector of a lane's Q values at p (vector aligned); ok = the lane
// stores and the row belongs to the work item.  keep: the next launch reads
// the values back (L2 evict-last).
template <class S, class T, int Q>
__device__ __forceinline__ void st_fast(S* p, const T (&v)[Q], bool ok, bool keep = false) {
    S w[Q];
#pragma unroll
    for (int j = 0; j < Q; ++j) w[j] = Storage<S>::st(v[j]);
    if (ok && store_ok(p, Q * (int)sizeof(S))) {
        if (keep) st_vec_keep<S, Q>(p, w);
        else st_vec<S, Q>(p, w);
    }
}

// How a strip stores the bands of a level.  kWhole: every storing lane whole
// aligned vectors; kHalves: the HL / HH bands start half a vector (of 4) off,
// two halves each; kColumns: column by column, for other starts and for the
// strips that the right border cuts.  One predicate per store and no branches:
// a lane-dependent branch per store made border strips, which are most strips
// of a small image, twice as long.
enum StoreMode { kWhole = 0, kHalves = 1, kColumns = 2 };

// A lane's Q values at p: whole vectors, or the first n of them.
template <class S, class T, int Q, int MODE>
__device__ __forceinline__ void st_band(S* p, const T (&v)[Q], bool ok, int n, bool keep = false) {
    if constexpr (MODE == kWhole) {
        st_fast<S, T, Q>(p, v, ok && n > 0, keep);
    } else {
        S w[Q];
#pragma unroll
        for (int j = 0; j < Q; ++j) w[j] = Storage<S>::st(v[j]);
        ok = ok && n > 0 && store_ok(p, n * (int)sizeof(S));
        if constexpr (MODE == kHalves && Q == 4) {
            if (ok) {
                st_vec<S, 2>(p, *reinterpret_cast<const S(*)[2]>(w));
                st_vec<S, 2>(p + 2, *reinterpret_cast<const S(*)[2]>(w + 2));
            }
        } else {
#pragma unroll
            for (int j = 0; j < Q; ++j)
                if (ok && j < n) p[j] = w[j];
        }
    }
}

// Per-level store state of one lane.
struct StoreGeo {
    int ne_r, no_r, ne_c;
    int g0;          // first quadruple column of this lane
    int r_lo, r_hi;  // rows of this level that this work item stores
    int n_e, n_o;    // columns this lane stores of the LL / LH and of the HL / HH bands
    int mode;        // warp-uniform StoreMode
};

// The bands of rows r .. r + R - 1 whose rows the item owns (and, with border
// rows, that exist); LAST: the LL leaves the chip too.
template <int E, class S, class T, int Q, int R, int MODE, bool LAST>
__device__ __forceinline__ void store_rows(const Block<T, Q, R>& b, int r, const StoreGeo& g, S* mallat,
                                           long long mpitch, S* ll, long long llpitch, bool keep) {
    constexpr int ME = MODE == kHalves ? kWhole : MODE;  // LL and LH start on a vector
    S* hl = mallat + (long long)r * mpitch + (g.g0 + g.ne_c);
    S* lh = hl + ((long long)g.ne_r * mpitch - g.ne_c);
    S* lrow = ll + (long long)r * llpitch + g.g0;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const bool in = r + k >= g.r_lo && r + k < g.r_hi;
        const bool even = in && (E == kInner || r + k < g.ne_r), odd = in && (E == kInner || r + k < g.no_r);
        st_band<S, T, Q, MODE>(hl, b.r[k].c[1], even, g.n_o);
        st_band<S, T, Q, ME>(lh, b.r[k].c[2], odd, g.n_e);
        st_band<S, T, Q, MODE>(lh + g.ne_c, b.r[k].c[3], odd, g.n_o);
        if constexpr (LAST) st_band<S, T, Q, ME>(lrow, b.r[k].c[0], even, g.n_e, keep);
        hl += mpitch;
        lh += mpitch;
        if constexpr (LAST) lrow += llpitch;
    }
}

__device__ __forceinline__ StoreGeo make_geo(int h, int w, int g0, int Q, int r_lo, int r_hi,
                                             bool lane_ok) {
    StoreGeo g;
    g.ne_r = (h + 1) >> 1;
    g.no_r = h >> 1;
    g.ne_c = (w + 1) >> 1;
    g.g0 = g0;
    g.r_lo = r_lo;
    g.r_hi = r_hi;
    g.n_e = lane_ok ? min(max(g.ne_c - g0, 0), Q) : 0;
    g.n_o = lane_ok ? min(max((w >> 1) - g0, 0), Q) : 0;
    const int al = g.ne_c & (Q - 1);  // where the HL / HH rows start, past a vector boundary
    const bool whole = __all_sync(kFull, (g.n_e == 0 || g.n_e == Q) && g.n_o == g.n_e);
    g.mode = !whole ? kColumns : al == 0 ? kWhole : Q == 4 && al == 2 ? kHalves : kColumns;
    return g;
}
// Pair two consecutive LL rows (even row e, odd row o) of Q values into a
// quadruple row of Q/2 columns for the next level.
template <class T, int Q>
__device__ __forceinline__ void pair_rows(const T (&e)[Q], const T (&o)[Q], Quads<T, Q / 2>& n) {
#pragma unroll
    for (int j = 0; j < Q / 2; ++j) {
        n.c[0][j] = e[2 * j];
        n.c[1][j] = e[2 * j + 1];
        n.c[2][j] = o[2 * j];
        n.c[3][j] = o[2 * j + 1];
    }
}

// Quadruple rows per slot (one TMA box of 2 SR image rows): 4, or 2 with 4
// columns per lane and at most 2 fused levels (the same 8 quadruples per
// lane per lifting step, and a box of the same bytes).
template <int NL, int Q1>
__host__ __device__ constexpr int fwd_slot_quads() { return (Q1 >= 4 && NL <= 2) ? 2 : 4; }

// All state of one warp's work item: the level engines, per-level geometry and
// the pending even LL rows, plus the static per-slot schedule.  Q1 quadruple
// columns per lane at level 1 (2 Q1 pixels), Q1/2 at level 2, Q1/4 at level 3.
template <class S, int SCH, int NL, int Q1>
struct FwdWarp {
    using T = typename Storage<S>::T;
    static constexpr int LAG = std::is_same<T, float>::value ? 2 : 1;
    static constexpr int Q2 = Q1 / 2 > 0 ? Q1 / 2 : 1;
    static constexpr int Q3 = Q1 / 4 > 0 ? Q1 / 4 : 1;
    static constexpr int BW = 64 * Q1;  // box width in pixels
    static constexpr int SR = fwd_slot_quads<NL, Q1>();  // quadruple rows per slot
    static_assert(NL <= 2 || SR == 4, "three fused levels need slots of 4 quadruple rows");
    Engine<T, Q1, SCH, true> e1;
    Engine<T, Q2, SCH, true> e2;
    Engine<T, Q3, SCH, true> e3;
    LevelCtx x1, x2, x3;
    StoreGeo s1, s2, s3;
    T pend1[Q1], pend2[Q2];
    S* mallat;
    S* ll;
    long long mpitch, llpitch;
    bool ll_keep;  // the next launch reads the LL back: store it L2 evict-last
    int lane;
    // border strips: columns outside the image that this lane fills with the
    // mirrored ones (element offsets within a row of the box, destination in
    // the low half; -1: none)
    int fix_l, fix_r;
    bool fix;        // warp-uniform: this strip has such columns
    int ref1, ref2;  // columns of the next level's input past which a row is mirrored again (0: no)

    // Columns outside the image take the mirrored ones (whole-sample symmetric
    // extension), in shared memory, before any lane reads them.
    __device__ __forceinline__ void extend_columns(S* sm) {
        // (every load before the first store, or the loads would wait for the
        // stores they might alias)
        S l[2 * SR], r[2 * SR];
        const int ls = (fix_l >> 16) & (BW - 1), rs = (fix_r >> 16) & (BW - 1);
#pragma unroll
        for (int k = 0; k < 2 * SR; ++k) {
            l[k] = sm[k * BW + ls];
            r[k] = sm[k * BW + rs];
        }
#pragma unroll
        for (int k = 0; k < 2 * SR; ++k) {
            if (fix_l >= 0) sm[k * BW + (fix_l & 0xffff)] = l[k];
            if (fix_r >= 0) sm[k * BW + (fix_r & 0xffff)] = r[k];
        }
        __syncwarp();
    }

    // The R LL rows of a level become the next level's input, which is mirrored
    // about its own last column n - 1.  The computed columns past it already
    // equal that for an odd width; an even one repeats its last column instead
    // (the border lies between two samples), so those columns are rewritten.
    // At the left border both agree unless the signal is shorter than the halo.
    template <int Q, int R>
    __device__ __forceinline__ void extend_ll(S* sm, Block<T, Q, R>& b, int g0, int n) {
        T* scratch = reinterpret_cast<T*>(sm);  // the slot's rows have been read
        const int gw = g0 - Q * lane;
        __syncwarp();
#pragma unroll
        for (int k = 0; k < R; ++k) st_vec<T, Q>(scratch + k * 32 * Q + Q * lane, b.r[k].c[0]);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            const int g = g0 + j;
            if (g < 0 || g >= n) {
                const int src = min(max(reflect(min(g, n + 15), n) - gw, 0), 32 * Q - 1);
#pragma unroll
                for (int k = 0; k < R; ++k) b.r[k].c[0][j] = scratch[k * 32 * Q + src];
            }
        }
        __syncwarp();
    }

    // One slot: level-1 input quadruple rows q0 .. q0+SR-1 (q0 a multiple of
    // fwd_row_align) in shared memory (2 SR image rows of BW pixels), pushed as
    // one block.  The rows every level emits, and how LL rows pair into the
    // next level's quadruple rows, are then fixed by the pipeline lag alone.
    // Level-2 input rows of the slot at q0: LL rows q0 - 2 .. q0 + SR - 3
    // paired into quadruple rows q0/2 - 1 .. q0/2 + SR/2 - 2.
    template <int R2>
    __device__ __forceinline__ void pair_level1(const Block<T, Q1, SR>& b1, Block<T, Q2, R2>& b2) {
        if constexpr (LAG == 2) {  // emitted rows q0-2 .. q0+SR-3
#pragma unroll
            for (int j = 0; j < R2; ++j) pair_rows<T, Q1>(b1.r[2 * j].c[0], b1.r[2 * j + 1].c[0], b2.r[j]);
        } else {  // emitted rows q0-1 .. q0+SR-2; row q0-2 was kept from the last slot
            pair_rows<T, Q1>(pend1, b1.r[0].c[0], b2.r[0]);
#pragma unroll
            for (int j = 1; j < R2; ++j) pair_rows<T, Q1>(b1.r[2 * j - 1].c[0], b1.r[2 * j].c[0], b2.r[j]);
            copy_arr(pend1, b1.r[SR - 1].c[0]);
        }
    }

    // The rows of level L that a push emitted, from row r on.
    template <int E, int L, int Q, int R>
    __device__ __forceinline__ void store_level(const Block<T, Q, R>& b, int r, const StoreGeo& g) {
        if (__builtin_expect(g.mode == kWhole, 1))
            store_rows<E, S, T, Q, R, kWhole, L == NL>(b, r, g, mallat, mpitch, ll, llpitch, ll_keep);
        else if (E == kInner && Q == 4 && g.mode == kHalves)
            store_rows<E, S, T, Q, R, kHalves, L == NL>(b, r, g, mallat, mpitch, ll, llpitch, ll_keep);
        else
            store_rows<E, S, T, Q, R, kColumns, L == NL>(b, r, g, mallat, mpitch, ll, llpitch, ll_keep);
    }

    template <int E>
    __device__ __forceinline__ void slot(S* sm, int q0) {
        if (__builtin_expect(fix, 0)) extend_columns(sm);
        Block<T, Q1, SR> b1;
#pragma unroll
        for (int k = 0; k < SR; ++k) {
            Quads<T, Q1>& row = b1.r[k];
            S ev[2 * Q1], od[2 * Q1];
            ld_vec<S, 2 * Q1>(ev, sm + (2 * k) * BW + 2 * Q1 * lane);
            ld_vec<S, 2 * Q1>(od, sm + (2 * k + 1) * BW + 2 * Q1 * lane);
#pragma unroll
            for (int j = 0; j < Q1; ++j) {
                row.c[0][j] = Storage<S>::ld(ev[2 * j]);
                row.c[1][j] = Storage<S>::ld(ev[2 * j + 1]);
                row.c[2][j] = Storage<S>::ld(od[2 * j]);
                row.c[3][j] = Storage<S>::ld(od[2 * j + 1]);
            }
        }
        e1.template push<E, SR>(b1, q0, x1);
        store_level<E, 1>(b1, q0 - LAG, s1);
        if constexpr (NL >= 2) {
            if (__builtin_expect(ref1 != 0, 0)) extend_ll(sm, b1, s1.g0, ref1);
            // level-2 input rows q0/2 - 1 .. q0/2 + R2 - 2 = LL rows q0 - 2 .. q0 + SR - 3
            constexpr int R2 = SR / 2;
            Block<T, Q2, R2> b2;
            pair_level1<R2>(b1, b2);
            const int in2 = q0 / 2 - 1;
            e2.template push<E, R2>(b2, in2, x2);
            store_level<E, 2>(b2, in2 - LAG, s2);
            if constexpr (NL >= 3) {
                static_assert(Q1 >= 4, "three fused levels need 4 columns per lane");
                if (__builtin_expect(ref2 != 0, 0)) extend_ll(sm, b2, s2.g0, ref2);
                Block<T, Q3, 1> b3;
                int in3;
                if constexpr (LAG == 2) {  // level-2 rows q0/2-3, q0/2-2; q0/2-4 kept
                    pair_rows<T, Q2>(pend2, b2.r[0].c[0], b3.r[0]);
                    copy_arr(pend2, b2.r[1].c[0]);
                    in3 = q0 / 4 - 2;
                } else {  // level-2 rows q0/2-2, q0/2-1
                    pair_rows<T, Q2>(b2.r[0].c[0], b2.r[1].c[0], b3.r[0]);
                    in3 = q0 / 4 - 1;
                }
                e3.template push<E, 1>(b3, in3, x3);
                store_level<E, 3>(b3, in3 - LAG, s3);
            }
        }
    }
};

// Rows of level l pushed in the slot of level-1 rows [q0, q0 + sr) lie in
// [lo, hi]; the interior code is valid if every stage row touched is at least
// one row away from the top and stays clear of the last odd row.
__device__ __forceinline__ bool rows_interior(int q0, int sr, int nl, int lag, const int* no_r) {
    int lo = q0, hi = q0 + sr - 1;
    for (int l = 0; l < nl; ++l) {
        if (lo - lag - 1 < 0 || hi + 1 >= no_r[l]) return false;
        lo = floordiv2(lo - lag) - 1;
        hi = floordiv2(hi - lag);
    }
    return true;
}

// One warp's work item `wid` of a launch described by `a` (input through the
// tensor map at `mapp`).
// Returns false if a bounded wait gave up (the status word is set).
template <class S, int SCH, int NL, int Q1>
__device__ __forceinline__ bool fwd_body(const CUtensorMap* mapp, const FusedArgs& a, int wid,
                                         unsigned char* smem_raw) {
    using FW = FwdWarp<S, SCH, NL, Q1>;
    using T = typename FW::T;
    constexpr int RHO = FW::LAG;
    constexpr int BW = FW::BW;
    constexpr int SR = FW::SR;
    constexpr int SLOT_ROWS = 2 * SR;  // image rows per TMA box
    static_assert(Engine<T, Q1, SCH, true>::LAG == RHO && Engine<T, 1, SCH, true>::LAG == RHO, "lag");

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;

    constexpr int kSlotElems = SLOT_ROWS * BW;
    static_assert(kFwdWarps * kFwdSlots * (kSlotElems * sizeof(S) + 8) <= kSmemBytes, "rings need an opt-in");
    S* ring = reinterpret_cast<S*>(smem_raw) + (size_t)warp * kFwdSlots * kSlotElems;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw + (size_t)kFwdWarps * kFwdSlots *
                                                              kSlotElems * sizeof(S)) +
                     warp * kFwdSlots;

    const int strip = wid % a.nstrips;
    const int xb = strip * a.valid_px - a.xoff;

    // rows of the last fused level this item produces, and the input rows it needs
    const int neN = (a.lv[NL - 1].h + 1) >> 1;
    int R0, R1;
    seg_rows(a, wid / a.nstrips, neN, R0, R1);
    int f = R0, e = R1 - 1;
#pragma unroll
    for (int l = NL; l >= 1; --l) {
        f -= RHO;
        e += RHO;
        if (l > 1) {
            f *= 2;
            e = 2 * e + 1;
        }
    }
    const int qstart = max(f, 0) & ~(fwd_row_align(NL) - 1);
    const int qend = e + 1;
    const int nslots = (qend - qstart + SR - 1) / SR;

    FW W;
    W.lane = lane;
    const bool lane_ok = lane >= a.lane_lo && lane < a.lane_hi;
    W.mallat = reinterpret_cast<S*>(a.mallat);
    W.mpitch = a.mallat_pitch;
    W.ll = reinterpret_cast<S*>(a.ll);
    W.llpitch = a.ll_pitch;
    W.ll_keep = a.ll_keep != 0;
    int no_r[3] = {0, 0, 0};
    bool active;  // both axes of every fused level
    {
        const int g1 = (xb >> 1) + Q1 * lane;
        W.x1 = make_ctx(g1, Q1, a.lv[0].h, a.lv[0].w, a.lv[0].s);
        W.s1 = make_geo(a.lv[0].h, a.lv[0].w, g1, Q1, R0 << (NL - 1), R1 << (NL - 1), lane_ok);
        no_r[0] = a.lv[0].h >> 1;
        active = a.lv[0].w > 1 && a.lv[0].h > 1;
    }
    if constexpr (NL >= 2) {
        const int g2 = (xb >> 2) + FW::Q2 * lane;
        W.x2 = make_ctx(g2, FW::Q2, a.lv[1].h, a.lv[1].w, a.lv[1].s);
        W.s2 = make_geo(a.lv[1].h, a.lv[1].w, g2, FW::Q2, R0 << (NL - 2), R1 << (NL - 2), lane_ok);
        no_r[1] = a.lv[1].h >> 1;
        active = active && a.lv[1].w > 1 && a.lv[1].h > 1;
    }
    if constexpr (NL >= 3) {
        const int g3 = (xb >> 3) + FW::Q3 * lane;
        W.x3 = make_ctx(g3, FW::Q3, a.lv[2].h, a.lv[2].w, a.lv[2].s);
        W.s3 = make_geo(a.lv[2].h, a.lv[2].w, g3, FW::Q3, R0, R1, lane_ok);
        no_r[2] = a.lv[2].h >> 1;
        active = active && a.lv[2].w > 1 && a.lv[2].h > 1;
        // A level of one row has no odd row, nor do the rows that the levels
        // above it compute before the image: their odd components, farther from
        // the image than two levels' are, would come through the zero
        // coefficient as NaNs where they are not finite.  (In every kernel this
        // made plain 16-bit launches 3 % longer.)
        if (a.lv[1].h == 1) W.x2.no_r = -(1 << 30);
        if (a.lv[2].h == 1) W.x3.no_r = -(1 << 30);
    }
    // columns outside the image: up to 32 on each side, one per lane (the
    // halo of three fused levels takes 28)
    const int w0 = a.lv[0].w;
    W.fix_l = W.fix_r = -1;
    if (xb + lane < 0) W.fix_l = lane | (min(max(reflect(xb + lane, w0) - xb, 0), BW - 1) << 16);
    if (w0 + lane < xb + BW)
        W.fix_r = (w0 + lane - xb) | (min(max(reflect(w0 + lane, w0) - xb, 0), BW - 1) << 16);
    W.fix = xb < 0 || xb + BW > w0;
    // a level of even width whose right border this box holds (a signal
    // shorter than its halo lies in one box, left border included)
    W.ref1 = NL >= 2 && !(w0 & 1) && xb + BW > w0 ? (w0 + 1) >> 1 : 0;
    W.ref2 = 0;
    if constexpr (NL >= 3) {
        const int w1 = a.lv[1].w;
        if (!(w1 & 1) && xb + BW > w0) W.ref2 = (w1 + 1) >> 1;
    }
    W.e1.init();
    if constexpr (NL >= 2) W.e2.init();
    if constexpr (NL >= 3) W.e3.init();
    set_store_windows(a.mallat, a.mallat_elems * (long long)sizeof(S), a.ll,
                      a.ll_elems * (long long)sizeof(S), a.err);

    // everything above came from the parameters: wait for the previous grid
    // (its output is this launch's input) only now
    grid_dependency_wait();

    // ---- TMA ring prologue
    const uint32_t ring_s = smem_u32(ring);
    const uint32_t bar_s = smem_u32(bars);
    constexpr uint32_t kSlotBytes = kSlotElems * sizeof(S);
    const int y0 = 2 * qstart;
    if (lane == 0) {
        for (int b = 0; b < kFwdSlots; ++b) mbar_init(bar_s + 8 * b, 1);
        fence_mbar_init();
        for (int s = 0; s < kFwdSlots && s < nslots; ++s) {
            mbar_arrive_expect_tx(bar_s + 8 * s, kSlotBytes);
            tma_load_2d(ring_s + s * kSlotBytes, mapp, xb, y0 + s * SLOT_ROWS, bar_s + 8 * s);
        }
    }
    __syncwarp();

    // the border-free slots form one run [si0, si1): the test holds from some
    // slot on (rows far enough from the top) and up to some slot (clear of the
    // bottom), so two scans find it instead of one test per slot
    int si0 = nslots, si1 = nslots;
    if (active) {
        si0 = 0;
        while (si0 < nslots && !rows_interior(qstart + SR * si0, SR, NL, RHO, no_r)) ++si0;
        si1 = nslots;
        while (si1 > si0 && !rows_interior(qstart + SR * (si1 - 1), SR, NL, RHO, no_r)) --si1;
    }

    bool failed = false;
    int s = 0;
    for (; s < nslots; ++s) {
        const int b = s % kFwdSlots;
        const bool ok = mbar_wait_bounded(bar_s + 8 * b, (s / kFwdSlots) & 1, kWaitBudget);
        if (!__all_sync(kFull, ok)) {  // keep the warp's control flow uniform
            failed = true;
            break;
        }
        const int q0 = qstart + SR * s;
        if (s >= si0 && s < si1)
            W.template slot<kInner>(ring + b * kSlotElems, q0);
        else
            W.template slot<kEdgeRows>(ring + b * kSlotElems, q0);
        fence_proxy_async_smem();  // every lane: its reads and writes before the refill
        __syncwarp();
        if (lane == 0 && s + kFwdSlots < nslots) {
            mbar_arrive_expect_tx(bar_s + 8 * b, kSlotBytes);
            tma_load_2d(ring_s + b * kSlotBytes, mapp, xb, y0 + (s + kFwdSlots) * SLOT_ROWS,
                        bar_s + 8 * b);
        }
    }
    if (failed) {
        if (lane == 0) atomicExch(a.err, -6);
        // drain the copies still in flight before the warp leaves
        for (int t = s; t < nslots && t < s + kFwdSlots; ++t)
            mbar_wait_bounded(bar_s + 8 * (t % kFwdSlots), (t / kFwdSlots) & 1, kWaitBudget);
        return false;
    }
    // every copy has landed: the barriers may be initialised again
    if (lane == 0)
        for (int b = 0; b < kFwdSlots; ++b) mbar_inval(bar_s + 8 * b);
    __syncwarp();
    return true;
}

}  // namespace dwt
