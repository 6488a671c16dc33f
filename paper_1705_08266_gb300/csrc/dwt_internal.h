// Host/device argument blocks shared by the C ABI and the kernel files.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dwt2d.h"

namespace dwt {

constexpr int kMaxFused = 3;  // levels fused in one streaming launch

// Lifting schemes: separable (Sec. 2), non-separable and its reduced form (Sec. 3).
enum Scheme { SCH_SEP = 0, SCH_NONSEP = 1, SCH_RED = 2 };

// Geometry of one warp-streaming launch (forward or inverse, 1..3 levels).
struct LevelArgs {
    int h, w;     // extent this level transforms (image or LL of the level before)
    float s[4];   // forward: scale of LL, HL, LH, HH; inverse: its reciprocal
};

struct FusedArgs {
    LevelArgs lv[kMaxFused];
    // Mallat coefficient array (forward: written; inverse: read), element pitch
    void* mallat;
    long long mallat_pitch;
    // forward: LL of the last fused level is written here;
    // inverse: LL of the coarsest fused level is read from here
    void* ll;
    long long ll_pitch;
    // inverse only: the reconstructed image (or LL of the finest fused level - 1)
    void* out;
    long long out_pitch;
    int nstrips, nsegs, segq;        // warp work items = nstrips * nsegs
    int seg_f;                       // segment order interleave (<= 1: top to bottom)
    int seg_lo;                      // first row segment of this launch (launches over a subset)
    // segments [0, nbig) have segq rows (taken in seg_f interleaved groups);
    // segments [nbig, nsegs) are shorter, segq2 rows each, below them, taken
    // last and top to bottom (nbig == nsegs: every segment has segq rows)
    int nbig, segq2;
    long long mallat_elems, ll_elems, out_elems;  // buffer extents (elements) for checked builds
    int valid_px, xoff;              // strip width in input pixels and left halo offset
    int lane_lo, lane_hi;            // lanes that store
    int* err;                        // device status word (0 = ok)
    int pdl;                         // host: launch with programmatic stream serialization
    int ll_keep;                     // forward: store the LL with an L2 evict-last policy
    int min_smem;                    // host: shared memory of a CTA at least (limits the resident warps)
};


// Where a multipass kernel reads or writes a level's coefficients.
struct Layout {
    const void* p;       // kind 0: interleaved image layout; kind 1: Mallat array (details)
    long long pitch;     // elements
    const void* ll;      // kind 1: the LL band (may be inside p)
    long long ll_pitch;  // elements
    int kind;
};

// One pass of the multipass (off-chip exchange) scheme.
struct PassArgs {
    int h, w;          // extent of the level
    Layout src, dst;
    float s[4];        // per-component scale applied on load (scale_in) or store (scale_out)
    float coef;        // float lifting coefficient of this step, sign included
    int scale_in, scale_out;
};

// One image (one level group) of a batched launch, in device memory.  The
// tensor maps (128-byte aligned) come first.  The forward uses m[0];
// the inverse m[0] (Mallat, level-1 box), m[1] (Mallat, level-2 box), m[2]
// (LL source).
struct BatchEntry {
    CUtensorMap m[3];
    FusedArgs args;
    int first_warp;  // first global warp of this entry in the launch (queue mode: in its queue)
    // queue mode: the entry's fusion depth, its done counter (image, level
    // group) and the counter of the group it consumes (-1: none) with the
    // number of work items that group has
    int nl, self, dep, dep_items;
};

// Persistent batched kernels (queue mode): `grid` one-warp CTAs take the
// `total` work items of a queue (entries of one direction and storage type,
// every level group, ordered by group) through the counter `head`; an item of
// a later group first waits (bounded) until done[dep] reaches dep_items.
// q1: quadruple columns per lane (2 or 4) of every item in the queue.
// Warps per SM that the queue kernels' register budget keeps resident.
__host__ __device__ constexpr int fwd_queue_resident(int q1) { return q1 >= 4 ? 8 : 12; }
__host__ __device__ constexpr int inv_queue_resident(int q1) { return q1 >= 4 ? 8 : 12; }
cudaError_t launch_fwd_queue(int elem, int scheme, int q1, const BatchEntry* table, int n, int total,
                             int* head, int* done, int* err, int grid, cudaStream_t st);
cudaError_t launch_inv_queue(int elem, int scheme, int q1, const BatchEntry* table, int n, int total,
                             int* head, int* done, int* err, int grid, cudaStream_t st);

// Kernel-geometry constants of the streaming forward kernel.
// warps per CTA: each warp is independent, so one-warp CTAs let the CTA
// scheduler refill an SM warp by warp (measured 1-4 % faster than 4)
constexpr int kFwdWarps = 1;
constexpr int kFwdSlots = 3;        // TMA ring depth per warp
constexpr int kFwdSlotRows = 8;     // image rows per TMA box (4 quadruple rows) with 2 columns per lane

// First quadruple row of a work item, forward: a multiple of this.  A slot of
// 1 or 2 fused levels may start at any row or pair of rows (the LL rows of the
// lag pair up all the same), which saves the halo up to a slot against starts
// at a multiple of the slot; three levels pair rows across slots.
__host__ __device__ constexpr int fwd_row_align(int nl) { return nl == 1 ? 1 : (nl == 2 ? 2 : 4); }
// The same for the inverse (two levels: a whole level-2 row).
__host__ __device__ constexpr int inv_row_align(int nl) { return nl == 1 ? 1 : 2; }

// Warps of a forward launch resident per SM, which its kernel's register budget
// and the host's waves are sized by: 16 (128 registers); 12 (168) at 4 quadruple
// columns per lane for two levels, and for one of float32 or in plain
// non-separable steps; 8 for three fused levels.  Two levels at 4 columns, 16
// and 12 warps: float32 8192^2 101.7 and 99.2 us, 1080 x 1920 12.7 and 11.1; 5/3
// 8192^2 103.8 and 92.9; 16-bit 5 levels of 1080 x 1920 34.0 and 29.0.
constexpr int fwd_resident(int scheme, int nl, int q1, bool f32) {
    return nl >= 3 ? 8 : (q1 >= 4 && (nl == 2 || f32 || scheme == SCH_NONSEP) ? 12 : 16);
}

// A large float32 forward launch keeps 12 warps per SM in flight instead of the
// 16 its registers allow: it is bound by HBM, and fewer rows in flight share
// DRAM pages better.  Each warp asks for more shared memory than its ring
// takes, so that 12 fit the 228 KB of an SM (1 KB of it per CTA reserved; at 4
// columns per lane the registers allow no more either).
// Two levels, us, 16 / 12 warps: 2 columns per lane 6000^2 57.3 / 54.4, 3000 x
// 20000 89.8 / 86.5; 4 columns 6000 x 20000 169 / 163.6, 16384^2 367 / 354 (2
// columns of 8192^2: 98.2 / 94.1, 10 warps 95.9, 8 warps 97.6).  A launch of one
// wave keeps 16 (4096^2 28.1 and 28.5), and so do the inverse (88.6 and 90.3),
// 5/3 (86.9 and 86.6) and 16-bit storage, which is bound by its arithmetic (78
// and 80).
constexpr int kFwdLargeResident = 12;
constexpr int kFwdLargeSmem = 17920;

// Warps of an inverse launch (1 or 2 fused levels) resident per SM, which its
// kernel's register budget and the host's waves are sized by: 16 (128
// registers) with 2 quadruple columns per lane, 12 (168) with 4 (slots of 2
// quadruple rows) and for the plain non-separable steps (48 multiply-adds per
// quadruple).  Registers come to an SM's four schedulers in whole warps, so a
// bound of 9 to 11 warps gives the registers of 12; 8 (204 registers) is slower
// but for the smallest launches: plain 9/7, 5 levels of 2160 x 3840 30.9 us at
// 12 and 32.8 at 8.
constexpr int inv_resident(int q1, int scheme) { return q1 <= 2 && scheme != SCH_NONSEP ? 16 : 12; }

// Image rows per TMA box of the forward kernel: 8, or 4 with 4 quadruple
// columns per lane and at most 2 fused levels.
int fwd_slot_rows(int nl, int q1);
size_t fwd_smem_bytes(int elem_bytes, int nl, int q1);

// Batched forward / inverse: entries of one element type, scheme, fusion
// depth (1 or 2) and quadruple columns per lane q1 (2 or 4); `grid` CTAs of
// kFwdWarps (forward) or kInvTmaWarps (inverse) warps.
// Rings stay below the 48 KB of shared memory that need an opt-in, so a launch
// is a plain kernel launch.
cudaError_t launch_fwd_batched(int elem, int scheme, int nl, int q1, const BatchEntry* table, int n,
                               int grid, cudaStream_t st, bool pdl);
cudaError_t launch_inv_batched(int elem, int scheme, int nl, int q1, const BatchEntry* table, int n,
                               int grid, cudaStream_t st, bool pdl);

// Launch `kernel` on `st`; with `pdl` the grid is launched with programmatic
// stream serialization (it may be scheduled while the previous kernel in the
// stream drains, and waits in griddepcontrol.wait before its first global
// access).  Only kernels that issue that wait may be launched with `pdl`.
template <class... P, class... A>
cudaError_t launch_kernel(void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t st,
                          bool pdl, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<A&&>(args)...);
}

// q1: quadruple columns per lane at the first fused level (2 or 4; 3 fused levels need 4)
cudaError_t launch_fwd_fused(int elem, int scheme, int nl, int q1, const CUtensorMap& map,
                             const FusedArgs& a, int grid, cudaStream_t st);
cudaError_t launch_inv_fused(int elem, int scheme, int nl, const FusedArgs& a, int grid,
                             cudaStream_t st);

// TMA-fed inverse for 1 or 2 fused levels: m1 / m2 map the Mallat array with
// boxes {32 q1 + 4, 4} and {16 q1 + 4, 2}; ml maps the LL source with the
// level-1 box (1 level) or the level-2 box (2 levels).
cudaError_t launch_inv_tma(int elem, int scheme, int nl, int q1, const CUtensorMap& m1,
                           const CUtensorMap& m2, const CUtensorMap& ml, const FusedArgs& a,
                           int grid, cudaStream_t st);
size_t inv_tma_smem_bytes(int elem_bytes, int nl, int q1);
// Level-1 quadruple rows per slot of the TMA inverse: 4, or 2 with 4 columns per lane.
int inv_slot_rows(int q1);
constexpr int kInvTmaWarps = 1;  // one-warp CTAs, as the forward

// One level of the separable convolution scheme (Sec. 2, Eq. 1).
struct ConvArgs {
    int h, w;
    const void* src;   // the level's input (image or LL), element pitch
    long long src_pitch;
    void* dst;         // Mallat array (detail bands of this level)
    long long dst_pitch;
    void* ll;          // LL output of this level
    long long ll_pitch;
    float h0[9];       // analysis low pass, centred (k = -4 .. 4)
    float g0[7];       // analysis high pass, centred (k = -3 .. 3)
};
cudaError_t launch_conv_fwd(int elem, const ConvArgs& a, cudaStream_t st);

// elem: 0 = float32, 1 = int32.  kind: the step (see dwt_multipass.cu).
cudaError_t launch_pass(int elem, int kind, bool fwd, const PassArgs& a, cudaStream_t st);

enum PassKind { P_TH = 0, P_TV, P_SH, P_SV, P_T, P_S, P_TR, P_SR };

// Workspace bytes a plan needs (0 for a null plan).
size_t plan_workspace_bytes(dwt2d_plan_t p);

// The argument checks of dwt2d_forward / dwt2d_inverse (buffers, alignment,
// pitches, 16-bit scale, src != dst), without any GPU work.
dwt2d_status check_transform_args(dwt2d_plan_t p, const void* src, int64_t src_pitch_bytes,
                                  const void* dst, int64_t dst_pitch_bytes, const void* ws,
                                  float scale);

}  // namespace dwt
