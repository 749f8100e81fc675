// Mixed-precision persistent ray caster for deep sparse octrees (sm_103a).
//
// One lane traces one ray (Sec. 6 of the paper): from the FP64 eye (Sec. 6.1)
// leaf by leaf through the octree, compositing front to back, until the
// transmittance drops below t_min or the ray leaves the canvas (Sec. 6.2).
//
// Cells are addressed by exact integer coordinates: the canvas is 2^31 units
// wide, mirrored on the axes the ray runs down, so that every ray runs upwards
// and leaves a cell [X, X + s) through a plane X_a + s. The new leaf is found
// from the neighbouring cell: a sibling in the same record, else the slot the
// parent's neighbour link names (the neighbour graph of Sec. 4.1.1, built at
// upload), or, in the stack traversal, the common ancestor's record kept on a
// per-lane stack of records by level; then a descent while the cell is
// internal. Down to the old cell's level the path is in the cell's own bits;
// below it, in the bits of the ray's position, formed once per descent.
//
// Precision (Sec. 6.1-6.3). The ray is evaluated around an anchor, its FP64
// position at parameter t_f held as whole units A_a and a rest, in the local
// parameter t' = (t - t_f) / extent:
//     t'(X) = (X - A_a - rest_a) / |d_a| 2^-31.
// X - A_a is an exact integer, so every error is relative to the way from the
// anchor: the paper's cell-local frame (origin at a cell) with its origin at
// the ray instead. The anchor moves, in FP64, where the ray descends more than
// K levels below the level its last anchor was set for, where it enters a leaf
// coarser than that level (for K < 16 also where it leaves that level's cell),
// and where a decision was open while the leaf was less than 2^-16 of the way
// from the anchor wide; the drift of Sec. 6.3 (e0 + 7.5 eps L) does not
// accumulate across anchors. Decisions (which face of the leaf the ray leaves
// by, which side of a mid-plane it is on) are screened in plain FP32 with a
// proven margin, and taken in FP64 from the exact planes when the screen cannot
// decide (the ray passes within about 2^-21 of its way from the anchor of an
// edge or a plane: a few steps in a hundred thousand). The time of the exit
// face, which sets the segment length, is a double-float: an unevaluated sum
// hi + lo of two FP32 words formed with error-free transformations (Dekker's
// product by fma), good to 2^-44 of itself and 2^-24 of a unit. A boundary
// between leaves of different value moves the pixel by at most 2 T max(sigma)
// |dt|; each ray carries a budget for these bounds, and a boundary whose bound
// would exceed it is recomputed in FP64.
//
// A step settles the boundary behind it, not the one ahead: the new leaf's value
// is asked for last and first needed in the next step, for the colour bound of
// the boundary it was entered by and then to composite the leaf before it, while
// the next link is on its way. One dependent load of a step's five or six thus
// leaves the chain that a single long ray waits for (a 256^2 view of the depth-8
// cube, whose longest ray crosses 283 leaves, one after the other: 491 -> 444 us).
// The new slot then takes one load after the link, whichever way it is found
// (398 -> 359 us; three, one after the other, before).
//
// What bounds it: instruction issue (0.83 of the issue slots on a reduced
// depth-24 stereo view, 28 of 32 warps resident), the loads being served by L1
// and L2; for views of few leaves per ray the FP64 pipe (0.82 busy on the opaque
// depth-16 view, the per-ray set-up); for small views the longest ray's chain
// (0.10 of the issue slots on the cube). So the step holds to integers and few
// words: against frames of cells with planes as FP32 dyadics and two-word
// reciprocals per axis, it issues 1.26 G instead of 1.98 G warp instructions on
// that reduced view (1.37 ms instead of 2.45), without spills at 64 registers
// (four blocks an SM), and the set-up takes 57 % fewer FP64 instructions (the
// opaque view 0.31 ms instead of 0.73; the depth-24 stereo pair of 2160^2 30.3 ms
// instead of 47.3).
//
// Compositing (emission-absorption reading of Sec. 6.2): per segment of signed
// length l in a leaf (sigma, rgb): a = 1 - exp(-sigma l) (opacity.cuh), C += T a rgb,
// T *= 1 - a, with a compensated (Kahan) FP32 sum for C and the transmittance
// kept as a running product (one rounding per leaf, unbiased).
//
// The per-lane counters of slot reads, leaf loads and record loads (the
// algorithmic bytes of a render) are a template option: a render that does
// not report them runs without them.
#include <cuda_fp16.h>

#include "canvox_internal.cuh"
#include "cells.cuh"
#include "opacity.cuh"

namespace canvox {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr float kEpsF = 3.5762786865234375e-07f;    // 6 * 2^-24: the exit-face screen's relative margin
constexpr float kEpsG = 9.765625e-04f;              // 2^-10 = 2^31 * 2^-41: its absolute margin per ih
constexpr float kEpsX = 7.152557373046875e-07f;     // 12 * 2^-24: the position's relative error bound, doubled
constexpr float kEpsU = 9.5367431640625e-07f;       // 2^-20: its absolute one, in units
constexpr float kEpsT = 1.1368683772161603e-13f;    // 2^-43 = 2 * 2^-44: factor 2 of the colour bound, times the time's
constexpr float kEpsI = 1.1920928955078125e-07f;    // 2^-23 = 2 * 2^-24: the same, per ih
constexpr float kFar = 65536.0f;                    // a cell this many sides from the anchor asks for a new anchor
constexpr int kBoxLevels = 16;                      // frames of fewer levels also end where the ray leaves their cell
constexpr uint32_t kLeft = 4u;                      // (Ray::entry)
constexpr float kMaxWay = 2147483520.0f;            // the largest float below 2^31
constexpr float kBigF = 1.0e28f;                    // time per unit of an axis the ray never crosses (d_a = 0)

// Resident 256-thread blocks per SM the register allocation must allow (occupancy knob).
#ifndef CANVOX_MIN_BLOCKS
#define CANVOX_MIN_BLOCKS 4
#endif

// 1 / x to about an ulp (one instruction).
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

extern __shared__ int32_t s_nodes[];  // copy of the tree's first records (kernel instance with kSmem)

// Child slot k of record rec: from the shared-memory copy of the tree's breadth-first prefix when the
// kernel keeps one and the record is in it (records [0, n_smem)), else through the read-only data cache.
template <bool kSmem, int kPool>
__device__ __forceinline__ int32_t load_slot(const Tree& T, int32_t n_smem, int32_t rec, int k) {
    if (kSmem && rec < n_smem) return s_nodes[rec * 8 + k];
    if (kPool == kSmallPool) return __ldg(byte_offset(T.nodes, (uint32_t)rec * 32u + (uint32_t)k * 4u));
    return __ldg(T.nodes + (int64_t)rec * 8 + k);
}
// Link of record rec past its face 2 ax + s.
template <int kPool>
__device__ __forceinline__ uint2 load_link(const Tree& T, int32_t rec, int ax, uint32_t s) {
    if (kPool == kSmallPool) return __ldg(byte_offset(T.ropes, (uint32_t)rec * 48u + (uint32_t)ax * 16u + s * 8u));
    return __ldg(T.ropes + (int64_t)rec * 6 + 2 * ax + (int)s);
}

// Two FP32 operations in one instruction, on the words of a 64-bit register.
typedef unsigned long long pair32;
__device__ __forceinline__ pair32 pack2(float a, float b) {
    pair32 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ pair32 add2(pair32 a, pair32 b) {
    pair32 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pair32 sub2(pair32 a, pair32 b) {
    pair32 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pair32 mul2(pair32 a, pair32 b) {
    pair32 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// Kahan's compensated sum s (its compensation in c) of two channels.
__device__ __forceinline__ void kahan_add2(pair32& s, pair32& c, pair32 x) {
    const pair32 old = s, y = sub2(x, c), t = add2(old, y);
    c = sub2(sub2(t, old), y);
    s = t;
}
__device__ __forceinline__ void kahan_add(float2& sc, float x) {
    const float y = __fsub_rn(x, sc.y);
    const float t = __fadd_rn(sc.x, y);
    sc.y = __fsub_rn(__fsub_rn(t, sc.x), y);
    sc.x = t;
}

constexpr int kBlock = 256;

// Per-lane state in shared memory: the colour sums and the error budget of every step, and what only re-anchoring,
// near-ties, start-up and the final write read. One 8-byte column per field and lane, so that every field of a
// lane is its base address plus a constant, and 8-byte accesses of a warp meet no bank conflict. 128 bytes a
// lane: four blocks stay within the 132 KB carve-out, which leaves 124 KB of the SM to L1.
enum Col {
    kColInv = 0,    // double: 1 / |d_a| (0 for d_a = 0), three columns
    kColDir = 3,    // double: |d_a|, three columns
    kColTf = 6,     // double: FP64 ray parameter at the anchor
    kColAcc = 7,    // float2: sums of the colour channels 0, 1; their Kahan terms; (sum, Kahan term) of channel 2
    kColPix = 10,   // uint32: output pixel within the view; then the view
    kColCnt = 11,   // uint32: anchors, FP64 boundaries
    kColSum = 14,   // uint32: rays, leaf steps
    kColG = 15,     // float: 2^-41 max_a 1 / |d_a| over the axes with d_a != 0, the exit screen's margin; uint32: slot reads
    kColIl = 12,    // float: low words of ih on axes 0, 1; then axis 2 and (uint32) the axes with d_a = 0
    kCols = 16
};
constexpr int kLaneShared = kCols * 8;
static_assert(kLaneShared <= 128, "per-lane shared record: 128 bytes keep four blocks within the 132 KB carve-out");

struct Ray {
    char* base;                 // the lane's shared columns
    float ih[3];                // 1 / |d_a|, in canvas sides per unit: the first of two FP32 words (zero axis: kBigF)
    float rr[3];                // - (the anchor position's part below a unit) * ih
    uint32_t X[3];              // low corner of the current cell: mirrored, in units
    int32_t A[3];               // the anchor: the ray's position at local time 0, rounded to a unit
    float cur_hi, cur_lo;       // local parameter of the current leaf's entry
    float ell, dt;              // the leaf before: its segment's length, and the time bound of the boundary that ends it
    float T;
    float err;                  // colour-error bound spent so far (the budget of the FP32 boundaries)
    int32_t sh, fs;             // the current cell's side is 2^sh units; that of the frame (anchor's neighbourhood) 2^fs
    uint32_t flip;              // axes with d_a < 0: the canvas is mirrored there, so every ray runs upwards
    uint32_t entry;             // axis of the face the current leaf was entered by; kLeft: the ray has left the canvas
    uint2 val, pval;            // values of the current leaf and of the one before
    int32_t pr;   // record holding the current leaf's slot (neighbour-link traversal)
    uint32_t kc;  // child index of the current leaf in pr (not mirrored)
    int32_t steps;
    // counters, summed over every ray the lane traces
    uint32_t n_leaf, n_rec;

    template <typename V>
    __device__ __forceinline__ V& col(int c) { return *reinterpret_cast<V*>(base + (size_t)c * (8 * kBlock)); }
    __device__ __forceinline__ double& inv64(int a) { return col<double>(kColInv + a); }
    __device__ __forceinline__ double& dir64(int a) { return col<double>(kColDir + a); }
    __device__ __forceinline__ double& tf() { return col<double>(kColTf); }
    __device__ __forceinline__ pair32& acc01(int i) { return col<pair32>(kColAcc + i); }
    __device__ __forceinline__ float2& acc2() { return col<float2>(kColAcc + 2); }
    __device__ __forceinline__ uint32_t& pix() { return col<uint32_t>(kColPix); }
    __device__ __forceinline__ uint32_t& view() { return (&col<uint32_t>(kColPix))[1]; }
    __device__ __forceinline__ uint32_t& n_rebase() { return col<uint32_t>(kColCnt); }
    __device__ __forceinline__ uint32_t& n_f64() { return (&col<uint32_t>(kColCnt))[1]; }
    __device__ __forceinline__ uint32_t& n_rays() { return col<uint32_t>(kColSum); }
    __device__ __forceinline__ uint32_t& n_steps() { return (&col<uint32_t>(kColSum))[1]; }
    __device__ __forceinline__ float& il(int a) { return (&col<float>(kColIl + (a >> 1)))[a & 1]; }
    __device__ __forceinline__ float& gscr() { return col<float>(kColG); }
    __device__ __forceinline__ uint32_t& n_reads() { return (&col<uint32_t>(kColG))[1]; }
    __device__ __forceinline__ uint32_t& zmask() { return (&col<uint32_t>(kColIl + 1))[1]; }
};

__device__ __forceinline__ double mirrored_eye(const MixedParams& P, uint32_t view, uint32_t flip, int a) {
    const double o = P.views[view].eye[a];
    return ((flip >> a) & 1u) ? -o : o;
}

// Canvas position of the plane at x units: exact, as every cell plane of the canvas is.
__device__ __forceinline__ double plane64(double unit, double half, uint32_t x) { return fma((double)x, unit, -half); }

// FP64 crossing time of the plane M on axis a.
__device__ __forceinline__ double time64(Ray& r, const MixedParams& P, int a, double M) {
    return (M - mirrored_eye(P, r.view(), r.flip, a)) * r.inv64(a);
}

// The ray is on the high side of the plane M of axis a just after parameter t (mirrored: it moves upwards; a ray
// that lies in the plane is on the high side of the canvas's own axis, which d_a = 0 never mirrors).
__device__ __forceinline__ uint32_t high64(Ray& r, const MixedParams& P, int a, double M, double t) {
    const double dist = M - mirrored_eye(P, r.view(), r.flip, a);
    if ((r.zmask() >> a) & 1u) return dist <= 0.0;
    return dist * r.inv64(a) <= t;
}

// Exit axis of the leaf with the far corner Y by the FP64 crossing times of its exact far planes, ties to the lowest
// axis. Taken on a few leaf steps in a hundred thousand (a ray within about 2^-22 of its way from the anchor of
// an edge), so it is kept out of line: its FP64 code then does not weigh on the register allocation of the step
// loop.
__device__ __noinline__ int exit_axis64(char* base, const View* views, double unit, double half, uint32_t flip,
                                        uint32_t Y0, uint32_t Y1, uint32_t Y2) {
    Ray r;
    r.base = base;
    double best = __longlong_as_double(0x7FF0000000000000ll);
    int ax = 0;
    const uint32_t zm = r.zmask();
    const View& V = views[r.view()];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if ((zm >> a) & 1u) continue;
        const double M = plane64(unit, half, a == 0 ? Y0 : (a == 1 ? Y1 : Y2));
        const double t = (M - (((flip >> a) & 1u) ? -V.eye[a] : V.eye[a])) * r.inv64(a);
        if (t < best) {
            best = t;
            ax = a;
        }
    }
    return ax;
}

// On an axis with d_a = 0 the anchor is the unit the eye is in, not the nearest one: the rest, which has no time there, is
// dropped, so an anchor rounded up to the cell's far plane would put that plane at distance 0 and local time 0 and have
// the ray leave by a face it runs along. Rounded down, every far plane is at least a unit ahead, at kBigF or later,
// past the time of every other face. (A branch of its own: few rays take it, and formed for every ray it cost the
// opaque 1920 x 1080 view 3 %.)
__device__ __forceinline__ void anchor_zero_axes(Ray& r, const View& V) {
    const uint32_t zm = r.zmask();
    if (zm == 0u) return;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (!((zm >> a) & 1u)) continue;
        const long long rest = __double_as_longlong(V.eye_rest[a]);  // (below 0: the sign bit set, and not -0)
        // (eye_unit is 0 only for an eye on the low face: a ray that meets the canvas has its eye within it on such an axis)
        r.A[a] = V.eye_unit[a] ? V.eye_unit[a] - (rest < 0 && (rest << 1) != 0 ? 1 : 0) : __double2int_rd(V.eye_rest[a]);
    }
}

// Anchor the ray at FP64 parameter t: local time 0, at the ray's position there, which is formed from the eye's
// (a whole number of units and a rest of a unit at most, so that it keeps its precision near the eye). On axis
// ax (the face just crossed; -1: none) it is the current cell's low plane exactly.
__device__ __forceinline__ void set_anchor(Ray& r, const MixedParams& P, const View& V, double t, int ax) {
    r.tf() = t;
    const double ts = t * P.inv_extent * 2147483648.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        uint32_t u = (uint32_t)V.eye_unit[a];
        double p = V.eye_rest[a];
        if ((r.flip >> a) & 1u) {
            p = u ? -p : 2147483648.0 - p;
            u = u ? 0x80000000u - u : 0u;
        }
        if (t != 0.0) p = fma(ts, r.dir64(a), p);
        if (a == ax) {
            u = r.X[a];
            p = 0.0;
        }
        // kept within 1 .. 2^31 - 1: every far plane is then less than 2^31 units ahead
        const int64_t x = (int64_t)u + (int64_t)__double2int_rn(p);
        r.A[a] = (int32_t)min(max(x, (int64_t)1), (int64_t)0x7FFFFFFF);
        // (with both words of the reciprocal: the rest's time then adds 2^-24 ih at most to an exit time's error)
        const float rest = (float)(p - (double)(int32_t)((uint32_t)r.A[a] - u));
        r.rr[a] = r.ih[a] == kBigF ? 0.0f : -__fmaf_rn(rest, r.ih[a], rest * r.il(a));
    }
    anchor_zero_axes(r, V);
    r.cur_hi = 0.0f;
    r.cur_lo = 0.0f;
    r.n_rebase() += 1;
}

// The anchor at the eye itself (of a view with the eye inside the canvas and eye_unit set): no FP64 arithmetic.
__device__ __forceinline__ void set_anchor_eye(Ray& r, const View& V) {
    r.tf() = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const bool m = (r.flip >> a) & 1u;
        const float rest = m ? -(float)V.eye_rest[a] : (float)V.eye_rest[a];
        r.A[a] = m ? (int32_t)(0x80000000u - (uint32_t)V.eye_unit[a]) : V.eye_unit[a];
        r.rr[a] = r.ih[a] == kBigF ? 0.0f : -__fmaf_rn(rest, r.ih[a], rest * r.il(a));
    }
    anchor_zero_axes(r, V);
    r.cur_hi = 0.0f;
    r.cur_lo = 0.0f;
    r.n_rebase() += 1;
}

// Composite the leaf before the current one. The length is not clamped at
// zero: a boundary can land slightly before the cursor (within its error
// bound), and only the signed lengths of consecutive segments telescope, so a
// boundary between two leaves of equal value then costs nothing.
__device__ __forceinline__ void composite(Ray& r) {
    if (r.pval.y >> 16) {
        const float s = hsig(r.pval);
        const float em = expm1_neg(s * r.ell);  // -a
        const float w = -r.T * em;
        pair32 s01 = r.acc01(0), c01 = r.acc01(1);
        float2 s2 = r.acc2();
        kahan_add2(s01, c01, mul2(pack2(w, w), pack2(hlo(r.pval.x), hhi(r.pval.x))));
        kahan_add(s2, w * hlo(r.pval.y));
        r.acc01(0) = s01;
        r.acc01(1) = c01;
        r.acc2() = s2;
        r.T = __fmaf_rn(r.T, em, r.T);  // T (1 - a)
    }
}

__device__ __forceinline__ void finish(Ray& r, const MixedParams& P) {
    const View& V = P.views[r.view()];
    float4 o;
    const float2 rg = r.col<float2>(kColAcc);
    o.x = rg.x + r.T * V.bg[0];
    o.y = rg.y + r.T * V.bg[1];
    o.z = r.acc2().x + r.T * V.bg[2];
    o.w = 1.0f - r.T;
    const int64_t pix = V.out_offset + (int64_t)r.pix();
    P.out[pix] = o;
    if (P.step_count) P.step_count[pix] = r.steps;
    r.n_rays() += 1;
    r.n_steps() += (uint32_t)r.steps;
}

// The ray's position on axis a at the local time th, in units, within the cell [X, X + s): its bits are the
// sides of every finer mid-plane at once. The way from the anchor, x = (th - rr) / ih, carries a relative error of
// at most 6 * 2^-24 (th for th + tl, rr, ih, the reciprocal, the product) and, where th and rr cancel, 2^-24 units;
// bits in which the ends of twice that interval differ, and all bits below them, are open (returned in `open`).
__device__ __forceinline__ uint32_t locate(const Ray& r, int a, float th, uint32_t s, uint32_t& open) {
    const float x = __fsub_rn(th, r.rr[a]) * rcp_approx(r.ih[a]);
    const float e = __fmaf_rn(fabsf(x), kEpsX, kEpsU);
    // from the cell's low corner
    const uint32_t l = (uint32_t)r.A[a] - r.X[a] + (uint32_t)__float2int_rd(__fsub_rn(x, e));
    const uint32_t h = (uint32_t)r.A[a] - r.X[a] + (uint32_t)__float2int_rd(__fadd_rn(x, e));
    // An interval that reaches past the cell, or lies past it, leaves every bit open: at a corner the next plane can come out
    // a little before the last one (an FP64 time from a far eye, around an anchor next to it), and the bits of a position
    // below the cell are those of its far end.
    open = (l ^ h) | ((l | h) & ~(s - 1u));
    return r.X[a] | (l & (s - 1u));
}

// Sides of the mid-planes of the cell that q's bits above `sh` name, on every axis but ax, just after FP64 time t:
// sets those bits of q (the bits below them are left open).
__device__ __forceinline__ void sides64(Ray& r, const MixedParams& P, int sh, int ax, double t, uint32_t q[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (a == ax) continue;
        const uint32_t lo = (q[a] >> sh) & ~1u;  // even: the cell's low half
        q[a] = (lo | high64(r, P, a, plane64(P.unit, P.tree.half, (lo + 1u) << sh), t)) << sh;
    }
}

// 1 / |d| in canvas sides per unit as two FP32 words, hi the leading 24 bits (truncated), lo the other 29 rounded.
// The reciprocal is at least about 1; one past the FP32 range gives infinity, which no screen decides on.
__device__ __forceinline__ void split_inv(double inv, float& hi, float& lo) {
    const long long b = __double_as_longlong(inv);
    const int e = (int)(b >> 52) - 1023 - kFix;  // exponent after the scaling by 2^-31
    if (e > 127) {
        hi = __int_as_float(0x7F800000);
        lo = 0.0f;
        return;
    }
    hi = __int_as_float(((e + 127) << 23) | ((int)(b >> 29) & 0x7FFFFF));
    lo = __int2float_rn((int)(b & 0x1FFFFFFF)) * __int_as_float((e + 127 - 52) << 23);
}

// Frame level for a leaf at level L that has descended past its frame, and for a ray's first frame at the eye's
// leaf: the level depth - K that holds the canvas's deepest leaves within K levels, kept within [L - K, L].
__device__ __forceinline__ int deep_frame(int L, int depth, int K) { return max(L - K, min(max(0, depth - K), L)); }

// Start ray g of the launch. Returns true if it has a leaf to step from.
template <bool kSmem, bool kRopes, bool kCount, int kPool>
__device__ bool ray_init(Ray& r, const MixedParams& P, unsigned long long g, int32_t* stk) {
    const Tree& T = P.tree;
    g += (unsigned long long)P.ray_base;
    int lo = 0, hi = P.n_views - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((unsigned long long)P.views[mid].ray_begin <= g) lo = mid;
        else hi = mid - 1;
    }
    const View& V = P.views[lo];
    const long long local = (long long)g - V.ray_begin;
    const unsigned tile = (unsigned)(local >> 5);  // tiles of one view fit 32 bits (width, height < 2^31)
    const int lane = (int)(local & 31);
    const unsigned ty = tile / (unsigned)V.tiles_x;
    const int wl = V.tile_wl;
    const int i = ((int)(tile - ty * (unsigned)V.tiles_x) << wl) + (lane & ((1 << wl) - 1));
    const int j = (int)ty * (32 >> wl) + (lane >> wl);
    if (i >= V.width || j >= V.height) return false;  // padding lane of a ragged tile
    r.view() = (uint32_t)lo;
    r.pix() = (uint32_t)j * (uint32_t)V.width + (uint32_t)i;
    r.acc01(0) = r.acc01(1) = 0;
    r.acc2() = make_float2(0.0f, 0.0f);
    r.T = 1.0f;
    r.err = 0.0f;
    r.steps = 0;
    // pixel-centre ray in FP64 (Sec. 6.1), mirrored so that it runs upwards on every axis. Signs, zeros and the FP32
    // words of the reciprocals are taken from the FP64 patterns by integer operations (this GPU's FP64 pipe, which
    // also converts, runs at 1/64 of the FP32 rate).
    double d[3];
    pixel_ray(V, i, j, d);
    r.flip = 0;
    uint32_t zmask = 0;
    float g_inv = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const long long bits = __double_as_longlong(d[a]);
        const long long mag = bits & 0x7FFFFFFFFFFFFFFFll;
        const double da = __longlong_as_double(mag);
        r.dir64(a) = da;
        if (mag != 0) {
            if (bits < 0) r.flip |= 1u << a;
            // (below 2^-1007 the reciprocal nears infinity, which is no time: 0 for a plane the eye is on, else past all)
            const double inv = mag > 0x0100000000000000ll ? rcp64(da) : 1.0e300;
            r.inv64(a) = inv;
            split_inv(inv, r.ih[a], r.il(a));
            g_inv = fmaxf(g_inv, r.ih[a]);
            if (!(r.ih[a] < kBigF)) {  // never crossed either, within FP32's range (no screen decides: g_inv)
                r.ih[a] = kBigF;
                r.il(a) = 0.0f;
            }
        } else {
            r.inv64(a) = 0.0;
            r.ih[a] = kBigF;
            r.il(a) = 0.0f;
            zmask |= 1u << a;
        }
    }
    r.zmask() = zmask;
    r.gscr() = kEpsG * g_inv;
    const EyePath& E = P.eye[lo];
    double t0 = 0.0;
    if (E.len == 0) {
        // an eye outside the canvas or on a cell plane: the ray's entry
        double t1 = __longlong_as_double(0x7FF0000000000000ll);
        bool miss = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double o = ((r.flip >> a) & 1u) ? -V.eye[a] : V.eye[a];
            if ((zmask >> a) & 1u) {
                if (!(o >= -T.half && o < T.half)) miss = true;
            } else {
                t0 = fmax(t0, (-T.half - o) * r.inv64(a));
                t1 = fmin(t1, (T.half - o) * r.inv64(a));
            }
        }
        if (miss || !(t0 < t1)) {
            finish(r, P);
            return false;
        }
    }
    if (E.len > 0 && V.eye_unit[0] > 0 && V.eye_unit[1] > 0 && V.eye_unit[2] > 0) set_anchor_eye(r, V);
    else set_anchor(r, P, V, t0, -1);
    r.pval = make_uint2(0u, 0u);  // (nothing before the first leaf)
    r.ell = r.dt = 0.0f;
    r.entry = 0;
    if (E.len > 0) {
        // the eye's leaf, located once for the view
        r.sh = kFix - E.len;
        if (kRopes) {
            r.pr = E.rec[E.len - 1];
            r.kc = (E.c[0] & 1u) | ((E.c[1] & 1u) << 1) | ((E.c[2] & 1u) << 2);
        } else {
            for (int l = 0; l < E.len; ++l) stk[l] = E.rec[l];
        }
        const uint32_t last = (1u << E.len) - 1u;
#pragma unroll
        for (int a = 0; a < 3; ++a) r.X[a] = (((r.flip >> a) & 1u) ? last - E.c[a] : E.c[a]) << (kFix - E.len);
        r.val = E.val;
        if (kCount) atomicAdd(&r.n_reads(), (uint32_t)(E.len));
        if (kCount) r.n_leaf += (uint32_t)E.stored;
    } else {
        // locate the leaf that holds r(t0+) from the root
        uint32_t q[3], open = 0u;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int32_t x = r.A[a];  // 1 .. 2^31 - 1, within a unit of the ray's entry
            q[a] = (uint32_t)x;
            open |= (uint32_t)(max(x - 2, 0) ^ (int32_t)min((uint32_t)x + 2u, 0x7FFFFFFFu));
        }
        int sh = kFix;
        int32_t rec = 0, slot = 0;
        do {
            rec = slot;
            if (!kRopes) stk[kFix - sh] = rec;
            --sh;
            if (open >> sh) sides64(r, P, sh, -1, t0, q);
            r.kc = (uint32_t)child_index_any(q, sh, r.flip);
            slot = load_slot<kSmem, kPool>(T, P.smem_records, rec, (int)r.kc);
            if (kCount) r.n_rec += 1;
        } while (slot > 0);
        r.pr = rec;
        r.sh = sh;
        if (kCount) atomicAdd(&r.n_reads(), (uint32_t)(kFix - sh));
        r.val = make_uint2(0u, 0u);
        if (slot < 0) {
            r.val = load_leaf<kPool>(T, rec, (int)r.kc, slot);
            if (kCount) r.n_leaf += 1;
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) r.X[a] = (q[a] >> sh) << sh;
    }
    // the frame a descent would settle in (depth - K, within [L - K, L]): rays that start in a deep subtree are not
    // anchored again on their first descent past the first leaf's frame
    r.fs = kFix - deep_frame(kFix - r.sh, T.depth, P.frame_levels);
    return true;
}

// One leaf step. Returns false once the ray is finished (its pixel written).
template <bool kSmem, bool kRopes, bool kCount, int kPool>
__device__ bool ray_step(Ray& r, const MixedParams& P, int32_t* stk) {
    const Tree& T = P.tree;
    // 1. exit of the current leaf: the far planes' distances from the anchor (exact integers) and their times.
    // F_a = fma(float(D_a), ih, rr) is within 3.01 * 2^-24 |F_a| + 2^-24 |rr| of the exact time of its words; when
    // the runner-up F_s exceeds the smallest F_b by more than 6 * 2^-24 (|F_s| + |F_b|) + gscr, F_b's face is the
    // exit face and only its double-float time is formed. Otherwise (a ray that passes within about 2^-22 of its way
    // from the anchor of an edge of the leaf) the face is chosen in FP64 from the exact planes.
    const uint32_t s = 1u << r.sh;
    const int32_t D0 = (int32_t)(r.X[0] + s - (uint32_t)r.A[0]);
    const int32_t D1 = (int32_t)(r.X[1] + s - (uint32_t)r.A[1]);
    const int32_t D2 = (int32_t)(r.X[2] + s - (uint32_t)r.A[2]);
    const float g0 = __int2float_rn(D0), g1 = __int2float_rn(D1), g2 = __int2float_rn(D2);
    int ax = 0;
    bool rebase = false, fexit = false;
    {
        const float F0 = __fmaf_rn(g0, r.ih[0], r.rr[0]);
        const float F1 = __fmaf_rn(g1, r.ih[1], r.rr[1]);
        const float F2 = __fmaf_rn(g2, r.ih[2], r.rr[2]);
        float Fb = F0;
        if (F1 < Fb) { ax = 1; Fb = F1; }
        if (F2 < Fb) { ax = 2; Fb = F2; }
        const float Fs = fmaxf(fminf(F0, F1), fminf(fmaxf(F0, F1), F2));  // the median: runner-up
        const bool clear = __fsub_rn(Fs, Fb) > __fmaf_rn(kEpsF, __fadd_rn(fabsf(Fs), fabsf(Fb)), r.gscr());
        if (!clear && !(r.entry & kLeft)) {
            ax = exit_axis64(r.base, P.views, P.unit, T.half, r.flip, r.X[0] + s, r.X[1] + s, r.X[2] + s);
            rebase = fabsf(pick(ax, g0, g1, g2)) > kFar * (float)s;
        }
    }
    const float ihx = pick(ax, r.ih[0], r.ih[1], r.ih[2]);
    float teh, tel;
    {
        // te = D ih + rr as hi + lo: D as two FP32 words, the product's error from one fma (Dekker). Within
        // 2^-45 |te| + 2^-25 ih. (dh at most the float below 2^31: rounded up to 2^31 itself, as for the canvas's far face
        // seen from its near one, it is past the largest integer, and the conversion back would leave dl a unit short.)
        const int32_t D = pick(ax, D0, D1, D2);
        const float dh = fminf(__int2float_rn(D), kMaxWay), dl = __int2float_rn(D - __float2int_rn(dh));
        const float p = __fmul_rn(dh, ihx);
        const float lo = __fadd_rn(__fmaf_rn(dh, r.il(ax),
                                             __fmaf_rn(dl, ihx, __fmaf_rn(dh, ihx, -p))),
                                   pick(ax, r.rr[0], r.rr[1], r.rr[2]));
        teh = __fadd_rn(p, lo);
        tel = __fsub_rn(lo, __fsub_rn(teh, p));
    }
    // 2. the neighbour across the exit face: its low corner is N on that axis. Its link is asked for here, and the
    //    boundary that ended the leaf before (whose other side, the current leaf's value, was still on its way when
    //    that leaf was left) is settled while the link arrives
    const uint32_t N = pick(ax, r.X[0], r.X[1], r.X[2]) + s;
    const bool linked = kRopes && !(N & s);  // not the high half of the same parent
    uint2 rp = make_uint2(0u, 0u);
    if (linked) rp = load_link<kPool>(T, r.pr, ax, ((r.flip >> ax) & 1u) ^ 1u);
    {
        const float bound = r.T * fmaxf(hsig(r.pval), hsig(r.val)) * r.dt;
        const float spent = r.err + (((r.val.x ^ r.pval.x) | (r.val.y ^ r.pval.y)) ? bound : 0.0f);
        if (spent > P.err_budget) {
            // the boundary in FP64: the low plane, on the axis it was entered by, of the current cell (past the
            // canvas, the canvas's far plane)
            const int a = (int)(r.entry & 3u);
            const double M = plane64(P.unit, T.half, pick(a, r.X[0], r.X[1], r.X[2]));
            const double tl = (time64(r, P, a, M) - r.tf()) * P.inv_extent;
            const float hi = (float)tl, lo = (float)(tl - (double)hi);
            r.ell += ((hi - r.cur_hi) + (lo - r.cur_lo)) * P.side;
            r.cur_hi = hi;
            r.cur_lo = lo;
            r.n_f64() += 1;
        } else {
            r.err = spent;
        }
    }
    composite(r);
    const bool done = (r.entry & kLeft) || (r.steps != 0 && r.T < P.t_min);
    if (done || r.steps >= P.steps) {
        if (!done) {
            atomicOr(&P.scratch->status, 1ull);
            atomicAdd(&P.scratch->stats[kStatStepLimited], 1ull);
        }
        finish(r, P);
        return false;
    }
    r.steps += 1;
    // 3. the current leaf's segment; where its end's time must be exact, in FP64 (formed anew where it is asked for
    //    twice, so that it is not carried through the descent)
    bool have64 = false;
    auto exact_time = [&]() {
        uint32_t x = N;
        asm volatile("" : "+r"(x));  // (formed here: hoisted out of the descent, it cost every step 9 % more instructions)
        const double t64 = time64(r, P, ax, plane64(P.unit, T.half, x));
        const double tl = (t64 - r.tf()) * P.inv_extent;
        teh = (float)tl;
        tel = (float)(tl - (double)teh);
        if (!have64) r.n_f64() += 1;
        have64 = true;
        return t64;
    };
    // 4. the new leaf: start at the neighbouring cell (a sibling, the parent's neighbour link, or the common ancestor on
    //    the stack), then descend while the cell is internal. The ray's way down to the old level is in the cell's own
    //    coordinates; below it, in the bits of the ray's position. Past the canvas the new leaf is an empty one, which
    //    only settles the last boundary (its link reads as an empty slot).
    uint32_t q[3] = {ax == 0 ? N : r.X[0], ax == 1 ? N : r.X[1], ax == 2 ? N : r.X[2]};
    const uint32_t left = N >> kFix;
    const int sh_old = r.sh;
    int lstar = 0;  // level of the common ancestor (stack traversal and counters only; -1 past the canvas)
    if (!kRopes || kCount) lstar = (kFix - 1) - (31 - __clz((N - s) ^ N));
    int32_t prec, slot;
    int kk, sh = sh_old;
    if (kRopes) {
        // one load for every lane: a sibling's slot, the slot a link names, or, where the parent's neighbour is an internal
        // cell (named by its own record), that of its child next to the old cell, which has a sibling's index; past the
        // canvas the root's, unused
        prec = r.pr;
        kk = (int)(r.kc ^ (1u << ax));
        if (kCount && linked && !left) r.n_rec += 1;
        const bool named = linked && !(rp.y & kLinkRecord);
        prec = linked ? (int32_t)rp.x : prec;
        kk = named ? (int)(rp.y >> 8) : kk;
        sh = named ? (int)(rp.y & 255u) : sh;
        slot = load_slot<kSmem, kPool>(T, P.smem_records, prec, kk);
        if (left) slot = 0;
        if (kCount && !left) r.n_rec += 1;
    } else {
        prec = kk = slot = 0;
        if (!left) {
            prec = stk[lstar];
            sh = kFix - 1 - lstar;
            for (;;) {
                kk = child_index_any(q, sh, r.flip);
                slot = load_slot<kSmem, kPool>(T, P.smem_records, prec, kk);
                if (kCount) r.n_rec += 1;
                if (slot <= 0 || sh == sh_old) break;
                stk[kFix - sh] = slot;
                prec = slot;
                --sh;
            }
        }
    }
    if (slot > 0) {
        // finer than the old cell: near side on the exit axis, the ray's position on the others
        uint32_t o0, o1, o2;
        const uint32_t q0 = locate(r, 0, teh, s, o0), q1 = locate(r, 1, teh, s, o1), q2 = locate(r, 2, teh, s, o2);
        q[0] = ax == 0 ? N : q0;
        q[1] = ax == 1 ? N : q1;
        q[2] = ax == 2 ? N : q2;
        const uint32_t open = (ax == 0 ? 0u : o0) | (ax == 1 ? 0u : o1) | (ax == 2 ? 0u : o2);
        do {
            if (!kRopes) stk[kFix - sh] = slot;
            --sh;
            if (open >> sh) {
                sides64(r, P, sh, ax, exact_time(), q);
                rebase = rebase || fabsf(teh) > kFar * ihx * (float)(1u << sh);
            }
            prec = slot;
            kk = child_index(q, sh, r.flip);
            slot = load_slot<kSmem, kPool>(T, P.smem_records, prec, kk);
            if (kCount) r.n_rec += 1;
        } while (slot > 0);
    }
    if (kCount && !left) atomicAdd(&r.n_reads(), (uint32_t)((uint32_t)(kFix - sh - lstar)));
    r.pval = r.val;
    r.val = make_uint2(0u, 0u);
    if (slot < 0) {
        r.val = load_leaf<kPool>(T, prec, kk, slot);
        if (kCount) r.n_leaf += 1;
    }
    rebase = rebase || (uint32_t)(r.fs - sh) > (uint32_t)P.frame_levels;
    if (P.frame_levels < kBoxLevels && (((N - s) ^ N) >> r.fs) != 0u) rebase = fexit = true;
    rebase = rebase && !left;
    if (kRopes) {
        r.pr = prec;
        r.kc = (uint32_t)kk;
    }
    r.entry = (uint32_t)ax | (left * kLeft);
    r.sh = sh;
#pragma unroll
    for (int a = 0; a < 3; ++a) r.X[a] = (q[a] >> sh) << sh;
    if (rebase) {
        const double te64 = exact_time();
        r.ell = ((teh - r.cur_hi) + (tel - r.cur_lo)) * P.side;
        // a leaf coarser than the frame takes the coarsest frame that holds it; a descent past the frame the deepest
        // one the canvas can need, so that deeper leaves do not anchor the ray again level by level
        const int L = kFix - sh;
        r.fs = kFix - (fexit || sh > r.fs ? max(0, L - P.frame_levels) : deep_frame(L, T.depth, P.frame_levels));
        set_anchor(r, P, P.views[r.view()], te64, ax);
    } else {
        r.ell = ((teh - r.cur_hi) + (tel - r.cur_lo)) * P.side;
        r.cur_hi = teh;
        r.cur_lo = tel;
    }
    r.dt = have64 ? 0.0f : __fmaf_rn(P.bound_t, fabsf(teh), P.bound_i * ihx);
    return true;
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    return v;
}

template <bool kSmem, bool kRopes, bool kCount, int kPool>
__global__ void __launch_bounds__(kBlock, CANVOX_MIN_BLOCKS) mixed_kernel(MixedParams P) {
    __shared__ double lanes[kCols * kBlock];
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the set-up launch (views, eye paths, queue head)
    if (kSmem) {
        for (int i = threadIdx.x; i < P.smem_records * 8; i += blockDim.x) s_nodes[i] = __ldg(P.tree.nodes + i);
        __syncthreads();
    }
    int32_t stk[kRopes ? 1 : kMaxDepth + 1];  // ancestors by level (stack traversal only)
    Ray r;
    r.base = reinterpret_cast<char*>(&lanes[threadIdx.x]);
    r.n_f64() = r.n_rebase() = r.n_rays() = r.n_steps() = 0;
    r.n_reads() = 0;
    r.n_leaf = r.n_rec = 0;
    const unsigned lane = threadIdx.x & 31u;
    bool alive = false;
    bool drained = false;
    for (;;) {
        unsigned busy = __ballot_sync(kFull, alive);
        if (!drained && __popc(busy) <= P.refill) {
            unsigned long long g = (unsigned long long)P.total_rays;
            if (P.per_block) {
                const unsigned w = threadIdx.x >> 5;
                if (w < (unsigned)P.per_block && lane < (unsigned)P.take)
                    g = (blockIdx.x * (unsigned)P.per_block + w) * (unsigned)P.take + lane;
                drained = true;
            } else {
                const unsigned idle = ~busy;
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(P.queue, (unsigned long long)__popc(idle));
                base = __shfl_sync(kFull, base, 0);
                if (base + __popc(idle) >= (unsigned long long)P.total_rays) drained = true;
                if (!alive) g = base + __popc(idle & ((1u << lane) - 1u));
            }
            if (g < (unsigned long long)P.total_rays) alive = ray_init<kSmem, kRopes, kCount, kPool>(r, P, g, stk);
            busy = __ballot_sync(kFull, alive);
            if (!drained && __popc(busy) <= P.refill) continue;
        }
        if (busy == 0u) {
            if (drained) break;
            continue;
        }
        do {
            if (alive) alive = ray_step<kSmem, kRopes, kCount, kPool>(r, P, stk);
            busy = __ballot_sync(kFull, alive);
            // (refill 0, the default: run until every lane is done; the uniform test skips the count)
        } while (busy != 0u && (drained || P.refill == 0 || __popc(busy) > P.refill));
    }
    const unsigned long long v[7] = {r.n_rays(), r.n_steps(), kCount ? r.n_reads() : 0u, kCount ? r.n_leaf : 0u,
                                     kCount ? r.n_rec : 0u, r.n_f64(), r.n_rebase()};
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const unsigned long long s = warp_sum(v[i]);
        if (lane == 0 && s) atomicAdd(&P.scratch->stats[i], s);
    }
}

}  // namespace

template <bool kRopes, bool kCount, int kPool>
cudaError_t launch_mixed_t(const MixedParams& p, int grid, int block, cudaStream_t s, bool after_setup) {
    void (*kernel)(MixedParams) = mixed_kernel<false, kRopes, kCount, kPool>;
    int smem = 0;
    if (p.smem_records > 0) {
        // static (per-lane records) plus dynamic shared memory passes the 48 KB default: always opt in
        kernel = mixed_kernel<true, kRopes, kCount, kPool>;
        smem = p.smem_records * 32;
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    // a captured launch keeps its plain edge: graph queries of callers need not know programmatic ones
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (!after_setup || cudaStreamIsCapturing(s, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone) {
        kernel<<<grid, block, smem, s>>>(p);
        return cudaGetLastError();
    }
    cudaLaunchAttribute overlap;
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cfg.attrs = &overlap;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

template <bool kRopes, bool kCount>
cudaError_t launch_mixed_w(const MixedParams& p, int grid, int block, cudaStream_t s, bool after_setup) {
    switch (pool_kind(p.tree)) {
        case kSmallPool: return launch_mixed_t<kRopes, kCount, kSmallPool>(p, grid, block, s, after_setup);
        case kPlainPool: return launch_mixed_t<kRopes, kCount, kPlainPool>(p, grid, block, s, after_setup);
        default: return launch_mixed_t<kRopes, kCount, kWrapPool>(p, grid, block, s, after_setup);
    }
}

cudaError_t launch_mixed(const MixedParams& params, int grid, int block, cudaStream_t s, bool after_setup) {
    MixedParams p = params;
    p.inv_extent = 1.0 / p.tree.extent;
    p.unit = p.tree.extent * 4.656612873077393e-10;  // 2^-31
    p.side = (float)p.tree.extent;
    p.bound_t = kEpsT * p.side;
    p.bound_i = kEpsI * p.side;
    p.steps = (int32_t)(p.step_limit < 0x7FFFFFFF ? p.step_limit : 0x7FFFFFFF);
    // Rays that fit the resident lanes are dealt out evenly, neighbouring ones to the warps of a block, instead of to
    // whichever warp asks first (the first blocks: some SMs then work for others). While half of the resident warps
    // would do, a warp takes half as many rays, down to one: a warp's steps follow every path that one of its lanes
    // takes, and a small launch waits for the longest ray's chain of steps. Beyond half, the FP64 set-up of a warp, the
    // same for one lane as for 32, and the shared issue slots cost more than that (256 x 256 pixels of the depth-24
    // canvas: 443 us with 16 rays a warp, 383 with 32). From the queue by 32, dealt out by 32 and by this rule, in us:
    // depth-8 cube 64 x 64 329, 323, 227, 128 x 128 363, 364, 307; depth-27 canvas 64 x 64 927, 867, 437, 128 x 128 1157,
    // 1136, 808; depth-24 canvas 128 x 128 409, 391, 350, 256 x 256 457, 383, 383; opaque paint 32 x 32 32, 31, 27, 64 x
    // 64 34, 30, 32, 128 x 128 36, 30, 34, 256 x 256 43, 35, 35.
    const int64_t room = (int64_t)grid * (block / 32);  // warps
    p.take = 32;
    while (p.refill == 0 && p.take > 1 && p.total_rays <= room / 2 * (p.take / 2)) p.take /= 2;
    const int64_t warps = (p.total_rays + p.take - 1) / p.take;
    p.per_block = warps <= room ? (int32_t)((warps + grid - 1) / grid) : 0;
    const bool ropes = p.use_ropes && p.tree.ropes;
    if (p.count_reads)
        return ropes ? launch_mixed_w<true, true>(p, grid, block, s, after_setup)
                     : launch_mixed_w<false, true>(p, grid, block, s, after_setup);
    return ropes ? launch_mixed_w<true, false>(p, grid, block, s, after_setup)
                 : launch_mixed_w<false, false>(p, grid, block, s, after_setup);
}

cudaError_t mixed_max_blocks_per_sm(int block, int smem_bytes, int* out) {
    // all instances share the register and static shared-memory budget
    if (smem_bytes <= 0)
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, mixed_kernel<false, true, true, kPlainPool>, block, 0);
    const cudaError_t e = cudaFuncSetAttribute(mixed_kernel<true, true, true, kPlainPool>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, mixed_kernel<true, true, true, kPlainPool>, block, smem_bytes);
}

}  // namespace canvox
