// FP64 twin of the mixed-precision traversal: the precision comparator.
//
// The same traversal as the mixed kernel (trace_mixed.cu): a persistent grid
// whose warps pop tiles of rays from one global queue, exact fixed-point cell
// corners in the mirrored canvas, the neighbour found as a sibling or through
// the parent's neighbour link (the neighbour graph of Sec. 4.1.1, built at
// upload), a descent while the cell is internal, front-to-back compositing to
// full opacity or the canvas exit (Sec. 6.2). What differs is the arithmetic:
// every crossing time, position and sum is FP64 (no anchor, no FP32 screen, no
// error budget). Timing this kernel beside the mixed one isolates what the
// single-precision decisions buy on this GPU, whose FP64 rate is a small
// fraction of its FP32 rate; the plain FP64 caster (trace_plain.cu) differs from
// the mixed kernel in its traversal too.
//
// A plane's time is (X - eye) / |d|, the difference in units taken between
// integers and the eye's rest below a unit (the ray's own 53 bits then count from
// the eye, not from the canvas's centre); the sides below the old cell's level
// are the bits of the position eye + t d. A ray leaves a leaf by the face with
// the smallest crossing time (ties to the lowest axis); a position on a plane is
// on the side the ray moves into, for d = 0 on the high side.
//
// What bounds it: the FP64 pipe, an instruction of which occupies an SM's unit
// for 16 cycles however few lanes take part, so the step counts them: two per
// axis for the exit times (an integer becomes a double by its bit pattern and
// one addition), compares, half-to-double conversions and the termination test on
// integer patterns, the opacity of thin leaves by its series, one position per
// descent instead of a plane and a time per level and axis. 28 FP64 instructions
// per warp and step (pipe 86 % busy): a depth-24 stereo pair of 540^2 with 205
// leaves a ray takes 6.25 ms, 15.6 ms with a plane and a time per level and axis,
// conversions and the library's opacity for every leaf.
#include <cuda_fp16.h>

#include "canvox_internal.cuh"
#include "cells.cuh"
#include "opacity.cuh"

namespace canvox {
namespace {

constexpr unsigned kFull64 = 0xFFFFFFFFu;
constexpr int kBlock64 = 256;

// Per-lane FP64 state that a step reads rarely, one 8-byte column per field and lane.
enum Col64 {
    kColC = 0,      // double: colour sums, three columns
    kColDs = 3,     // double: |d_a| in units per length
    kColRest = 6,   // double: the eye's rest below a unit (mirrored)
    kColAt = 9,     // uint32: output pixel, view
    kCols64 = 10
};

struct Ray64 {
    char* base;             // the lane's shared columns
    double iu[3], nr[3];    // t(X) = (X - U) iu + nr; axis with d = 0: 0 and a time past every other
    double t;               // parameter where the current leaf is entered
    double T;               // transmittance
    uint32_t X[3], U[3];    // low corner of the current cell, the eye in whole units (mirrored)
    int32_t L;
    uint32_t flip;
    uint2 val;
    int32_t pr;   // record holding the current leaf's slot
    uint32_t kc;  // child index of the current leaf in pr
    int32_t steps;
    uint32_t n_rays, n_steps, n_reads, n_leaf, n_rec;

    template <typename V>
    __device__ __forceinline__ V& col(int c) { return *reinterpret_cast<V*>(base + (size_t)c * (8 * kBlock64)); }
    __device__ __forceinline__ double& C(int i) { return col<double>(kColC + i); }
    __device__ __forceinline__ double& ds(int a) { return col<double>(kColDs + a); }
    __device__ __forceinline__ double& rest(int a) { return col<double>(kColRest + a); }
    __device__ __forceinline__ uint32_t& pix() { return col<uint32_t>(kColAt); }
    __device__ __forceinline__ uint32_t& view() { return (&col<uint32_t>(kColAt))[1]; }
};

// A binary16 value as a double, through its float (a normal one or zero) by exponent arithmetic.
__device__ __forceinline__ double half_to_double(unsigned h) {
    const uint32_t f = __float_as_uint(half_bits_to_float(h));
    const uint32_t m = f & 0x7FFFFFFFu;
    const long long d = ((long long)m << 29) + (m ? 0x3800000000000000ll : 0ll);
    return __longlong_as_double(d | ((long long)(f >> 31) << 63));
}

// Composite the current leaf over [r.t, te].
__device__ __forceinline__ void composite64(Ray64& r, double te) {
    if (r.val.y >> 16) {
        const double em = expm1_neg64(half_to_double(r.val.y >> 16) * (te - r.t));  // -(1 - e^{-sigma l})
        const double w = -r.T * em;
        r.C(0) = fma(w, half_to_double(r.val.x & 0xFFFFu), r.C(0));
        r.C(1) = fma(w, half_to_double(r.val.x >> 16), r.C(1));
        r.C(2) = fma(w, half_to_double(r.val.y & 0xFFFFu), r.C(2));
        r.T = fma(r.T, em, r.T);
    }
}

__device__ __forceinline__ void finish64(Ray64& r, const MixedParams& P) {
    const View& V = P.views[r.view()];
    float4 o;
    o.x = (float)(r.C(0) + r.T * (double)V.bg[0]);
    o.y = (float)(r.C(1) + r.T * (double)V.bg[1]);
    o.z = (float)(r.C(2) + r.T * (double)V.bg[2]);
    o.w = (float)(1.0 - r.T);
    const int64_t pix = V.out_offset + (int64_t)r.pix();
    P.out[pix] = o;
    if (P.step_count) P.step_count[pix] = r.steps;
    r.n_rays += 1;
    r.n_steps += (uint32_t)r.steps;
}

// The ray's position on axis a at parameter t: the unit it lies in, kept within [X, X + s).
__device__ __forceinline__ uint32_t locate64(Ray64& r, int a, double t, uint32_t X, uint32_t s) {
    const int32_t n = __double2int_rd(fma(t, r.ds(a), r.rest(a)));
    const int64_t rel = (int64_t)r.U[a] + n - (int64_t)X;
    return X + (uint32_t)min(max(rel, (int64_t)0), (int64_t)s - 1);
}

// Start ray g of the launch. Returns true if it has a leaf to step from.
template <int kPool>
__device__ bool init64(Ray64& r, const MixedParams& P, unsigned long long g) {
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
    const unsigned tile = (unsigned)(local >> 5);
    const int lane = (int)(local & 31);
    const unsigned ty = tile / (unsigned)V.tiles_x;
    const int wl = V.tile_wl;
    const int i = ((int)(tile - ty * (unsigned)V.tiles_x) << wl) + (lane & ((1 << wl) - 1));
    const int j = (int)ty * (32 >> wl) + (lane >> wl);
    if (i >= V.width || j >= V.height) return false;
    r.view() = (uint32_t)lo;
    r.pix() = (uint32_t)j * (uint32_t)V.width + (uint32_t)i;
    r.C(0) = r.C(1) = r.C(2) = 0.0;
    r.T = 1.0;
    r.steps = 0;
    double d[3];
    pixel_ray(V, i, j, d);
    r.flip = 0;
    double t0 = 0.0, t1 = __longlong_as_double(0x7FF0000000000000ll);
    bool miss = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const bool neg = d[a] < 0.0;
        if (neg) r.flip |= 1u << a;
        uint32_t u = (uint32_t)V.eye_unit[a];
        double rest = V.eye_rest[a];
        if (neg) {
            // (an eye outside: from the face it looks at, whose distance keeps its own precision)
            rest = u ? -rest : (T.half - V.eye[a]) * (P.inv_extent * 2147483648.0);
            u = u ? 0x80000000u - u : 0u;
        }
        r.U[a] = u;
        r.rest(a) = rest;
        const double da = fabs(d[a]), o = neg ? -V.eye[a] : V.eye[a];
        r.ds(a) = da * (P.inv_extent * 2147483648.0);
        if (da != 0.0) {
            // (smaller components are never crossed: a time of 1e200 per length keeps the products below finite)
            const double inv = da > 1.0e-200 ? rcp64(da) : 1.0e200;
            r.iu[a] = P.unit * inv;
            r.nr[a] = -rest * r.iu[a];
            t0 = fmax(t0, (-T.half - o) * inv);
            t1 = fmin(t1, (T.half - o) * inv);
        } else {
            r.iu[a] = 0.0;
            r.nr[a] = 1.0e300;
            if (!(o >= -T.half && o < T.half)) miss = true;
        }
    }
    if (miss || !(t0 < t1)) {
        finish64(r, P);
        return false;
    }
    r.t = t0;
    r.steps = 1;
    const EyePath& E = P.eye[lo];
    if (E.len > 0) {  // (t0 is 0 for an eye inside the canvas)
        r.L = E.len;
        r.pr = E.rec[E.len - 1];
        r.kc = (E.c[0] & 1u) | ((E.c[1] & 1u) << 1) | ((E.c[2] & 1u) << 2);
        const uint32_t last = (1u << E.len) - 1u;
#pragma unroll
        for (int a = 0; a < 3; ++a) r.X[a] = (((r.flip >> a) & 1u) ? last - E.c[a] : E.c[a]) << (kFix - E.len);
        r.val = E.val;
        r.n_reads += r.L;
        r.n_leaf += (uint32_t)E.stored;
        return true;
    }
    // locate the leaf that holds r(t0+) from the root
    uint32_t q[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) q[a] = locate64(r, a, t0, 0u, 0x80000000u);
    int sh = kFix;
    int32_t rec = 0, slot = 0;
    do {
        rec = slot;
        --sh;
        r.kc = (uint32_t)child_index_any(q, sh, r.flip);
        slot = __ldg(T.nodes + (int64_t)rec * 8 + r.kc);
        r.n_rec += 1;
    } while (slot > 0);
    r.pr = rec;
    r.L = kFix - sh;
    r.n_reads += r.L;
    r.val = make_uint2(0u, 0u);
    if (slot < 0) {
        r.val = load_leaf<kPool>(T, rec, (int)r.kc, slot);
        r.n_leaf += 1;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) r.X[a] = (q[a] >> sh) << sh;
    return true;
}

// One leaf step. Returns false once the ray is finished (its pixel written).
template <int kPool>
__device__ bool step64(Ray64& r, const MixedParams& P) {
    const Tree& T = P.tree;
    // 1. exit face: the smallest FP64 crossing time of the exact far planes (ties to the lowest axis)
    const uint32_t s = 1u << (kFix - r.L);
    const double t0 = fma(uint_to_double(r.X[0] + s - r.U[0]), r.iu[0], r.nr[0]);
    const double t1 = fma(uint_to_double(r.X[1] + s - r.U[1]), r.iu[1], r.nr[1]);
    const double t2 = fma(uint_to_double(r.X[2] + s - r.U[2]), r.iu[2], r.nr[2]);
    int ax = 0;
    double te = t0;
    if (less_pos(t1, te)) { ax = 1; te = t1; }
    if (less_pos(t2, te)) { ax = 2; te = t2; }
    // 2. the neighbour across the exit face: its low corner is N on that axis
    const uint32_t N = pick(ax, r.X[0], r.X[1], r.X[2]) + s;
    if ((N >> kFix) != 0u) {  // leaving the canvas
        composite64(r, te);
        finish64(r, P);
        return false;
    }
    const int lstar = (kFix - 1) - (31 - __clz((N - s) ^ N));
    uint32_t q[3] = {ax == 0 ? N : r.X[0], ax == 1 ? N : r.X[1], ax == 2 ? N : r.X[2]};
    const int sh_old = kFix - r.L;
    int32_t prec = r.pr;
    int kk = (int)(r.kc ^ (1u << ax)), sh = sh_old;
    if (!(N & s)) {  // not the high half of the same parent
        const uint2 rp = __ldg(T.ropes + (int64_t)r.pr * 6 + 2 * ax + (int)(((r.flip >> ax) & 1u) ^ 1u));
        r.n_rec += 1;
        prec = (int32_t)rp.x;
        // (an internal neighbour is named by its own record: its child next to the old cell has a sibling's index)
        if (!(rp.y & kLinkRecord)) {
            kk = (int)(rp.y >> 8);
            sh = (int)(rp.y & 255u);
        }
    }
    int32_t slot = __ldg(T.nodes + (int64_t)prec * 8 + kk);
    r.n_rec += 1;
    // 3. finer than the old cell: near side on the exit axis, the ray's position at te on the others
    if (slot > 0) {
        const uint32_t q0 = locate64(r, 0, te, r.X[0], s), q1 = locate64(r, 1, te, r.X[1], s),
                       q2 = locate64(r, 2, te, r.X[2], s);
        q[0] = ax == 0 ? N : q0;
        q[1] = ax == 1 ? N : q1;
        q[2] = ax == 2 ? N : q2;
        do {
            --sh;
            prec = slot;
            kk = child_index(q, sh, r.flip);
            slot = __ldg(T.nodes + (int64_t)prec * 8 + kk);
            r.n_rec += 1;
        } while (slot > 0);
    }
    r.n_reads += (uint32_t)(kFix - sh - lstar);
    uint2 nval = make_uint2(0u, 0u);
    if (slot < 0) {
        nval = load_leaf<kPool>(T, prec, kk, slot);
        r.n_leaf += 1;
    }
    // 4. composite the current leaf, then terminate or advance
    composite64(r, te);
    if (less_pos(r.T, (double)P.t_min)) {
        finish64(r, P);
        return false;
    }
    if (r.steps >= P.step_limit) {
        atomicOr(&P.scratch->status, 1ull);
        atomicAdd(&P.scratch->stats[kStatStepLimited], 1ull);
        finish64(r, P);
        return false;
    }
    r.L = kFix - sh;
#pragma unroll
    for (int a = 0; a < 3; ++a) r.X[a] = (q[a] >> sh) << sh;
    r.val = nval;
    r.pr = prec;
    r.kc = (uint32_t)kk;
    r.t = te;
    r.steps += 1;
    return true;
}

__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull64, v, o);
    return v;
}

template <int kPool>
__global__ void __launch_bounds__(kBlock64, 3) fp64links_kernel(MixedParams P) {
    __shared__ double lanes[kCols64 * kBlock64];
    Ray64 r;
    r.base = reinterpret_cast<char*>(&lanes[threadIdx.x]);
    r.n_rays = r.n_steps = r.n_reads = r.n_leaf = r.n_rec = 0;
    const unsigned lane = threadIdx.x & 31u;
    bool alive = false;
    bool drained = false;
    for (;;) {
        unsigned busy = __ballot_sync(kFull64, alive);
        if (!drained && __popc(busy) <= P.refill) {
            const unsigned idle = ~busy;
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(P.queue, (unsigned long long)__popc(idle));
            base = __shfl_sync(kFull64, base, 0);
            if (base + __popc(idle) >= (unsigned long long)P.total_rays) drained = true;
            if (!alive) {
                const unsigned long long g = base + __popc(idle & ((1u << lane) - 1u));
                if (g < (unsigned long long)P.total_rays) alive = init64<kPool>(r, P, g);
            }
            busy = __ballot_sync(kFull64, alive);
            if (!drained && __popc(busy) <= P.refill) continue;
        }
        if (busy == 0u) {
            if (drained) break;
            continue;
        }
        do {
            if (alive) alive = step64<kPool>(r, P);
            busy = __ballot_sync(kFull64, alive);
        } while (busy != 0u && (drained || __popc(busy) > P.refill));
    }
    const unsigned long long v[5] = {r.n_rays, r.n_steps, r.n_reads, r.n_leaf, r.n_rec};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const unsigned long long s = warp_sum64(v[i]);
        if (lane == 0 && s) atomicAdd(&P.scratch->stats[i], s);
    }
}

}  // namespace

cudaError_t launch_fp64links(const MixedParams& params, int grid, int block, cudaStream_t s) {
    if (!params.tree.ropes) return cudaErrorInvalidValue;
    MixedParams p = params;
    p.inv_extent = 1.0 / p.tree.extent;
    p.unit = p.tree.extent * 4.656612873077393e-10;  // 2^-31
    if (p.tree.n_wrap > 0) fp64links_kernel<kWrapPool><<<grid, block, 0, s>>>(p);
    else fp64links_kernel<kPlainPool><<<grid, block, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t fp64links_max_blocks_per_sm(int block, int* out) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, fp64links_kernel<kPlainPool>, block, 0);
}

}  // namespace canvox
