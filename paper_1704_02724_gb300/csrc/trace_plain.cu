// Plain single-precision-type ray casters (one launch per view), and the small
// kernels around the traversal: the pool hash, the eye leaf of each view, and
// the neighbour links built at upload.
//
// These are the baselines the mixed kernel is measured against: the ray, the
// cell planes and the compositing are all in one type R, in canvas
// coordinates, and every step locates the leaf from the root (no stack, no
// local frame). With R = double this is the plain FP64 GPU path; with
// R = float it is the canvas-coordinate FP32 traversal that Sec. 6.3 and the
// canvas-coordinate panel of its accuracy figure show drifting at depth.
// Planes are formed from integer cell coordinates, c * w_L - E/2, so a plane has
// one rounded value at every level and the located leaf always lies ahead of t.
// The FP64 caster can also mark the records and stored leaves it reads (the
// footprint of a frame, canvox_footprint).
#include <cuda_fp16.h>

#include "canvox_internal.cuh"
#include "cells.cuh"

namespace canvox {
namespace {

template <typename R>
struct Num;
template <>
struct Num<double> {
    static __device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
    static __device__ __forceinline__ double rsqrt_(double x) { return rsqrt(x); }
    static __device__ __forceinline__ double expm1_(double x) { return expm1(x); }
    static __device__ __forceinline__ double exp_(double x) { return exp(x); }
    static __device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }
    static __device__ __forceinline__ double inf() { return __longlong_as_double(0x7FF0000000000000ll); }
};
template <>
struct Num<float> {
    static __device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
    static __device__ __forceinline__ float rsqrt_(float x) { return rsqrtf(x); }
    static __device__ __forceinline__ float expm1_(float x) { return expm1f(x); }
    static __device__ __forceinline__ float exp_(float x) { return expf(x); }
    static __device__ __forceinline__ float pow2(int e) { return __int_as_float((127 + e) << 23); }
    static __device__ __forceinline__ float inf() { return __int_as_float(0x7F800000); }
};

__device__ __forceinline__ float h2f(unsigned short h) { return __half2float(__ushort_as_half(h)); }

// Set bit i of a footprint bitset (read through L2 first: most bits are already set).
__device__ __forceinline__ void mark_bit(uint32_t* bits, long long i) {
    const uint32_t m = 1u << (i & 31);
    uint32_t* w = bits + (i >> 5);
    if (!(__ldcg(w) & m)) atomicOr(w, m);
}

struct PlainCount {
    unsigned long long steps, leaf_loads, rec_loads;
};

// kWrap: the canvas has more than 2^31 leaves (slots hold leaf numbers modulo 2^31); an instance
// without it reads the number straight from the slot.
template <typename R, bool kWrap>
__device__ __forceinline__ PlainCount plain_ray(const PlainParams& P, long long idx) {
    using N = Num<R>;
    const View& V = *P.view;
    const int i = (int)(idx % V.width), j = (int)(idx / V.width);
    const Tree& T = P.tree;
    const R E = (R)T.extent, half = (R)T.half;
    // pixel-centre ray: the camera model's FP64 ray, rounded to R
    R o[3], d[3], inv[3], nod[3];
    {
        double dd[3];
        pixel_ray(V, i, j, dd);
        for (int a = 0; a < 3; ++a) {
            o[a] = (R)V.eye[a];
            d[a] = (R)dd[a];
        }
    }
    R t0 = 0, t1 = N::inf();
    bool miss = false;
    for (int a = 0; a < 3; ++a) {
        if (d[a] != (R)0) {
            inv[a] = (R)1 / d[a];
            nod[a] = -o[a] * inv[a];
            const R ta = N::fma_(-half, inv[a], nod[a]), tb = N::fma_(half, inv[a], nod[a]);
            t0 = fmax(t0, d[a] > 0 ? ta : tb);
            t1 = fmin(t1, d[a] > 0 ? tb : ta);
        } else {
            inv[a] = 0;
            nod[a] = o[a];
            if (!(o[a] >= -half && o[a] < half)) miss = true;
        }
    }
    R C[3] = {0, 0, 0}, Tr = 1;
    int steps = 0;
    unsigned long long rec_loads = 0, leaf_loads = 0;
    if (!miss && t0 < t1) {
        R t = t0;
        for (;;) {
            if (steps >= P.step_limit) {
                atomicOr(&P.scratch->status, 1ull);
                atomicAdd(&P.scratch->stats[kStatStepLimited], 1ull);
                break;
            }
            // locate the leaf holding r(t+) from the root
            unsigned cc[3] = {0u, 0u, 0u};
            int lev = 0;
            int32_t rec = 0, slot;
            int64_t li = 0;  // number of the located leaf (slot < 0)
            for (;;) {
                const R w = E * N::pow2(-(lev + 1));
                int k = 0;
                for (int a = 0; a < 3; ++a) {
                    const R M = N::fma_((R)(2u * cc[a] + 1u), w, -half);
                    unsigned b;
                    if (d[a] == (R)0) {
                        b = nod[a] >= M;
                    } else {
                        const R tm = N::fma_(M, inv[a], nod[a]);
                        b = d[a] > 0 ? (tm <= t) : (tm > t);
                    }
                    cc[a] = 2u * cc[a] + b;
                    k |= (int)b << a;
                }
                slot = __ldg(T.nodes + (long long)rec * 8 + k);
                rec_loads += 1;
                if (slot > 0) {
                    rec = slot;
                    ++lev;
                } else {
                    if (slot < 0) li = kWrap ? leaf_index(T, rec, k, slot) : -(int64_t)slot - 1;
                    break;
                }
            }
            if (P.mark_rec) mark_bit(P.mark_rec, rec);
            const int L = lev + 1;
            const R w = E * N::pow2(-L);
            R te = N::inf();
            for (int a = 0; a < 3; ++a) {
                if (d[a] == (R)0) continue;
                const R F = N::fma_((R)(cc[a] + (d[a] > 0 ? 1u : 0u)), w, -half);
                const R ta = N::fma_(F, inv[a], nod[a]);
                te = fmin(te, ta);
            }
            te = fmin(te, t1);
            steps += 1;
            if (slot < 0) {
                const uint2 q = __ldg(T.leaves + li);
                leaf_loads += 1;
                if (P.mark_leaf) mark_bit(P.mark_leaf, li);
                const R s = (R)h2f((unsigned short)(q.y >> 16));
                if (s > (R)0) {
                    const R l = te - t;
                    const R a = -N::expm1_(-s * l);
                    C[0] += Tr * a * (R)h2f((unsigned short)(q.x & 0xFFFFu));
                    C[1] += Tr * a * (R)h2f((unsigned short)(q.x >> 16));
                    C[2] += Tr * a * (R)h2f((unsigned short)(q.y & 0xFFFFu));
                    Tr *= N::exp_(-s * l);
                }
            }
            if (Tr < (R)P.t_min || te >= t1) break;
            t = te;
        }
    }
    float4 out;
    out.x = (float)(C[0] + Tr * (R)V.bg[0]);
    out.y = (float)(C[1] + Tr * (R)V.bg[1]);
    out.z = (float)(C[2] + Tr * (R)V.bg[2]);
    out.w = (float)(1 - Tr);
    const long long pix = V.out_offset + idx;
    if (P.out) P.out[pix] = out;
    if (P.step_count) P.step_count[pix] = steps;
    return PlainCount{(unsigned long long)steps, leaf_loads, rec_loads};
}

template <typename R, bool kWrap>
__global__ void __launch_bounds__(256) plain_kernel(PlainParams P, long long n_pixels) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    PlainCount c = {0ull, 0ull, 0ull};
    const bool valid = idx < n_pixels;
    if (valid) c = plain_ray<R, kWrap>(P, idx);
    // counters in canvox_stats order: rays, steps, slot reads (not tracked here), leaf loads, record loads
    unsigned long long vals[5] = {valid ? 1ull : 0ull, c.steps, 0ull, c.leaf_loads, c.rec_loads};
    for (int q = 0; q < 5; ++q) {
        unsigned long long s = vals[q];
        for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, off);
        if ((threadIdx.x & 31) == 0 && s) atomicAdd(&P.scratch->stats[q], s);
    }
}

__device__ __forceinline__ void add_warp_sum(unsigned long long acc, unsigned long long* out) {
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, off);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}

__device__ __forceinline__ unsigned long long leaf_terms(const uint2* leaves, long long first, long long n) {
    unsigned long long acc = 0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint2 q = leaves[i];
        acc += elem_hash(2ull, (unsigned long long)(first + i), ((unsigned long long)q.y << 32) | q.x);
    }
    return acc;
}

// The whole pools: 16 bytes a load, so that the loads and four chains of multiplications of a thread overlap (one
// element a load took 1.2 ms for 3.2 GB).
__global__ void __launch_bounds__(256) hash_kernel(Tree t, unsigned long long* out) {
    unsigned long long acc = 0;
    const long long stride = (long long)gridDim.x * blockDim.x, first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int4* nodes = reinterpret_cast<const int4*>(t.nodes);
    for (long long i = first; i < 2 * t.n_rec; i += stride) {
        const int4 q = __ldg(nodes + i);
        acc += elem_hash(1ull, (unsigned long long)(4 * i), (unsigned long long)(uint32_t)q.x);
        acc += elem_hash(1ull, (unsigned long long)(4 * i + 1), (unsigned long long)(uint32_t)q.y);
        acc += elem_hash(1ull, (unsigned long long)(4 * i + 2), (unsigned long long)(uint32_t)q.z);
        acc += elem_hash(1ull, (unsigned long long)(4 * i + 3), (unsigned long long)(uint32_t)q.w);
    }
    const uint4* leaves = reinterpret_cast<const uint4*>(t.leaves);
    for (long long i = first; i < t.n_leaf / 2; i += stride) {
        const uint4 q = __ldg(leaves + i);
        acc += elem_hash(2ull, (unsigned long long)(2 * i), ((unsigned long long)q.y << 32) | q.x);
        acc += elem_hash(2ull, (unsigned long long)(2 * i + 1), ((unsigned long long)q.w << 32) | q.z);
    }
    if (first == 0 && (t.n_leaf & 1)) {
        const uint2 q = t.leaves[t.n_leaf - 1];
        acc += elem_hash(2ull, (unsigned long long)(t.n_leaf - 1), ((unsigned long long)q.y << 32) | q.x);
    }
    add_warp_sum(acc, out);
}

__global__ void hash_leaves_kernel(const uint2* leaves, long long first, long long n, unsigned long long* out) {
    add_warp_sum(leaf_terms(leaves, first, n), out);
}

// The leaf holding the eye of view V, or len = 0 when the eye is outside the
// canvas or exactly on a mid-plane of its path (then the ray's direction
// decides the side and every ray locates its own start).
__device__ __forceinline__ void eye_path(const Tree& t, const View& V, EyePath& E) {
    E.len = 0;
    E.stored = 0;
    E.val = make_uint2(0u, 0u);
    for (int a = 0; a < 3; ++a)
        if (!(V.eye[a] > -t.half && V.eye[a] < t.half)) return;  // (on the low face the direction decides)
    int32_t rec = 0;
    const int32_t* unit = V.eye_unit;
    // The eye in whole units (set for an eye inside the canvas) and an exactly signed rest: the bits of the unit it is in are
    // its path, and the path's first mid-plane that it lies on is the lowest bit of a whole number of units. So the chain
    // has no FP64 (fma and three comparisons a level), only the loads: 3 us less of a render at depth 16 (a view of
    // 32 x 32 pixels 29.5 -> 26.3 us), 9 us at depths 24 and 27.
    uint32_t v[3];
    int on = kMaxDepth + 1;
    for (int a = 0; a < 3; ++a) {
        const long long rest = __double_as_longlong(V.eye_rest[a]);
        const bool zero = (rest << 1) == 0;
        v[a] = (uint32_t)unit[a] - (rest < 0 && !zero ? 1u : 0u);
        if (zero) on = min(on, kFix - __ffs(unit[a]));
    }
    for (int lev = 0; lev < kMaxDepth; ++lev) {
        E.rec[lev] = rec;
        if (lev == on) return;
        const int sh = kFix - 1 - lev;
        const int k = (int)(((v[0] >> sh) & 1u) | (((v[1] >> sh) & 1u) << 1) | (((v[2] >> sh) & 1u) << 2));
        const int32_t slot = __ldg(t.nodes + (long long)rec * 8 + k);
        if (slot > 0) {
            rec = slot;
            continue;
        }
        if (slot < 0) {
            E.val = t.leaves[leaf_index(t, rec, k, slot)];
            E.stored = 1;
        }
        for (int a = 0; a < 3; ++a) E.c[a] = v[a] >> sh;
        E.len = lev + 1;
        return;
    }
}

// One thread per view.
__global__ void eye_path_kernel(Tree t, const View* views, int n_views, EyePath* out) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < n_views) eye_path(t, views[v], out[v]);
}

// One block per view: a render's set-up in one launch. A copy of the view table, a memset and the eye paths, as three
// stream operations, and a plain launch of the traversal after them took 9 us more of a render: 407 -> 398 us (256 x
// 256 pixels of the depth-8 cube), 320 -> 310 us (1920 x 1080 inside opaque paint). Two sizes of the argument
// block, as the launch copies all of it: 0.9 KB for a frame's few views, 13.8 KB (the most that fits in a launch's 32 KB
// with room to spare) up to 64.
template <int kViews>
struct ViewArgs {
    View v[kViews];
};
template <int kViews>
__global__ void __launch_bounds__(64) setup_kernel(const __grid_constant__ ViewArgs<kViews> args, Tree t, View* views,
                                                   EyePath* eye, unsigned long long* scratch, int scratch_words) {
    asm volatile("griddepcontrol.launch_dependents;");  // (the traversal's blocks may take their places)
    const int v = blockIdx.x;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(&args.v[v]);
    uint32_t* dst = reinterpret_cast<uint32_t*>(views + v);
    for (int i = threadIdx.x; i < (int)(sizeof(View) / 4); i += blockDim.x) dst[i] = src[i];
    if (v == 0)
        for (int i = threadIdx.x; i < scratch_words; i += blockDim.x) scratch[i] = 0ull;
    if (threadIdx.x == 0) eye_path(t, args.v[v], eye[v]);
}
static_assert(sizeof(View) % 4 == 0 && sizeof(ViewArgs<kSetupViews>) <= 32000, "kernel arguments end at 32764 bytes");

template <int kViews>
cudaError_t setup_launch(const Tree& t, const View* host_views, int n, View* views, EyePath* eye, Scratch* scratch,
                         int words, cudaStream_t s) {
    ViewArgs<kViews> a;
    for (int v = 0; v < n; ++v) a.v[v] = host_views[v];
    setup_kernel<kViews><<<n, 64, 0, s>>>(a, t, views, eye, reinterpret_cast<unsigned long long*>(scratch), words);
    return cudaGetLastError();
}

// Neighbour links (the paper's neighbour graph of Sec. 4.1.1, kept per record).
// ropes[r][2a + s] names the cell across face (axis a, s = 1 high / 0 low) of
// record r's cell: the same-level neighbour if it exists, else the coarser leaf
// that covers it, as (record holding its slot, (child index << 8) | the shift of its side, 31 - level),
// or, for an internal neighbour, as (its own record, kLinkRecord | the same),
// which saves a ray the load of its slot; outside the canvas as (0, kLinkRecord),
// which reads as an empty slot. One launch per level, parents before
// children: a child's link is its sibling inside the parent, or the parent's
// link, refined to the adjacent child when that neighbour is an internal cell.
// Bound by memory (32 B of slots and 48 B of links read and 48 B written per
// record); a lane per slot, so that slots are read and the children's links,
// which follow one another, are written side by side, 16 bytes at a time: 38.8 M
// records in 2.5 ms with a lane per record, 8-byte stores 384 bytes apart.
__global__ void __launch_bounds__(256) rope_level_kernel(const int32_t* nodes, uint2* ropes, long long lo, long long hi,
                                                         int level) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long r = lo + (t >> 3);
    const int k = (int)(t & 7);
    if (r >= hi) return;
    if (level == 0 && k < 6) ropes[k] = make_uint2(0u, kLinkRecord);
    const int32_t v = nodes[8 * r + k];
    if (v <= 0) return;
    uint2 R[6];
    if (level == 0) {
        for (int f = 0; f < 6; ++f) R[f] = make_uint2(0u, kLinkRecord);
    } else {
        const uint4* p = reinterpret_cast<const uint4*>(ropes + 6 * r);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const uint4 q = p[a];
            R[2 * a] = make_uint2(q.x, q.y);
            R[2 * a + 1] = make_uint2(q.z, q.w);
        }
    }
    uint4* out = reinterpret_cast<uint4*>(ropes + 6 * (long long)v);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const uint32_t kk = (uint32_t)(k ^ (1 << a));
        const bool high = (k >> a) & 1;
        const uint32_t where = (kk << 8) | (uint32_t)(kFix - (level + 1));
        // the sibling inside r, and the cell past r's face on the child's side
        const int32_t ov = nodes[8 * r + kk];
        const uint2 own = ov > 0 ? make_uint2((uint32_t)ov, kLinkRecord | where) : make_uint2((uint32_t)r, where);
        uint2 far = high ? R[2 * a + 1] : R[2 * a];
        if ((far.y & kLinkRecord) && far.x != 0u) {
            const int32_t cv = nodes[(long long)(int)far.x * 8 + kk];
            far = cv > 0 ? make_uint2((uint32_t)cv, kLinkRecord | where) : make_uint2(far.x, where);
        }
        out[a] = high ? make_uint4(own.x, own.y, far.x, far.y) : make_uint4(far.x, far.y, own.x, own.y);
    }
}

}  // namespace

cudaError_t launch_rope_level(const int32_t* nodes, uint2* ropes, int64_t lo, int64_t hi, int level, cudaStream_t s) {
    if (hi <= lo) return cudaSuccess;
    const long long n = 8 * (hi - lo);
    rope_level_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(nodes, ropes, lo, hi, level);
    return cudaGetLastError();
}

cudaError_t launch_eye_paths(const Tree& t, const View* views, int n_views, EyePath* out, cudaStream_t s) {
    if (n_views <= 0) return cudaSuccess;
    eye_path_kernel<<<(n_views + 63) / 64, 64, 0, s>>>(t, views, n_views, out);
    return cudaGetLastError();
}

cudaError_t launch_setup(const Tree& t, const View* host_views, int n, View* views, EyePath* eye, Scratch* scratch,
                         int queues, cudaStream_t s) {
    if (n < 1 || n > kSetupViews) return cudaErrorInvalidValue;
    const int words = (int)(sizeof(Scratch) / 8) + queues - 1;
    if (n <= 4) return setup_launch<4>(t, host_views, n, views, eye, scratch, words, s);
    return setup_launch<kSetupViews>(t, host_views, n, views, eye, scratch, words, s);
}

cudaError_t launch_plain(const PlainParams& p, int precision, long long n_pixels, cudaStream_t s) {
    if (n_pixels <= 0) return cudaSuccess;
    const int block = 256;
    const long long grid = (n_pixels + block - 1) / block;
    if (grid > 0x7FFFFFFFll) return cudaErrorInvalidValue;
    const bool wrap = p.tree.n_wrap > 0;
    if (precision == CANVOX_PREC_FP32) {
        if (wrap) plain_kernel<float, true><<<(unsigned)grid, block, 0, s>>>(p, n_pixels);
        else plain_kernel<float, false><<<(unsigned)grid, block, 0, s>>>(p, n_pixels);
    } else {
        if (wrap) plain_kernel<double, true><<<(unsigned)grid, block, 0, s>>>(p, n_pixels);
        else plain_kernel<double, false><<<(unsigned)grid, block, 0, s>>>(p, n_pixels);
    }
    return cudaGetLastError();
}

cudaError_t launch_hash(const Tree& t, unsigned long long* out, cudaStream_t s) {
    hash_kernel<<<152 * 8, 256, 0, s>>>(t, out);
    return cudaGetLastError();
}

cudaError_t launch_hash_leaves(const uint2* leaves, int64_t first, int64_t n, unsigned long long* out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int64_t blocks = (n + 255) / 256;
    hash_leaves_kernel<<<(unsigned)(blocks < 1024 ? blocks : 1024), 256, 0, s>>>(leaves, first, n, out);
    return cudaGetLastError();
}

}  // namespace canvox
