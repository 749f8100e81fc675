// Device-side stamp painter: spherical brush stamps -> canonical octree pools on the GPU.
//
// The brush model of Sec. 5: a stamp refines every cell it partially covers
// down to its target depth (the smallest k with E 2^-k <= r/10, about ten
// cells across the radius, Sec. 5.2), paints cells that lie inside the sphere
// whole, and paints the finest partially covered cells by their centre; a
// cell that is already refined when the stamp arrives is descended instead.
// Paint values are blended additively (Sec. 5.1): rgb' = B m + (1-m) C with
// m = B_a / (B_a + C_a), a' = B_a + C_a, in FP32 with every operation rounded
// separately. Leaves are then rounded to FP16, eight identical siblings merge
// into one leaf, and the pools are written in breadth-first order (Sec. 4.1.1:
// eight children per allocation unit, index-based pools).
//
// The stamps are applied in order, but the result has a closed form that is
// computed level by level without replaying them:
//   * cell C is refined iff some stamp partially covers it and has its target
//     depth below C (firstref(C) = the first such stamp, else none);
//   * a stamp s descends through C iff C is refined by the time s arrives,
//     i.e. firstref(C) <= s;
//   * a leaf's value is the blend, in stamp order, of the stamps that paint
//     it: s paints leaf X when, walking down X's ancestors from the root, the
//     first cell s does not descend through lies inside s, or is partially
//     covered and has its centre inside s.
// Each level keeps, per refined cell, the ordered list of stamps that still
// descend (undecided) or already paint its whole subtree (painted). Eight lanes
// take a cell, one per child, and walk its list in order: at stamp s a child
// knows whether an earlier stamp (or s itself) refines it, so one pass gives its
// firstref, its blend and which stamps its own list keeps; that decision is left
// as two bits per stamp and child, from which the next level's lists are written.
// Lists of more than 512 entries, 128 on levels of few cells (near the root every
// stamp is on them; around a room, its stamps) are cut into items that octets take
// in parallel: first the least refining stamp per child, then the decisions.
// Geometry is FP32 with a proven margin, retaken in FP64 with the same operations
// and order as the host painter inside the margin, so the pools are identical.
//
// What bounds it: near the root the latency of few octets walking lists, on the
// levels of millions of cells instruction issue and the gathers of the stamps'
// records. A lane per child suits the short lists most cells have: with a warp
// per cell and a lane per stamp (32 stamps at a time, two passes), a list of five
// left 27 lanes idle and its children were taken one after the other: the depth-24
// table of 210,000 stamps took 251 ms then and 35 ms now (expand_last 11.2 ms of it,
// expand_count 8, their issue slots 66-69 % used at 33 of 36 resident warps), the
// 1,000 stamps of the depth-8 cube with the read-back 7.5 and 1.6 ms.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include <cuda_fp16.h>

#include "canvox_internal.cuh"

namespace canvox {
namespace {

constexpr uint64_t kInternal = 1ull << 63;  // child slot: internal cell, low bits = index at the next level
constexpr uint64_t kNotCollapsed = 1ull << 63;
constexpr unsigned kFullMask = 0xFFFFFFFFu;
constexpr int kCells = 16;              // cells per block of the octet kernels (128 threads)
// Lists longer than this are cut into items, on levels of up to kFewCells cells and on those of more. A level of few cells
// waits for the octet with the longest list (0.25 us an entry: 70-220 us for 300-500 entries on the levels where a room
// begins), and the five launches for long lists cost some 30 us: 128 entries. With kLongFew 64, or kFewCells 4,096 or
// 65,536, the painting session took the same within 1 %; with more cells the octets of other cells hide a list of 512.
constexpr int64_t kFewCells = 16384;
constexpr int64_t kLongFew = 128, kLongMany = 512;
constexpr int kItemMin = 16, kItemMax = 128;  // ... of so many entries (item_size), one octet each
constexpr int32_t kNoStamp = 0x7FFFFFFF;

// Totals of a level on the device: the next level's entries and cells, its longest list, how many of its lists are
// longer than kLongFew and than kLongMany and their entries, and find_long's two counters.
enum { kTotEnt = 0, kTotCells = 1, kTotLongest = 2, kTotLong = 3, kLongCtr = 7, kTotWords = 9 };

// What a child box test reads of a stamp: the centre as two FP32 words per axis, the squared radius (both scaled by the
// power of two that brings the canvas to a side in [1, 2), so that no FP32 square leaves its range), the target depth.
struct StampRec {
    float ch[3], cl0;
    float cl1, cl2, r2;
    int32_t kt;
};
static_assert(sizeof(StampRec) == 32, "two 16-byte loads, one L2 sector");

struct StampDev {
    const double* c;       // [n][3]
    const double* r2;      // [n]
    const StampRec* rec;   // [n]
    const float4* rgba;    // [n]
};

__device__ __forceinline__ double sq(double x) { return __dmul_rn(x, x); }

// Squared distances from the sphere centre to the box [lo, lo + h]^3 and to its farthest corner.
__device__ __forceinline__ void box_dist2(const double* c, const double lo[3], double h, double& dmin2, double& dmax2) {
    dmin2 = 0.0;
    dmax2 = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double l = lo[a], u = __dadd_rn(lo[a], h);
        if (c[a] < l) dmin2 = __dadd_rn(dmin2, sq(__dsub_rn(l, c[a])));
        else if (c[a] > u) dmin2 = __dadd_rn(dmin2, sq(__dsub_rn(c[a], u)));
        dmax2 = __dadd_rn(dmax2, fmax(sq(__dsub_rn(c[a], l)), sq(__dsub_rn(u, c[a]))));
    }
}

__device__ __forceinline__ void blend(float4& C, float4 B) {
    const float s = __fadd_rn(B.w, C.w);
    if (s == 0.0f) return;
    const float m = __fdiv_rn(B.w, s);
    const float om = __fsub_rn(1.0f, m);
    C.x = __fadd_rn(__fmul_rn(B.x, m), __fmul_rn(om, C.x));
    C.y = __fadd_rn(__fmul_rn(B.y, m), __fmul_rn(om, C.y));
    C.z = __fadd_rn(__fmul_rn(B.z, m), __fmul_rn(om, C.z));
    C.w = s;
}

// FP16 leaf key (R | G << 16 | B << 32 | sigma << 48), 0 when sigma rounds to zero.
__device__ __forceinline__ uint64_t leaf_key(float4 v) {
    const float r = fminf(fmaxf(v.x, 0.0f), 1.0f), g = fminf(fmaxf(v.y, 0.0f), 1.0f), b = fminf(fmaxf(v.z, 0.0f), 1.0f);
    const float a = fminf(fmaxf(v.w, 0.0f), 60000.0f);
    const uint64_t ha = __half_as_ushort(__float2half_rn(a));
    if (ha == 0) return 0;
    return (uint64_t)__half_as_ushort(__float2half_rn(r)) | ((uint64_t)__half_as_ushort(__float2half_rn(g)) << 16) |
           ((uint64_t)__half_as_ushort(__float2half_rn(b)) << 32) | (ha << 48);
}

struct LevelIn {
    int64_t n;              // refined cells at this level
    int32_t level;
    const uint32_t* coord;  // [n][3]
    const int64_t* off;     // [n + 1]
    const int32_t* ent;     // s: descends, ~s: paints the whole cell
    int64_t limit;          // longer lists are cut into items
    double h;               // side of the children
    float hf;               // the same scaled as the stamps' records are (NaN: a canvas for FP64 alone)
};

// How a stamp covers a box.
enum { kOut = 0, kIn = 1, kPartCentreIn = 2, kPartCentreOut = 3 };

// The box of one child. Its low corner is j h with the integer j = child coordinate - 2^level, formed for the screen
// as two FP32 words without FP64 (whose pipe, converting and adding, bounded the levels of millions of cells at 74 %
// busy): j as two words too (the second 0 up to 2^24), the product's error from one fma. Within 2^-46 of the
// corner's own size of the exact one.
struct Child {
    uint32_t cc[3];      // child coordinates
    float lh[3], ll[3];  // low corner
    float uh[3], ul[3];  // high corner
    float hh;            // half side
    float a;             // the sum of the corners' sizes (the larger of the two per axis)
};

// j h as two FP32 words
__device__ __forceinline__ void plane_words(int32_t j, float hf, float& hi, float& lo) {
    const float jh = __int2float_rn(j), jl = __int2float_rn(j - __float2int_rn(jh));
    const float p = __fmul_rn(jh, hf), t = __fmaf_rn(jl, hf, __fmaf_rn(jh, hf, -p));
    hi = __fadd_rn(p, t);
    lo = __fsub_rn(t, __fsub_rn(hi, p));
}

__device__ __forceinline__ Child child_box(const LevelIn& L, int64_t i, int k) {
    Child B;
    B.hh = 0.5f * L.hf;
    B.a = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        B.cc[a] = 2u * L.coord[3 * i + a] + ((k >> a) & 1u);
        const int32_t j = (int32_t)B.cc[a] - (1 << L.level);
        plane_words(j, L.hf, B.lh[a], B.ll[a]);
        plane_words(j + 1, L.hf, B.uh[a], B.ul[a]);
        B.a += fmaxf(fabsf(B.lh[a]), fabsf(B.uh[a]));
    }
    return B;
}

// The cover of stamp v in FP64, in the host painter's operations and order (its skipped terms are +0, which is
// exact). Taken on about one test in ten thousand, so it is kept out of line.
__device__ __noinline__ int cover64(const double* c, double r2, uint32_t c0, uint32_t c1, uint32_t c2, double h,
                                    double half) {
    double dmin[3], dmax[3], cen[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double lo = fma((double)(a == 0 ? c0 : (a == 1 ? c1 : c2)), h, -half), up = __dadd_rn(lo, h);
        const double A = sq(__dsub_rn(c[a], lo)), B = sq(__dsub_rn(c[a], up));
        dmin[a] = c[a] < lo ? A : (c[a] > up ? B : 0.0);
        dmax[a] = fmax(A, B);
        cen[a] = sq(__dsub_rn(__dadd_rn(lo, 0.5 * h), c[a]));
    }
    if (__dadd_rn(__dadd_rn(dmin[0], dmin[1]), dmin[2]) >= r2) return kOut;
    if (__dadd_rn(__dadd_rn(dmax[0], dmax[1]), dmax[2]) <= r2) return kIn;
    return __dadd_rn(__dadd_rn(cen[0], cen[1]), cen[2]) < r2 ? kPartCentreIn : kPartCentreOut;
}

// The cover of a stamp, screened in FP32 (-1: open). The difference x of the centre and a face's plane, formed from two
// words each (the plane's within 2^-46 of it, the centre's within 2^-48), is within 2^-22.9 |x| + 2^-44.5 p of the exact
// one, p the plane's size: next to a plane the words cancel exactly. So with A the sum of the planes' sizes and n that
// of the distances outside the box per axis, the squared distance to the box is within 2^-21.1 of itself + 2^-43.5 A n +
// 2^-88 A^2 (margin twice that and more). With m >= |x| + 2 h on every axis the squared distances to the far corner and
// the centre are within 2^-20.9 (m + 2^-22 A)^2 (margin 2^-18). Without kExact the difference to the high face is formed
// from the one to the low face, which is off by 2^-23 m: the squared distance to the box is then within 2^-21.4 m n +
// 3 2^-44.8 m^2 + 2^-22 of itself. That leaves the stamps of a room that a plane of a far coarser cell crosses to FP64
// (half of all tests on such a cell's list, 1 us an entry instead of 0.3), but next to cells of the stamps' own size
// decides as many with fewer instructions and registers: expand_count
// took 7.1 ms with kExact and 6.5 ms without over the levels of six paintings of 13,000 stamps.
// Every comparison is false for a NaN or an infinite margin, which leaves it open.
template <bool kExact>
__device__ __forceinline__ int cover32(const Child& B, const StampRec& R, bool centre) {
    const float cl[3] = {R.cl0, R.cl1, R.cl2};
    float dmin2 = 0.0f, dmax2 = 0.0f, cen2 = 0.0f, m = 12.0f * B.hh + 2.384185791015625e-07f * B.a, n = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float dl = __fadd_rn(__fsub_rn(R.ch[a], B.lh[a]), __fsub_rn(cl[a], B.ll[a]));
        const float du = kExact ? __fadd_rn(__fsub_rn(R.ch[a], B.uh[a]), __fsub_rn(cl[a], B.ul[a]))
                                : __fsub_rn(dl, 2.0f * B.hh);
        const float dc = __fsub_rn(dl, B.hh);
        const float near = fmaxf(fmaxf(-dl, du), 0.0f), far = fmaxf(fabsf(dl), fabsf(du));
        dmin2 = fmaf(near, near, dmin2);
        dmax2 = fmaf(far, far, dmax2);
        cen2 = fmaf(dc, dc, cen2);
        m += fabsf(dl);
        n += near;
    }
    // 2^-20 (dmin2 + r2) + 2^-42 A (n + 2^-44 A), or 2^-20 m n + 2^-41 m^2 + 2^-21 (dmin2 + r2)
    const float e = kExact ? fmaf(9.5367431640625e-07f, dmin2 + R.r2,
                                  2.2737367544323206e-13f * B.a * fmaf(5.684341886080802e-14f, B.a, n))
                           : fmaf(m, fmaf(4.547473508864641e-13f, m, 9.5367431640625e-07f * n),
                                  4.76837158203125e-07f * (dmin2 + R.r2));
    if (dmin2 > R.r2 + e) return kOut;
    if (!(dmin2 < R.r2 - e)) return -1;
    const float margin = fmaf(3.814697265625e-06f * m, m, 2.384185791015625e-07f * R.r2);  // 2^-18 m^2 + 2^-22 r2
    const float lo = R.r2 - margin, hi = R.r2 + margin;
    if (dmax2 < lo) return kIn;
    if (!(dmax2 > hi)) return -1;
    if (!centre || cen2 < lo) return kPartCentreIn;
    return cen2 > hi ? kPartCentreOut : -1;
}

// Eight list entries of an octet: lane k loads entry q0 + k and its stamp's record, so the octet's eight loads are in
// flight at once (one entry after the other, each step of the walk waits for an entry and then for its record, 2.7 us
// a step on a level of few cells). The records are staged in shared memory, padded so that the four octets of a warp
// read different banks; on the long lists the next eight are loaded while these are used.
struct Entries {
    int64_t q0, e;  // [q0, q0 + m) of the list that ends at e
    int32_t v;      // lane k's entry
    int m;
    float4 x, y;    // its record
};
constexpr int kStageRow = 17;  // float4 per octet: eight records and a pad
constexpr int kColourRow = 25; // the same with the eight stamps' colours
__device__ __forceinline__ void load_entries(Entries& E, const LevelIn& L, const StampDev& S, int k) {
    E.m = (int)max((int64_t)0, min((int64_t)8, E.e - E.q0));
    E.v = k < E.m ? L.ent[E.q0 + k] : -1;
    if (E.v >= 0) {
        const float4* r = reinterpret_cast<const float4*>(S.rec + E.v);
        E.x = __ldg(r);
        E.y = __ldg(r + 1);
    }
}
__device__ __forceinline__ void stage_entries(const Entries& E, float4* row, int k) {
    row[2 * k] = E.x;
    row[2 * k + 1] = E.y;
}
__device__ __forceinline__ StampRec staged(const float4* row, int j) {
    StampRec R;
    const float4 x = row[2 * j], y = row[2 * j + 1];
    R.ch[0] = x.x;
    R.ch[1] = x.y;
    R.ch[2] = x.z;
    R.cl0 = x.w;
    R.cl1 = y.x;
    R.cl2 = y.y;
    R.r2 = y.z;
    R.kt = __float_as_int(y.w);
    return R;
}

template <bool kExact>
__device__ __forceinline__ int cover(const StampDev& S, int32_t v, const StampRec& R, const Child& B, double h,
                                     double half, bool centre) {
    const int c = cover32<kExact>(B, R, centre);
    return c >= 0 ? c : cover64(S.c + 3 * (int64_t)v, S.r2[v], B.cc[0], B.cc[1], B.cc[2], h, half);
}

enum { kDrop = 0, kPaint = 1, kKeep = 2 };

// Squared radius, target depth (the smallest k with extent 2^-k <= r/10, at most depth) and record of each stamp.
__global__ void stamp_prep(const double* c, const double* r, int64_t n, int32_t depth, double extent, double scale,
                           double* r2, StampRec* rec) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const double rs = r[s];
    const double rr = __dmul_rn(rs, rs);
    r2[s] = rr;
    const double tgt = __ddiv_rn(rs, 10.0);
    int32_t k = 0;
    double w = extent;
    while (k < depth && w > tgt) {
        w = __dmul_rn(w, 0.5);
        ++k;
    }
    float h[3], l[3];
    for (int a = 0; a < 3; ++a) {
        const double x = c[3 * s + a] * scale;
        h[a] = (float)x;
        l[a] = (float)(x - (double)h[a]);
    }
    StampRec R;
    R.ch[0] = h[0];
    R.ch[1] = h[1];
    R.ch[2] = h[2];
    R.cl0 = l[0];
    R.cl1 = l[1];
    R.cl2 = l[2];
    R.r2 = (float)(rr * scale * scale);
    R.kt = k;
    rec[s] = R;
}

// ---------------------------------------------------------------------------
// Long lists: items of item_size entries, one octet (eight lanes, one per child) each.
// ---------------------------------------------------------------------------

// Entries per item of a level. An octet takes 0.3 us an entry when few are in flight and long_sums 1 us per 32 items of
// a list, which meet at the square root of a tenth of the list's length; more than 65,536 items fill the chip
// whatever their length, and each takes 64 bytes. On lists of
// 3,000 stamps 24 items of 128 kept an item's octet busy for 40 us a level and the rest of the chip idle; 192 of 16 take
// 8.7 us (a painting of 13,000 stamps opened and appended to twice: 22.1 -> 19.1 ms).
int item_size(int64_t longest, int64_t n_ent) {
    int item = kItemMin;
    while (item < kItemMax && (10 * (int64_t)item * item < longest || 65536 * (int64_t)item < n_ent)) item *= 2;
    return item;
}

struct LongCell {
    int64_t cell, b, e;  // its list [b, e)
    int64_t item;        // its first item
};
struct Item {
    int64_t cell, b, e;
    int64_t p;  // long cell
};

// Cells with lists longer than the limit, their items, and no refining stamp yet; tot[kLongCtr] counts the cells, the
// next word their items.
__global__ void __launch_bounds__(256) find_long(LevelIn L, int item, LongCell* cells, Item* items, int32_t* fr,
                                                 long long* tot) {
    __shared__ LongCell s_cell[256];
    __shared__ int64_t s_p[256];
    __shared__ int s_n;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t b = i < L.n ? L.off[i] : 0, e = i < L.n ? L.off[i + 1] : 0;
    if (e - b > L.limit) {
        unsigned long long* ctr = reinterpret_cast<unsigned long long*>(tot + kLongCtr);
        const int64_t p = (int64_t)atomicAdd(&ctr[0], 1ull);
        const LongCell C{i, b, e, (int64_t)atomicAdd(&ctr[1], (unsigned long long)((e - b + item - 1) / item))};
        const int j = atomicAdd(&s_n, 1);
        cells[p] = s_cell[j] = C;
        s_p[j] = p;
    }
    __syncthreads();
    for (int j = 0; j < s_n; ++j) {
        const LongCell C = s_cell[j];
        const int64_t p = s_p[j];
        for (int64_t q = threadIdx.x; C.b + q * item < C.e; q += blockDim.x)
            items[C.item + q] = Item{C.cell, C.b + q * item, min(C.e, C.b + (q + 1) * item), p};
        if (threadIdx.x < 8) fr[8 * p + threadIdx.x] = kNoStamp;
    }
}

// The least stamp of each item that refines each child (entries are in stamp order, so the first that does).
__global__ void __launch_bounds__(128) long_first(LevelIn L, StampDev S, double half, const Item* items,
                                                  const long long* tot, int32_t* fr) {
    __shared__ float4 s_rec[16 * kStageRow];
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3;
    const int lane = threadIdx.x & 31, k = threadIdx.x & 7, lc = L.level + 1;
    float4* row = s_rec + (threadIdx.x >> 3) * kStageRow;
    const bool mine = w < tot[kLongCtr + 1];
    const Item I = mine ? items[w] : Item{0, 0, 0, 0};
    const Child B = child_box(L, I.cell, k);
    int32_t first = kNoStamp;
    Entries E{I.b, I.e, -1, 0, {}, {}};
    load_entries(E, L, S, k);
    while (__any_sync(kFullMask, E.m > 0 && first == kNoStamp)) {
        const Entries C = E;
        stage_entries(C, row, k);
        __syncwarp();
        E.q0 += 8;
        load_entries(E, L, S, k);
        for (int j = 0; j < 8; ++j) {
            const int32_t v = __shfl_sync(kFullMask, C.v, (lane & 24) + j);
            if (v < 0 || first != kNoStamp) continue;
            const StampRec R = staged(row, j);
            if (R.kt > lc && cover<true>(S, v, R, B, L.h, half, false) >= kPartCentreIn) first = v;
        }
        __syncwarp();
    }
    if (mine && first != kNoStamp) atomicMin(&fr[8 * I.p + k], first);
}

// Decision bits of one entry for the octet's eight children: low byte kept, high byte painted.
__device__ __forceinline__ unsigned decision_bits(int c) {
    const unsigned keep = __ballot_sync(kFullMask, c != kDrop), paint = __ballot_sync(kFullMask, c == kPaint);
    const int o = threadIdx.x & 24;
    return ((keep >> o) & 0xFFu) | (((paint >> o) & 0xFFu) << 8);
}

// Per item: the entries' decisions, and per child how many a refined child keeps or paint one that stays a leaf.
__global__ void __launch_bounds__(128) long_count(LevelIn L, StampDev S, double half, const Item* items,
                                                  const long long* tot, const int32_t* fr, uint16_t* cls,
                                                  int32_t* icnt) {
    __shared__ float4 s_rec[16 * kStageRow];
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3;
    const int lane = threadIdx.x & 31, k = threadIdx.x & 7;
    float4* row = s_rec + (threadIdx.x >> 3) * kStageRow;
    const bool mine = w < tot[kLongCtr + 1];
    const Item I = mine ? items[w] : Item{0, 0, 0, 0};
    const Child B = child_box(L, I.cell, k);
    const int32_t f = mine ? fr[8 * I.p + k] : kNoStamp;
    int32_t n = 0;
    Entries E{I.b, I.e, -1, 0, {}, {}};
    load_entries(E, L, S, k);
    while (__any_sync(kFullMask, E.m > 0)) {
        const Entries C = E;
        stage_entries(C, row, k);
        __syncwarp();
        E.q0 += 8;
        load_entries(E, L, S, k);
        const int mm = __reduce_max_sync(kFullMask, C.m);
        unsigned own = 0;
        for (int j = 0; j < mm; ++j) {
            const int32_t v = __shfl_sync(kFullMask, C.v, (lane & 24) + j);
            int c = kDrop;
            if (j < C.m) {
                if (v < 0) {
                    c = kPaint;
                } else {
                    const bool refined = f <= v;
                    const int x = cover<true>(S, v, staged(row, j), B, L.h, half, !refined);
                    c = x == kIn ? kPaint : (x == kOut ? kDrop : (refined ? kKeep : (x == kPartCentreIn ? kPaint : kDrop)));
                }
            }
            const unsigned bits = decision_bits(c);
            if (k == j) own = bits;
            n += f != kNoStamp ? c != kDrop : c == kPaint;
        }
        if (k < C.m) cls[C.q0 + k] = (uint16_t)own;
        __syncwarp();
    }
    if (mine) icnt[8 * w + k] = n;
}

// One block per long cell: the items' counts become exclusive sums per child; the child's total and slot, and (a warp per
// child) for a painted child that stays a leaf the blend, in order, of the stamps that paint it.
constexpr int kSumRows = 32;  // items at a time (a lane per item and child)
__global__ void __launch_bounds__(8 * kSumRows) long_sums(LevelIn L, StampDev S, const LongCell* cells, int item,
                                                          const long long* tot, const int32_t* fr, const uint16_t* cls,
                                                          int32_t* icnt, uint64_t* slot, int32_t* cnt) {
    __shared__ int32_t s_x[8][kSumRows + 1];
    const int64_t p = blockIdx.x;
    const int k = threadIdx.x & 7, row = threadIdx.x >> 3, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (p >= tot[kLongCtr]) return;
    const LongCell C = cells[p];
    const int64_t ni = (C.e - C.b + item - 1) / item;
    int32_t sum = 0;  // warp w sums child w's items
    for (int64_t j = 0; j < ni; j += kSumRows) {
        int32_t* x = icnt + 8 * (C.item + j + row) + k;
        s_x[k][row] = j + row < ni ? *x : 0;
        __syncthreads();
        const int32_t own = s_x[warp][lane];
        int32_t pre = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(kFullMask, pre, o);
            if (lane >= o) pre += u;
        }
        s_x[warp][lane] = sum + pre - own;
        sum += __shfl_sync(kFullMask, pre, 31);
        __syncthreads();
        if (j + row < ni) *x = s_x[k][row];
        __syncthreads();
    }
    const int64_t t = 8 * C.cell + warp;
    if (fr[8 * p + warp] != kNoStamp) {
        if (lane == 0) {
            slot[t] = kInternal;
            cnt[t] = sum;
        }
        return;
    }
    float4 val = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t base = C.b; sum != 0 && base < C.e; base += 32) {
        const int64_t q = base + lane;
        const bool paints = q < C.e && ((cls[q] >> (8 + warp)) & 1u);
        const int32_t v = paints ? L.ent[q] : 0;
        unsigned m = __ballot_sync(kFullMask, paints);
        while (m) {  // every lane folds the same sequence
            const int32_t x = __shfl_sync(kFullMask, v, __ffs(m) - 1);
            m &= m - 1;
            blend(val, S.rgba[x < 0 ? ~x : x]);
        }
    }
    if (lane == 0) {
        slot[t] = leaf_key(val);
        cnt[t] = 0;
    }
}

// One octet per item: its kept entries at the child's list start plus the counts of the cell's earlier items.
__global__ void __launch_bounds__(128) long_write(LevelIn L, const Item* items, const long long* tot, const uint64_t* slot,
                                                  const uint16_t* cls, const int32_t* icnt, const int64_t* noff,
                                                  int32_t* nent) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3;
    const int k = threadIdx.x & 7;
    if (w >= tot[kLongCtr + 1]) return;
    const Item I = items[w];
    const uint64_t s = slot[8 * I.cell + k];
    if (!(s & kInternal)) return;
    int64_t pos = noff[s & ~kInternal] + icnt[8 * w + k];
    for (int64_t q = I.b; q < I.e; ++q) {
        const unsigned bits = cls[q];
        if ((bits >> k) & 1u) {
            const int32_t v = L.ent[q];
            nent[pos++] = (v >= 0 && ((bits >> (8 + k)) & 1u)) ? ~v : v;
        }
    }
}

// ---------------------------------------------------------------------------
// Every cell: one octet each (16 cells a block).
// ---------------------------------------------------------------------------

// Sums of a block of the octet kernels (entries and cells of the next level), then their exclusive sums over the
// blocks (scan_sums).
struct BlockSum {
    int64_t ent, cells;
};

// Sum of x over the warp.
__device__ __forceinline__ int64_t warp_total(int64_t x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(kFullMask, x, o);
    return x;
}

// The children of every cell: slot (internal, or the leaf's key), list length, the entries' decisions; the block's
// sums; in tot the longest list and the long ones. Cells with long lists only add their sums here.
template <bool kExact>
__global__ void __launch_bounds__(8 * kCells, 9) expand_count(LevelIn L, StampDev S, double half, uint64_t* slot,
                                                           int32_t* cnt, uint16_t* cls, BlockSum* bs, long long* tot) {
    __shared__ float4 s_rec[kCells * kColourRow];
    __shared__ int64_t s_ent[kCells / 4], s_int[kCells / 4];
    const int64_t i = (int64_t)blockIdx.x * kCells + (threadIdx.x >> 3);
    const int lane = threadIdx.x & 31, k = threadIdx.x & 7, lc = L.level + 1;
    int64_t b = 0, e = 0;
    if (i < L.n) {
        b = L.off[i];
        e = L.off[i + 1];
    }
    const bool is_long = e - b > L.limit;
    if (is_long) e = b;
    int32_t n = 0;
    bool found = false;
    float4 val = make_float4(0.f, 0.f, 0.f, 0.f);
    if (__any_sync(kFullMask, b < e)) {
        const Child B = child_box(L, i < L.n ? i : 0, k);
        float4* row = s_rec + (threadIdx.x >> 3) * kColourRow;
        Entries C{b, e, -1, 0, {}, {}};
        for (; __any_sync(kFullMask, C.q0 < C.e); C.q0 += 8) {
            load_entries(C, L, S, k);  // (most lists are short: no loads ahead, which cost registers)
            // (the colours too: asked for by the child that an entry paints, each was a wait; 1 % of a depth-24 paint)
            if (k < C.m) row[16 + k] = __ldg(S.rgba + (C.v < 0 ? ~C.v : C.v));
            stage_entries(C, row, k);
            __syncwarp();
            const int mm = __reduce_max_sync(kFullMask, C.m);
            unsigned own = 0;
            for (int j = 0; j < mm; ++j) {
                const int32_t v = __shfl_sync(kFullMask, C.v, (lane & 24) + j);
                int c = kDrop;
                if (j < C.m) {
                    if (v < 0) {
                        c = kPaint;
                    } else {
                        const StampRec R = staged(row, j);
                        const bool refines = found || R.kt > lc;
                        const int x = cover<kExact>(S, v, R, B, L.h, half, !refines);
                        if (x == kIn) {
                            c = kPaint;
                        } else if (x != kOut) {
                            found = refines;  // (the first stamp that partially covers it with a deeper target)
                            c = refines ? kKeep : (x == kPartCentreIn ? kPaint : kDrop);
                        }
                    }
                }
                const unsigned bits = decision_bits(c);
                if (k == j) own = bits;
                n += c != kDrop;
                if (c == kPaint && !found) blend(val, row[16 + j]);
            }
            if (k < C.m) cls[C.q0 + k] = (uint16_t)own;
            __syncwarp();
        }
    }
    const int64_t t = 8 * i + k;
    if (i < L.n) {
        if (is_long) {
            found = slot[t] == kInternal;
            n = cnt[t];
        } else {
            if (!found) n = 0;
            slot[t] = found ? kInternal : leaf_key(val);
            cnt[t] = n;
        }
    }
    if (n > kLongFew) {
        unsigned long long* lists = reinterpret_cast<unsigned long long*>(tot + kTotLong);
        for (int x = 0; x < (n > kLongMany ? 4 : 2); ++x) atomicAdd(&lists[x], (x & 1) ? (unsigned long long)n : 1ull);
    }
    const int32_t longest = __reduce_max_sync(kFullMask, n);
    const int64_t ents = longest < (1 << 26) ? (int64_t)__reduce_add_sync(kFullMask, n) : warp_total(n);
    const int ints = __popc(__ballot_sync(kFullMask, found));
    if (lane == 0) {
        s_ent[threadIdx.x >> 5] = ents;
        s_int[threadIdx.x >> 5] = ints;
        if (longest > kLongFew) atomicMax(&tot[kTotLongest], (long long)longest);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        BlockSum x{0, 0};
        for (int w = 0; w < kCells / 4; ++w) {
            x.ent += s_ent[w];
            x.cells += s_int[w];
        }
        bs[blockIdx.x] = x;
    }
}

// The children of the cells of the level above the deepest: leaves all, each the blend of the stamps that hold its centre
// (one that holds the whole leaf holds its centre too, and one that does not touch it does not: also in FP64, whose
// rounding is monotone), in order. A distance instead of three, and neither decisions nor lists: 28.8 million cells of
// the depth-24 table take 11.2 ms instead of 18.9 (expand_count), bound by the waits for records (69 % of the issue slots).
__global__ void __launch_bounds__(8 * kCells, 9) expand_last(LevelIn L, StampDev S, double half, uint64_t* slot) {
    __shared__ float4 s_rec[kCells * kColourRow];
    const int64_t i = (int64_t)blockIdx.x * kCells + (threadIdx.x >> 3);
    const int lane = threadIdx.x & 31, k = threadIdx.x & 7;
    int64_t b = 0, e = 0;
    if (i < L.n) {
        b = L.off[i];
        e = L.off[i + 1];
    }
    const bool is_long = e - b > L.limit;
    if (is_long) e = b;
    float4 val = make_float4(0.f, 0.f, 0.f, 0.f);
    if (__any_sync(kFullMask, b < e)) {
        // the leaf's centre, (2 j + 1) h / 2, as two words per axis, and the margin's terms (cover32)
        const uint32_t* coord = L.coord + 3 * (i < L.n ? i : 0);
        float mh[3], ml[3], A = 0.0f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const uint32_t cc = 2u * coord[a] + ((k >> a) & 1u);
            plane_words(2 * ((int32_t)cc - (1 << L.level)) + 1, 0.5f * L.hf, mh[a], ml[a]);
            A += fabsf(mh[a]);
        }
        const float g1 = 2.2737367544323206e-13f * A, g2 = 5.684341886080802e-14f * A;  // 2^-42, 2^-44
        float4* row = s_rec + (threadIdx.x >> 3) * kColourRow;
        Entries C{b, e, -1, 0, {}, {}};
        for (; __any_sync(kFullMask, C.q0 < C.e); C.q0 += 8) {
            load_entries(C, L, S, k);
            if (k < C.m) row[16 + k] = __ldg(S.rgba + (C.v < 0 ? ~C.v : C.v));
            stage_entries(C, row, k);
            __syncwarp();
            const int mm = __reduce_max_sync(kFullMask, C.m);
            for (int j = 0; j < mm; ++j) {
                const int32_t v = __shfl_sync(kFullMask, C.v, (lane & 24) + j);
                if (j >= C.m) continue;
                bool paints = v < 0;
                if (!paints) {
                    const StampRec R = staged(row, j);
                    const float x0 = __fadd_rn(__fsub_rn(R.ch[0], mh[0]), __fsub_rn(R.cl0, ml[0]));
                    const float x1 = __fadd_rn(__fsub_rn(R.ch[1], mh[1]), __fsub_rn(R.cl1, ml[1]));
                    const float x2 = __fadd_rn(__fsub_rn(R.ch[2], mh[2]), __fsub_rn(R.cl2, ml[2]));
                    const float cen2 = fmaf(x2, x2, fmaf(x1, x1, x0 * x0)), d = cen2 - R.r2;
                    const float n = fabsf(x0) + fabsf(x1) + fabsf(x2);
                    const float margin = fmaf(9.5367431640625e-07f, cen2 + R.r2, g1 * (n + g2));  // 2^-20 (cen2 + r2) + ...
                    paints = d < 0.0f;
                    if (!(fabsf(d) > margin)) {
                        const int x = cover64(S.c + 3 * (int64_t)v, S.r2[v], 2u * coord[0] + (k & 1u),
                                              2u * coord[1] + ((k >> 1) & 1u), 2u * coord[2] + ((k >> 2) & 1u), L.h, half);
                        paints = x == kIn || x == kPartCentreIn;
                    }
                }
                if (paints) blend(val, row[16 + j]);
            }
            __syncwarp();
        }
    }
    if (i < L.n && !is_long) slot[8 * i + k] = leaf_key(val);
}

// Exclusive sums over the blocks, two levels: within kScanItems of them in place, and over those groups (sup).
constexpr int kScanThreads = 1024, kScanPer = 4, kScanItems = kScanThreads * kScanPer;

// Exclusive sums of x over the block's threads; *total = the block's sum.
__device__ __forceinline__ BlockSum block_scan(BlockSum x, BlockSum* total) {
    __shared__ BlockSum s_w[kScanThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    BlockSum v = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t a = __shfl_up_sync(kFullMask, v.ent, o), c = __shfl_up_sync(kFullMask, v.cells, o);
        if (lane >= o) {
            v.ent += a;
            v.cells += c;
        }
    }
    __syncthreads();
    if (lane == 31) s_w[w] = v;
    __syncthreads();
    if (w == 0) {
        BlockSum y = lane < (int)(blockDim.x >> 5) ? s_w[lane] : BlockSum{0, 0};
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t a = __shfl_up_sync(kFullMask, y.ent, o), c = __shfl_up_sync(kFullMask, y.cells, o);
            if (lane >= o) {
                y.ent += a;
                y.cells += c;
            }
        }
        s_w[lane] = y;
    }
    __syncthreads();
    if (w > 0) {
        v.ent += s_w[w - 1].ent;
        v.cells += s_w[w - 1].cells;
    }
    *total = s_w[(blockDim.x >> 5) - 1];
    return BlockSum{v.ent - x.ent, v.cells - x.cells};
}

// (with a single group, tot gets the whole sums here and scan_sup is not needed)
__global__ void __launch_bounds__(kScanThreads) scan_groups(BlockSum* bs, int64_t n, BlockSum* sup, long long* tot) {
    const int64_t g = (int64_t)blockIdx.x * kScanItems + (int64_t)threadIdx.x * kScanPer;
    BlockSum x[kScanPer], sum{0, 0};
#pragma unroll
    for (int j = 0; j < kScanPer; ++j) {
        x[j] = g + j < n ? bs[g + j] : BlockSum{0, 0};
        sum.ent += x[j].ent;
        sum.cells += x[j].cells;
    }
    BlockSum total;
    BlockSum pre = block_scan(sum, &total);
#pragma unroll
    for (int j = 0; j < kScanPer; ++j) {
        if (g + j < n) bs[g + j] = pre;
        pre.ent += x[j].ent;
        pre.cells += x[j].cells;
    }
    if (threadIdx.x == 0) {
        sup[blockIdx.x] = gridDim.x == 1 ? BlockSum{0, 0} : total;
        if (gridDim.x == 1) {
            tot[kTotEnt] = total.ent;
            tot[kTotCells] = total.cells;
        }
    }
}

// Exclusive sums over the groups (one block); tot[0], tot[1] = the whole sums.
__global__ void __launch_bounds__(kScanThreads) scan_sup(BlockSum* sup, int64_t n, long long* tot) {
    BlockSum carry{0, 0};
    for (int64_t base = 0; base < n; base += kScanThreads) {
        const int64_t g = base + threadIdx.x;
        const BlockSum x = g < n ? sup[g] : BlockSum{0, 0};
        BlockSum total;
        const BlockSum pre = block_scan(x, &total);
        if (g < n) sup[g] = BlockSum{carry.ent + pre.ent, carry.cells + pre.cells};
        carry.ent += total.ent;
        carry.cells += total.cells;
    }
    if (threadIdx.x == 0) {
        tot[kTotEnt] = carry.ent;
        tot[kTotCells] = carry.cells;
    }
}

// The next level: each refined child's index (into its slot), coordinates, list start and list, and with pid the
// partition it belongs to. The lists of long cells are left to long_write.
__global__ void __launch_bounds__(8 * kCells) expand_write(LevelIn L, uint64_t* slot, const int32_t* cnt, const uint16_t* cls,
                                                           const BlockSum* bs, const BlockSum* sup, const long long* tot,
                                                           const int32_t* pid, uint32_t* ncoord, int64_t* noff, int32_t* nent, int32_t* npid) {
    __shared__ int64_t s_ent[kCells / 4];
    __shared__ int s_int[kCells / 4];
    const int64_t i = (int64_t)blockIdx.x * kCells + (threadIdx.x >> 3);
    const int lane = threadIdx.x & 31, k = threadIdx.x & 7, warp = threadIdx.x >> 5;
    const int64_t t = 8 * i + k;
    const bool internal = i < L.n && slot[t] == kInternal;
    const int64_t n = internal ? cnt[t] : 0;
    // offsets: the block's, the earlier warps', the earlier lanes'
    int64_t pre = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t u = __shfl_up_sync(kFullMask, pre, o);
        if (lane >= o) pre += u;
    }
    const unsigned im = __ballot_sync(kFullMask, internal);
    if (lane == 31) {
        s_ent[warp] = pre;
        s_int[warp] = __popc(im);
    }
    __syncthreads();
    const BlockSum base = bs[blockIdx.x], group = sup[blockIdx.x / kScanItems];
    int64_t w = base.ent + group.ent + pre - n, j = base.cells + group.cells + __popc(im & ((1u << lane) - 1u));
    for (int q = 0; q < warp; ++q) {
        w += s_ent[q];
        j += s_int[q];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) noff[tot[kTotCells]] = tot[kTotEnt];
    if (internal) {
        slot[t] = kInternal | (uint64_t)j;
        ncoord[3 * j] = 2u * L.coord[3 * i] + (k & 1u);
        ncoord[3 * j + 1] = 2u * L.coord[3 * i + 1] + ((k >> 1) & 1u);
        ncoord[3 * j + 2] = 2u * L.coord[3 * i + 2] + ((k >> 2) & 1u);
        noff[j] = w;
        if (pid) npid[j] = pid[i];
    }
    int64_t b = 0, e = 0;
    if (i < L.n) {
        b = L.off[i];
        e = L.off[i + 1];
        if (e - b > L.limit) e = b;
    }
    for (int64_t q0 = b; __any_sync(kFullMask, q0 < e); q0 += 8) {
        const int m = (int)max((int64_t)0, min((int64_t)8, e - q0));
        const int32_t vv = k < m ? L.ent[q0 + k] : 0;
        const int own = k < m ? (int)cls[q0 + k] : 0;
        const int mm = __reduce_max_sync(kFullMask, m);
        for (int x = 0; x < mm; ++x) {
            const int32_t v = __shfl_sync(kFullMask, vv, (lane & 24) + x);
            const int bits = __shfl_sync(kFullMask, own, (lane & 24) + x);
            if (internal && ((bits >> k) & 1)) nent[w++] = (v >= 0 && ((bits >> (8 + k)) & 1)) ? ~v : v;
        }
    }
}

// Stamps that touch the canvas, in order (the root's list).
__global__ void root_flags(StampDev S, int64_t n, double extent, double half, int64_t* flag) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const double lo[3] = {-half, -half, -half};
    double dmin2, dmax2;
    box_dist2(S.c + 3 * s, lo, extent, dmin2, dmax2);
    flag[s] = dmin2 < S.r2[s] ? 1 : 0;
}
__global__ void root_write(int64_t n, const int64_t* flag_scan, const int64_t* flag, int32_t* ent) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s < n && flag[s]) ent[flag_scan[s]] = (int32_t)s;
}

// Merge of identical siblings, bottom-up, an octet per cell (a lane per child): ckey = the common key of the eight
// children, else kNotCollapsed. A cell that does not collapse survives as a record; place = its rank among its
// block's surviving cells and the rank of its first leaf among the block's (kSurvives, bits 16.., bits 0..15), and
// the block's sums of both.
constexpr int kMergeCells = 32;  // cells per block (256 threads)
constexpr uint32_t kSurvives = 1u << 31;
__global__ void __launch_bounds__(8 * kMergeCells) collapse_level(int64_t n, const uint64_t* slot, const uint64_t* ckey_next,
                                                                  uint64_t* ckey, bool is_root, uint32_t* place,
                                                                  BlockSum* bs) {
    __shared__ uint32_t s_sum[kMergeCells];  // leaves | survives << 16 per cell
    const int64_t t = (int64_t)blockIdx.x * (8 * kMergeCells) + threadIdx.x, i = t >> 3;
    const int o = threadIdx.x & 24, k = threadIdx.x & 7;
    uint64_t key = 0;
    if (i < n) {
        const uint64_t v = slot[t];
        key = (v & kInternal) ? ckey_next[v & ~kInternal] : v;
    }
    const uint64_t k0 = __shfl_sync(kFullMask, key, o);
    const unsigned eq = (__ballot_sync(kFullMask, key == k0 && key != kNotCollapsed) >> o) & 0xFFu;
    const unsigned lf = (__ballot_sync(kFullMask, key != kNotCollapsed && key != 0) >> o) & 0xFFu;
    const bool same = eq == 0xFFu && !is_root, surv = i < n && !same;
    if (k == 0) {
        if (i < n) ckey[i] = same ? k0 : kNotCollapsed;
        s_sum[threadIdx.x >> 3] = surv ? (1u << 16) | __popc(lf) : 0u;
    }
    __syncthreads();
    if (threadIdx.x < kMergeCells) {
        const uint32_t own = s_sum[threadIdx.x];
        uint32_t pre = own;
#pragma unroll
        for (int d = 1; d < kMergeCells; d <<= 1) {
            const uint32_t u = __shfl_up_sync(kFullMask, pre, d);
            if ((int)threadIdx.x >= d) pre += u;
        }
        const int64_t c = (int64_t)blockIdx.x * kMergeCells + threadIdx.x;
        if (c < n) place[c] = (pre - own) | (own ? kSurvives : 0u);
        if (threadIdx.x == kMergeCells - 1) bs[blockIdx.x] = BlockSum{(int64_t)(pre & 0xFFFFu), (int64_t)(pre >> 16)};
    }
}

// Where a level's surviving cells go: place, the blocks' exclusive sums and the groups'.
struct Ranks {
    const uint32_t* place;
    const BlockSum* bs;
    const BlockSum* sup;
};
__device__ __forceinline__ int64_t record_rank(const Ranks& R, int64_t c) {
    const int64_t b = c / kMergeCells;
    return R.bs[b].cells + R.sup[b / kScanItems].cells + ((R.place[c] >> 16) & 0x7FFFu);
}

// Pool rows of the surviving records of one level, a lane per slot.
// Leaf numbers (breadth-first slot order) are written modulo 2^31; the slot position 8 r + k of each leaf
// whose number is a nonzero multiple m 2^31 goes to wraps[m - 1].
__global__ void __launch_bounds__(8 * kMergeCells) write_level(int64_t n, const uint64_t* slot, const uint64_t* ckey_next,
                                                               Ranks own, Ranks next, int64_t rec_base,
                                                               int64_t next_rec_base, int64_t leaf_base, int32_t* nodes,
                                                               uint2* leaves, int64_t* wraps) {
    const int64_t t = (int64_t)blockIdx.x * (8 * kMergeCells) + threadIdx.x, i = t >> 3;
    const int o = threadIdx.x & 24, k = threadIdx.x & 7;
    uint32_t pl = 0;
    uint64_t v = 0, key = 0;
    if (i < n) {
        pl = own.place[i];
        v = slot[t];
        key = (v & kInternal) ? ckey_next[v & ~kInternal] : v;
    }
    const bool leaf = key != kNotCollapsed && key != 0;
    const unsigned lf = (__ballot_sync(kFullMask, leaf) >> o) & 0xFFu;
    if (!(pl & kSurvives)) return;
    const BlockSum b = own.bs[blockIdx.x], g = own.sup[blockIdx.x / kScanItems];
    const int64_t r = rec_base + b.cells + g.cells + ((pl >> 16) & 0x7FFFu);
    int32_t out = 0;
    if (leaf) {
        const int64_t l = leaf_base + b.ent + g.ent + (pl & 0xFFFFu) + __popc(lf & ((1u << k) - 1u));
        leaves[l] = make_uint2((uint32_t)key, (uint32_t)(key >> 32));
        const int64_t low = l & 0x7FFFFFFFll;
        out = -(int32_t)low - 1;
        if (low == 0 && l > 0) wraps[(l >> 31) - 1] = 8 * r + k;
    } else if (key == kNotCollapsed) {
        out = (int32_t)(next_rec_base + record_rank(next, (int64_t)(v & ~kInternal)));
    }
    nodes[8 * r + k] = out;
}

// In-place exclusive scan of int64 (three phases; block sums scanned recursively).
constexpr int kScanBlock = 1024;
__global__ void scan_block(int64_t* d, int64_t n, int64_t* sums) {
    __shared__ int64_t s[kScanBlock];
    const int64_t g = (int64_t)blockIdx.x * kScanBlock + threadIdx.x;
    const int64_t x = g < n ? d[g] : 0;
    s[threadIdx.x] = x;
    __syncthreads();
    for (int o = 1; o < kScanBlock; o <<= 1) {
        const int64_t y = threadIdx.x >= (unsigned)o ? s[threadIdx.x - o] : 0;
        __syncthreads();
        s[threadIdx.x] += y;
        __syncthreads();
    }
    if (g < n) d[g] = s[threadIdx.x] - x;
    if (threadIdx.x == kScanBlock - 1) sums[blockIdx.x] = s[threadIdx.x];
}
__global__ void scan_add(int64_t* d, int64_t n, const int64_t* sums) {
    const int64_t g = (int64_t)blockIdx.x * kScanBlock + threadIdx.x;
    if (g < n) d[g] += sums[blockIdx.x];
}

}  // namespace

// ---------------------------------------------------------------------------
// Device memory of the painter: a memory pool of its own. From the device allocator an array costs 30-50 us and a free
// 30 us (0.3 and 0.5 ms a GB), from the pool 1.5 us each, so what a level needs only while it is painted is one
// allocation. Everything runs on the legacy default stream, which orders frees and reuse. After a paint the pool keeps
// what the last two paintings (their appends among them) had live at once, whichever is more, and room for the gaps
// between arrays (with_gaps), but no more than a kPoolShare-th of the device's free memory; the rest is given back. The
// same paintings, changed and painted again, then allocate nothing: the depth-24 table of 210,000 stamps, 6 GB live at once,
// takes 35.3 ms, with an eighth of that for the gaps 36.5, and a session of appends 12.8 and 13.2. An allocation of the
// library that finds no memory gets what is not live (paint_pool_trim), and canvox_release destroys the pool.
// ---------------------------------------------------------------------------
namespace {
constexpr size_t kPoolShare = 16;
// 1.16 to 1.21 of the bytes live were reserved for paintings of 0.6 and 6 GB, and 72 MB more than the 62 MB of a small one
// (the pool takes the device's memory 32 MiB at a time).
size_t with_gaps(size_t live) { return live + live / 4 + ((size_t)64 << 20); }
size_t g_live_before = 0;  // the painting's before the last
cudaMemPool_t g_pool = nullptr;

cudaError_t pool_ready() {
    if (g_pool) return cudaSuccess;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    cudaMemPoolProps props;
    std::memset(&props, 0, sizeof(props));
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    e = cudaMemPoolCreate(&g_pool, &props);
    if (e != cudaSuccess) {
        g_pool = nullptr;
        return e;
    }
    uint64_t keep = ~0ull;  // nothing is given back at the synchronisations of a paint
    return cudaMemPoolSetAttribute(g_pool, cudaMemPoolAttrReleaseThreshold, &keep);
}

void pool_trim(size_t keep) {
    if (g_pool && cudaDeviceSynchronize() == cudaSuccess) cudaMemPoolTrimTo(g_pool, keep);
}

// The most bytes live at once since the mark was last set back (to what is live then).
uint64_t pool_high_water() {
    uint64_t high = 0;
    if (!g_pool || cudaMemPoolGetAttribute(g_pool, cudaMemPoolAttrUsedMemHigh, &high) != cudaSuccess) return 0;
    return high;
}
void new_painting() {
    g_live_before = (size_t)pool_high_water();
    uint64_t zero = 0;
    if (g_pool) cudaMemPoolSetAttribute(g_pool, cudaMemPoolAttrUsedMemHigh, &zero);
}

template <typename T>
cudaError_t dalloc(T** p, int64_t n) {
    *p = nullptr;
    cudaError_t e = pool_ready();
    if (e != cudaSuccess) return e;
    const size_t bytes = sizeof(T) * (size_t)(n > 0 ? n : 1);
    e = cudaMallocFromPoolAsync(reinterpret_cast<void**>(p), bytes, g_pool, 0);
    if (e == cudaErrorMemoryAllocation) {  // once more, with what the pool does not hold live and the canvas before
        cudaGetLastError();
        canvas_spares_free();
        pool_trim(0);
        e = cudaMallocFromPoolAsync(reinterpret_cast<void**>(p), bytes, g_pool, 0);
    }
    return e;
}
void dfree(void* p) {
    if (p) cudaFreeAsync(p, 0);
}
}  // namespace

void paint_pool_trim() { pool_trim(0); }

void paint_pool_release() {
    if (!g_pool) return;
    cudaDeviceSynchronize();
    cudaMemPoolDestroy(g_pool);
    g_pool = nullptr;
    g_live_before = 0;
}

// Exclusive scan of d[0..n) in place; returns the total through *total (synchronous).
cudaError_t scan_i64(int64_t* d, int64_t n, int64_t* total) {
    if (n <= 0) {
        *total = 0;
        return cudaSuccess;
    }
    const int64_t nb = (n + kScanBlock - 1) / kScanBlock;
    int64_t* sums = nullptr;
    cudaError_t e = dalloc(&sums, nb + 1);
    if (e != cudaSuccess) return e;
    scan_block<<<(unsigned)nb, kScanBlock>>>(d, n, sums);
    e = cudaGetLastError();
    int64_t t = 0;
    if (e == cudaSuccess) {
        if (nb > 1) {
            e = scan_i64(sums, nb, &t);  // sums becomes the block offsets
            if (e == cudaSuccess) {
                scan_add<<<(unsigned)nb, kScanBlock>>>(d, n, sums);
                e = cudaGetLastError();
            }
        } else {
            e = cudaMemcpy(&t, sums, sizeof(int64_t), cudaMemcpyDeviceToHost);
        }
    }
    dfree(sums);
    *total = t;
    return e;
}

namespace {

struct DevBuf {
    std::vector<void*> ptrs;
    ~DevBuf() {
        for (void* p : ptrs) dfree(p);
    }
    template <typename T>
    cudaError_t alloc(T** p, int64_t n) {
        const cudaError_t e = dalloc(p, n);
        if (e == cudaSuccess) ptrs.push_back(*p);
        return e;
    }
};

// Arrays in one allocation: sizes first, then alloc(), then the same calls of take().
struct Arena {
    size_t bytes = 0;
    unsigned char* base = nullptr;
    template <typename T>
    void size(int64_t n) {
        bytes += (sizeof(T) * (size_t)n + 255) / 256 * 256;
    }
    template <typename T>
    T* take(int64_t n) {
        T* p = reinterpret_cast<T*>(base);
        base += (sizeof(T) * (size_t)n + 255) / 256 * 256;
        return p;
    }
};

unsigned blocks_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

void scan_sums(BlockSum* bs, int64_t n, BlockSum* sup, long long* tot) {
    const int64_t ng = (n + kScanItems - 1) / kScanItems;
    scan_groups<<<(unsigned)ng, kScanThreads>>>(bs, n, sup, tot);
    if (ng > 1) scan_sup<<<1, kScanThreads>>>(sup, ng, tot);
}

// ---------------------------------------------------------------------------
// Partitions for appends. The refined cells of one level P (the partition level)
// split the tree: breadth-first order keeps each one's subtree contiguous within
// every deeper level, in the order of the partitions. Stamps appended later do
// not change what any earlier stamp does (a cell's first refining stamp can only
// appear among the new ones), so a partition whose stamp list at level P is
// unchanged keeps its whole subtree, and only the others are painted again.
// ---------------------------------------------------------------------------

// off[p] = first index of partition p in the (nondecreasing) partition ids of one level, p = 0 .. nseg.
__global__ void seg_offsets(int64_t n, const int32_t* pid, int64_t nseg, int64_t* off) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p > nseg) return;
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (pid[mid] < p) lo = mid + 1;
        else hi = mid;
    }
    off[p] = lo;
}

__global__ void iota32(int64_t n, int32_t* v) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) v[i] = (int32_t)i;
}

// Morton code of a level-P cell: its child indices k = x + 2y + 4z from the root down, 3 bits per level (the
// breadth-first order of the level).
__device__ __forceinline__ uint64_t morton(const uint32_t* c, int P) {
    uint64_t m = 0;
    for (int b = P - 1; b >= 0; --b)
        m = (m << 3) | (uint64_t)(((c[0] >> b) & 1u) | (((c[1] >> b) & 1u) << 1) | (((c[2] >> b) & 1u) << 2));
    return m;
}
__global__ void morton_codes(int64_t n, const uint32_t* coord, int P, uint64_t* code) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) code[i] = morton(coord + 3 * i, P);
}

// One warp per new partition: the old partition with the same cell and the same stamp list (entry for entry),
// else -1.
__global__ void match_partitions(int64_t n_new, const uint32_t* coord_new, const int64_t* off_new,
                                 const int32_t* ent_new, int64_t n_old, const uint64_t* code_old,
                                 const int64_t* off_old, const int32_t* ent_old, int P, int32_t* reuse) {
    const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (p >= n_new) return;  // warp-uniform
    const uint64_t m = morton(coord_new + 3 * p, P);
    int64_t lo = 0, hi = n_old;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (code_old[mid] < m) lo = mid + 1;
        else hi = mid;
    }
    int32_t q = -1;
    if (lo < n_old && code_old[lo] == m) {
        const int64_t bn = off_new[p], en = off_new[p + 1], bo = off_old[lo], eo = off_old[lo + 1];
        bool same = en - bn == eo - bo;
        for (int64_t j = lane; same && j < en - bn; j += 32)
            if (ent_new[bn + j] != ent_old[bo + j]) same = false;
        same = __all_sync(kFullMask, same);
        if (same) q = (int32_t)lo;
    }
    if (lane == 0) reuse[p] = q;
}

// Cells `sel` of a level (their coordinates and stamp lists) gathered into a new level; dst_off = exclusive scan of
// the selected lists' lengths.
__global__ void gather_cells(int64_t m, const int32_t* sel, const uint32_t* coord, const int64_t* off,
                             const int32_t* ent, const int64_t* dst_off, uint32_t* ncoord, int64_t* noff, int32_t* nent) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= m) return;
    const int64_t i = sel[r], b = off[i], e = off[i + 1], d = dst_off[r];
    if (lane < 3) ncoord[3 * r + lane] = coord[3 * i + lane];
    if (lane == 0) noff[r] = d;
    for (int64_t j = lane; j < e - b; j += 32) nent[d + j] = ent[b + j];
}
__global__ void list_lengths(int64_t m, const int32_t* sel, const int64_t* off, int64_t* len) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < m) len[r] = off[sel[r] + 1] - off[sel[r]];
}

// Per level (a block each) and new partition p, the first cell of p: the exclusive sums of the cell counts, from the
// kept subtree (reuse[p] = q) or the repainted one (rep[p] = r); dst[n] = total[level] = the level's cells.
struct PartLevels {
    const int64_t *old[kMaxDepth], *rep[kMaxDepth];  // first cells per old and repainted partition (null: no such level)
    int64_t* dst[kMaxDepth];
};
__global__ void __launch_bounds__(kScanThreads) part_offsets(int64_t n, const int32_t* reuse, const int32_t* rep,
                                                             const __grid_constant__ PartLevels levels, int64_t* total) {
    const int64_t *off_old = levels.old[blockIdx.x], *off_rep = levels.rep[blockIdx.x];
    int64_t* dst = levels.dst[blockIdx.x];
    int64_t carry = 0;
    for (int64_t base = 0; base < n; base += kScanThreads) {
        const int64_t p = base + threadIdx.x;
        int64_t c = 0;
        if (p < n) {
            const int32_t q = reuse[p];
            if (q >= 0) c = off_old ? off_old[q + 1] - off_old[q] : 0;
            else if (off_rep) c = off_rep[rep[p] + 1] - off_rep[rep[p]];
        }
        BlockSum sum;
        const BlockSum pre = block_scan(BlockSum{c, 0}, &sum);
        if (p < n) dst[p] = carry + pre.ent;
        carry += sum.ent;
    }
    if (threadIdx.x == 0) dst[n] = total[blockIdx.x] = carry;
}

// The assembled level: each cell's eight slots copied from its source, internal children renumbered to the
// assembled next level (same partition, same position within it).
__global__ void assemble_level(int64_t n_dst, int64_t n_part, const int64_t* dst_off, const int64_t* dst_off_next,
                               const int32_t* reuse, const int32_t* rep, const uint64_t* slot_old,
                               const int64_t* off_old, const int64_t* off_old_next, const uint64_t* slot_rep,
                               const int64_t* off_rep, const int64_t* off_rep_next, uint64_t* slot_dst) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 8 * n_dst) return;
    const int64_t j = t >> 3;
    int64_t lo = 0, hi = n_part;  // the partition p with dst_off[p] <= j < dst_off[p + 1]
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (dst_off[mid] <= j) lo = mid;
        else hi = mid;
    }
    const int64_t p = lo, local = j - dst_off[p];
    const int32_t q = reuse[p];
    uint64_t v;
    int64_t src_next;
    if (q >= 0) {
        v = slot_old[8 * (off_old[q] + local) + (t & 7)];
        src_next = (v & kInternal) ? off_old_next[q] : 0;
    } else {
        const int32_t r = rep[p];
        v = slot_rep[8 * (off_rep[r] + local) + (t & 7)];
        src_next = (v & kInternal) ? off_rep_next[r] : 0;
    }
    if (v & kInternal) v = kInternal | (uint64_t)((int64_t)(v & ~kInternal) - src_next + dst_off_next[p]);
    slot_dst[t] = v;
}

}  // namespace

#define PCK(call)                                    \
    do {                                             \
        cudaError_t e_ = (call);                     \
        if (e_ != cudaSuccess) return e_;            \
    } while (0)

namespace {

// Merge of identical siblings and the breadth-first pools of the painted levels (slots[l]: 8 child slots per
// refined cell of level l), with the positions where leaf numbers pass multiples of 2^31.
cudaError_t finish_pools(const std::vector<uint64_t*>& slots, const std::vector<int64_t>& ncell, int32_t** d_nodes_out,
                         uint2** d_leaves_out, int64_t* n_rec_out, int64_t* n_leaf_out,
                         std::vector<int64_t>* level_begin, int64_t* wrap_out, int32_t* n_wrap_out) {
    DevBuf buf;
    // bottom-up merge of identical siblings, with every level's ranks
    const size_t nl = slots.size();
    std::vector<uint64_t*> ckey(nl + 1, nullptr);
    std::vector<Ranks> ranks(nl + 1);
    const auto blocks = [](int64_t nc) { return (nc + kMergeCells - 1) / kMergeCells; };
    const auto groups = [&](int64_t nc) { return (blocks(nc) + kScanItems - 1) / kScanItems; };
    Arena A;
    for (int64_t nc : ncell) {
        A.size<uint64_t>(nc);
        A.size<uint32_t>(nc);
        A.size<BlockSum>(blocks(nc));
        A.size<BlockSum>(groups(nc));
    }
    A.size<uint64_t>(2);
    A.size<long long>(2 * (int64_t)nl + 2);
    A.size<int64_t>(kMaxWraps);
    PCK(buf.alloc(&A.base, (int64_t)A.bytes));
    ckey[nl] = A.take<uint64_t>(2);  // below the deepest level: no refined cells
    ranks[nl] = Ranks{nullptr, nullptr, nullptr};
    long long* d_tot = A.take<long long>(2 * (int64_t)nl + 2);
    int64_t* d_wraps = A.take<int64_t>(kMaxWraps);
    for (size_t l = nl; l-- > 0;) {
        const int64_t nc = ncell[l], nb = blocks(nc), ng = groups(nc);
        ckey[l] = A.take<uint64_t>(nc);
        uint32_t* place = A.take<uint32_t>(nc);
        BlockSum *bs = A.take<BlockSum>(nb), *sup = A.take<BlockSum>(ng);
        collapse_level<<<(unsigned)nb, 8 * kMergeCells>>>(nc, slots[l], ckey[l + 1], ckey[l], l == 0, place, bs);
        scan_sums(bs, nb, sup, d_tot + 2 * l);
        PCK(cudaGetLastError());
        ranks[l] = Ranks{place, bs, sup};
    }
    std::vector<long long> tot(2 * nl);
    PCK(cudaMemcpy(tot.data(), d_tot, sizeof(long long) * tot.size(), cudaMemcpyDeviceToHost));
    // breadth-first numbering: records level by level, leaves in slot order
    std::vector<int64_t> rec_base(nl + 1, 0), leaf_base(nl + 1, 0);
    for (size_t l = 0; l < nl; ++l) {
        leaf_base[l + 1] = leaf_base[l] + tot[2 * l];
        rec_base[l + 1] = rec_base[l] + tot[2 * l + 1];
    }
    const int64_t n_rec = rec_base[nl], n_leaf = leaf_base[nl];
    if (n_rec > 0x7FFFFFFFll || n_leaf > kMaxLeaves) return cudaErrorMemoryAllocation;  // beyond the pool format
    const int32_t n_wrap = n_leaf > 0 ? (int32_t)((n_leaf - 1) >> 31) : 0;
    int32_t* d_nodes = nullptr;
    uint2* d_leaves = nullptr;
    PCK(canvas_malloc(kPoolNodes, reinterpret_cast<void**>(&d_nodes), sizeof(int32_t) * 8 * (size_t)n_rec));
    cudaError_t e = canvas_malloc(kPoolLeaves, reinterpret_cast<void**>(&d_leaves), sizeof(uint2) * (size_t)(n_leaf > 0 ? n_leaf : 1));
    if (e != cudaSuccess) {
        cudaFree(d_nodes);
        return e;
    }
    for (size_t l = 0; l < nl; ++l) {
        const int64_t nc = ncell[l];
        write_level<<<blocks_for(nc, kMergeCells), 8 * kMergeCells>>>(nc, slots[l], ckey[l + 1], ranks[l], ranks[l + 1],
                                                                       rec_base[l], rec_base[l + 1], leaf_base[l],
                                                                       d_nodes, d_leaves, d_wraps);
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess && n_wrap > 0)
        e = cudaMemcpy(wrap_out, d_wraps, sizeof(int64_t) * (size_t)n_wrap, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) {
        cudaFree(d_nodes);
        cudaFree(d_leaves);
        return e;
    }
    *n_wrap_out = n_wrap;
    *d_nodes_out = d_nodes;
    *d_leaves_out = d_leaves;
    *n_rec_out = n_rec;
    *n_leaf_out = n_leaf;
    level_begin->clear();
    for (size_t l = 0; l <= nl; ++l)
        if (l == 0 || rec_base[l] > rec_base[l - 1]) level_begin->push_back(rec_base[l]);
    return cudaSuccess;
}

}  // namespace

namespace {

// The power of two that brings the canvas side to [1, 2). NaN past 2^+-400, where the FP64 squares themselves come near
// the end of their range and the FP32 screen, which would not, is left out (every comparison with a NaN is open).
double screen_scale(double extent) {
    const int e = std::ilogb(extent);
    return e < -400 || e > 400 ? std::nan("") : std::ldexp(1.0, -e);
}

// Refined cells of one level with their ordered stamp lists (device arrays owned here).
struct Level {
    int64_t n = 0;
    int64_t n_ent = 0;    // entries of all lists
    int64_t longest = 0;  // the longest list (0: none is longer than kLongFew)
    int64_t long_cells[2] = {0, 0}, long_ent[2] = {0, 0};  // at most: lists longer than kLongFew, kLongMany; their entries
    int32_t level = 0;
    uint32_t* coord = nullptr;  // [n][3]
    int64_t* off = nullptr;     // [n + 1]
    int32_t* ent = nullptr;     // s: descends, ~s: paints the whole cell
    bool few() const { return n <= kFewCells; }
    int64_t limit() const { return few() ? kLongFew : kLongMany; }
    LevelIn in(double extent) const {
        const double h = std::ldexp(extent, -(level + 1));
        return LevelIn{n, level, coord, off, ent, limit(), h, (float)(h * screen_scale(extent))};
    }
    void free() {
        dfree(coord);
        dfree(off);
        dfree(ent);
        coord = nullptr;
        off = nullptr;
        ent = nullptr;
        n = 0;
    }
};

// Expand one level: the eight child slots of each cell (*slot_out, handed to the caller: a leaf key, or
// kInternal | index in the next level) and the next level's refined cells with their lists; with pid (the cells'
// partitions) also the next level's (*npid).
cudaError_t expand(const Level& L, const StampDev& S, double extent, double half, int depth, uint64_t** slot_out,
                   Level* next, const int32_t* pid, int32_t** npid) {
    DevBuf buf;
    const int64_t nch = 8 * L.n, nb = (L.n + kCells - 1) / kCells, ng = (nb + kScanItems - 1) / kScanItems;
    // cells with long lists: an octet per item of a list
    const bool longs = L.longest > L.limit();
    const int item = item_size(L.longest, L.n_ent), few = L.few() ? 0 : 1;
    const int64_t nlong = longs ? L.long_cells[few] : 0, ni = longs ? L.long_ent[few] / item + nlong : 0;
    const bool last = L.level + 1 == depth;  // (the children are leaves all)
    const int64_t n_cnt = last && !longs ? 0 : nch, n_cls = last && !longs ? 0 : L.n_ent;
    Arena A;
    A.size<int32_t>(n_cnt);
    A.size<uint16_t>(n_cls);
    A.size<BlockSum>(nb);
    A.size<BlockSum>(ng);
    A.size<long long>(kTotWords);
    A.size<LongCell>(nlong);
    A.size<Item>(ni);
    A.size<int32_t>(8 * ni);
    A.size<int32_t>(8 * nlong);
    PCK(buf.alloc(&A.base, (int64_t)A.bytes));
    int32_t* cnt = A.take<int32_t>(n_cnt);
    uint16_t* cls = A.take<uint16_t>(n_cls);
    BlockSum *bs = A.take<BlockSum>(nb), *sup = A.take<BlockSum>(ng);
    long long* tot = A.take<long long>(kTotWords);
    LongCell* cells = A.take<LongCell>(nlong);
    Item* items = A.take<Item>(ni);
    int32_t *icnt = A.take<int32_t>(8 * ni), *fr = A.take<int32_t>(8 * nlong);
    uint64_t* slot;
    PCK(dalloc(&slot, nch));
    *slot_out = slot;
    const LevelIn in = L.in(extent);
    PCK(cudaMemsetAsync(tot, 0, kTotWords * sizeof(long long), 0));
    if (longs) {
        find_long<<<blocks_for(L.n, 256), 256>>>(in, item, cells, items, fr, tot);
        long_first<<<blocks_for(ni, 16), 128>>>(in, S, half, items, tot, fr);
        long_count<<<blocks_for(ni, 16), 128>>>(in, S, half, items, tot, fr, cls, icnt);
        long_sums<<<(unsigned)nlong, 8 * kSumRows>>>(in, S, cells, item, tot, fr, cls, icnt, slot, cnt);
        PCK(cudaGetLastError());
    }
    if (last) {
        expand_last<<<(unsigned)nb, 8 * kCells>>>(in, S, half, slot);
        next->n = 0;
        next->level = depth;
        return cudaGetLastError();
    }
    (L.few() ? expand_count<true> : expand_count<false>)<<<(unsigned)nb, 8 * kCells>>>(in, S, half, slot, cnt, cls, bs, tot);
    scan_sums(bs, nb, sup, tot);
    PCK(cudaGetLastError());
    long long h_tot[kTotWords];
    PCK(cudaMemcpy(h_tot, tot, sizeof(h_tot), cudaMemcpyDeviceToHost));
    next->n = h_tot[kTotCells];
    next->n_ent = h_tot[kTotEnt];
    next->longest = h_tot[kTotLongest];
    for (int x = 0; x < 2; ++x) {
        next->long_cells[x] = h_tot[kTotLong + 2 * x];
        next->long_ent[x] = h_tot[kTotLong + 2 * x + 1];
    }
    next->level = L.level + 1;
    if (next->n == 0) return cudaSuccess;  // no internal child: the slots are all leaf keys
    PCK(dalloc(&next->coord, 3 * next->n));
    PCK(dalloc(&next->off, next->n + 1));
    PCK(dalloc(&next->ent, next->n_ent));
    if (pid) PCK(dalloc(npid, next->n));
    expand_write<<<(unsigned)nb, 8 * kCells>>>(in, slot, cnt, cls, bs, sup, tot, pid, next->coord, next->off, next->ent,
                                               pid ? *npid : nullptr);
    if (longs) long_write<<<blocks_for(ni, 16), 128>>>(in, items, tot, slot, cls, icnt, next->off, next->ent);
    return cudaGetLastError();
}

// Paint down from L (its arrays are freed on the way): slots and cell counts per level, until no refined cell is
// left, or up to level `stop` (that level's cells are then left unexpanded in *rest). With track, the cells of L
// are partitions 0 .. L.n - 1 and offs receives, per painted level, the first cell of each partition.
cudaError_t paint_down(Level L, const StampDev& S, double extent, double half, int depth, int stop, bool track,
                       std::vector<uint64_t*>* slots, std::vector<int64_t>* ncell, Level* rest,
                       std::vector<int64_t*>* offs) {
    const int64_t nseg = L.n;
    int32_t* pid = nullptr;
    cudaError_t e = cudaSuccess;
    if (track && L.n > 0) {
        e = dalloc(&pid, L.n);
        if (e == cudaSuccess) iota32<<<blocks_for(L.n, 256), 256>>>(L.n, pid);
    }
    while (e == cudaSuccess && L.n > 0 && L.level != stop) {
        uint64_t* slot = nullptr;
        int32_t* npid = nullptr;
        Level next;
        e = expand(L, S, extent, half, depth, &slot, &next, pid, &npid);
        if (slot) {
            slots->push_back(slot);
            ncell->push_back(L.n);
        }
        if (e == cudaSuccess && track) {
            int64_t* off = nullptr;
            e = dalloc(&off, nseg + 1);
            if (e == cudaSuccess) {
                offs->push_back(off);
                seg_offsets<<<blocks_for(nseg + 1, 256), 256>>>(L.n, pid, nseg, off);
                e = cudaGetLastError();
            }
        }
        dfree(pid);
        pid = npid;
        L.free();
        L = next;
        if (e != cudaSuccess) L.free();
    }
    dfree(pid);
    if (e == cudaSuccess && L.n > 0 && L.level == stop) {
        *rest = L;
    } else {
        L.free();
        rest->n = 0;
        rest->level = stop;
    }
    return e == cudaSuccess ? cudaDeviceSynchronize() : e;
}

}  // namespace

// What the painter keeps of a painted canvas for appends: the level-P cells (Morton codes and stamp lists) and
// the slots of every level from P down, with each partition's first cell per level.
struct PaintCache {
    int32_t depth = 0;
    double extent = 0.0;
    int64_t n_stamps = 0;       // stamps painted
    int64_t nP = 0;             // refined cells at the partition level
    uint64_t* code = nullptr;   // [nP] Morton codes (ascending)
    int64_t* lst_off = nullptr; // [nP + 1]
    int32_t* lst_ent = nullptr; // their stamp lists
    std::vector<uint64_t*> slots;  // levels P, P + 1, ...
    std::vector<int64_t> ncell;
    std::vector<int64_t*> off;     // per level: [nP + 1] first cell of each partition
};

void paint_cache_free(PaintCache* c) {
    if (!c) return;
    dfree(c->code);
    dfree(c->lst_off);
    dfree(c->lst_ent);
    for (auto* p : c->slots) dfree(p);
    for (auto* p : c->off) dfree(p);
    delete c;
}

namespace {

constexpr int kPartLevel = 5;  // partition level: up to 32,768 partitions

void free_all(std::vector<uint64_t*>& v) {
    for (auto* p : v) dfree(p);
    v.clear();
}
void free_all(std::vector<int64_t*>& v) {
    for (auto* p : v) dfree(p);
    v.clear();
}

// The root with the stamps [0, n) that touch the canvas, in order.
cudaError_t root_level(const StampDev& S, int64_t n, double extent, double half, Level* root) {
    DevBuf buf;
    int64_t *flag, *flag_scan, n_root = 0;
    PCK(buf.alloc(&flag, n));
    PCK(buf.alloc(&flag_scan, n));
    if (n > 0) {
        root_flags<<<blocks_for(n, 256), 256>>>(S, n, extent, half, flag);
        PCK(cudaGetLastError());
        PCK(cudaMemcpy(flag_scan, flag, sizeof(int64_t) * (size_t)n, cudaMemcpyDeviceToDevice));
        PCK(scan_i64(flag_scan, n, &n_root));
    }
    root->n = 1;
    root->n_ent = root->longest = n_root;
    for (int x = 0; x < 2; ++x) {
        root->long_cells[x] = 1;
        root->long_ent[x] = n_root;
    }
    root->level = 0;
    PCK(dalloc(&root->coord, 3));
    PCK(dalloc(&root->off, 2));
    PCK(dalloc(&root->ent, n_root));
    PCK(cudaMemset(root->coord, 0, 3 * sizeof(uint32_t)));
    const int64_t off0[2] = {0, n_root};
    PCK(cudaMemcpy(root->off, off0, sizeof(off0), cudaMemcpyHostToDevice));
    if (n > 0) {
        root_write<<<blocks_for(n, 256), 256>>>(n, flag_scan, flag, root->ent);
        PCK(cudaGetLastError());
    }
    return cudaDeviceSynchronize();
}

// Per-level partition offsets and slots of the appended canvas, from the kept subtrees (reuse[p] >= 0) and the
// repainted ones (rep[p] >= 0).
cudaError_t assemble(int64_t n_part, const int32_t* reuse, const int32_t* rep, const PaintCache& old,
                     const std::vector<uint64_t*>& slots_r, const std::vector<int64_t*>& offs_r,
                     std::vector<uint64_t*>* slots, std::vector<int64_t>* ncell, std::vector<int64_t*>* offs) {
    DevBuf buf;
    const size_t depth_max = std::max(old.slots.size(), slots_r.size());
    if (n_part == 0 || depth_max == 0) return cudaDeviceSynchronize();
    int64_t* d_total;
    PCK(buf.alloc(&d_total, (int64_t)depth_max));
    PartLevels levels = {};
    for (size_t d = 0; d < depth_max; ++d) {
        int64_t* off;
        PCK(dalloc(&off, n_part + 1));
        offs->push_back(off);
        levels.old[d] = d < old.off.size() ? old.off[d] : nullptr;
        levels.rep[d] = d < offs_r.size() ? offs_r[d] : nullptr;
        levels.dst[d] = off;
    }
    part_offsets<<<(unsigned)depth_max, kScanThreads>>>(n_part, reuse, rep, levels, d_total);
    PCK(cudaGetLastError());
    std::vector<int64_t> total(depth_max);
    PCK(cudaMemcpy(total.data(), d_total, sizeof(int64_t) * depth_max, cudaMemcpyDeviceToHost));
    for (size_t d = 0; d < depth_max && total[d] > 0; ++d) ncell->push_back(total[d]);
    for (size_t d = ncell->size(); d < depth_max; ++d) dfree((*offs)[d]);
    offs->resize(ncell->size());
    for (size_t d = 0; d < ncell->size(); ++d) {
        uint64_t* slot;
        PCK(dalloc(&slot, 8 * (*ncell)[d]));
        slots->push_back(slot);
        const bool last = d + 1 == ncell->size();
        assemble_level<<<blocks_for(8 * (*ncell)[d], 256), 256>>>(
            (*ncell)[d], n_part, (*offs)[d], last ? nullptr : (*offs)[d + 1], reuse, rep,
            d < old.slots.size() ? old.slots[d] : nullptr, d < old.off.size() ? old.off[d] : nullptr,
            d + 1 < old.off.size() ? old.off[d + 1] : nullptr, d < slots_r.size() ? slots_r[d] : nullptr,
            d < offs_r.size() ? offs_r[d] : nullptr, d + 1 < offs_r.size() ? offs_r[d + 1] : nullptr, slot);
        PCK(cudaGetLastError());
    }
    return cudaDeviceSynchronize();
}

}  // namespace

cudaError_t paint_pools(int32_t depth, double extent, const double* d_c, const double* d_r, const float4* d_rgba,
                        int64_t n, PaintCache** cache, int32_t** d_nodes_out, uint2** d_leaves_out, int64_t* n_rec_out,
                        int64_t* n_leaf_out, std::vector<int64_t>* level_begin, int64_t* wrap_out,
                        int32_t* n_wrap_out) {
    const double half = 0.5 * extent;
    PaintCache* old = *cache;
    *cache = nullptr;
    // an append: the same canvas, and the stamps the cache was painted with come first in the table
    const bool append = old && old->depth == depth && old->extent == extent && old->n_stamps <= n;
    if (!append) new_painting();
    DevBuf buf;
    // squared radii and target depths (the host painter's integer loop, in the same FP64 operations)
    double* d_r2;
    StampRec* d_rec;
    cudaError_t e = buf.alloc(&d_r2, n);
    if (e == cudaSuccess) e = buf.alloc(&d_rec, n);
    if (e == cudaSuccess && n > 0) {
        stamp_prep<<<blocks_for(n, 256), 256>>>(d_c, d_r, n, depth, extent, screen_scale(extent), d_r2, d_rec);
        e = cudaGetLastError();
    }
    const StampDev S{d_c, d_r2, d_rec, d_rgba};
    // levels 0 .. P - 1 from the root (always painted: every stamp reaches the root's list)
    std::vector<uint64_t*> slots_top, slots_bot, slots_r;
    std::vector<int64_t> ncell_top, ncell_bot, ncell_r;
    std::vector<int64_t*> offs_bot, offs_r;
    Level root, partP, rep_lvl, unused;
    PaintCache* nc = nullptr;
    if (e == cudaSuccess) e = root_level(S, n, extent, half, &root);
    if (e == cudaSuccess) e = paint_down(root, S, extent, half, depth, kPartLevel, false, &slots_top, &ncell_top, &partP, nullptr);
    else root.free();
    if (e == cudaSuccess) {
        nc = new PaintCache();
        nc->depth = depth;
        nc->extent = extent;
        nc->n_stamps = n;
        nc->nP = partP.n;
        e = dalloc(&nc->code, partP.n);
        if (e == cudaSuccess && partP.n > 0) {
            morton_codes<<<blocks_for(partP.n, 256), 256>>>(partP.n, partP.coord, kPartLevel, nc->code);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess && !append) {
        // a full paint: every partition painted, a copy of their lists kept
        Level start = partP;
        int64_t* keep_off = nullptr;
        int32_t* keep_ent = nullptr;
        e = dalloc(&keep_off, partP.n + 1);
        if (e == cudaSuccess) e = dalloc(&keep_ent, 1);
        if (e == cudaSuccess && partP.n > 0) {
            int64_t n_ent = 0;
            e = cudaMemcpy(&n_ent, partP.off + partP.n, sizeof(int64_t), cudaMemcpyDeviceToHost);
            dfree(keep_ent);
            keep_ent = nullptr;
            if (e == cudaSuccess) e = dalloc(&keep_ent, n_ent);
            if (e == cudaSuccess)
                e = cudaMemcpy(keep_ent, partP.ent, sizeof(int32_t) * (size_t)n_ent, cudaMemcpyDeviceToDevice);
            if (e == cudaSuccess)
                e = cudaMemcpy(keep_off, partP.off, sizeof(int64_t) * (size_t)(partP.n + 1), cudaMemcpyDeviceToDevice);
        }
        nc->lst_off = keep_off;
        nc->lst_ent = keep_ent;
        if (e == cudaSuccess)
            e = paint_down(start, S, extent, half, depth, -1, true, &slots_bot, &ncell_bot, &unused, &offs_bot);
        else
            start.free();
        partP = Level();
    } else if (e == cudaSuccess) {
        // an append: keep the partitions whose cell and stamp list are unchanged, paint the others again
        int32_t *reuse = nullptr, *rep = nullptr, *sel = nullptr;
        int64_t* len = nullptr;
        const int64_t np = partP.n;
        std::vector<int32_t> h_reuse((size_t)np), h_rep((size_t)np, -1), h_sel;
        e = buf.alloc(&reuse, np);
        if (e == cudaSuccess && np > 0) {
            match_partitions<<<blocks_for(32 * np, 256), 256>>>(np, partP.coord, partP.off, partP.ent, old->nP, old->code,
                                                                old->lst_off, old->lst_ent, kPartLevel, reuse);
            e = cudaGetLastError();
            if (e == cudaSuccess)
                e = cudaMemcpy(h_reuse.data(), reuse, sizeof(int32_t) * (size_t)np, cudaMemcpyDeviceToHost);
        }
        for (int64_t p = 0; p < np; ++p)
            if (h_reuse[(size_t)p] < 0) {
                h_rep[(size_t)p] = (int32_t)h_sel.size();
                h_sel.push_back((int32_t)p);
            }
        const int64_t m = (int64_t)h_sel.size();
        if (e == cudaSuccess) e = buf.alloc(&rep, np);
        if (e == cudaSuccess) e = buf.alloc(&sel, m);
        if (e == cudaSuccess) e = buf.alloc(&len, m + 1);
        if (e == cudaSuccess && np > 0) e = cudaMemcpy(rep, h_rep.data(), sizeof(int32_t) * (size_t)np, cudaMemcpyHostToDevice);
        if (e == cudaSuccess && m > 0) e = cudaMemcpy(sel, h_sel.data(), sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice);
        // the repainted partitions as one level
        rep_lvl.n = m;
        rep_lvl.level = kPartLevel;
        if (e == cudaSuccess && m > 0) {
            list_lengths<<<blocks_for(m, 256), 256>>>(m, sel, partP.off, len);
            int64_t n_ent = 0;
            e = scan_i64(len, m, &n_ent);
            rep_lvl.n_ent = n_ent;
            rep_lvl.longest = partP.longest;
            for (int x = 0; x < 2; ++x) {
                rep_lvl.long_cells[x] = partP.long_cells[x];
                rep_lvl.long_ent[x] = partP.long_ent[x];
            }
            if (e == cudaSuccess) e = cudaMemcpy(len + m, &n_ent, sizeof(int64_t), cudaMemcpyHostToDevice);
            if (e == cudaSuccess) e = dalloc(&rep_lvl.coord, 3 * m);
            if (e == cudaSuccess) e = dalloc(&rep_lvl.off, m + 1);
            if (e == cudaSuccess) e = dalloc(&rep_lvl.ent, n_ent);
            if (e == cudaSuccess) {
                gather_cells<<<blocks_for(32 * m, 256), 256>>>(m, sel, partP.coord, partP.off, partP.ent, len,
                                                               rep_lvl.coord, rep_lvl.off, rep_lvl.ent);
                e = cudaGetLastError();
            }
            if (e == cudaSuccess)
                e = cudaMemcpy(rep_lvl.off + m, &n_ent, sizeof(int64_t), cudaMemcpyHostToDevice);
        }
        if (e == cudaSuccess)
            e = paint_down(rep_lvl, S, extent, half, depth, -1, true, &slots_r, &ncell_r, &unused, &offs_r);
        else
            rep_lvl.free();
        if (e == cudaSuccess) e = assemble(np, reuse, rep, *old, slots_r, offs_r, &slots_bot, &ncell_bot, &offs_bot);
        free_all(slots_r);
        free_all(offs_r);
        // the new level-P lists are kept
        nc->lst_off = partP.off;
        nc->lst_ent = partP.ent;
        dfree(partP.coord);
        partP = Level();
    }
    paint_cache_free(old);
    if (e == cudaSuccess) {
        std::vector<uint64_t*> all(slots_top);
        all.insert(all.end(), slots_bot.begin(), slots_bot.end());
        std::vector<int64_t> cells(ncell_top);
        cells.insert(cells.end(), ncell_bot.begin(), ncell_bot.end());
        e = finish_pools(all, cells, d_nodes_out, d_leaves_out, n_rec_out, n_leaf_out, level_begin, wrap_out, n_wrap_out);
    }
    free_all(slots_top);
    partP.free();
    size_t spare = 0, total = 0;
    if (cudaMemGetInfo(&spare, &total) != cudaSuccess) spare = 0;
    const size_t live = std::max((size_t)pool_high_water(), g_live_before);
    pool_trim(std::min(with_gaps(live), spare / kPoolShare));
    if (e == cudaSuccess) {
        nc->slots = slots_bot;
        nc->ncell = ncell_bot;
        nc->off = offs_bot;
        *cache = nc;
    } else {
        free_all(slots_bot);
        free_all(offs_bot);
        paint_cache_free(nc);
    }
    return e;
}

}  // namespace canvox
