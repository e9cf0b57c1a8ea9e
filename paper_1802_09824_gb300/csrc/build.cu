// Tree build on the GPU: keys, sort, leaves, target groups, frames.
//
// Sec. 3.2 ("Tree building"): each particle is labelled with its ground cell
// index (i N_side + j) N_side + k, particles are ordered by that index and,
// inside a ground cell, by a Morton (or Peano-Hilbert, Sec. 4.1) key, so that
// every octree node is one contiguous run of particles.  Leaves are the
// largest cells holding at most leaf_max particles (the N_pp of Sec. 3.1, the
// leaf size of Sec. 4.4); a level of the hierarchy is level_bits key bits:
// 3 gives the octree cells, 1 splits every octree level into its three
// binary sub-levels (half, quarter cell), which are key prefixes too.
//
// Leaf rule, evaluated independently for every particle k: k starts a leaf
// iff k is the first particle of a ground cell, or the smallest cell that
// holds both k-1 and k (their common key prefix) has more than leaf_max
// particles -- then k-1 and k lie in different children of a cell that had
// to be split.  Particles with identical keys (a finest cell) that number
// more than leaf_max are cut into runs of leaf_max from the run's start.
//
// Positions are stored relative to a reference point of their leaf in FP32
// (the FP64 wrap and the reference points are the only FP64 data on the
// device), and a second copy relative to the reference point of their target
// group, derived from the first by one FP32 add of the FP64-computed offset,
// exactly as the PP kernel shifts source particles, so that a particle seen
// as target and as source has bitwise the same coordinates.
#include <algorithm>
#include <climits>
#include <cmath>

#include "checks.cuh"
#include "curve.cuh"
#include "handles.cuh"

namespace phpp {
namespace {

__device__ __forceinline__ int find_box(const int32_t *box_first, int nb, int64_t i)
{
    int lo = 0, hi = nb - 1;          // largest b with box_first[b] <= i
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (box_first[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ double wrap_coord(double x, double L)
{
    // x - L floor(x / L), each operation rounded once (no contraction); a
    // coordinate already in [0, L) is returned as is, which is what the
    // formula gives for it (floor = 0), without the FP64 divide
    if (x >= 0.0 && x < L) return x;
    double f = floor(__ddiv_rn(x, L));
    return __dsub_rn(x, __dmul_rn(L, f));
}

__device__ __forceinline__ uint32_t quant_coord(double xw, double S, int T)
{
    // floor(xw S) of a wrapped (finite, non-negative) coordinate, clamped
    const int q = __double2int_rd(__dmul_rn(xw, S));
    const int top = (1 << T) - 1;
    return (uint32_t)(q < 0 ? 0 : (q > top ? top : q));
}

// The widening of an FP32 number with integer operations (the FP64 pipe, which
// conversions share, has two lanes an SM here; a subnormal still goes there).
__device__ __forceinline__ double widen(float x)
{
    const uint32_t b = __float_as_uint(x), e = (b >> 23) & 0xffu;
    if (e == 0 && (b & 0x7fffffu)) return (double)x;
    const uint32_t hi = (b & 0x80000000u) | (e ? ((e + 896u) << 20) | ((b & 0x7fffffu) >> 3) : 0u);
    return __hiloint2double((int)hi, (int)(b << 29));
}

// The reverse where it is exact: true if x is a normal FP32 number or zero.
__device__ __forceinline__ bool narrow(double x, float &f)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x), e = (hi >> 20) & 0x7ffu;
    const bool zero = !((hi & 0x7fffffffu) | lo);
    f = __uint_as_float((hi & 0x80000000u) | (zero ? 0u : ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29)));
    return zero || (!(lo & 0x1fffffffu) && e >= 897u && e <= 1150u);
}

// Wrapped coordinate of an FP32 input: the in-box test runs in FP32 (x < L
// exactly when x < L_up), so only the multiply of the key and the widening
// to FP64 remain on the FP64 pipe for particles already in the box.
__device__ __forceinline__ double wrap_f32(float x, const BoxDev &bx)
{
    if (x >= 0.f && x < bx.L_up) return widen(x);
    return wrap_coord((double)x, bx.L);
}

// quant_coord of an FP32 coordinate in [0, L) without FP64: x S as a
// double-float product (the product's rounding error taken exactly by an FMA),
// off by at most 2^-25 (S_lo's rounding and one FP32 rounding of the low
// part, x S < 2^21).  The floor is taken from it when its fraction lies at
// least 1e-6 off an integer, 40 times that, else the FP64 product decides
// (false).
__device__ __forceinline__ bool quant_f32(float x, const BoxDev &bx, int T, uint32_t &q)
{
    const float p = x * bx.S_hi;
    const float lo = fmaf(x, bx.S_lo, fmaf(x, bx.S_hi, -p));
    float fl = floorf(p), fr = (p - fl) + lo;
    if (fr < 0.f) {
        fr += 1.f;
        fl -= 1.f;
    } else if (fr >= 1.f) {
        fr -= 1.f;
        fl += 1.f;
    }
    const int i = (int)fl, top = (1 << T) - 1;
    q = (uint32_t)(i < 0 ? 0 : (i > top ? top : i));
    return fr >= 1e-6f && fr <= 1.f - 1e-6f;
}

// Particle i's coordinates wrapped into [0, L) in FP64 (non-finite input
// counts as 0 and is reported once per particle through `bad`).
template <int kPosType>
__device__ __forceinline__ void wrapped_pos(const void *pos, int64_t i, const BoxDev &bx, double &x, double &y,
                                            double &z, bool &bad)
{
    if (kPosType == PH_F64) {
        const double *p = static_cast<const double *>(pos) + 3 * i;
        x = p[0]; y = p[1]; z = p[2];
        bad = !(isfinite(x) && isfinite(y) && isfinite(z));
        if (bad) x = y = z = 0.0;
        x = wrap_coord(x, bx.L);
        y = wrap_coord(y, bx.L);
        z = wrap_coord(z, bx.L);
    } else {
        const float *p = static_cast<const float *>(pos) + 3 * i;
        float fx = p[0], fy = p[1], fz = p[2];
        bad = !(isfinite(fx) && isfinite(fy) && isfinite(fz));
        if (bad) fx = fy = fz = 0.f;
        x = wrap_f32(fx, bx);
        y = wrap_f32(fy, bx);
        z = wrap_f32(fz, bx);
    }
}

template <int kPosType>
__global__ void k_keys(const void *pos, int64_t n, const int32_t *box_first, int nb, const BoxDev *boxes, int T,
                       int key_kind, uint64_t *keys, int32_t *vals, SortCounts sc, uint32_t *status)
{
    chain_begin();
    // (the loop's bound is the block's, so that its warps stay whole)
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x; i0 < n; i0 += (int64_t)gridDim.x * blockDim.x) {
        const bool in = i0 + threadIdx.x < n;
        const int64_t i = in ? i0 + threadIdx.x : n - 1;
        const int bi = nb > 1 ? find_box(box_first, nb, i) : 0;
        const BoxDev &bx = boxes[bi];
        uint32_t qx = 0, qy = 0, qz = 0;
        bool done = false;
        if (kPosType == PH_F32) {
            const float *p = static_cast<const float *>(pos) + 3 * i;
            const float x = p[0], y = p[1], z = p[2];
            done = x >= 0.f && x < bx.L_up && y >= 0.f && y < bx.L_up && z >= 0.f && z < bx.L_up;   // (NaN: no)
            done = done && quant_f32(x, bx, T, qx) && quant_f32(y, bx, T, qy) && quant_f32(z, bx, T, qz);
        }
        if (!done) {
            double x, y, z;
            bool bad;
            wrapped_pos<kPosType>(pos, i, bx, x, y, z, bad);
            if (bad) atomicOr(status, ST_NONFINITE);
            qx = quant_coord(x, bx.S, T);
            qy = quant_coord(y, bx.S, T);
            qz = quant_coord(z, bx.S, T);
        }
        const int b = bx.b;
        const uint32_t lm = (1u << b) - 1u;
        uint64_t ground = ((uint64_t)(qx >> b) * bx.nside + (qy >> b)) * bx.nside + (qz >> b);
        uint64_t local = key_kind == PH_KEY_HILBERT ? hilbert3(qx & lm, qy & lm, qz & lm, b)
                                                    : interleave3(qx & lm, qy & lm, qz & lm);
        uint64_t boxbits = 3 * T < 64 ? ((uint64_t)bi << (3 * T)) : 0ull;
        const uint64_t key = boxbits | (ground << (3 * b)) | local;
        if (in) {
            keys[i] = key;
            vals[i] = (int32_t)i;
        }
        count_digit(sc.hist, (int)(key & ((1u << kSortBits) - 1u)) * sc.row + (int)(i >> sc.tile_shift), in);
    }
}

__device__ __forceinline__ int box_of_cell(const BoxDev *boxes, int nb, int c)
{
    int lo = 0, hi = nb - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (boxes[mid].cell_base <= c) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int64_t lower_bound_u64(const uint64_t *a, int64_t lo, int64_t hi, uint64_t v)
{
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// First particle of every ground cell (a search in the sorted keys).
__device__ __forceinline__ void cell_starts(const uint64_t *keys, int64_t n, const BoxDev *boxes, int nb, int n_cells,
                                            int T, int c, int32_t *cell_first)
{
    if (c >= n_cells) {
        if (c == n_cells) cell_first[c] = (int32_t)n;
        return;
    }
    const int bi = box_of_cell(boxes, nb, c);
    const BoxDev &bx = boxes[bi];
    const uint64_t boxbits = 3 * T < 64 ? ((uint64_t)bi << (3 * T)) : 0ull;
    const uint64_t pre = boxbits | ((uint64_t)(c - bx.cell_base) << (3 * bx.b));
    cell_first[c] = (int32_t)lower_bound_u64(keys, bx.first, (int64_t)bx.first + bx.n, pre);
}

// The particles in sorted order, wrapped, and (the last blocks, one thread a
// cell) the first particle of every ground cell: both read only the sorted
// keys and rows, so they share a launch.
template <int kPosType>
__global__ void k_gather(const void *pos, const float *mass, int64_t n, const uint64_t *keys, const int32_t *perm,
                         const BoxDev *boxes, int T, double *xw, float *mass_sorted, uint32_t *status, int cell_blocks,
                         int nb, int n_cells, int32_t *cell_first)
{
    chain_begin();
    const int blocks = (int)gridDim.x - cell_blocks;
    if ((int)blockIdx.x >= blocks) {
        cell_starts(keys, n, boxes, nb, n_cells, T, ((int)blockIdx.x - blocks) * (int)blockDim.x + (int)threadIdx.x,
                    cell_first);
        return;
    }
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)blocks * blockDim.x) {
        int64_t i = perm[k];
        if (!in_bounds(i, n, BS_BUILD_ROW)) i = 0;
        const int bi = 3 * T < 64 ? (int)(keys[k] >> (3 * T)) : 0;
        const BoxDev &bx = boxes[bi];
        double x, y, z;
        bool bad;
        wrapped_pos<kPosType>(pos, i, bx, x, y, z, bad);
        xw[3 * k + 0] = x;
        xw[3 * k + 1] = y;
        xw[3 * k + 2] = z;
        float m = mass ? mass[i] : bx.mass_default;
        if (!isfinite(m)) {
            atomicOr(status, ST_NONFINITE);
            m = 0.f;
        }
        mass_sorted[k] = m;
    }
}

// The leaves and groups are numbered in two passes over the particles, one
// contiguous chunk a block: k_flags marks the starts (see the leaf rule in the
// file comment) and counts them per chunk, k_starts adds up the counts of the
// chunks before its own and numbers them.  Two launches where flags, two
// three-kernel scans and a kernel for the first particles took eight (with the
// merged launches below and k_offsets, per step: 1000 particles 187 -> 132 us,
// 4096 102 -> 77 us, 50,021 472 -> 413 us, 128^3 lattice 4121 -> 4079 us).
constexpr int kMaxChunks = 2048;

struct Chunks {
    int blocks;
    int64_t size;            // particles a block, a multiple of kThreads
};

inline Chunks chunks_of(int64_t n)
{
    const int64_t tiles = (n + kThreads - 1) / kThreads;
    const int64_t per = (tiles + kMaxChunks - 1) / kMaxChunks;
    return Chunks{(int)((tiles + per - 1) / per), per * kThreads};
}

// Sums of two values over the block (every thread gets them).
__device__ __forceinline__ int2 block_sum2(int a, int b)
{
    __shared__ int2 s_w[kThreads / 32];
    a = __reduce_add_sync(0xffffffffu, a);
    b = __reduce_add_sync(0xffffffffu, b);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = make_int2(a, b);
    __syncthreads();
    int2 t = make_int2(0, 0);
#pragma unroll
    for (int w = 0; w < kThreads / 32; w++) {
        t.x += s_w[w].x;
        t.y += s_w[w].y;
    }
    __syncthreads();
    return t;
}

__global__ void __launch_bounds__(kThreads) k_flags(const uint64_t *keys, int64_t n, int64_t chunk, const BoxDev *boxes,
                                                    int T, int leaf_max, int level_bits, const int32_t *cell_first,
                                                    uint8_t *starts, int2 *chunk_count)
{
    chain_begin();
    const int64_t lo = blockIdx.x * chunk, end = lo + chunk < n ? lo + chunk : n;
    int nl = 0, ngr = 0;
    for (int64_t k = lo + threadIdx.x; k < end; k += kThreads) {
        const uint64_t Bk = keys[k];
        const int bi = 3 * T < 64 ? (int)(Bk >> (3 * T)) : 0;
        const BoxDev &bx = boxes[bi];
        const int b = bx.b;
        const uint64_t cellpre = Bk >> (3 * b);
        const int cell = bx.cell_base + (int)(cellpre & ((1ull << (3 * bx.g)) - 1ull));
        // target groups: runs of group_size inside each ground cell
        const int64_t cf = cell_first[cell];
        const int gf = (int)(k - cf) % bx.group_size == 0 ? 1 : 0;
        int lf;
        if (k == 0) {
            lf = 1;
        } else {
            const uint64_t A = keys[k - 1];
            if ((A >> (3 * b)) != cellpre || (3 * T < 64 && (A >> (3 * T)) != (Bk >> (3 * T)))) {
                lf = 1;   // new box or new ground cell
            } else {
                const uint64_t x = A ^ Bk;
                if (x == 0) {
                    // identical keys: a finest cell; cut into runs of leaf_max
                    // from its first particle if it is too full
                    int64_t lo = k - 1, step = 1;
                    while (lo - step >= 0 && keys[lo - step] == Bk) { lo -= step; step <<= 1; }
                    int64_t a = lo - step < 0 ? 0 : lo - step;  // keys[a] may or may not equal Bk
                    lo = lower_bound_u64(keys, a, lo + 1, Bk);
                    int64_t hi = k, st2 = 1;
                    while (hi + st2 < n && keys[hi + st2] == Bk) { hi += st2; st2 <<= 1; }
                    int64_t e = hi + st2 < n ? hi + st2 : n;
                    hi = lower_bound_u64(keys, hi, e, Bk + 1);   // first index > Bk
                    lf = (hi - lo > leaf_max && ((k - lo) % leaf_max) == 0) ? 1 : 0;
                } else {
                    const int hb = 63 - __clzll((long long)x);
                    const int sh = level_bits * (hb / level_bits + 1);   // prefix shift of the common cell
                    const uint64_t P = Bk >> sh;
                    // is the common cell (holding k-1 and k) larger than leaf_max?
                    bool big;
                    const int64_t far = k - 1 - leaf_max;
                    if (far >= 0 && (keys[far] >> sh) == P) {
                        big = true;
                    } else {
                        int64_t lo = far < 0 ? 0 : far + 1, hi = k - 1;   // first index with prefix P
                        while (lo < hi) {
                            int64_t mid = (lo + hi) >> 1;
                            if ((keys[mid] >> sh) < P) lo = mid + 1; else hi = mid;
                        }
                        const int64_t q = lo + leaf_max;
                        big = q < n && (keys[q] >> sh) == P;
                    }
                    lf = big ? 1 : 0;
                }
            }
        }
        starts[k] = (uint8_t)(lf | (gf << 1));
        nl += lf;
        ngr += gf;
    }
    const int2 t = block_sum2(nl, ngr);
    if (threadIdx.x == 0) chunk_count[blockIdx.x] = t;
}

// The leaf and the group of every particle, the first particle of every leaf
// and group, and their numbers.
__global__ void __launch_bounds__(kThreads) k_starts(const uint8_t *starts, int64_t n, int64_t chunk,
                                                     const int2 *chunk_count, int32_t *leaf_of, int32_t *group_of,
                                                     int32_t *lfirst, int32_t *gfirst, int32_t *counts)
{
    chain_begin();
    __shared__ int2 s_w[2][kThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned le = 0xffffffffu >> (31 - lane);
    int2 run = make_int2(0, 0);
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += kThreads) {
        const int2 c = chunk_count[b];
        run.x += c.x;
        run.y += c.y;
    }
    run = block_sum2(run.x, run.y);   // starts before this chunk
    const int64_t lo = blockIdx.x * chunk, end = lo + chunk < n ? lo + chunk : n;
    for (int64_t base = lo; base < end; base += kThreads) {
        const int64_t k = base + threadIdx.x;
        const int f = k < end ? starts[k] : 0;
        const unsigned lb = __ballot_sync(0xffffffffu, f & 1), gb = __ballot_sync(0xffffffffu, f & 2);
        int2 *sw = s_w[((base - lo) / kThreads) & 1];   // alternating, so one barrier a tile
        if (lane == 0) sw[w] = make_int2(__popc(lb), __popc(gb));
        __syncthreads();
        int2 at = run;
#pragma unroll
        for (int ww = 0; ww < kThreads / 32; ww++) {
            const int2 c = sw[ww];
            if (ww < w) {
                at.x += c.x;
                at.y += c.y;
            }
            run.x += c.x;
            run.y += c.y;
        }
        if (k < end) {
            const int l = at.x + __popc(lb & le) - 1, g = at.y + __popc(gb & le) - 1;
            leaf_of[k] = l;
            group_of[k] = g;
            if ((f & 1) && in_bounds(l, n, BS_BUILD_ROW)) lfirst[l] = (int32_t)k;
            if ((f & 2) && in_bounds(g, n, BS_BUILD_ROW)) gfirst[g] = (int32_t)k;
        }
    }
    if (end == n && threadIdx.x == 0) {
        lfirst[run.x] = (int32_t)n;
        gfirst[run.y] = (int32_t)n;
        counts[0] = run.x;
        counts[1] = run.y;
    }
}

// Orders doubles like their values when compared as signed 64-bit integers.
__device__ __forceinline__ long long dkey(double x)
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

__device__ __forceinline__ double dkey_inv(long long k)
{
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
}

// Smallest and largest of the lanes' values, 64-bit integers, by two 32-bit
// warp reductions each: the high words, then the low words of those that hold
// the extreme one.
__device__ __forceinline__ long long warp_min(long long v)
{
    const int h = (int)(v >> 32), mh = __reduce_min_sync(0xffffffffu, h);
    const unsigned ml = __reduce_min_sync(0xffffffffu, h == mh ? (unsigned)v : 0xffffffffu);
    return ((long long)mh << 32) | ml;
}

__device__ __forceinline__ long long warp_max(long long v)
{
    const int h = (int)(v >> 32), mh = __reduce_max_sync(0xffffffffu, h);
    const unsigned ml = __reduce_max_sync(0xffffffffu, h == mh ? (unsigned)v : 0u);
    return ((long long)mh << 32) | ml;
}

struct BoxTable {
    const int32_t *first, *count;
    double *ref;
    float4 *r4, *c4, *h4;
    int32_t *cell_of, *box_of;   // groups only
};

struct FrameArgs {               // leaves only: the particles in their frames
    const float *mass_sorted;
    const int32_t *leaf_of, *group_of;
    const float4 *group_r4;
    float4 *pos_leaf, *pos_group;
    int64_t n;
};

// Bounding box of each leaf (or group): FP64 reference point near the box
// centre, FP32 half extents around it rounded up, FP32 reference point
// relative to the ground cell's lower corner; and for the leaves the
// particles' positions in their leaf's and group's frames.
//
// The reference point is the centre rounded to a multiple of U = 2^(e-24),
// the FP32 spacing of the box's largest |coordinate| (2^(e-1) <= m < 2^e),
// so that an FP32 coordinate minus it is exact; rounding to a multiple of U
// is done as (c + 1.5 2^52 U) - 1.5 2^52 U (round half to even).  Being a
// multiple of U below 2^e in magnitude, it is itself an FP32 number: r4
// holds that exact FP32 copy.
//
// A block takes kBoxes consecutive boxes: a warp reduces the extents of four
// of them (coordinates as integers ordered like the doubles, dkey), then one
// thread an axis does the FP64 arithmetic of all (a warp per box would spend
// the narrow FP64 pipe on idle lanes), then the leaves' particles, one
// contiguous run, are written in their frames.  An FP32 coordinate takes an
// FP32 subtraction there: the difference of two FP32 numbers rounded once,
// as the FP64 one rounded to FP32 is.  (Extents by segmented warp reductions
// and global atomics, the boxes and the frames as three launches took 88 us
// for 2 M particles, now 62 us; the 128^3 lattice step 4046 -> 4014 us.)
constexpr int kBoxes = 32;

template <bool kLeaves>
__device__ __forceinline__ void box_block(const BoxTable &t, const FrameArgs &fr, const uint64_t *keys,
                                          const BoxDev *boxes, int T, const double *xw, int block, int blocks)
{
    __shared__ int s_first[kBoxes + 1];
    __shared__ long long s_ext[kBoxes][6];
    __shared__ float s_ref[kBoxes][3], s_c[kBoxes][3], s_h[kBoxes][3];
    __shared__ double s_refd[kLeaves ? kBoxes : 1][3];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int count = *t.count;
    for (int l0 = block * kBoxes; l0 < count; l0 += blocks * kBoxes) {
        const int nb = count - l0 < kBoxes ? count - l0 : kBoxes;
        if (threadIdx.x <= nb) s_first[threadIdx.x] = t.first[l0 + threadIdx.x];
        __syncthreads();
        constexpr int kPer = kBoxes / (kThreads / 32);
        // the first 32 particles of the warp's boxes in flight together
        double x[kPer][3];
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            const int b = w * kPer + q;
            const int k = b < nb ? s_first[b] + lane : 0;
            const bool in = b < nb && k < s_first[b + 1];
#pragma unroll
            for (int d = 0; d < 3; d++) x[q][d] = in ? xw[3 * (int64_t)k + d] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            const int b = w * kPer + q;
            if (b >= nb) break;
            const int f1 = s_first[b + 1];
            int k = s_first[b] + lane;
            long long lo[3], hi[3];
#pragma unroll
            for (int d = 0; d < 3; d++) {
                lo[d] = k < f1 ? dkey(x[q][d]) : LLONG_MAX;
                hi[d] = k < f1 ? lo[d] : LLONG_MIN;
            }
            for (k += 32; k < f1; k += 32)
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    const long long v = dkey(xw[3 * (int64_t)k + d]);
                    lo[d] = v < lo[d] ? v : lo[d];
                    hi[d] = v > hi[d] ? v : hi[d];
                }
            __syncwarp();
#pragma unroll
            for (int d = 0; d < 3; d++) {
                lo[d] = warp_min(lo[d]);
                hi[d] = warp_max(hi[d]);
            }
            if (lane == 0) {
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    s_ext[b][d] = lo[d];
                    s_ext[b][3 + d] = hi[d];
                }
            }
        }
        __syncthreads();
        if (threadIdx.x < 3 * nb) {
            const int b = threadIdx.x / 3, d = threadIdx.x % 3;
            const uint64_t key = keys[s_first[b]];
            const int bi = 3 * T < 64 ? (int)(key >> (3 * T)) : 0;
            const BoxDev &bx = boxes[bi];
            const uint32_t ground = (uint32_t)((key >> (3 * bx.b)) & ((1ull << (3 * bx.g)) - 1ull));
            const uint32_t gc = d == 2 ? ground % bx.nside
                                       : d == 1 ? (ground / bx.nside) % bx.nside : ground / (bx.nside * bx.nside);
            const double vlo = dkey_inv(s_ext[b][d]), vhi = dkey_inv(s_ext[b][3 + d]);
            const double m = fmax(fabs(vlo), fabs(vhi));
            const int ex = (int)((__double_as_longlong(m) >> 52) & 0x7ff) - 1022;   // m = f 2^ex, f in [0.5, 1)
            const double C = __longlong_as_double(((long long)(ex + 28 + 1023) << 52) | (1ll << 51));
            const double cen = __dmul_rn(0.5, __dadd_rn(vlo, vhi));
            const double r = __dsub_rn(__dadd_rn(cen, C), C);
            const double half = fmax(__dsub_rn(vhi, r), __dsub_rn(r, vlo));
            t.ref[3 * (int64_t)(l0 + b) + d] = r;
            if (kLeaves) s_refd[kLeaves ? b : 0][d] = r;
            s_ref[b][d] = __double2float_rn(r);   // exact
            s_c[b][d] = __double2float_rn(__dsub_rn(r, __dmul_rn((double)gc, bx.h)));
            s_h[b][d] = __double2float_ru(half);
            if (!kLeaves && d == 0) {
                t.cell_of[l0 + b] = bx.cell_base + (int)ground;
                t.box_of[l0 + b] = bi;
            }
        }
        __syncthreads();
        if (threadIdx.x < nb) {
            const int b = threadIdx.x, l = l0 + b, f0 = s_first[b];
            t.r4[l] = make_float4(s_ref[b][0], s_ref[b][1], s_ref[b][2], 0.f);
            t.c4[l] = make_float4(s_c[b][0], s_c[b][1], s_c[b][2], __int_as_float(f0));   // w: first particle
            t.h4[l] = make_float4(s_h[b][0], s_h[b][1], s_h[b][2], __int_as_float(s_first[b + 1] - f0));   // w: particles
        }
        if (kLeaves) {
            for (int k = s_first[0] + threadIdx.x; k < s_first[nb]; k += kThreads) {
                int b = fr.leaf_of[k] - l0;
                int64_t g = fr.group_of[k];
                if (!in_bounds(b, nb, BS_BUILD_ROW)) b = 0;
                if (!in_bounds(g, fr.n, BS_BUILD_ROW)) g = 0;
                const float4 gr4 = fr.group_r4[g];
                const float grf[3] = {gr4.x, gr4.y, gr4.z};
                float p[3], q[3];
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    const double v = xw[3 * (int64_t)k + d];
                    float vf;
                    p[d] = narrow(v, vf) ? __fsub_rn(vf, s_ref[b][d])
                                         : __double2float_rn(__dsub_rn(v, s_refd[kLeaves ? b : 0][d]));
                    // the same FP32 offset (the rounded difference of the two exact FP32
                    // reference points) and FP32 add as the PP kernel's source shift
                    q[d] = __fadd_rn(p[d], __fsub_rn(s_ref[b][d], grf[d]));
                }
                const float m = fr.mass_sorted[k];
                fr.pos_leaf[k] = make_float4(p[0], p[1], p[2], m);
                fr.pos_group[k] = make_float4(q[0], q[1], q[2], m);
            }
        }
        __syncthreads();   // the tables are rewritten for the next boxes
    }
}

// The boxes of the groups (the first `blocks` blocks) and the first leaf of
// every ground cell (the rest, one thread a cell): independent of each other,
// one launch.  A cell's first particle starts a leaf; an empty cell takes the
// next cell's.
__global__ void __launch_bounds__(kThreads) k_groups(BoxTable groups, int blocks, const uint64_t *keys,
                                                     const BoxDev *boxes, int T, const double *xw, int64_t n,
                                                     const int32_t *cell_first, const int32_t *leaf_of,
                                                     const int32_t *n_leaves, int n_cells, int32_t *cell_leaf_first)
{
    chain_begin();
    if ((int)blockIdx.x < blocks) {
        box_block<false>(groups, FrameArgs{}, keys, boxes, T, xw, blockIdx.x, blocks);
    } else {
        const int c = ((int)blockIdx.x - blocks) * (int)blockDim.x + (int)threadIdx.x;
        if (c <= n_cells) cell_leaf_first[c] = cell_first[c] < n ? leaf_of[cell_first[c]] : *n_leaves;
    }
}

// The boxes of the leaves and the particles in their frames (after k_groups).
__global__ void __launch_bounds__(kThreads) k_leaves(BoxTable leaves, FrameArgs fr, const uint64_t *keys,
                                                     const BoxDev *boxes, int T, const double *xw)
{
    chain_begin();
    box_block<true>(leaves, fr, keys, boxes, T, xw, blockIdx.x, gridDim.x);
}

// Tree part (theta > 0): one particle per leaf carrying the leaf's mass at
// its mass centre, sum(m x) / sum(m) over the leaf's wrapped positions in
// FP64 (summed in particle order), stored after the N particles of pos_leaf
// relative to the leaf's reference point like the leaf's own particles.  A
// massless leaf keeps its reference point.
__global__ void k_leaf_mass(const int32_t *first, const int32_t *n_leaves, const double *xw, const float *mass,
                            const double *ref, int64_t n, float4 *pos_leaf)
{
    chain_begin();
    const int count = *n_leaves;
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < count; l += gridDim.x * blockDim.x) {
        const int a = first[l], e = first[l + 1];
        double M = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
        for (int k = a; k < e; k++) {
            const double m = mass[k];
            M = __dadd_rn(M, m);
            sx = __dadd_rn(sx, __dmul_rn(m, xw[3 * (int64_t)k]));
            sy = __dadd_rn(sy, __dmul_rn(m, xw[3 * (int64_t)k + 1]));
            sz = __dadd_rn(sz, __dmul_rn(m, xw[3 * (int64_t)k + 2]));
        }
        const double *r = ref + 3 * (int64_t)l;
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        if (M > 0.0) {
            q.x = __double2float_rn(__dsub_rn(__ddiv_rn(sx, M), r[0]));
            q.y = __double2float_rn(__dsub_rn(__ddiv_rn(sy, M), r[1]));
            q.z = __double2float_rn(__dsub_rn(__ddiv_rn(sz, M), r[2]));
            q.w = __double2float_rn(M);
        }
        pos_leaf[n + l] = q;
    }
}

inline int grid_for(int64_t n, int threads = kThreads, int cap = 152 * 16)
{
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    return (int)(b < cap ? b : cap);
}

// Active-particle mode: flag the groups that hold at least one particle
// flagged active (flags in caller order, perm maps sorted -> caller row).
__global__ void k_group_active(const int32_t *gfirst, const int32_t *n_groups, const int32_t *perm,
                               const uint8_t *active, int32_t *gflag)
{
    const int ng = *n_groups;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += gridDim.x * blockDim.x) {
        int f = 0;
        for (int j = gfirst[g]; j < gfirst[g + 1] && !f; j++) f = active[perm[j]] ? 1 : 0;
        gflag[g] = f;
    }
}

// The flagged groups in order, and their number into *n_active.
__global__ void k_active_list(const int32_t *gflag, const int32_t *gscan, const int32_t *n_groups, int32_t *list,
                              int32_t *n_active)
{
    const int ng = *n_groups;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += gridDim.x * blockDim.x)
        if (gflag[g]) list[gscan[g]] = g;
    if (blockIdx.x == 0 && threadIdx.x == 0) *n_active = gscan[ng];
}

}  // namespace

// h(u) = exp(u^2) erfc(u) + 2u/sqrt(pi), so that Eq. (split) is f = exp(-u^2) h(u)
// with u = s / 2R_s.  Chebyshev interpolation of h on [0, U] at deg+1 nodes,
// returned as monomial coefficients in t = 2u/U - 1.
void fit_factor_poly(double U, int deg, float *coef)
{
    const int n = deg + 1;
    double f[kMaxPoly + 1], c[kMaxPoly + 1];
    for (int k = 0; k < n; k++) {
        double t = std::cos(M_PI * (k + 0.5) / n);
        double u = 0.5 * (t + 1.0) * U;
        f[k] = std::exp(u * u) * std::erfc(u) + 2.0 * u / std::sqrt(M_PI);
    }
    for (int j = 0; j < n; j++) {
        double s = 0.0;
        for (int k = 0; k < n; k++) s += f[k] * std::cos(j * M_PI * (k + 0.5) / n);
        c[j] = 2.0 * s / n;
    }
    c[0] *= 0.5;
    // monomial coefficients: sum_j c_j T_j(t), T_{j+1} = 2t T_j - T_{j-1}
    double m[kMaxPoly + 1] = {0}, Tm1[kMaxPoly + 2] = {0}, T0[kMaxPoly + 2] = {0}, T1[kMaxPoly + 2] = {0};
    T0[0] = 1.0;                    // T_0
    for (int j = 0; j < n; j++) {
        const double *Tj = j == 0 ? T0 : T1;
        for (int k = 0; k <= j; k++) m[k] += c[j] * Tj[k];
        if (j == 0) {
            T1[1] = 1.0;            // T_1 = t
            for (int k = 0; k <= kMaxPoly; k++) Tm1[k] = T0[k];
        } else {
            double Tn[kMaxPoly + 2] = {0};
            for (int k = 0; k <= j; k++) Tn[k + 1] += 2.0 * T1[k];
            for (int k = 0; k <= j; k++) Tn[k] -= Tm1[k];
            for (int k = 0; k <= kMaxPoly; k++) { Tm1[k] = T1[k]; T1[k] = Tn[k]; }
        }
    }
    for (int k = 0; k <= kMaxPoly; k++) coef[k] = k < n ? (float)m[k] : 0.f;
}

// (1 - f)/u^3 as a function of v = u^2, u = r / 2R_s: entire, since
// 1 - f = erf(u) - (2u/sqrt(pi)) exp(-u^2) = (4/sqrt(pi)) sum (-1)^n u^(2n+3) / (n! (2n+3)).
static double one_minus_f_over_u3(double v)
{
    if (v < 1.0) {
        double term = 1.0, s = 0.0;
        for (int n = 0; n < 24; n++) {
            s += term / (2 * n + 3);
            term *= -v / (n + 1);
        }
        return 4.0 / std::sqrt(M_PI) * s;
    }
    const double u = std::sqrt(v);
    return (std::erf(u) - 2.0 * u / std::sqrt(M_PI) * std::exp(-v)) / (u * v);
}

// The exact kernel's inverse-distance form of the softened short-range weight
// W = f(r) (r^2 + eps^2)^(-3/2).  In units of 2R_s, with v = r^2, e = eps^2,
// x = v + e: W = x^(-3/2) - (1 - e/x)^(3/2) E(v), E(v) = (1 - f)/v^(3/2)
// entire.  (1 - e/x)^(3/2) = 1 - 1.5 e/x + kappa (e/x)^2 up to its third
// order, so the second term is b1/x + b2/x^2 (the singular parts of E times
// that expansion) plus a function smooth in x, interpolated by a degree-9
// polynomial P in x at the zeros of the weighted minimax error curve for
// U = 2.25 (weight x^(3/2): the error in units of the Newtonian term), scaled
// to [0, U^2].  kappa = 0.46 instead of the Taylor 0.375 evens the rest out
// over r ~ eps.  Error in units of the Newtonian term: 8e-8 at U = 2.25, 1.2e-7
// at U = 2.3, and 1.1e-7 at r < eps for eps = 2R_s / 64.  The general form's
// 3.5e-7 (its degree-10 polynomial and ex2) is relative to the weight, which is
// f = 0.0175 of the Newtonian term at the cutoff for U = 2.25; in FP32 no fit
// changes that, since the terms subtracted here are rounded (dense_group).
// The kernel evaluates (1 - k) W = Y (y (x Y - k) + b1' + b2' Y) + P', with
// y = rsqrt(x), Y = y^2 and k = 5/3: (x Y - k) / (1 - k) = 1 + 1.5 (1 - x Y)
// corrects the three-fold error of an SFU rsqrt in y^3 to second order.  k is
// the FP32 number nearest 5/3 and 1 - k is taken of that number, so its
// rounding leaves no bias in the Newtonian term (6e-8 with an exact -2/3).
void fit_inverse_form(BoxDev &bx, double G, double rcut, double rs)
{
    constexpr int n = kInvDeg + 1;
    static const double node[n] = {0.05768249, 0.14244654, 0.25282438, 0.38132087, 0.51875132,
                                   0.65494475, 0.77953489, 0.88282818, 0.95665679, 0.99511833};
    const double kappa = 0.46;
    const double s2 = bx.s2, unit = 4.0 * rs * rs * s2;   // scaled x = unit * (x in units of 2R_s)
    const double e = (double)bx.eps2s / unit;
    const double V = rcut * rcut / (4.0 * rs * rs);
    const double E0 = 4.0 / (3.0 * std::sqrt(M_PI)), E1 = -0.6 * E0, E2 = 3.0 / 14.0 * E0;
    const double a0 = E0 - E1 * e + E2 * e * e, a1 = E1 - 2.0 * E2 * e;   // E(x - e) = a0 + a1 x + ...
    const double b1 = -1.5 * e * a0 + kappa * e * e * a1, b2 = kappa * e * e * a0;
    // Newton's divided differences in t = (x - zc) / (V / 2), zc = e + V / 2,
    // expanded to monomials
    double t[n], d[n], m[n] = {0};
    for (int k = 0; k < n; k++) {
        const double v = node[k] * V, x = v + e;
        t[k] = 2.0 * node[k] - 1.0;
        d[k] = std::pow(1.0 - e / x, 1.5) * one_minus_f_over_u3(v) - b1 / x - b2 / (x * x);
    }
    for (int j = 1; j < n; j++)
        for (int k = n - 1; k >= j; k--) d[k] = (d[k] - d[k - 1]) / (t[k] - t[k - j]);
    for (int k = n - 1; k >= 0; k--) {
        for (int j = n - 1; j > 0; j--) m[j] = m[j - 1] - t[k] * m[j];
        m[0] = d[k] - t[k] * m[0];
    }
    const double su = std::sqrt(unit);
    const double mk = (double)kInvK - 1.0;
    double scale = mk / (unit * su);
    for (int k = 0; k < n; k++) {
        bx.inv_poly[k] = (float)(m[k] * scale);
        scale *= 2.0 / (V * unit);
    }
    bx.inv_b1 = (float)(b1 * mk / su);
    bx.inv_b2 = (float)(b2 * mk * su);
    bx.inv_zc = (float)(-(e + 0.5 * V) * unit);
    bx.inv_cut = (float)(rcut * rcut * s2 + (double)bx.eps2s);
    bx.sc = (float)std::sqrt(s2);
    bx.inv_g = (float)(-G * s2 / mk);
}

size_t build_temp_bytes() { return kMaxChunks * sizeof(int2); }

// Enqueue the whole leaf/group build for the particles already in device
// memory (pos, mass).  The handle's box table and buffers are set up.
int build_leaves_device(ph_leaves *h, const void *pos, int pos_type, const float *mass, cudaStream_t s)
{
    const int64_t n = h->n;
    const int nb = h->n_boxes;
    const int T = h->key_bits;
    const BoxDev *boxes = static_cast<const BoxDev *>(h->boxes.p);
    const int32_t *box_first = static_cast<const int32_t *>(h->box_first.p);
    uint32_t *status = static_cast<uint32_t *>(h->status.p);
    uint64_t *keys = static_cast<uint64_t *>(h->keys.p);
    int32_t *vals = static_cast<int32_t *>(h->vals.p);
    if (n > 0) {
        int rc = sort_begin(n, h->temp.p, s);
        if (rc) return rc;
        const SortCounts sc = sort_counts(n, h->temp.p);
        if (pos_type == PH_F64)
            launch_chained(true, k_keys<PH_F64>, grid_for(n), kThreads, 0, s, pos, n, box_first, nb, boxes, T,
                           h->key_kind, keys, vals, sc, status);
        else
            launch_chained(true, k_keys<PH_F32>, grid_for(n), kThreads, 0, s, pos, n, box_first, nb, boxes, T,
                           h->key_kind, keys, vals, sc, status);
        bool alt = false;
        int box_bits = 0;
        while ((1 << box_bits) < nb) box_bits++;
        int bits = 3 * T + box_bits;
        bits = (bits + kSortBits - 1) / kSortBits * kSortBits;
        rc = radix_sort_pairs(keys, vals, static_cast<uint64_t *>(h->keys_alt.p),
                                  static_cast<int32_t *>(h->vals_alt.p), n, bits, h->temp.p, s, &alt);
        if (rc) return rc;
        h->keys_in_alt = alt;
    } else {
        h->keys_in_alt = false;
    }
    const uint64_t *sk = static_cast<const uint64_t *>(h->keys_in_alt ? h->keys_alt.p : h->keys.p);
    const int32_t *perm = static_cast<const int32_t *>(h->keys_in_alt ? h->vals_alt.p : h->vals.p);
    double *xw = static_cast<double *>(h->xw.p);
    float *ms = static_cast<float *>(h->mass_sorted.p);
    int32_t *cell_first = static_cast<int32_t *>(h->cell_first.p);
    int32_t *cell_leaf_first = static_cast<int32_t *>(h->cell_leaf_first.p);
    int32_t *lfirst = static_cast<int32_t *>(h->leaf_first.p), *gfirst = static_cast<int32_t *>(h->group_first.p);
    int32_t *cnt = static_cast<int32_t *>(h->counts.p);   // leaves, groups, active groups
    if (n == 0) {
        // no particles: no leaves, no groups, every cell empty
        int rc = cuda_check(cudaMemsetAsync(cnt, 0, 2 * sizeof(int32_t), s), "clear counts");
        if (!rc) rc = cuda_check(cudaMemsetAsync(lfirst, 0, sizeof(int32_t), s), "clear leaves");
        if (!rc) rc = cuda_check(cudaMemsetAsync(gfirst, 0, sizeof(int32_t), s), "clear groups");
        if (!rc) rc = cuda_check(cudaMemsetAsync(cell_first, 0, 4 * (size_t)(h->n_cells + 1), s), "clear cells");
        if (!rc) rc = cuda_check(cudaMemsetAsync(cell_leaf_first, 0, 4 * (size_t)(h->n_cells + 1), s), "clear cells");
        return rc;
    }
    const int cell_blocks = (h->n_cells + kThreads) / kThreads;   // one thread a cell, and one for the end
    if (pos_type == PH_F64)
        launch_chained(true, k_gather<PH_F64>, grid_for(n) + cell_blocks, kThreads, 0, s, pos, mass, n, sk, perm, boxes,
                       T, xw, ms, status, cell_blocks, nb, h->n_cells, cell_first);
    else
        launch_chained(true, k_gather<PH_F32>, grid_for(n) + cell_blocks, kThreads, 0, s, pos, mass, n, sk, perm, boxes,
                       T, xw, ms, status, cell_blocks, nb, h->n_cells, cell_first);
    const Chunks ch = chunks_of(n);
    uint8_t *starts = static_cast<uint8_t *>(h->starts.p);
    int2 *chunk_count = static_cast<int2 *>(h->temp.p);   // (the sort is done with it)
    launch_chained(true, k_flags, ch.blocks, kThreads, 0, s, sk, n, ch.size, boxes, T, h->max_leaf, h->level_bits,
                   cell_first, starts, chunk_count);
    int32_t *leaf_of = static_cast<int32_t *>(h->leaf_of.p), *group_of = static_cast<int32_t *>(h->group_of.p);
    launch_chained(true, k_starts, ch.blocks, kThreads, 0, s, starts, n, ch.size, chunk_count, leaf_of, group_of, lfirst,
                   gfirst, cnt);
    double *lref = static_cast<double *>(h->leaf_ref.p);
    float4 *lr4 = static_cast<float4 *>(h->leaf_r4.p), *gr4 = static_cast<float4 *>(h->group_r4.p);
    float4 *pos_leaf = static_cast<float4 *>(h->pos_leaf.p);
    const BoxTable lt{lfirst, cnt, lref, lr4, static_cast<float4 *>(h->leaf_c4.p),
                      static_cast<float4 *>(h->leaf_h4.p), nullptr, nullptr};
    const BoxTable gt{gfirst, cnt + 1, static_cast<double *>(h->group_ref.p), gr4,
                      static_cast<float4 *>(h->group_c4.p), static_cast<float4 *>(h->group_h4.p),
                      static_cast<int32_t *>(h->group_cell.p), static_cast<int32_t *>(h->group_box.p)};
    const FrameArgs fr{ms, leaf_of, group_of, gr4, pos_leaf, static_cast<float4 *>(h->pos_group.p), n};
    // at most one part-filled group a ground cell; up to n leaves
    const int64_t most = std::min<int64_t>(n, n / h->group_size + h->n_cells);
    const int gb = grid_for(most, kBoxes), lb = grid_for(n, kBoxes);
    launch_chained(true, k_groups, gb + cell_blocks, kThreads, 0, s, gt, gb, sk, boxes, T, xw, n, cell_first, leaf_of,
                   cnt, h->n_cells, cell_leaf_first);
    launch_chained(true, k_leaves, lb, kThreads, 0, s, lt, fr, sk, boxes, T, xw);
    if (h->tree_leaves) {
        launch_chained(true, k_leaf_mass, grid_for(n), kThreads, 0, s, lfirst, cnt, xw, ms, lref, n, pos_leaf);
    }
    int rc = 0;
    if (h->active) {
        // the groups to sum in active-particle mode (buffers sized by the caller)
        int32_t *gact = static_cast<int32_t *>(h->group_act.p), *gacts = static_cast<int32_t *>(h->group_act_scan.p);
        k_group_active<<<grid_for(n), kThreads, 0, s>>>(gfirst, cnt + 1, perm, h->active, gact);
        count_launch();
        rc = scan_exclusive_i32(gact, gacts, n, cnt + 1, h->temp.p, s);
        if (rc) return rc;
        k_active_list<<<grid_for(n), kThreads, 0, s>>>(gact, gacts, cnt + 1,
                                                       static_cast<int32_t *>(h->active_list.p), cnt + 2);
        count_launch();
    }
    return cuda_check(cudaGetLastError(), "build kernels");
}

}  // namespace phpp
