// Stable LSD radix sort of (64-bit key, 32-bit value) pairs, 8-bit digits.
//
// One pass is one kernel, two for more than kDirectTiles tiles.  The counts
// of a pass's digits per tile are made by whoever writes its input: the
// caller counts the first digit as it makes the keys, each pass counts the
// next digit at the tile a key lands in (one L2 atomic a key).  A tile ranks
// its keys stably (warp by warp, 32 keys at a time),
// reorders them by digit in shared memory and writes each digit's run after
// the keys of earlier tiles, with consecutive threads on consecutive
// positions.  The earlier tiles' counts it adds up itself (up to
// kDirectTiles: a row of 64 counts a digit, in L2), or reads from a scan of
// the counts (k_digit_scan) that runs between the passes.
// Bound by latency up to ~10^5 keys and by L2 traffic and atomics above.
// Measured against one count, three scan and one scatter kernel a pass: a
// pass of 4096 keys 27 -> 9 us, of 2 M keys 46 -> 26 us; per step, 1000
// particles 253 -> 187 us, 4096 140 -> 102 us, 50,021 552 -> 472 us.
#include <algorithm>
#include <utility>

#include "checks.cuh"
#include "phpp_internal.cuh"

namespace phpp {
namespace {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kBins = 1 << kSortBits;
constexpr int kDirectTiles = 64;

// The lanes holding the same digit (0 .. kBins): one ballot a bit (a pass of
// 2 M keys took 7 us longer with __match_any_sync).
__device__ __forceinline__ unsigned same_digit(int d)
{
    unsigned m = 0xffffffffu;
#pragma unroll
    for (int b = 0; b <= kSortBits; b++) {
        const unsigned set = __ballot_sync(0xffffffffu, (d >> b) & 1);
        m &= (d >> b) & 1 ? set : ~set;
    }
    return m;
}

// Exclusive scan of one int per thread over the block.
__device__ __forceinline__ int block_excl(int v, int *s_wsum)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s_wsum[w] = incl;
    __syncthreads();
    int base = 0;
#pragma unroll
    for (int ww = 0; ww < kSortWarps; ww++) base += ww < w ? s_wsum[ww] : 0;
    __syncthreads();
    return base + incl - v;
}

// Exclusive prefix over the tiles of one digit's counts, and its total.
__global__ void __launch_bounds__(kSortThreads) k_digit_scan(const int32_t *hist, int row, int32_t *offs, int32_t *total)
{
    chain_begin();
    __shared__ int s_wsum[kSortWarps];
    __shared__ int s_sum;
    const int32_t *h = hist + (int64_t)blockIdx.x * row;
    int32_t *o = offs + (int64_t)blockIdx.x * row;
    int run = 0;
    for (int b = 0; b < row; b += 4 * kSortThreads) {
        const int t = b + 4 * threadIdx.x;
        int4 v = make_int4(0, 0, 0, 0);
        if (t < row) v = *reinterpret_cast<const int4 *>(h + t);
        const int mine = v.x + v.y + v.z + v.w;
        int e = run + block_excl(mine, s_wsum);
        if (threadIdx.x == kSortThreads - 1) s_sum = e + mine;
        if (t < row) *reinterpret_cast<int4 *>(o + t) = make_int4(e, e + v.x, e + v.x + v.y, e + v.x + v.y + v.z);
        __syncthreads();
        run = s_sum;
        __syncthreads();
    }
    if (threadIdx.x == 0) total[blockIdx.x] = run;
}

__global__ void __launch_bounds__(kSortThreads) k_clear(int4 *p, int n)
{
    chain_begin();
    for (int i = blockIdx.x * kSortThreads + threadIdx.x; i < n; i += gridDim.x * kSortThreads)
        p[i] = make_int4(0, 0, 0, 0);
}

struct PassArgs {
    const uint64_t *keys;
    const int32_t *vals;
    uint64_t *keys_out;
    int32_t *vals_out;
    int64_t n;
    int shift, ntiles, row;
    const int32_t *hist;     // [kBins][row] this pass's digit counts per tile
    const int32_t *offs;     // [kBins][row] their prefixes, and the totals [kBins] (k_digit_scan)
    const int32_t *total;
    int32_t *hist_next;      // the next digit's counts (NULL in the last pass)
    int32_t *hist_clear;     // the counts of the pass after that, cleared here
};

// kItems: rounds of 32 keys per warp (tile of 256 kItems keys).
template <int kItems, bool kDirect>
__global__ void __launch_bounds__(kSortThreads) k_radix_pass(PassArgs a)
{
    chain_begin();
    constexpr int kTile = kSortThreads * kItems;
    __shared__ uint16_t cnt[kSortWarps][kBins];   // (a tile has at most 2048 keys)
    __shared__ int32_t s_off[kBins];            // output position of the tile's first key of each digit
    __shared__ int32_t s_start[kBins];          // its first slot in the tile
    __shared__ int32_t s_wsum[kSortWarps];
    __shared__ uint64_t s_key[kTile];
    __shared__ int32_t s_val[kTile];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int d = lane; d < kBins; d += 32) cnt[w][d] = 0;
    // warp w owns keys [base, base + 32 kItems), 32 per round, in order
    const int64_t tile0 = (int64_t)blockIdx.x * kTile;
    const int64_t base = tile0 + (int64_t)w * 32 * kItems;
    uint64_t k_[kItems];
    int32_t v_[kItems];
    int32_t d_[kItems];
    int32_t r_[kItems];
#pragma unroll
    for (int r = 0; r < kItems; r++) {
        const int64_t i = base + r * 32 + lane;
        const bool ok = i < a.n;
        k_[r] = ok ? a.keys[i] : 0ull;
        v_[r] = ok ? a.vals[i] : 0;
        d_[r] = ok ? (int)((k_[r] >> a.shift) & (kBins - 1)) : kBins;   // kBins = no key
    }
    if (a.hist_clear)
        for (int i = blockIdx.x * kSortThreads + threadIdx.x; i < kBins * a.row; i += a.ntiles * kSortThreads)
            a.hist_clear[i] = 0;
    {
        // this thread's digit: the keys of earlier tiles, and all of them
        int before = 0, all = 0;
        if (kDirect) {
            const int32_t *h = a.hist + (int64_t)threadIdx.x * a.row;
            for (int t = 0; t < a.row; t += 4) {
                const int4 c = *reinterpret_cast<const int4 *>(h + t);
                all += c.x + c.y + c.z + c.w;
                before += (t < (int)blockIdx.x ? c.x : 0) + (t + 1 < (int)blockIdx.x ? c.y : 0) +
                          (t + 2 < (int)blockIdx.x ? c.z : 0) + (t + 3 < (int)blockIdx.x ? c.w : 0);
            }
        } else {
            before = a.offs[(int64_t)threadIdx.x * a.row + blockIdx.x];
            all = a.total[threadIdx.x];
        }
        s_off[threadIdx.x] = before + block_excl(all, s_wsum);
    }
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < kItems; r++) {
        const unsigned peers = same_digit(d_[r]);
        const int leader = __ffs(peers) - 1;
        int old = 0;
        if (d_[r] < kBins && lane == leader) {
            old = cnt[w][d_[r]];
            cnt[w][d_[r]] = (uint16_t)(old + __popc(peers));
        }
        r_[r] = __shfl_sync(0xffffffffu, old, leader) + __popc(peers & lt);
        __syncwarp();
    }
    __syncthreads();
    {   // per digit: exclusive prefix of the per-warp counts over warps, then of
        // the totals over digits
        const int d = threadIdx.x;
        int run = 0;
#pragma unroll
        for (int ww = 0; ww < kSortWarps; ww++) {
            const int c = cnt[ww][d];
            cnt[ww][d] = (uint16_t)run;
            run += c;
        }
        s_start[d] = block_excl(run, s_wsum);
    }
    __syncthreads();
    // the tile in digit order in shared memory ...
#pragma unroll
    for (int r = 0; r < kItems; r++) {
        if (d_[r] < kBins) {
            const int slot = s_start[d_[r]] + cnt[w][d_[r]] + r_[r];
            s_key[slot] = k_[r];
            s_val[slot] = v_[r];
        }
    }
    __syncthreads();
    // ... then written out slot by slot: consecutive threads write consecutive
    // positions of a digit's run
    const int tile_n = a.n - tile0 < kTile ? (int)(a.n - tile0) : kTile;
    for (int s0 = 0; s0 < tile_n; s0 += kSortThreads) {
        const int slot = s0 + threadIdx.x;
        const bool ok = slot < tile_n;
        const uint64_t key = ok ? s_key[slot] : 0ull;
        const int d = (int)((key >> a.shift) & (kBins - 1));
        const int pos = ok ? s_off[d] + (slot - s_start[d]) : 0;
        const bool in = ok && in_bounds(pos, a.n, BS_SORT_OUT);
        if (in) {
            a.keys_out[pos] = key;
            a.vals_out[pos] = s_val[slot];
        }
        if (a.hist_next)
            count_digit(a.hist_next, (int)((key >> (a.shift + kSortBits)) & (kBins - 1)) * a.row + pos / kTile, in);
    }
}

struct SortLayout {
    int tile, ntiles, row;
    size_t counts;           // bytes of one [kBins][row] array
};

// Tile of 512 keys up to 32,768, 1024 up to 65,536, else 2048: small sorts
// need the blocks (4096 keys in tiles of 2048 are two blocks of eight serial
// rounds), large ones the longer runs per digit.
SortLayout layout_for(int64_t n)
{
    SortLayout l;
    l.tile = n <= 64 * 512 ? 512 : n <= 64 * 1024 ? 1024 : 2048;
    l.ntiles = (int)std::max<int64_t>((n + l.tile - 1) / l.tile, 1);
    l.row = (l.ntiles + 3) & ~3;
    l.counts = (size_t)kBins * l.row * sizeof(int32_t);
    return l;
}

template <int kItems, bool kDirect>
void launch_pass(const PassArgs &a, cudaStream_t s)
{
    launch_chained(true, k_radix_pass<kItems, kDirect>, a.ntiles, kSortThreads, 0, s, a);
}

}  // namespace

size_t sort_temp_bytes(int64_t n)
{
    const SortLayout l = layout_for(n);
    return 4 * l.counts + kBins * sizeof(int32_t) + 256;
}

SortCounts sort_counts(int64_t n, void *temp)
{
    const SortLayout l = layout_for(n);
    return SortCounts{static_cast<int32_t *>(temp), l.row, l.tile == 512 ? 9 : l.tile == 1024 ? 10 : 11};
}

int sort_begin(int64_t n, void *temp, cudaStream_t s)
{
    const int words = (int)(2 * layout_for(n).counts / sizeof(int4));
    k_clear<<<std::min((words + 1023) / 1024, 152 * 4), kSortThreads, 0, s>>>(static_cast<int4 *>(temp), words);
    count_launch();
    return cuda_check(cudaGetLastError(), "clear digit counts");
}

int radix_sort_pairs(uint64_t *keys, int32_t *vals, uint64_t *keys_alt, int32_t *vals_alt, int64_t n, int bits,
                     void *temp, cudaStream_t s, bool *result_in_alt)
{
    *result_in_alt = false;
    if (n <= 1) return PH_OK;
    const SortLayout l = layout_for(n);
    char *t = static_cast<char *>(temp);
    // three count arrays in turn: a pass reads one, fills the next and clears
    // the one after (the first two start cleared, sort_begin)
    int32_t *hist[3];
    for (int k = 0; k < 3; k++) hist[k] = reinterpret_cast<int32_t *>(t + k * l.counts);
    int32_t *offs = reinterpret_cast<int32_t *>(t + 3 * l.counts);
    int32_t *total = reinterpret_cast<int32_t *>(t + 4 * l.counts);
    const bool direct = l.ntiles <= kDirectTiles;
    uint64_t *kin = keys, *kout = keys_alt;
    int32_t *vin = vals, *vout = vals_alt;
    bool alt = false;
    for (int shift = 0, p = 0; shift < bits; shift += kSortBits, p++) {
        PassArgs a;
        a.keys = kin;
        a.vals = vin;
        a.keys_out = kout;
        a.vals_out = vout;
        a.n = n;
        a.shift = shift;
        a.ntiles = l.ntiles;
        a.row = l.row;
        a.hist = hist[p % 3];
        a.offs = offs;
        a.total = total;
        const bool last = shift + kSortBits >= bits;
        a.hist_next = last ? nullptr : hist[(p + 1) % 3];
        a.hist_clear = last ? nullptr : hist[(p + 2) % 3];
        if (!direct) {
            launch_chained(true, k_digit_scan, kBins, kSortThreads, 0, s, a.hist, l.row, offs, total);
        }
        if (l.tile == 512) launch_pass<2, true>(a, s);
        else if (l.tile == 1024) launch_pass<4, true>(a, s);
        else if (direct) launch_pass<8, true>(a, s);
        else launch_pass<8, false>(a, s);
        std::swap(kin, kout);
        std::swap(vin, vout);
        alt = !alt;
    }
    *result_in_alt = alt;
    return cuda_check(cudaGetLastError(), "radix sort launch");
}

}  // namespace phpp
