// sort.cu -- Alg. 1 CreateTiles, DuplicateWithKeys, SortByKeys and
// IdentifyTileRanges.
//
// The instance key is (global tile index, camera depth), the lists ordered as
// by a stable sort of the full key in emission order.  Every instance of one
// projected row carries the same depth, so neither path sorts instances by it.
//
// The binned path (the default up to 40960 tiles per view) lists every row in
// the 8x8-tile super-tiles that its rectangle meets, sorts each super-tile's
// list by (depth bits, row) on its own (k_cell_count, k_cell_scan,
// k_cell_scatter, k_unit_sort; with few rows k_small_lists), and filters it into
// its tiles' lists in order:
// the first 512 to 2048 entries by a saturation head (k_head_count), the rest in
// parallel segments (k_tail_count), the counts turned into ranges by one
// look-back pass (k_tile_ranges) and the lists written by one pass
// (k_tile_write).  With culling on, a list holds only the tiles the opacity footprint
// reaches and ends where every pixel of the tile has certainly saturated (tile
// saturation, below); neither changes a result.
//
// The radix path sorts the rows by the IEEE bits of their depth (positive
// floats order like their bit patterns), emits the instances in that row order
// and radix-sorts the tile digits stably.  Its passes are single-pass
// "onesweep"-style: one 8-bit digit per pass, partitions of 4096 keys taken in
// ticket order by persistent CTAs, local ranking of the keys of a warp
// (digit-bit ballots or a match instruction) with shared-memory counters, and a
// decoupled look-back across partitions whose waits are bounded
// (SPLAT_ERR_TIMEOUT on expiry).
#include <algorithm>

#include "splat_internal.cuh"

namespace splat {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 16;
constexpr int kSortPart = kSortThreads * kSortItems;  // keys per partition
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanPart = kScanThreads * kScanItems;
constexpr int kDupChunk = 2048;  // instance slots per duplicate work item
constexpr int kDupThreads = 256;

constexpr int kLookWindow = 8;  // predecessors a look-back thread reads per step
constexpr uint32_t kFlagAgg = 1u << 30;
constexpr uint32_t kFlagPrefix = 2u << 30;
constexpr uint32_t kValMask = (1u << 30) - 1;

// Exclusive scan of one value per thread across a 256-thread block.
__device__ __forceinline__ unsigned long long block_excl_scan256_u64(unsigned long long v, unsigned long long* s_tmp,
                                                                     unsigned long long* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_tmp[warp] = x;
    __syncthreads();
    unsigned long long wsum = 0, all = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const unsigned long long t = s_tmp[w];
        if (w < warp) wsum += t;
        all += t;
    }
    __syncthreads();
    *total = all;
    return wsum + x - v;
}

// WARPS warps
template <int WARPS>
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* s_tmp, uint32_t* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_tmp[warp] = x;
    __syncthreads();
    uint32_t wsum = 0, all = 0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
        const uint32_t t = s_tmp[w];
        if (w < warp) wsum += t;
        all += t;
    }
    __syncthreads();
    if (total) *total = all;
    return wsum + x - v;
}

__device__ __forceinline__ uint32_t block_excl_scan256(uint32_t v, uint32_t* s_tmp, uint32_t* total)
{
    return block_excl_scan<8>(v, s_tmp, total);
}

// ---------------------------------------------------------------------------
// Depth keys of the projected rows + histograms of their 4 digits
// ---------------------------------------------------------------------------

struct DepthArgs {
    splat_proj proj;
    int64_t n_rows;
    uint32_t* keys;
    uint32_t* vals;
    uint32_t* dhist;        // [4][256] digit counts (zeroed)
    uint32_t* zero_a;
    int64_t n_zero_a;
    unsigned long long* zero_b;
    int64_t n_zero_b;
};

__global__ void __launch_bounds__(256) k_depth_keys(DepthArgs a)
{
    __shared__ uint32_t s_hist[4][kRadix];
    for (int i = threadIdx.x; i < 4 * kRadix; i += blockDim.x) (&s_hist[0][0])[i] = 0;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t gt = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t r = gt; r < a.n_rows; r += stride) {
        const float depth = ((const float4*)a.proj.rgb_depth)[r].w;
        const uint32_t k = a.proj.n_tiles[r] > 0 ? __float_as_uint(depth) : 0xffffffffu;
        a.keys[r] = k;
        a.vals[r] = (uint32_t)r;
#pragma unroll
        for (int p = 0; p < 4; ++p) atomicAdd(&s_hist[p][(k >> (8 * p)) & 0xff], 1u);
    }
    for (int64_t i = gt; i < a.n_zero_a; i += stride) a.zero_a[i] = 0;
    for (int64_t i = gt; i < a.n_zero_b; i += stride) a.zero_b[i] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < 4 * kRadix; i += blockDim.x) {
        const uint32_t c = (&s_hist[0][0])[i];
        if (c) atomicAdd(&a.dhist[i], c);
    }
}

// ---------------------------------------------------------------------------
// One onesweep radix pass (8-bit digit at `shift`)
// ---------------------------------------------------------------------------

struct PassArgs {
    const uint32_t* keys_in;
    const uint32_t* vals_in;
    uint32_t* keys_out;  // may be null (keys not needed after this pass)
    uint32_t* vals_out;
    const int64_t* n_dev;  // element count on the device (null: n_host)
    int64_t n_host;
    int64_t cap;
    const uint32_t* hist;  // [256] digit counts of this pass
    uint32_t* lb;          // [parts][256] look-back words of this pass (zeroed)
    uint32_t* lb_next;     // [parts][256] zeroed here for the next pass (may be null)
    uint32_t* ticket;
    int32_t* status;
    int stage;
    int shift;
    int64_t spin_limit;
    int ballot_rank;       // rank by digit-bit ballots (many distinct digits per warp) instead of match
};

template <bool BALLOT>
__global__ void __launch_bounds__(kSortThreads) k_onesweep(PassArgs a)
{
    __shared__ uint32_t s_keys[kSortPart];
    __shared__ uint32_t s_vals[kSortPart];
    __shared__ uint32_t s_whist[kSortWarps][kRadix];
    __shared__ uint32_t s_dstart[kRadix];
    __shared__ uint32_t s_base[kRadix];
    __shared__ uint32_t s_tmp[8];
    __shared__ int64_t s_ticket;

    if (block_failed(a.status)) return;
    const int64_t n = a.n_dev ? min(*a.n_dev, a.cap) : a.n_host;
    if (n <= 0) return;
    const int64_t parts = (n + kSortPart - 1) / kSortPart;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = lanemask_lt();
    const uint32_t gofs = block_excl_scan256(a.hist[tid], s_tmp, nullptr);  // first output position of digit tid

    for (;;) {
        if (tid == 0) s_ticket = atomicAdd(a.ticket, 1u);
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) s_whist[w][tid] = 0;
        __syncthreads();
        const int64_t ticket = s_ticket;
        if (ticket >= parts) break;
        const int64_t base = ticket * kSortPart;
        const int64_t wbase = base + (int64_t)warp * 32 * kSortItems;
        // keys of this warp's share of the partition: its items j * 32 + lane < wrem
        const int64_t wr = n - wbase;
        const int wrem = wr <= 0 ? 0 : (wr >= 32 * kSortItems ? 32 * kSortItems : (int)wr);
        const uint32_t* kin = a.keys_in + wbase;
        const uint32_t* vin = a.vals_in + wbase;

        uint32_t k[kSortItems], v[kSortItems], r[kSortItems];
#pragma unroll
        for (int j = 0; j < kSortItems; ++j) {
            const bool ok = j * 32 + lane < wrem;
            k[j] = ok ? kin[j * 32 + lane] : 0u;
            v[j] = ok ? vin[j * 32 + lane] : 0u;
        }
        // warp-level stable ranking, items in (j, lane) order.  The lanes holding
        // the same digit: with BALLOT, one ballot per digit bit (a constant
        // cost, for digits that take many values in a warp); otherwise a match
        // instruction (fast when the warp holds few distinct digits, slow with many)
#pragma unroll
        for (int j = 0; j < kSortItems; ++j) {
            const bool ok = j * 32 + lane < wrem;
            const uint32_t dj = (k[j] >> a.shift) & 0xff;
            const unsigned valid = __ballot_sync(0xffffffffu, ok);
            unsigned same = valid;
            if (BALLOT) {
#pragma unroll
                for (int bit = 0; bit < 8; ++bit) {
                    const unsigned bb = __ballot_sync(0xffffffffu, (dj >> bit) & 1u);
                    same &= ((dj >> bit) & 1u) ? bb : ~bb;
                }
            }
            r[j] = 0;
            if (ok) {
                const uint32_t d = dj;
                const unsigned peers = BALLOT ? same : __match_any_sync(valid, d);
                const int leader = __ffs(peers) - 1;
                uint32_t prev = 0;
                if (lane == leader) {
                    prev = s_whist[warp][d];
                    s_whist[warp][d] = prev + __popc(peers);
                }
                prev = __shfl_sync(peers, prev, leader);
                r[j] = prev + __popc(peers & lt);
            }
            __syncwarp();
        }
        __syncthreads();
        // per digit: exclusive prefix over warps, partition count
        const int d = tid;
        uint32_t cnt = 0;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) {
            const uint32_t c = s_whist[w][d];
            s_whist[w][d] = cnt;
            cnt += c;
        }
        uint32_t* my = a.lb + ticket * kRadix + d;
        st_relaxed(my, (ticket == 0 ? kFlagPrefix : kFlagAgg) | cnt);
        if (a.lb_next) a.lb_next[ticket * kRadix + d] = 0;
        s_dstart[d] = block_excl_scan256(cnt, s_tmp, nullptr);
        // decoupled look-back for digit d, kLookWindow predecessors per step
        // (independent loads): all partitions of a pass usually run in one wave,
        // so a walk of one predecessor per L2 round trip would make the last
        // partition wait for about half the partition count of round trips
        uint32_t excl = 0;
        if (ticket > 0) {
            int64_t j = ticket - 1;  // nearest predecessor not yet added
            int64_t spins = 0;
            for (;;) {
                uint32_t w[kLookWindow];
#pragma unroll
                for (int q = 0; q < kLookWindow; ++q)
                    w[q] = j - q >= 0 ? ld_relaxed(a.lb + (j - q) * kRadix + d) : kFlagPrefix;
                // add the published words from the nearest one back, up to and
                // including the first inclusive prefix, or up to the first word
                // not yet published
                int q = 0;
                bool found = false;
#pragma unroll
                for (int t = 0; t < kLookWindow; ++t) {
                    if (found || q < t) continue;  // stopped at an earlier word
                    const uint32_t flag = w[t] & ~kValMask;
                    if (flag == 0) continue;       // not yet published: q stays at t
                    excl += w[t] & kValMask;
                    q = t + 1;
                    found = flag == kFlagPrefix;
                }
                if (found) break;
                j -= q;
                if (q == 0) {
                    if (++spins > a.spin_limit) {
                        set_status(a.status, SPLAT_ERR_TIMEOUT, a.stage, ticket);
                        break;
                    }
                    if (spins > 64) __nanosleep(64);
                }
            }
            st_relaxed(my, kFlagPrefix | ((excl + cnt) & kValMask));
        }
        s_base[d] = gofs + excl - s_dstart[d];
        __syncthreads();
        // local scatter into digit order
#pragma unroll
        for (int j = 0; j < kSortItems; ++j) {
            if (j * 32 + lane < wrem) {
                const uint32_t dd = (k[j] >> a.shift) & 0xff;
                const uint32_t pos = s_dstart[dd] + s_whist[warp][dd] + r[j];
                s_keys[pos] = k[j];
                s_vals[pos] = v[j];
            }
        }
        __syncthreads();
        const int nvalid = (int)min((int64_t)kSortPart, n - base);
        for (int i = tid; i < nvalid; i += kSortThreads) {
            const uint32_t key = s_keys[i];
            const uint32_t out = s_base[(key >> a.shift) & 0xff] + i;
            if (out >= (uint64_t)n) continue;  // only after a timed-out look-back
            const uint32_t val = s_vals[i];
            if (a.keys_out) a.keys_out[out] = key;
            a.vals_out[out] = val;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Exclusive scan of the tile counts in depth order (A5) + chunk starts for
// the load-balanced duplication + capacity check.
// ---------------------------------------------------------------------------

struct ScanArgs {
    const uint32_t* rows;      // [n_rows] depth-sorted rows
    const uint32_t* n_tiles;   // [n_rows] per row
    int64_t n_rows;
    uint32_t* offsets;         // [n_rows] exclusive prefix (saturated at 2^32-1)
    uint32_t* chunk_row;       // [n_chunks_max] first sorted position of each duplicate chunk
    int64_t n_chunks_max;
    unsigned long long* lb;    // [parts] look-back words (zeroed)
    uint32_t* ticket;
    int64_t* n_instances;      // out: K
    int64_t* n_needed;         // out (may be null): K as the capacity needed
    int64_t capacity;
    int32_t* status;
    int64_t spin_limit;
};

__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(ScanArgs a)
{
    __shared__ unsigned long long s_tmp64[8];
    __shared__ int64_t s_ticket;
    __shared__ unsigned long long s_excl;
    constexpr unsigned long long kA = 1ull << 62, kP = 2ull << 62, kM = (1ull << 62) - 1;
    if (block_failed(a.status)) return;  // the row order is not valid after a failed sort
    const int64_t parts = (a.n_rows + kScanPart - 1) / kScanPart;
    const int tid = threadIdx.x;
    for (;;) {
        if (tid == 0) s_ticket = atomicAdd(a.ticket, 1u);
        __syncthreads();
        const int64_t ticket = s_ticket;
        if (ticket >= parts) break;
        const int64_t base = ticket * kScanPart;
        // blocked layout: thread tid owns the kScanItems consecutive rows from base + tid * kScanItems,
        // so one block scan of the per-thread sums serves the whole partition
        const int64_t i0 = base + (int64_t)tid * kScanItems;
        uint32_t c[kScanItems];
        if (i0 + kScanItems <= a.n_rows) {
            const uint4* r4 = (const uint4*)(a.rows + i0);
#pragma unroll
            for (int q = 0; q < kScanItems / 4; ++q) {
                const uint4 r = r4[q];
                c[4 * q + 0] = a.n_tiles[r.x];
                c[4 * q + 1] = a.n_tiles[r.y];
                c[4 * q + 2] = a.n_tiles[r.z];
                c[4 * q + 3] = a.n_tiles[r.w];
            }
        } else {
#pragma unroll
            for (int j = 0; j < kScanItems; ++j) c[j] = i0 + j < a.n_rows ? a.n_tiles[a.rows[i0 + j]] : 0u;
        }
        unsigned long long tsum = 0;
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) tsum += c[j];
        unsigned long long running;
        const unsigned long long texcl = block_excl_scan256_u64(tsum, s_tmp64, &running);
        const unsigned long long agg = running;
        if (tid < 32) {
            // decoupled look-back by one warp: lane l reads predecessor j - l, so
            // one round trip covers 32 of them (all partitions usually run in one
            // wave, and a walk of one predecessor per round trip would make the
            // last partition wait for about half the partition count of them)
            const int lane = tid;
            unsigned long long excl = 0;
            if (lane == 0) st_relaxed64(a.lb + ticket, (ticket == 0 ? kP : kA) | agg);
            if (ticket > 0) {
                int64_t j = ticket - 1, spins = 0;  // nearest predecessor not yet added
                for (;;) {
                    const bool in = j - lane >= 0;
                    const unsigned long long s = in ? ld_relaxed64(a.lb + (j - lane)) : kP;
                    const unsigned long long flag = s & ~kM;
                    // the published words from the nearest one back, up to and
                    // including the first inclusive prefix or up to the first
                    // word not yet published
                    const unsigned pend = __ballot_sync(0xffffffffu, flag == 0);
                    const unsigned pref = __ballot_sync(0xffffffffu, flag == kP);
                    const int first_pend = pend ? __ffs(pend) - 1 : 32;
                    const int first_pref = pref ? __ffs(pref) - 1 : 32;
                    const bool found = first_pref < first_pend;
                    const int take = found ? first_pref + 1 : first_pend;
                    unsigned long long v = lane < take ? (s & kM) : 0ull;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                    excl += v;
                    if (found) break;
                    j -= take;
                    if (take == 0) {
                        if (++spins > a.spin_limit) {
                            if (lane == 0) set_status(a.status, SPLAT_ERR_TIMEOUT, SPLAT_STAGE_SCAN, ticket);
                            break;
                        }
                        if (spins > 64) __nanosleep(64);
                    }
                }
                if (lane == 0) st_relaxed64(a.lb + ticket, kP | ((excl + agg) & kM));
            }
            if (lane == 0) s_excl = excl;
            if (lane == 0 && ticket == parts - 1) {
                const int64_t K = (int64_t)(excl + agg);
                *a.n_instances = K;
                if (a.n_needed) *a.n_needed = K;
                if (K > a.capacity) set_status(a.status, SPLAT_ERR_CAPACITY, SPLAT_STAGE_SCAN, K);
            }
        }
        __syncthreads();
        const unsigned long long excl = s_excl;
        unsigned long long off = excl + texcl;
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) {
            const int64_t idx = i0 + j;
            if (idx < a.n_rows) {
                a.offsets[idx] = off > 0xffffffffull ? 0xffffffffu : (uint32_t)off;
                if (c[j] != 0) {
                    // chunks whose first slot falls inside [off, off + c)
                    const unsigned long long lo = (off + kDupChunk - 1) / kDupChunk;
                    const unsigned long long hi = (off + c[j] - 1) / kDupChunk;
                    for (unsigned long long q = lo; q <= hi && q < (unsigned long long)a.n_chunks_max; ++q)
                        a.chunk_row[q] = (uint32_t)idx;
                }
            }
            off += c[j];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// DuplicateWithKeys: one (tile, row) instance per tile of each row's
// rectangle, rows in depth order, tiles row major; + tile-digit histograms.
// ---------------------------------------------------------------------------

struct DupArgs {
    splat_proj proj;
    const uint32_t* rows;      // depth-sorted rows
    const uint32_t* offsets;
    const uint32_t* chunk_row;
    int64_t n_rows;
    const int64_t* n_instances;
    int64_t capacity;
    uint32_t* keys_out;
    uint32_t* vals_out;
    uint32_t* hist;            // [tile_passes][256]
    int tile_passes;
    uint32_t* zero;            // first tile-pass look-back buffer
    int32_t* status;
    int tile_base[SPLAT_MAX_VIEWS];
    int TX[SPLAT_MAX_VIEWS];
};

__global__ void __launch_bounds__(kDupThreads) k_duplicate(DupArgs a)
{
    __shared__ uint32_t s_off[kDupChunk + 1];
    __shared__ uint32_t s_base[kDupChunk + 1];
    __shared__ uint32_t s_w[kDupChunk + 1];
    __shared__ uint32_t s_tx[kDupChunk + 1];
    __shared__ uint32_t s_row[kDupChunk + 1];
    __shared__ uint32_t s_hist[4][kRadix];
    if (status_failed(a.status)) return;
    const int64_t K = min(*a.n_instances, a.capacity);
    const int tid = threadIdx.x;
    for (int i = tid; i < 4 * kRadix; i += kDupThreads) (&s_hist[0][0])[i] = 0;
    {
        const int64_t nz = ((K + kSortPart - 1) / kSortPart) * kRadix;
        for (int64_t i = blockIdx.x * (int64_t)kDupThreads + tid; i < nz; i += (int64_t)gridDim.x * kDupThreads)
            a.zero[i] = 0;
    }
    const int64_t chunks = (K + kDupChunk - 1) / kDupChunk;
    const int64_t N = a.proj.n;
    __syncthreads();
    for (int64_t c = blockIdx.x; c < chunks; c += gridDim.x) {
        const int64_t s0 = c * kDupChunk;
        const int64_t s1 = min(s0 + kDupChunk, K);
        const int64_t j0 = a.chunk_row[c];
        int64_t j1 = (c + 1 < chunks) ? (int64_t)a.chunk_row[c + 1] : j0 + (s1 - s0) - 1;
        j1 = min(j1, a.n_rows - 1);
        j1 = min(j1, j0 + kDupChunk);  // a chunk spans at most kDupChunk + 1 rows
        const int cnt = (int)(j1 - j0 + 1);
        for (int q = tid; q < cnt; q += kDupThreads) {
            const int64_t j = j0 + q;
            const uint32_t row = a.rows[j];
            const int v = (int)(row / N);
            const int4 rc = ((const int4*)a.proj.rect)[row];
            s_off[q] = a.offsets[j];
            s_base[q] = (uint32_t)(a.tile_base[v] + rc.y * a.TX[v] + rc.x);
            s_w[q] = (uint32_t)max(rc.z - rc.x, 1);
            s_tx[q] = (uint32_t)a.TX[v];
            s_row[q] = row;
        }
        __syncthreads();
        for (int64_t s = s0 + tid; s < s1; s += kDupThreads) {
            // last q with s_off[q] <= s
            int lo = 0, hi = cnt - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if ((int64_t)s_off[mid] <= s) lo = mid; else hi = mid - 1;
            }
            const uint32_t l = (uint32_t)(s - s_off[lo]);
            const uint32_t w = s_w[lo];
            const uint32_t ty = l / w, tx = l - ty * w;
            const uint32_t key = s_base[lo] + ty * s_tx[lo] + tx;
            a.keys_out[s] = key;
            a.vals_out[s] = s_row[lo];
            for (int p = 0; p < a.tile_passes; ++p) atomicAdd(&s_hist[p][(key >> (8 * p)) & 0xff], 1u);
        }
        __syncthreads();
    }
    for (int i = tid; i < a.tile_passes * kRadix; i += kDupThreads) {
        const uint32_t h = (&s_hist[0][0])[i];
        if (h) atomicAdd(&a.hist[i], h);
    }
}

// IdentifyTileRanges: [start, end) of each tile's run in the sorted keys.
__global__ void __launch_bounds__(256) k_ranges(const uint32_t* keys, const int64_t* n_instances, int64_t capacity,
                                                uint2* ranges, int32_t* status)
{
    if (status_failed(status)) return;
    const int64_t K = min(*n_instances, capacity);
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < K; s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = keys[s];
        if (s == 0 || keys[s - 1] != k) ranges[k].x = (uint32_t)s;
        if (s == K - 1 || keys[s + 1] != k) ranges[k].y = (uint32_t)(s + 1);
    }
}

// ---------------------------------------------------------------------------
// Super-tile lists (level 1 of the binned path).  A row enters the list of
// every 8x8-tile super-tile its tile rectangle meets; a list is ordered by
// (depth bits, row).  An MSD bucket sort with every list on its own:
//
//   k_cell_count    adds each entry to its cell = (super-tile, depth bin), one
//                   reduction per entry, and packs the row's super-rectangle and
//                   key into 8 bytes for the scatter.  Bins are equal steps of
//                   the depth bits over the range of a sample of the view's rows
//                   (depths outside fall into the first or last bin), or runs
//                   between samples where the rows lie on few depths; a bin's
//                   entries are contiguous in the list's order
//   k_cell_scan     block per super-tile: cell starts, the lists' ranges, K1, and
//                   the sort units: runs of bins of about kUnit / 2 entries
//   k_cell_scatter  writes each entry (row, key) into its cell, in any order
//   k_unit_sort     sorts the units in shared memory (sort_unit below): before the
//                   head count the units that hold the head's entries of a
//                   list, after it the others, of the super-tiles with a list that
//                   did not end in the head
//
// What bounds these kernels is latency and the one L2 atomic per entry.  They
// replaced a radix sort of all rows by depth (four onesweep passes), a scan of
// the rows' super-tile counts and a stable split of the entries by super-tile:
// that chain of dependent passes took 130 us for a single view of any size below
// 300k rows, and sorted every list to its end though a dense list is only read
// up to its saturation.  All are exact: (depth bits, row) is unique in a list, so
// the order does not depend on the arrival order in a cell.
// ---------------------------------------------------------------------------

// a row's super-rectangle is packed into four bytes (CellArgs::rec)
static_assert((kMaxImage / kTile + 7) / 8 <= 255, "super-tile coordinates in a byte");
constexpr int64_t kBinMaxTiles = 40960;  // per view: the binned path's default range
constexpr int kSplitMaxSmem = 200 * 1024;
constexpr int kMaxBins = 1024;           // depth bins per super-tile
constexpr int kUnit = 2048;              // entries a block sorts in shared memory
constexpr int kUnitThreads = 256, kPer = kUnit / kUnitThreads;
constexpr int kUnitStep = kUnit / 2;     // a unit starts at the first bin start at or after each multiple
constexpr int kSortBuckets = 2048;
constexpr int kSortBucketBits = 11;
constexpr uint32_t kCrowded = 48;        // entries in one bucket above which a unit takes a second counting pass
constexpr uint32_t kWholeUnit = 0xffffffffu;
constexpr int kRowsPerThread = 2;         // of k_cell_count: 256 kRowsPerThread rows per block
constexpr int kScatterRounds = 4;         // 32-entry rounds of a warp whose atomics are in flight together
constexpr int kHeadEntries = 512;        // entries of a list a head CTA takes at a time, in order
constexpr int kLongList = 4096;          // lists of more entries than this may get kLongHead of them in the head
constexpr int kLongHead = 2048;

// Entries of a list of n that the head pass may go through before the tail: the
// certified end of a tile's list can only fall inside them.  What lies past the
// ends is neither sorted nor counted nor written (figures: k_head_count).
__host__ __device__ __forceinline__ uint32_t head_reach(uint32_t n, int long_heads)
{
    return min(n, (uint32_t)(long_heads && n > (uint32_t)kLongList ? kLongHead : kHeadEntries));
}

struct CellArgs {
    splat_proj proj;
    int V, bin_bits, nbins;        // nbins = 2^bin_bits depth bins
    int copies;                    // of the cells (a power of two); a view's b-th run of 512 rows uses copy b % copies
    int64_t n;                     // rows per view
    uint2* range;                  // [V] first depth bits and shift of the views' bins (kSplitBins: by split), from
                                   // k_cell_count
    unsigned long long* split;     // [V][kSplits] bounds of the views' bins where kSplitBins
    int super_base[SPLAT_MAX_VIEWS + 1];
    int STX[SPLAT_MAX_VIEWS];
    uint2* rec;                    // [V * n] (super-rectangle x0 | y0 << 8 | x1 << 16 | y1 << 24, depth bits)
    uint32_t* cell;                // [copies][total_super][nbins] entry counts (zeroed), then cursors
    uint2* entries;                // out: (row, depth bits) of the lists' entries, by cell
    int64_t capacity;
    // k_cell_scan
    unsigned long long* lb;        // [total_super] look-back words (zeroed)
    uint32_t* ticket;              // (zeroed)
    uint2* sranges;                // out: [total_super] [start, end) of each list, (0, 0) when empty
    int64_t* K1;                   // out: entries of all lists
    uint4* queue;                  // out: units (start, end, super-tile, part or kWholeUnit); those of the
                                   // head from the front, the others from the back
    uint32_t* n_queue;             // [2] their counts (zeroed)
    int64_t queue_cap;
    int total_super;
    int long_heads;                // head_reach
    int32_t* status;
    int64_t spin_limit;
    // zeroed by k_cell_count (the results of a call that stops early)
    uint2* ranges;
    int64_t total_tiles;
    int64_t* n_instances;
    int64_t* n_needed;             // may be null
};

constexpr uint32_t kSplitBins = 32;  // range.y of a view whose bins are bounded by kSplits sampled entries
constexpr int kSplits = 256;         // samples per view, one per thread of the count

// An entry's place in a list's order, rows counted inside the view.
__device__ __forceinline__ unsigned long long place_of(uint32_t key, uint32_t i)
{
    return (unsigned long long)key << 32 | i;
}

// Bin of row i of a view; monotone in (key, i).  range: first depth bits, shift.  split: kSplits ascending bounds
// in shared memory, for kSplitBins.
__device__ __forceinline__ uint32_t depth_bin(uint2 range, int nbins, uint32_t key, uint32_t i,
                                              const unsigned long long* split)
{
    if (range.y == kSplitBins) {
        const unsigned long long e = place_of(key, i);
        uint32_t at = 0;  // bounds at or before e, 256 counting as 255
#pragma unroll
        for (int step = kSplits / 2; step > 0; step >>= 1)
            if (split[at + step - 1] <= e) at += step;
        if (nbins < 4 * kSplits) return nbins >= kSplits ? at : at * (uint32_t)nbins / kSplits;
        // four equal steps between two bounds
        const unsigned long long lo = at > 0 ? split[at - 1] : 0ull, w = (split[at] - lo) >> 2;
        return 4u * at + (e >= lo + w) + (e >= lo + 2 * w) + (e >= lo + 3 * w);
    }
    return key > range.x ? min((key - range.x) >> range.y, (uint32_t)nbins - 1u) : 0u;
}

// Depth bins of view v: equal steps of the depth bits over their range among 256
// of its rows, one per thread, one from each of 256 runs of rows (at a scattered
// place in the run: rows may come in a regular order).  About one row in 128 lies
// outside; a camera far from a small scene, whose depths share their leading bits,
// gets as fine a division as any other (bins of a fixed part of an octave held a
// list's whole depth range: 1060 against 340 us for 1M Gaussians seen from 40 times
// their extent).  Where many pairs of samples share a bin, the rows lie on few
// depths: a plane that faces the camera, a flat scene.  The samples themselves,
// ordered by depth and row, bound the bins then, so that no bin of a list gets
// long, whatever the depths: a long bin is sorted by blocks that each read all of
// it.  1M rows in 128x128, all at one depth 1332 -> 240 us, at two 815 -> 282; 300k
// 276 -> 106 and 257 -> 104 (the radix sort of all rows took 283 and 200).  The test of
// the samples costs nothing that shows.
__device__ __forceinline__ uint2 sample_range(const CellArgs& a, int v, uint32_t (*s_mm)[8], unsigned long long* s_split)
{
    const uint32_t tid = threadIdx.x;
    const uint32_t step = a.n >= kSplits ? (uint32_t)(a.n / kSplits) : 1u;
    const uint32_t i = tid * step + (tid * 0x9e3779b9u >> 8) % step;
    uint32_t lo = 0xffffffffu, hi = 0u;
    if (i < a.n) {
        const int64_t r = (int64_t)v * a.n + i;
        const uint32_t nt = a.proj.n_tiles[r];
        const uint32_t key = __float_as_uint(((const float4*)a.proj.rgb_depth)[r].w);
        if (nt > 0) lo = hi = key;
    }
    const bool seen = lo <= hi;
    const uint32_t key = lo;
    uint32_t* s_key = (uint32_t*)s_split;
    s_key[tid] = key;
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((tid & 31) == 0) {
        s_mm[0][tid >> 5] = lo;
        s_mm[1][tid >> 5] = hi;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        lo = min(lo, s_mm[0][w]);
        hi = max(hi, s_mm[1][w]);
    }
    if (lo > hi) return make_uint2(0u, 31u);  // none visible in the sample
    const uint2 range = make_uint2(lo, (uint32_t)min(31, max(0, 32 - __clz(hi - lo) - a.bin_bits)));
    // pairs of a scattered pairing (neighbours may be alike): a share p of the samples in one bin makes 256 p^2 of
    // them, a sixth 7; rows spread evenly over the bins make one in four batches of 1024 bins, and 4 of 64
    const uint32_t other = s_key[(77u * tid + 31u) & 255u];
    const int pairs = __syncthreads_count(seen && other != 0xffffffffu &&
                                          depth_bin(range, a.nbins, key, 0u, nullptr) ==
                                              depth_bin(range, a.nbins, other, 0u, nullptr));
    if (pairs < (a.nbins >= kSplits ? 8 : 32)) return range;
    // order the samples by counting the smaller ones; those not seen come last
    const unsigned long long e = seen ? place_of(key, i) : place_of(0xffffffffu, 0xffffff00u + tid);
    s_split[kSplits + tid] = e;
    __syncthreads();
    int at = 0;
    for (int q = 0; q < kSplits; ++q) at += s_split[kSplits + q] < e;
    s_split[at] = e;
    __syncthreads();
    return make_uint2(0u, kSplitBins);
}

// The cells of the rows of count block `block` (the same in k_cell_count and k_cell_scatter).
// Atomics on one cell, and on cells that share a sector, go one after the
// other; where a batch has few super-tiles, or most rows lie in a few of them,
// several copies of the cells spread them.
__device__ __forceinline__ uint32_t* cell_copy(const CellArgs& a, unsigned block)
{
    return a.cell + ((size_t)(block & (a.copies - 1)) * a.total_super << a.bin_bits);
}

// Two rows per thread, blockIdx.y the view.  Each lane walks its own
// super-rectangle: the reductions return nothing, so a warp only pays issue
// slots for its widest row (sharing the entries out over the lanes, as the
// scatter does, costs the same on wide splats and more on small ones).
__global__ void __launch_bounds__(256) k_cell_count(CellArgs a)
{
    wait_for_previous_kernel();
    __shared__ uint32_t s_mm[2][8];
    __shared__ unsigned long long s_split[2 * kSplits];
    const int v = blockIdx.y;
    const int64_t gt = ((int64_t)v * gridDim.x + blockIdx.x) * 256 + threadIdx.x;
    for (int64_t t = gt; t < a.total_tiles; t += (int64_t)gridDim.x * gridDim.y * 256) a.ranges[t] = make_uint2(0u, 0u);
    if (gt == 0) {
        *a.n_instances = 0;
        if (a.n_needed) *a.n_needed = 0;
    }
    if (status_failed(a.status)) return;
    // (all at once: most rows are visible, and the loads' latency bounds the kernel)
    uint32_t nt[kRowsPerThread];
    int4 rc[kRowsPerThread];
    float depth[kRowsPerThread];
#pragma unroll
    for (int q = 0; q < kRowsPerThread; ++q) {
        const int64_t i = (blockIdx.x * kRowsPerThread + q) * 256ll + threadIdx.x, r = (int64_t)v * a.n + i;
        nt[q] = 0u;
        if (i < a.n) {
            nt[q] = a.proj.n_tiles[r];
            rc[q] = ((const int4*)a.proj.rect)[r];
            depth[q] = ((const float4*)a.proj.rgb_depth)[r].w;
        }
    }
    const uint2 range = sample_range(a, v, s_mm, s_split);
    uint32_t* cells = cell_copy(a, blockIdx.x);
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) a.range[v] = range;
        if (range.y == kSplitBins) a.split[v * kSplits + threadIdx.x] = s_split[threadIdx.x];
    }
#pragma unroll
    for (int q = 0; q < kRowsPerThread; ++q) {
        const int64_t i = (blockIdx.x * kRowsPerThread + q) * 256ll + threadIdx.x;
        if (i >= a.n) continue;
        uint32_t pack = 0u, key = 0u;
        if (nt[q] > 0) {
            key = __float_as_uint(depth[q]);
            const int x0 = rc[q].x >> 3, y0 = rc[q].y >> 3, x1 = (rc[q].z + 7) >> 3, y1 = (rc[q].w + 7) >> 3;
            if (x1 > x0 && y1 > y0) {
                pack = (uint32_t)x0 | (uint32_t)y0 << 8 | (uint32_t)x1 << 16 | (uint32_t)y1 << 24;
                const uint32_t bin = depth_bin(range, a.nbins, key, (uint32_t)i, s_split);
                for (int y = y0; y < y1; ++y) {
                    uint32_t* c = cells + (size_t)(a.super_base[v] + y * a.STX[v]) * a.nbins + bin;
                    for (int x = x0; x < x1; ++x) atomicAdd(c + (size_t)x * a.nbins, 1u);
                }
            }
        }
        a.rec[(int64_t)v * a.n + i] = make_uint2(pack, key);
    }
}

// First index of the ascending p[0 .. n) with p[index] >= x (n when none).
__device__ __forceinline__ int lower_bound(const uint32_t* p, int n, uint32_t x)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        const int m = (lo + hi) >> 1;
        if (p[m] < x) lo = m + 1;
        else hi = m;
    }
    return lo;
}

// Block per super-tile, taken in ticket order (look-back over the super-tiles).
__global__ void __launch_bounds__(256) k_cell_scan(CellArgs a)
{
    wait_for_previous_kernel();
    __shared__ uint32_t s_p[kMaxBins + 1];  // first entry of each bin, relative to the list
    __shared__ uint32_t s_tmp[8];
    __shared__ unsigned long long s_excl;
    __shared__ int s_gs;
    constexpr unsigned long long kA = 1ull << 62, kP = 2ull << 62, kM = (1ull << 62) - 1;
    if (block_failed(a.status)) return;
    const int tid = threadIdx.x;
    if (tid == 0) s_gs = (int)atomicAdd(a.ticket, 1u);
    __syncthreads();
    const int gs = s_gs;
    if (gs >= a.total_super) return;
    uint32_t* cell = a.cell + (size_t)gs * a.nbins;
    const size_t copy_stride = (size_t)a.total_super << a.bin_bits;
    uint32_t c[4] = {0u, 0u, 0u, 0u};
    const bool quad = a.nbins == kMaxBins;  // four bins per thread, else one
    for (int k = 0; k < a.copies; ++k) {
        if (quad) {
            const uint4 q = ((const uint4*)(cell + k * copy_stride))[tid];
            c[0] += q.x; c[1] += q.y; c[2] += q.z; c[3] += q.w;
        } else if (tid < a.nbins) {
            c[0] += cell[k * copy_stride + tid];
        }
    }
    uint32_t n;
    uint32_t p = block_excl_scan256(c[0] + c[1] + c[2] + c[3], s_tmp, &n);
    if (quad) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            s_p[4 * tid + q] = p;
            p += c[q];
        }
    } else if (tid < a.nbins) {
        s_p[tid] = p;
    }
    if (tid == 0) s_p[a.nbins] = n;
    if (tid < 32) {  // decoupled look-back by one warp, 32 predecessors per round trip
        unsigned long long excl = 0;
        if (tid == 0) st_relaxed64(a.lb + gs, (gs == 0 ? kP : kA) | n);
        if (gs > 0) {
            int64_t j = gs - 1, spins = 0;
            for (;;) {
                const unsigned long long w = j - tid >= 0 ? ld_relaxed64(a.lb + (j - tid)) : kP;
                const unsigned long long flag = w & ~kM;
                const unsigned pend = __ballot_sync(0xffffffffu, flag == 0);
                const unsigned pref = __ballot_sync(0xffffffffu, flag == kP);
                const int first_pend = pend ? __ffs(pend) - 1 : 32;
                const int first_pref = pref ? __ffs(pref) - 1 : 32;
                const bool found = first_pref < first_pend;
                const int take = found ? first_pref + 1 : first_pend;
                unsigned long long x = tid < take ? (w & kM) : 0ull;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                excl += x;
                if (found) break;
                j -= take;
                if (take == 0) {
                    if (++spins > a.spin_limit) {
                        if (tid == 0) set_status(a.status, SPLAT_ERR_TIMEOUT, SPLAT_STAGE_SCAN, gs);
                        break;
                    }
                    if (spins > 64) __nanosleep(64);
                }
            }
            if (tid == 0) st_relaxed64(a.lb + gs, kP | ((excl + n) & kM));
        }
        if (tid == 0) {
            s_excl = excl;
            if (gs == a.total_super - 1) {
                const int64_t K1 = (int64_t)(excl + n);
                *a.K1 = K1;
                if (K1 > a.capacity) set_status(a.status, SPLAT_ERR_CAPACITY, SPLAT_STAGE_SCAN, K1);
            }
        }
    }
    __syncthreads();
    // (starts past 2^32 only arise with K1 beyond any capacity: the check above reports them)
    const uint32_t start = (uint32_t)s_excl;
    if (quad) {  // a bin's copies follow one another
        uint4 at = make_uint4(start + s_p[4 * tid], start + s_p[4 * tid + 1], start + s_p[4 * tid + 2],
                              start + s_p[4 * tid + 3]);
        for (int k = 0; k < a.copies; ++k) {
            uint4* q = (uint4*)(cell + k * copy_stride) + tid;
            const uint4 x = a.copies > 1 ? *q : make_uint4(0u, 0u, 0u, 0u);
            *q = at;
            at.x += x.x; at.y += x.y; at.z += x.z; at.w += x.w;
        }
    } else if (tid < a.nbins) {
        uint32_t at = start + s_p[tid];
        for (int k = 0; k < a.copies; ++k) {
            const uint32_t x = cell[k * copy_stride + tid];
            cell[k * copy_stride + tid] = at;
            at += x;
        }
    }
    if (tid == 0) a.sranges[gs] = n ? make_uint2(start, start + n) : make_uint2(0u, 0u);
    if (n <= (uint32_t)kUnit) return;  // one unit, sorted with the head's without a queue entry
    const uint32_t steps = (n + kUnitStep - 1) / kUnitStep;
    for (uint32_t k = tid; k < steps; k += 256) {
        const uint32_t u0 = s_p[lower_bound(s_p, a.nbins, k * kUnitStep)];
        const uint32_t u1 = s_p[lower_bound(s_p, a.nbins, (k + 1) * kUnitStep)];
        if (u0 >= u1) continue;  // inside a bin of more than kUnitStep entries
        const int q = u0 < head_reach(n, a.long_heads) ? 0 : 1;
        const uint32_t parts = u1 - u0 <= (uint32_t)kUnit ? 1u : (u1 - u0 + kUnitStep - 1) / kUnitStep;
        const uint32_t at = atomicAdd(&a.n_queue[q], parts);
        for (uint32_t g = 0; g < parts; ++g) {
            const int64_t slot = q ? a.queue_cap - 1 - (int64_t)(at + g) : (int64_t)(at + g);
            if (slot >= 0 && slot < a.queue_cap)  // (it holds every unit of lists within the capacity)
                a.queue[slot] = make_uint4(start + u0, start + u1, (uint32_t)gs, parts == 1 ? kWholeUnit : g);
        }
    }
}

// A warp takes 32 rows and shares their entries out over its lanes: the
// position of each comes back from an atomic on its cell's cursor, and a row's
// entries one after the other would wait for one another's.
__global__ void __launch_bounds__(256) k_cell_scatter(CellArgs a)
{
    wait_for_previous_kernel();
    if (status_failed(a.status)) return;  // includes K1 above the capacity
    const int v = blockIdx.y, lane = threadIdx.x & 31;
    const int64_t i = blockIdx.x * 256ll + threadIdx.x;
    const uint32_t row = (uint32_t)((int64_t)v * a.n + i);
    const uint2 rec = i < a.n ? a.rec[row] : make_uint2(0u, 0u);
    const uint32_t x0 = rec.x & 255u, y0 = rec.x >> 8 & 255u, w = (rec.x >> 16 & 255u) - x0;
    const uint32_t c = w * ((rec.x >> 24) - y0);
    // first cell of the row, and of its entries' order in the warp: lane l owns [e, e + c)
    const uint32_t cell0 = (uint32_t)(a.super_base[v] + (int)y0 * a.STX[v] + (int)x0);
    const uint2 range = a.range[v];
    __shared__ unsigned long long s_split[kSplits];
    if (range.y == kSplitBins) {  // (block-uniform)
        s_split[threadIdx.x] = a.split[v * kSplits + threadIdx.x];
        __syncthreads();
    }
    const uint32_t bin = depth_bin(range, a.nbins, rec.y, (uint32_t)i, s_split);
    uint32_t* cells = cell_copy(a, blockIdx.x / kRowsPerThread);
    uint32_t e = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, e, o);
        if (lane >= o) e += y;
    }
    const uint32_t E = __shfl_sync(0xffffffffu, e, 31);
    e -= c;
    for (uint32_t s0 = 0; s0 < E; s0 += 32 * kScatterRounds) {
        uint32_t pos[kScatterRounds], srow[kScatterRounds], skey[kScatterRounds];
#pragma unroll
        for (int q = 0; q < kScatterRounds; ++q) {  // the rounds' atomics are in flight together
            pos[q] = 0xffffffffu;
            if (s0 + 32 * q >= E) continue;  // warp-uniform
            const uint32_t s = s0 + 32 * q + lane;
            // the row of entry s: the last lane whose first entry is at or before it
            int src = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(0xffffffffu, e, src + step) <= s) src += step;
            const uint32_t k = s - __shfl_sync(0xffffffffu, e, src);
            const int sw = (int)__shfl_sync(0xffffffffu, w, src);
            const uint32_t sc = __shfl_sync(0xffffffffu, cell0, src), sbin = __shfl_sync(0xffffffffu, bin, src);
            skey[q] = __shfl_sync(0xffffffffu, rec.y, src);
            srow[q] = row - (uint32_t)(lane - src);
            // k / sw: an approximate quotient of (k + 1/2) / sw (off by at most one), then corrected
            int ky = sw ? (int)__fdividef((float)k + 0.5f, (float)sw) : 0, kx = (int)k - ky * sw;
            if (kx < 0) {
                --ky;
                kx += sw;
            } else if (kx >= sw && sw) {
                ++ky;
                kx -= sw;
            }
            if (s < E)
                pos[q] = atomicAdd(cells + (size_t)(sc + (uint32_t)(ky * a.STX[v] + kx)) * a.nbins + sbin, 1u);
        }
#pragma unroll
        for (int q = 0; q < kScatterRounds; ++q)
            if (pos[q] < (uint64_t)a.capacity) a.entries[pos[q]] = make_uint2(srow[q], skey[q]);
    }
}

constexpr int log2_of(int x) { return x > 1 ? 1 + log2_of(x / 2) : 0; }

struct SortArgs {
    const uint2* sranges;
    int total_super;
    const unsigned long long* entries;  // (row, depth bits) as one word: depth bits << 32 | row
    uint32_t* list;                     // out: the lists' rows in order
    const uint4* queue;
    const uint32_t* n_queue;
    int64_t queue_cap;
    const uint2* sat_head;              // the head count's ended tiles (second pass)
    int32_t* status;
};

// Of a block of THREADS that sorts kPer entries per thread, into as many buckets.
template <int THREADS>
struct SortSmem {
    static constexpr int kEntries = kPer * THREADS;
    unsigned long long e[kEntries];
    uint32_t h[kEntries + 4];   // bucket counts, then first positions; [kEntries]: the total
    uint32_t h2[kEntries + 4];  // the same of the second level
    uint16_t at[kEntries];      // arrival in a second-level bucket
    uint32_t red[4][THREADS / 32], tmp[THREADS / 32];
    uint32_t n;
    bool taken;                 // a part's entries are all in e
};
using UnitSmem = SortSmem<kUnitThreads>;

// Bounds of a key range and the right shift that maps its differences to
// 2^bits buckets (at least half of them used), order preserved.
struct KeyRange {
    unsigned long long lo;
    int shift;
};

__device__ __forceinline__ KeyRange key_range(unsigned long long lo, unsigned long long hi, int bits)
{
    return {lo, max(0, 64 - bits - __clzll((long long)(hi - lo)))};
}

__device__ __forceinline__ uint32_t key_bucket(const KeyRange& r, unsigned long long e)
{
    return (uint32_t)((e - r.lo) >> r.shift);
}

// Block-wide key range from the threads' own extremes of the depth bits and,
// should all depths be equal, of the rows.
template <int THREADS>
__device__ __forceinline__ void block_bounds(SortSmem<THREADS>& s, uint32_t dmin, uint32_t dmax, uint32_t rmin, uint32_t rmax,
                                             unsigned long long& lo, unsigned long long& hi)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    dmin = __reduce_min_sync(0xffffffffu, dmin);
    dmax = __reduce_max_sync(0xffffffffu, dmax);
    rmin = __reduce_min_sync(0xffffffffu, rmin);
    rmax = __reduce_max_sync(0xffffffffu, rmax);
    if (lane == 0) {
        s.red[0][warp] = dmin;
        s.red[1][warp] = dmax;
        s.red[2][warp] = rmin;
        s.red[3][warp] = rmax;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) {
        dmin = min(dmin, s.red[0][w]);
        dmax = max(dmax, s.red[1][w]);
        rmin = min(rmin, s.red[2][w]);
        rmax = max(rmax, s.red[3][w]);
    }
    lo = (unsigned long long)dmin << 32 | (dmin == dmax ? rmin : 0u);
    hi = (unsigned long long)dmax << 32 | (dmin == dmax ? rmax : 0xffffffffu);
}

// h: bucket counts -> first positions, the last the total; returns
// (block-uniform) whether a bucket is crowded.
template <int THREADS>
__device__ __forceinline__ bool scan_buckets(SortSmem<THREADS>& s, uint32_t* h)
{
    static_assert(kPer == 8, "eight buckets per thread");
    uint4* h4 = (uint4*)h + 2 * threadIdx.x;
    const uint4 c = h4[0], d = h4[1];
    const uint32_t mx = max(max(max(c.x, c.y), max(c.z, c.w)), max(max(d.x, d.y), max(d.z, d.w)));
    const uint32_t sc = c.x + c.y + c.z + c.w;
    uint32_t total;
    const uint32_t x = block_excl_scan<THREADS / 32>(sc + d.x + d.y + d.z + d.w, s.tmp, &total), y = x + sc;
    h4[0] = make_uint4(x, x + c.x, x + c.x + c.y, x + c.x + c.y + c.z);
    h4[1] = make_uint4(y, y + d.x, y + d.x + d.y, y + d.x + d.y + d.z);
    if (threadIdx.x == 0) h[kPer * THREADS] = total;
    return __syncthreads_or(mx > kCrowded);
}

// The second-level position of entry e, whose bucket is b: the bucket's first
// position, in a crowded bucket plus a share of its length linear in the row.
template <int THREADS>
__device__ __forceinline__ uint32_t second_level(const SortSmem<THREADS>& s, uint32_t b, uint32_t row, uint32_t rmin, int up)
{
    const uint32_t p = s.h[b], c = s.h[b + 1] - p;
    return c > kCrowded ? p + __umulhi((row - rmin) << up, c) : p;
}

// Sorts the P (a power of two) values of e in shared memory.
template <int THREADS>
__device__ __forceinline__ void sort_bitonic(unsigned long long* e, int P)
{
    for (int size = 2; size <= P; size <<= 1) {
        for (int step = size >> 1; step > 0; step >>= 1) {
            for (int t = threadIdx.x; t < P / 2; t += THREADS) {
                const int i = 2 * t - (t & (step - 1)), j = i + step;
                const unsigned long long x = e[i], y = e[j];
                if ((x > y) == ((i & size) == 0)) {
                    e[i] = y;
                    e[j] = x;
                }
            }
            __syncthreads();
        }
    }
}

// Sorts a unit of n <= kPer THREADS entries, entry t + THREADS k in e[k] of thread
// t, and writes their rows to dst: one counting-sort pass over buckets linear in
// the key (about one entry each), then every entry counts the smaller ones of its
// bucket.  Where a bucket is crowded (many equal depths: means stored in 16 bits
// seen along an axis, planes facing the camera), a second counting pass spreads
// the crowded buckets' entries over their positions by row; should such a bucket
// hold different depths, or the rows crowd as well, the unit is sorted
// bitonically.  (The second pass keeps its arrivals in shared memory: in
// registers they made the common path spill, 78 -> 118 us for the rest of the
// lists of 1M Gaussians at 4 x 2704x2028.)
template <int THREADS>
__device__ __forceinline__ void sort_unit(SortSmem<THREADS>& s, const unsigned long long (&e)[kPer], int n,
                                          uint32_t* dst)
{
    const int tid = threadIdx.x;
    uint32_t dmin = 0xffffffffu, dmax = 0u, rmin = 0xffffffffu, rmax = 0u;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if (tid + THREADS * k < n) {
            const uint32_t d = (uint32_t)(e[k] >> 32), r = (uint32_t)e[k];
            dmin = min(dmin, d);
            dmax = max(dmax, d);
            rmin = min(rmin, r);
            rmax = max(rmax, r);
        }
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) s.h[tid + THREADS * k] = 0u;
    unsigned long long lo, hi;
    block_bounds(s, dmin, dmax, rmin, rmax, lo, hi);
    const KeyRange kr = key_range(lo, hi, log2_of(kPer * THREADS));
    uint32_t at[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k)
        if (tid + THREADS * k < n) at[k] = atomicAdd(&s.h[key_bucket(kr, e[k])], 1u);
    __syncthreads();
    const bool crowded = scan_buckets(s, s.h);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if (tid + THREADS * k < n) {
            const uint32_t b = key_bucket(kr, e[k]);
            s.e[s.h[b] + at[k]] = e[k];
        }
    }
    __syncthreads();
    if (!crowded) {
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            if (tid + THREADS * k < n) {
                const uint32_t b = key_bucket(kr, e[k]), j1 = s.h[b + 1];
                uint32_t j = s.h[b], r = j;
                for (; j < j1; ++j) r += s.e[j] < e[k];
                at[k] = r;
            }
        }
        __syncthreads();
        uint32_t* rows = (uint32_t*)s.e;
#pragma unroll
        for (int k = 0; k < kPer; ++k)
            if (tid + THREADS * k < n) rows[at[k]] = (uint32_t)e[k];
        __syncthreads();
        for (int i = tid; i < n; i += THREADS) dst[i] = rows[i];
    } else {
        rmin = 0xffffffffu;
        rmax = 0u;
        for (int w = 0; w < THREADS / 32; ++w) {  // the block's bounds of the rows, as block_bounds left the warps'
            rmin = min(rmin, s.red[2][w]);
            rmax = max(rmax, s.red[3][w]);
        }
        const int up = __clz(max(1u, rmax - rmin));
        for (int i = tid; i < kPer * THREADS; i += THREADS) s.h2[i] = 0u;
        __syncthreads();
        bool mixed = false;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            if (tid + THREADS * k < n) {
                const uint32_t b = key_bucket(kr, e[k]);
                const uint32_t p = second_level(s, b, (uint32_t)e[k], rmin, up);
                mixed |= s.h[b + 1] - s.h[b] > kCrowded && (s.e[s.h[b]] >> 32) != (e[k] >> 32);
                s.at[tid + THREADS * k] = (uint16_t)atomicAdd(&s.h2[p], 1u);
            }
        }
        mixed = __syncthreads_or(mixed);
        if (!mixed) mixed = scan_buckets(s, s.h2);
        if (!mixed) {
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                if (tid + THREADS * k < n) {
                    const uint32_t p = second_level(s, key_bucket(kr, e[k]), (uint32_t)e[k], rmin, up);
                    s.e[s.h2[p] + s.at[tid + THREADS * k]] = e[k];
                }
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                if (tid + THREADS * k < n) {
                    const uint32_t p = second_level(s, key_bucket(kr, e[k]), (uint32_t)e[k], rmin, up);
                    const uint32_t j1 = s.h2[p + 1];
                    uint32_t j = s.h2[p], r = j;
#pragma unroll 1
                    for (; j < j1; ++j) r += s.e[j] < e[k];
                    dst[r] = (uint32_t)e[k];
                }
            }
        } else {
            int P = 2;
            while (P < n) P <<= 1;
            for (int i = n + tid; i < P; i += THREADS) s.e[i] = ~0ull;
            __syncthreads();
            sort_bitonic<THREADS>(s.e, P);
            for (int i = tid; i < n; i += THREADS) dst[i] = (uint32_t)s.e[i];
        }
    }
    __syncthreads();
}

// f(entry) for every one of src[0 .. n), eight loads in flight per thread (with
// one a long unit is bound by their latency: 545 -> 160 us for a view whose
// 300k rows all share one depth).
template <typename F>
__device__ __forceinline__ void each_entry(const unsigned long long* src, uint32_t n, F f)
{
    for (uint32_t i0 = threadIdx.x; i0 < n; i0 += 8 * kUnitThreads) {
        unsigned long long x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = i0 + (uint32_t)kUnitThreads * k < n ? src[i0 + (uint32_t)kUnitThreads * k] : 0ull;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (i0 + (uint32_t)kUnitThreads * k < n) f(x[k]);
    }
}

// Bucket counts (scanned, in s.h) of those of src[0 .. n) within [lo, hi].
__device__ __forceinline__ KeyRange count_range(UnitSmem& s, const unsigned long long* src, uint32_t n,
                                                unsigned long long lo, unsigned long long hi)
{
    const KeyRange kr = key_range(lo, hi, kSortBucketBits);
    for (int k = threadIdx.x; k < kSortBuckets; k += kUnitThreads) s.h[k] = 0u;
    __syncthreads();
    each_entry(src, n, [&](unsigned long long e) {
        if (e >= lo && e <= hi) atomicAdd(&s.h[(e - lo) >> kr.shift], 1u);
    });
    __syncthreads();
    scan_buckets(s, s.h);
    return kr;
}

// Part g of a unit of more than kUnit entries (one depth bin of a crowded
// list): the parts' blocks each read the whole unit and take the entries between
// two of its sorted samples, about kUnitStep of them, so that any number of
// blocks share a long unit without waiting for one another.  (Samples, not equal
// steps of the key: where many entries share one depth next to others, the steps
// would hold them all in one part: 84 ms for 500k of them.)
// Sets the value range [lo, hi] of the part, the number of its entries and their
// first position in the unit, and leaves the entries in s.e if they are no more
// than kUnit.
__device__ __noinline__ void part_range(UnitSmem& s, const unsigned long long* src, uint32_t n, uint32_t g,
                                        unsigned long long& lo, unsigned long long& hi, uint32_t& left, uint32_t& out)
{
    const uint32_t tid = threadIdx.x, parts = (n + kUnitStep - 1) / kUnitStep;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const unsigned long long i = tid + kUnitThreads * k;
        s.e[i] = src[i * n / kUnit];
    }
    __syncthreads();
    sort_bitonic<kUnitThreads>(s.e, kUnit);
    lo = g > 0 ? s.e[(unsigned long long)g * kUnit / parts] : 0ull;
    hi = g + 1 < parts ? s.e[(unsigned long long)(g + 1) * kUnit / parts] - 1 : ~0ull;
    if (tid == 0) s.n = s.red[0][0] = 0u;
    __syncthreads();
    uint32_t below = 0u;
    each_entry(src, n, [&](unsigned long long e) {
        below += e < lo;
        if (e >= lo && e <= hi) {
            const uint32_t at = atomicAdd(&s.n, 1u);
            if (at < (uint32_t)kUnit) s.e[at] = e;
        }
    });
    below = __reduce_add_sync(0xffffffffu, below);
    if ((tid & 31) == 0) atomicAdd(&s.red[0][0], below);
    __syncthreads();
    left = s.n;
    out = s.red[0][0];
    if (tid == 0) s.taken = left <= (uint32_t)kUnit;
    __syncthreads();
}

// The first up to kUnit entries by value of a part's `left` ones in [lo, hi] into
// s.e, unless part_range left them there: returns their number and the value top up to which they go (0: none).  A
// part that holds more than kUnit (one crowded bucket) goes through several of
// these, each found by counting again over ever finer buckets (entries are unique,
// so this ends).
__device__ __noinline__ uint32_t take_range(UnitSmem& s, const unsigned long long* src, uint32_t n, uint32_t left,
                                            unsigned long long& lo, unsigned long long hi, unsigned long long& top)
{
    const int tid = threadIdx.x;
    top = hi;
    if (s.taken) return left;
    uint32_t m = left;
    while (m > (uint32_t)kUnit && lo < top) {
        const KeyRange kr = count_range(s, src, n, lo, top);
        // the buckets below b hold at most kUnit entries, those up to and including b more
        const int b = lower_bound(s.h, kSortBuckets, kUnit + 1) - 1;
        m = s.h[b];
        if (m == 0) {  // bucket b alone holds too many
            m = s.h[b + 1];
            lo += (unsigned long long)b << kr.shift;
            top = min(top, lo + (1ull << kr.shift) - 1);
        } else {
            top = lo + ((unsigned long long)b << kr.shift) - 1;
        }
        __syncthreads();
    }
    m = min(min(m, left), (uint32_t)kUnit);
    if (m == 0) return 0u;  // (not for consistent counts: bounds the loop whatever the buffer holds)
    if (tid == 0) s.n = 0u;
    __syncthreads();
    each_entry(src, n, [&](unsigned long long x) {
        if (x >= lo && x <= top) {
            const uint32_t at = atomicAdd(&s.n, 1u);
            if (at < (uint32_t)kUnit) s.e[at] = x;
        }
    });
    __syncthreads();
    return m;
}

// REST false: the lists of at most kUnit entries and the longer lists' units
// that hold their head's entries; true: the longer lists' other units,
// where a tile's list goes on past the head.
template <bool REST>
__global__ void __launch_bounds__(kUnitThreads, 4) k_unit_sort(SortArgs a)
{
    wait_for_previous_kernel();
    __shared__ UnitSmem s;
    if (status_failed(a.status)) return;
    const uint32_t direct = REST ? 0u : (uint32_t)a.total_super;
    const uint32_t items = direct + a.n_queue[REST ? 1 : 0];
    for (uint32_t it = blockIdx.x; it < items; it += gridDim.x) {
        uint32_t st, en, part = kWholeUnit;
        if (!REST && it < direct) {
            const uint2 rg = a.sranges[it];
            st = rg.x;
            en = rg.y - rg.x <= (uint32_t)kUnit ? rg.y : rg.x;
        } else {
            const int64_t q = it - direct;
            const uint4 u = a.queue[REST ? a.queue_cap - 1 - q : q];
            st = u.x;
            en = u.y;
            part = u.w;
            if (REST) {
                const uint2 sat = a.sat_head[u.z];
                if ((sat.x & sat.y) == 0xffffffffu) continue;  // every list of the super-tile ended in the head
            }
        }
        if (st >= en) continue;  // (block-uniform)
        const uint32_t n = en - st;
        unsigned long long lo = 0ull, hi = ~0ull;
        uint32_t left = n, out = 0u;
        if (part != kWholeUnit) part_range(s, a.entries + st, n, part, lo, hi, left, out);
        while (left > 0) {  // (block-uniform) once for a whole unit
            uint32_t m = left;
            unsigned long long top = hi;
            unsigned long long e[kPer];
            if (part == kWholeUnit) {
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    const uint32_t i = threadIdx.x + kUnitThreads * k;
                    e[k] = i < n ? a.entries[st + i] : 0ull;
                }
            } else {
                m = take_range(s, a.entries + st, n, left, lo, hi, top);
                if (m == 0) break;
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    const uint32_t i = threadIdx.x + kUnitThreads * k;
                    e[k] = i < m ? s.e[i] : 0ull;
                }
                __syncthreads();
            }
            sort_unit(s, e, (int)m, a.list + st + out);
            out += m;
            left -= m;
            lo = top + 1;
        }
    }
}

// The sorted super-tile lists of a call with few rows, in one kernel: a block per
// super-tile reads every row of its view, keeps the entries of its own list in
// shared memory and sorts them there (sort_unit).  The list starts behind the
// entries of the super-tiles before it, which the block counts from the same
// rectangles (and those of the earlier views), so blocks do not wait for one
// another.  A block also clears what the later passes count in.  Where a call is as
// small as this, the kernels above are bound by their launches and first loads:
// 4096 rows in 128x128 sort in 40 us instead of 50, 8192 rows in 1600x1400 (143
// super-tiles) in 48 instead of 60.
constexpr int kSmallThreads = 1024;
constexpr int64_t kSmallRows = kPer * kSmallThreads;  // a list holds at most every row

struct SmallArgs {
    CellArgs c;
    uint32_t* list;  // out: the lists' rows in order
    uint32_t* zero;  // cleared
    int n_zero;
};

__global__ void __launch_bounds__(kSmallThreads) k_small_lists(SmallArgs s)
{
    wait_for_previous_kernel();
    extern __shared__ __align__(16) unsigned char smem[];
    SortSmem<kSmallThreads>& m = *(SortSmem<kSmallThreads>*)smem;
    const CellArgs& a = s.c;
    const int tid = threadIdx.x, lane = tid & 31, gs = blockIdx.x;
    for (int64_t t = gs * (int64_t)kSmallThreads + tid; t < a.total_tiles; t += (int64_t)gridDim.x * kSmallThreads)
        a.ranges[t] = make_uint2(0u, 0u);
    if (gs == 0) {
        for (int i = tid; i < s.n_zero; i += kSmallThreads) s.zero[i] = 0u;
        if (tid == 0) {
            *a.n_instances = 0;
            if (a.n_needed) *a.n_needed = 0;
        }
    }
    if (tid == 0) m.n = 0u;
    if (block_failed(a.status)) return;  // (the last super-tile's block sets it)
    int v = 0;
    for (int q = 1; q < a.V; ++q)
        if (gs >= a.super_base[q]) v = q;
    const int ls = gs - a.super_base[v], sy = ls / a.STX[v], sx = ls - sy * a.STX[v];
    // rows of this view and the views before it, at most 4 kPer per thread, four with all their loads in flight
    const int first = (int)(v * a.n), end = first + (int)a.n;
    uint32_t before = 0u;  // entries of the lists before this one
    for (int r0 = tid; r0 - tid < end; r0 += 4 * kSmallThreads) {
        uint32_t nt[4];
        int4 rc[4];
        float depth[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int r = r0 + kSmallThreads * k;
            nt[k] = 0u;
            if (r < end) {
                nt[k] = a.proj.n_tiles[r];
                rc[k] = ((const int4*)a.proj.rect)[r];
                depth[k] = ((const float4*)a.proj.rgb_depth)[r].w;
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int r = r0 + kSmallThreads * k;
            bool in = false;
            if (nt[k] > 0) {
                const int x0 = rc[k].x >> 3, y0 = rc[k].y >> 3, x1 = (rc[k].z + 7) >> 3, y1 = (rc[k].w + 7) >> 3;
                if (x1 > x0 && y1 > y0) {
                    const int w = x1 - x0;
                    if (r < first) {
                        before += (uint32_t)(w * (y1 - y0));
                    } else {
                        const bool row_in = sy >= y0 && sy < y1;
                        before += (uint32_t)(w * min(max(sy - y0, 0), y1 - y0) + (row_in ? min(max(sx - x0, 0), w) : 0));
                        in = row_in && sx >= x0 && sx < x1;
                    }
                }
            }
            const unsigned hits = __ballot_sync(0xffffffffu, in);
            if (!hits) continue;
            uint32_t at = 0u;
            if (lane == 0) at = atomicAdd(&m.n, (uint32_t)__popc(hits));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(hits & lanemask_lt());
            if (in) m.e[at] = (unsigned long long)__float_as_uint(depth[k]) << 32 | (uint32_t)r;
        }
    }
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0) m.tmp[tid >> 5] = before;
    __syncthreads();
    const uint32_t n = m.n;
    uint32_t start = __reduce_add_sync(0xffffffffu, m.tmp[lane]);
    if (tid == 0) {
        a.sranges[gs] = n ? make_uint2(start, start + n) : make_uint2(0u, 0u);
        if (gs == a.total_super - 1) {
            const int64_t K1 = (int64_t)start + n;
            *a.K1 = K1;
            if (K1 > a.capacity) set_status(a.status, SPLAT_ERR_CAPACITY, SPLAT_STAGE_SCAN, K1);
        }
    }
    if (!n || (int64_t)start + n > a.capacity) return;  // (block-uniform)
    unsigned long long e[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const uint32_t i = tid + kSmallThreads * k;
        e[k] = i < n ? m.e[i] : 0ull;
    }
    __syncthreads();
    sort_unit<kSmallThreads>(m, e, (int)n, s.list + start);
}

// Tiles in decreasing order of list length for the compositing kernels'
// scheduling (the longest first, so that the last wave of warps is short):
// classes of eight per power of two (the three bits after the leading one),
// a counting sort over the classes in two grid-wide passes (class counts,
// then each tile's slot from its class start and a class cursor), the order
// inside a class unspecified.  Greedy scheduling of the bench scene's measured
// walks on the compositing kernels' 2432 warp slots ends 7.7% above the ideal
// with one class per power of two and 2.9% above with eight (2.8% with the
// exact order).  cls[0..kOrderClasses): counts, then as many cursors, all zero
// on entry.  Lanes of a warp in the same class touch its counter once.
constexpr uint32_t kOrderClasses = 32 * 8 + 1;  // class 0: empty lists

__device__ __forceinline__ uint32_t length_class(uint32_t c)
{
    if (!c) return 0u;
    const int e = 31 - __clz(c);  // c in [2^e, 2^(e+1))
    const uint32_t f = (e >= 3 ? c >> (e - 3) : c << (3 - e)) & 7u;
    return 1u + 8u * (uint32_t)e + f;
}

__device__ __forceinline__ uint32_t tile_class(const uint2* ranges, int i)
{
    const uint2 r = ranges[i];
    return length_class(r.y - r.x);
}

template <bool SCATTER>
__global__ void __launch_bounds__(256) k_tile_order(const uint2* ranges, int n, uint32_t* cls, uint32_t* order,
                                                    int32_t* status)
{
    wait_for_previous_kernel();
    __shared__ uint32_t s_start[kOrderClasses];
    __shared__ uint32_t s_tmp[8];
    if (status_failed(status)) return;
    const int lane = threadIdx.x & 31;
    if (SCATTER) {
        // class starts, the longest class first: thread t takes class
        // kOrderClasses - 1 - t; the empty lists (class 0) go last
        const uint32_t cb = kOrderClasses - 1u - threadIdx.x;
        uint32_t total;
        const uint32_t ex = block_excl_scan256(cls[cb], s_tmp, &total);
        s_start[cb] = ex;
        if (threadIdx.x == 0) s_start[0] = total;
        __syncthreads();
    }
    const int stride = gridDim.x * blockDim.x;
    for (int i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < n; i0 += stride) {  // warp-uniform
        const int i = i0 + lane;
        const uint32_t c = i < n ? tile_class(ranges, i) : kOrderClasses;
        const unsigned peers = __match_any_sync(0xffffffffu, c);
        const int leader = __ffs(peers) - 1;
        uint32_t base = 0;
        if (lane == leader && c < kOrderClasses)
            base = atomicAdd(&cls[SCATTER ? kOrderClasses + c : c], (uint32_t)__popc(peers));
        if (SCATTER) {
            base = __shfl_sync(0xffffffffu, base, leader);
            if (c < kOrderClasses) order[s_start[c] + base + __popc(peers & lanemask_lt())] = (uint32_t)i;
        }
    }
}

// counted: the class counts are already in place (and the cursors zero), from
// the binned path's tile ranges
static cudaError_t launch_tile_order(const splat_bins& bins, int64_t total_tiles, uint32_t* cls, int32_t* status,
                                     const LaunchCtx& ctx, bool counted = false)
{
    if (!bins.tile_order || total_tiles <= 0) return cudaSuccess;
    const int n = (int)total_tiles;
    const int blocks = (int)std::min<int64_t>((total_tiles + 255) / 256, (int64_t)ctx.num_sms * 4);
    if (!counted) {
        cudaError_t e = cudaMemsetAsync(cls, 0, 2 * kOrderClasses * sizeof(uint32_t), ctx.stream);
        if (e != cudaSuccess) return e;
        count_launch();
        launch_kernel(k_tile_order<false>, blocks, 256, 0, ctx.stream, (const uint2*)bins.ranges, n, cls, bins.tile_order, status);
    }
    count_launch();
    launch_kernel(k_tile_order<true>, blocks, 256, 0, ctx.stream, (const uint2*)bins.ranges, n, cls, bins.tile_order, status);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Tile level.  Counting passes over each super-tile's list (the head in order,
// the tail in segments) give every tile's counts, k_tile_ranges turns them
// into ranges (and K), and the writing passes emit the lists.
// ---------------------------------------------------------------------------

struct TileArgs {
    splat_proj proj;
    int V;
    int64_t n_rows;
    int total_tiles;
    int tile_base[SPLAT_MAX_VIEWS + 1];
    int TX[SPLAT_MAX_VIEWS], TY[SPLAT_MAX_VIEWS];
    uint32_t* tile_total;
    // per-super-tile filter
    const uint32_t* list;             // rows grouped by super-tile, depth order inside
    const uint2* sranges;             // [total_super]
    int total_super;
    int super_base[SPLAT_MAX_VIEWS + 1];
    int STX[SPLAT_MAX_VIEWS];
    const uint2* ranges;              // tile ranges (cursor starts)
    uint32_t* vals_out;
    uint32_t* keys_out;               // may be null
    int cull;                         // drop tiles the opacity footprint cannot reach
    int W[SPLAT_MAX_VIEWS], H[SPLAT_MAX_VIEWS];
    uint2* sat_head;                  // [total_super] tiles (bit 8 r + c) whose lists ended in the head
    uint2* n_head;                    // [total_super] entries the head's two halves (tile rows 0-3, 4-7) went through
    int long_heads;                   // head_reach
    uint32_t* seg_base;               // [total_super + 1] first tail segment of each super-tile
    uint32_t* seg_super;              // [segments] super-tile of each tail segment
    uint32_t* seg_cnt;                // [segments][64] per-segment tile counts, then offsets
    uint2* mask;                      // coverage: 8 bytes per super-tile list entry, by groups of 32 entries of
                                      // a head or segment: word t of a full group holds the entries listed in
                                      // tile t (bit e: entry e); a last, partial group keeps one word pair per
                                      // entry (bit t: listed in tile t)
    uint32_t* ticket;                 // [3] tickets of the writing and tail counting passes, head count
                                      // CTAs done (zeroed)
    int32_t* status;
    unsigned long long* stats;        // diagnostic (may be null): [4] super-tiles whose lists ended in
                                      // the head for some tiles and continue in tail segments for others,
                                      // [5] tail segments
};

// Tile saturation.  Every pixel of a tile stops its walk before the first
// entry that would take its transmittance T below 1e-4 (Alg. 1), so the
// entries of a tile list that come after the point where T is certainly below
// that bound at every pixel of the tile are never read.  For each (entry,
// tile) the count pass takes a lower bound of the alpha the compositing
// kernels compute at every pixel of the tile (clipped to the image):
// alpha_max exp(-q/2) with q the largest value of the conic's quadratic form
// over the tile's corners (the form is convex), q enlarged to cover FP32
// rounding, provided the bound passes the 1/255 skip with a margin and the
// conic is far enough from singular that the kernels' evaluation of the power
// cannot round to the wrong side of 0.  The head pass sums -ln(1 - alpha)
// over each tile's list in order, in fixed point (rounded down), and ends the
// list after the batch of 32 entries that takes the sum past -ln(1e-4) with a
// margin for the rounding of the T products (a product of (1 - alpha) below
// e^-9.25 at every pixel; the kernels' T rounds by about 2^-23 an update, which
// the margin covers for 2e5 updates, and a cut falls within the first
// kLongHead entries of a list).  The sums are exact integers, so the
// cut does not depend on the order of any reduction.
constexpr float kSatScale = 65536.f;                       // fixed point of -ln(1 - alpha)
constexpr uint32_t kSatThreshold = (uint32_t)(9.25 * 65536);  // -ln(1e-4) = 9.2103 plus the margin

// Terms of an entry's quadratic form that depend only on the tile row's pixel
// rows [ylo, yhi] (shared by the tiles of the row).
struct SatRow {
    float a, B0, B1, C0, C1, Bm, Cm, px, amax;
};

__device__ __forceinline__ SatRow sat_row(const float4& co, float px, float py, float ylo, float yhi)
{
    const float b2 = 2.f * co.y, dy0 = py - ylo, dy1 = py - yhi, my = fmaxf(fabsf(dy0), fabsf(dy1));
    SatRow r;
    r.a = co.x;
    r.B0 = b2 * dy0;
    r.B1 = b2 * dy1;
    r.C0 = co.z * dy0 * dy0;
    r.C1 = co.z * dy1 * dy1;
    r.Bm = fabsf(b2) * my;
    r.Cm = co.z * my * my;
    r.px = px;
    r.amax = co.w;
    return r;
}

// Saturation weight of one (entry, tile): -ln(1 - alpha_lb) in fixed point,
// rounded down, for the tile's pixel columns [xlo, xhi]; 0 when the bound does
// not pass the 1/255 skip with a margin.
__device__ __forceinline__ uint32_t sat_weight(const SatRow& r, float xlo, float xhi)
{
    const float dx0 = r.px - xlo, dx1 = r.px - xhi;
    // q = a dx^2 + 2 b dx dy + c dy^2 at the four corners
    const float q00 = fmaf(dx0, fmaf(r.a, dx0, r.B0), r.C0), q01 = fmaf(dx0, fmaf(r.a, dx0, r.B1), r.C1);
    const float q10 = fmaf(dx1, fmaf(r.a, dx1, r.B0), r.C0), q11 = fmaf(dx1, fmaf(r.a, dx1, r.B1), r.C1);
    const float qmax = fmaxf(fmaxf(q00, q01), fmaxf(q10, q11));
    const float mx = fmaxf(fabsf(dx0), fabsf(dx1));
    const float qabs = fmaf(mx, fmaf(r.a, mx, r.Bm), r.Cm);  // bounds |a dx^2| + |2 b dx dy| + |c dy^2|
    const float qhi = fmaf(1e-5f, qabs, qmax) + 1e-6f;
    const float alpha = fminf(r.amax * __expf(-0.5f * qhi) * (1.f - 1e-5f), 0.98999f);
    if (!(alpha >= kAlphaMin * 1.002f)) return 0u;
    const float nl = -__log2f(1.f - alpha) * 0.69314718f;  // -ln(1 - alpha)
    const float w = fmaf(nl, 1.f - 1e-4f, -2e-5f);
    return w > 0.f ? (uint32_t)(w * kSatScale) : 0u;
}

constexpr int kFilterSeg = 1024;  // list entries per tail segment (one CTA): 32 groups of 32

// First entry (relative to the list) of the tail of a super-tile with open tiles:
// where the head left its open halves (sat: ended tiles, nh: n_head).
__device__ __forceinline__ uint32_t tail_start(uint2 sat, uint2 nh)
{
    return min(sat.x != 0xffffffffu ? nh.x : 0xffffffffu, sat.y != 0xffffffffu ? nh.y : 0xffffffffu);
}

// one block of 512 threads (the last of the head count): tail segments per
// list, exclusive scan -> seg_base
__device__ __forceinline__ void seg_plan(const TileArgs& a, uint32_t* s_tmp)
{
    uint32_t carry = 0;
    for (int base = 0; base < a.total_super; base += 512) {
        const int gs = base + threadIdx.x;
        uint32_t c = 0;
        if (gs < a.total_super) {  // the tail: what the head pass left, unless every list ended in it
            const uint2 rg = a.sranges[gs], sat = a.sat_head[gs];
            const uint32_t rest = (sat.x & sat.y) == 0xffffffffu ? 0u : rg.y - rg.x - tail_start(sat, a.n_head[gs]);
            c = (rest + kFilterSeg - 1) / kFilterSeg;
        }
        uint32_t tot;
        const uint32_t ex = block_excl_scan<16>(c, s_tmp, &tot);
        if (gs < a.total_super) {
            a.seg_base[gs] = carry + ex;
            for (uint32_t q = 0; q < c; ++q) a.seg_super[carry + ex + q] = (uint32_t)gs;
            if (a.stats && c > 0) {  // some of its tiles closed in the head, others open in the tail
                int v = 0;
                for (int q = 1; q < a.V; ++q)
                    if (gs >= a.super_base[q]) v = q;
                const int ls = gs - a.super_base[v], sy = ls / a.STX[v], sx = ls - sy * a.STX[v];
                const int nx = min(8, a.TX[v] - 8 * sx), ny = min(8, a.TY[v] - 8 * sy);
                const uint32_t in_grid = (1u << nx) - 1u;
                const uint2 sat = a.sat_head[gs];
                bool closed = false, open = false;
                for (int r = 0; r < ny; ++r) {
                    const uint32_t b = ((r < 4 ? sat.x >> (8 * r) : sat.y >> (8 * (r - 4))) & 0xffu) & in_grid;
                    closed |= b != 0u;
                    open |= b != in_grid;
                }
                if (closed && open) atomicAdd(a.stats + 4, 1ull);
            }
        }
        carry += tot;
    }
    if (threadIdx.x == 0) {
        a.seg_base[a.total_super] = carry;
        if (a.stats) atomicAdd(a.stats + 5, (unsigned long long)carry);
    }
}

// Tile totals, offsets and ranges in one pass over the tiles in global order,
// kRangeTiles per block taken in ticket order, kRangeTiles / 256 consecutive
// tiles per thread.  A tile's total is its head count plus its counts in the
// tail segments of its super-tile, whose entries become the tile-relative
// offsets of the segments; the exclusive scan of the totals across blocks
// (decoupled look-back) gives every tile's range [start, start + total) and
// leaves the start in tile_total.  The last block also writes K, checks it
// against the capacity and reports the capacity the call needed.
constexpr int kRangeTileItems = 1;
constexpr int kRangeTiles = 256 * kRangeTileItems;

struct TileRangeArgs {
    unsigned long long* lb;  // [blocks] look-back words (zeroed)
    uint32_t* ticket;        // (zeroed)
    uint2* ranges;
    int64_t* K_out;
    int64_t capacity;
    const int64_t* K_super;  // entries of the super-tile lists, which share the capacity
    int64_t* needed;         // may be null
    uint32_t* cls;           // [kOrderClasses] tiles per list-length class for the tile order (zeroed), or null
    uint32_t* order;         // the tile order, where one block holds every tile (else null)
    int64_t spin_limit;
};

__global__ void __launch_bounds__(256) k_tile_ranges(TileArgs a, TileRangeArgs r)
{
    wait_for_previous_kernel();
    __shared__ unsigned long long s_tmp64[8];
    __shared__ unsigned long long s_excl;
    __shared__ int64_t s_ticket;
    __shared__ uint32_t s_cls[kOrderClasses];
    constexpr unsigned long long kA = 1ull << 62, kP = 2ull << 62, kM = (1ull << 62) - 1;
    if (block_failed(a.status)) return;
    const int tid = threadIdx.x;
    if (tid == 0) s_ticket = atomicAdd(r.ticket, 1u);
    for (int c = tid; c < (int)kOrderClasses; c += blockDim.x) s_cls[c] = 0u;
    __syncthreads();
    const int64_t blk = s_ticket, nblk = ((int64_t)a.total_tiles + kRangeTiles - 1) / kRangeTiles;
    if (blk >= nblk) return;
    const int64_t t0 = blk * kRangeTiles + (int64_t)tid * kRangeTileItems;
    uint32_t cnt[kRangeTileItems];
    unsigned long long tsum = 0;
#pragma unroll
    for (int q = 0; q < kRangeTileItems; ++q) {
        const int64_t t = t0 + q;
        uint32_t run = 0;
        if (t < a.total_tiles) {
            int v = 0;
            for (int w = 1; w < a.V; ++w)
                if (t >= a.tile_base[w]) v = w;
            const int local = (int)(t - a.tile_base[v]);
            const int ty = local / a.TX[v], tx = local - ty * a.TX[v];
            const int gs = a.super_base[v] + (ty >> 3) * a.STX[v] + (tx >> 3), lt = (ty & 7) * 8 + (tx & 7);
            run = a.tile_total[t];  // the head's count: the tail segments follow it
            // the segments' counts, four loads in flight at a time, become their offsets
            const uint32_t g1 = a.seg_base[gs + 1];
            for (uint32_t g = a.seg_base[gs]; g < g1; g += 4) {
                uint32_t c[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) c[u] = g + u < g1 ? a.seg_cnt[(size_t)(g + u) * 64 + lt] : 0u;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (g + u < g1) a.seg_cnt[(size_t)(g + u) * 64 + lt] = run;
                    run += c[u];
                }
            }
        }
        cnt[q] = run;
        tsum += run;
        if (r.cls && t < a.total_tiles) atomicAdd(&s_cls[length_class(run)], 1u);  // as tile_class
    }
    unsigned long long agg;
    const unsigned long long texcl = block_excl_scan256_u64(tsum, s_tmp64, &agg);
    if (tid < 32) {  // decoupled look-back by one warp, 32 predecessors per round trip
        const int lane = tid;
        unsigned long long excl = 0;
        if (lane == 0) st_relaxed64(r.lb + blk, (blk == 0 ? kP : kA) | agg);
        if (blk > 0) {
            int64_t j = blk - 1, spins = 0;
            for (;;) {
                const unsigned long long w = j - lane >= 0 ? ld_relaxed64(r.lb + (j - lane)) : kP;
                const unsigned long long flag = w & ~kM;
                const unsigned pend = __ballot_sync(0xffffffffu, flag == 0);
                const unsigned pref = __ballot_sync(0xffffffffu, flag == kP);
                const int first_pend = pend ? __ffs(pend) - 1 : 32;
                const int first_pref = pref ? __ffs(pref) - 1 : 32;
                const bool found = first_pref < first_pend;
                const int take = found ? first_pref + 1 : first_pend;
                unsigned long long x = lane < take ? (w & kM) : 0ull;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                excl += x;
                if (found) break;
                j -= take;
                if (take == 0) {
                    if (++spins > r.spin_limit) {
                        if (lane == 0) set_status(a.status, SPLAT_ERR_TIMEOUT, SPLAT_STAGE_DUPLICATE, blk);
                        break;
                    }
                    if (spins > 64) __nanosleep(64);
                }
            }
            if (lane == 0) st_relaxed64(r.lb + blk, kP | ((excl + agg) & kM));
        }
        if (lane == 0) {
            s_excl = excl;
            if (blk == nblk - 1) {
                const int64_t K = (int64_t)(excl + agg);
                *r.K_out = K;
                if (K > r.capacity) set_status(a.status, SPLAT_ERR_CAPACITY, SPLAT_STAGE_DUPLICATE, K);
                if (r.needed) *r.needed = max(K, *r.K_super);
            }
        }
    }
    __syncthreads();
    if (r.order) {  // (block-uniform) k_tile_order's slots: the classes' starts, the longest first, then cursors
        __shared__ uint32_t s_tmp[8];
        const uint32_t cb = kOrderClasses - 1u - tid;
        uint32_t total;
        const uint32_t ex = block_excl_scan256(s_cls[cb], s_tmp, &total);
        s_cls[cb] = ex;
        if (tid == 0) s_cls[0] = total;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kRangeTileItems; ++q)
            if (t0 + q < a.total_tiles) r.order[atomicAdd(&s_cls[length_class(cnt[q])], 1u)] = (uint32_t)(t0 + q);
    } else if (r.cls) {
        for (int c = tid; c < (int)kOrderClasses; c += blockDim.x)
            if (s_cls[c]) atomicAdd(&r.cls[c], s_cls[c]);
    }
    // slots past 2^32 only arise with K beyond any capacity: the check above reports them
    uint32_t st = (uint32_t)(s_excl + texcl);
#pragma unroll
    for (int q = 0; q < kRangeTileItems; ++q) {
        const int64_t t = t0 + q;
        if (t < a.total_tiles) {
            r.ranges[t] = cnt[q] ? make_uint2(st, st + cnt[q]) : make_uint2(0u, 0u);
            a.tile_total[t] = st;
        }
        st += cnt[q];
    }
}

// Tile columns [lo, hi) of the super-tile's tile row with pixel rows
// [vlo, vlo + 15] that an entry is listed in, as bits: its rectangle's columns
// [x0, x1), with culling on narrowed to the tiles its opacity footprint reaches.
__device__ __forceinline__ uint32_t row_columns(int x0, int x1, int tx0, float vlo, const float4& g0, const float4& g1,
                                                bool cull)
{
    if (cull) {
        float ul, ur;
        if (!ellipse_band_extent(g0, g1, vlo, vlo + (float)(kTile - 1), ul, ur)) return 0u;
        // tiles [16 tx, 16 tx + 15] meeting [ul, ur]
        const float fl = ceilf((ul - (float)(kTile - 1)) * (1.f / kTile));
        const float fh = floorf(ur * (1.f / kTile));
        x0 = max(x0, (int)fminf(fmaxf(fl, -1.f), 1.0e6f) - tx0);
        x1 = min(x1, (int)fminf(fmaxf(fh, -2.f), 1.0e6f) + 1 - tx0);
    }
    return x1 > x0 ? (1u << x1) - (1u << x0) : 0u;
}

// Footprint constants of a projected row, the squared radius enlarged by a
// margin that covers FP32 rounding (the compositing kernels skip
// power < log(1/(255 alpha_max))).
__device__ __forceinline__ void footprint(const float2& xy, const float4& co, float4& g0, float4& g1)
{
    const float R2 = -2.f * __logf(__fdividef(kAlphaMin, co.w)) * 1.0001f + 2e-3f;
    ellipse_consts(xy.x, xy.y, co.x, co.y, co.z, R2, g0, g1);
}

// 32 x 32 bit matrix transpose over the warp: bit e of lane t's result is bit t
// of lane e's argument.
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x, int lane)
{
    auto step = [&](int j, uint32_t low) {
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
        x = (lane & j) ? ((x & ~low) | ((y >> j) & low)) : ((x & low) | ((y << j) & ~low));
    };
    step(16, 0x0000ffffu);
    step(8, 0x00ff00ffu);
    step(4, 0x0f0f0f0fu);
    step(2, 0x33333333u);
    step(1, 0x55555555u);
    return x;
}

// Tile columns (of [tx0, tx0 + 8), as bits) of a tile row that lie wholly inside
// the footprint: those between its chords at the row's first and last pixel row
// (the footprint is convex).  Only these can have a saturation weight, which
// needs every pixel of the tile to pass the alpha skip.
__device__ __forceinline__ uint32_t inner_columns(const float4& g0, const float4& g1, float ylo, float yhi, int tx0,
                                                  float xmax_img)
{
    const float d0 = g0.y - ylo, d1 = g0.y - yhi;
    const float q0 = g0.z - g1.w * d0 * d0, q1 = g0.z - g1.w * d1 * d1;
    if (!(q0 > 0.f && q1 > 0.f)) return 0u;
    const float s0 = sqrt_approx(q0), s1 = sqrt_approx(q1);
    const float c0 = g0.x + g1.z * d0, c1 = g0.x + g1.z * d1;  // chord centres
    const float l = fmaxf(c0 - s0, c1 - s1), r = fminf(c0 + s0, c1 + s1);
    const float fl = ceilf(l * (1.f / kTile));
    // the image's last column of tiles ends at its last pixel
    const float fr = r >= xmax_img ? 1.0e6f : floorf((r - (float)(kTile - 1)) * (1.f / kTile));
    const int lo = max((int)fminf(fmaxf(fl, -1.f), 1.0e6f) - tx0, 0);
    const int hi = min((int)fminf(fmaxf(fr, -2.f), 1.0e6f) + 1 - tx0, 8);
    return hi > lo ? (1u << hi) - (1u << lo) : 0u;
}

// Head pass, counting: the first entries of each super-tile's list (head_reach),
// kHeadEntries at a time while one of its tiles is open, one CTA per half of the
// super-tile (four tile rows, 32 tiles), one thread per entry and one warp per
// group of 32 of them.  A thread finds the tiles of its half that its entry is
// listed in (a 32-bit mask) and, with culling on, adds the entry's saturation
// weight in each to the sum of (group, tile) in shared memory.  The warp then
// transposes its 32 masks, which leaves lane t with tile t's entries: counts are
// population counts, with no ballot per column.  One warp (lane t: tile t) goes
// through the groups in order, ends tile t's list after the group that takes its
// sum past the threshold and counts the entries up to there; the groups' words
// are written with the entries past an end taken out, so that the write pass
// runs on the words alone.  The last CTA to finish plans the tail segments
// (seg_plan).
// With long heads a half goes on past its first window while every open tile of
// it is on its way to close within the reach (one that stays open keeps the tail
// alive, and a window costs about what three windows of the tail cost); its tail
// starts where it stopped.  On 1M Gaussians at 4 x 2704x2028 the lists shrink
// from 87M to 23M instances: head 139 -> 305 us, but the rest of the lists' sort
// 78 -> 33, tail 259 -> 54, writes 237 -> 85.  The rule does not weigh the saving
// against the windows: on 300k at 4 x 1352x1014 the head takes 75 us instead of 42
// and the passes behind it save about 18 (the sort 8 us slower in the step).
// Batches of fewer super-tiles than two per SM keep short heads: there the tail's
// parallel segments are faster.
// Bound by the entries' gathers (three sectors each) and by issue.  One CTA per
// tile row with its entries queued per row and a warp per tile column re-read
// every entry eight times and evaluated the weights on the few lanes listed in
// the column: 173 us on 1M Gaussians at 4 x 2704x2028, 50 us on 300k at
// 4 x 1352x1014.
__global__ void __launch_bounds__(kHeadEntries, 2) k_head_count(TileArgs a)
{
    wait_for_previous_kernel();
    constexpr int kGroups = kHeadEntries / 32;
    __shared__ uint32_t s_sum[kGroups][32];  // saturation weights of each (group, tile)
    __shared__ uint32_t s_word[kGroups][32];
    __shared__ int s_cut[32];                // last group of each tile's list in this window (-1: ended before it)
    __shared__ uint32_t s_tmp[16];
    __shared__ bool s_on;                    // the half goes on to another window
    __shared__ bool s_last;
    if (status_failed(a.status)) return;
    const int tid = threadIdx.x, lane = tid & 31, g = tid >> 5;
    const int gs = (int)(blockIdx.x >> 1), half = (int)(blockIdx.x & 1);
    int v = 0;
    for (int q = 1; q < a.V; ++q)
        if (gs >= a.super_base[q]) v = q;
    const int ls = gs - a.super_base[v];
    const int sy = ls / a.STX[v], sx = ls - sy * a.STX[v];
    const int TX = a.TX[v], TY = a.TY[v];
    const int ty0 = sy * 8 + 4 * half, tx0 = sx * 8;
    const uint2 rgs = a.sranges[gs];
    const int reach = (int)head_reach(rgs.y - rgs.x, a.long_heads);
    const float xmax_img = (float)(a.W[v] - 1), ymax_img = (float)(a.H[v] - 1);
    // warp 0, lane t: the state of tile t of the half
    const int ty = ty0 + (lane >> 3), tx = tx0 + (lane & 7);
    const bool in = ty < TY && tx < TX;
    uint32_t cnt = 0u, sum = 0u;
    bool ended = !in;  // tiles outside the grid count as ended
    s_sum[g][lane] = 0u;
    __syncthreads();
    int w0 = 0;
    while (w0 < reach) {
        const int n = min(reach - w0, kHeadEntries);
        uint32_t m = 0u;
        if (tid < n) {
            const uint32_t row = a.list[rgs.x + w0 + tid];
            const int4 rc = ((const int4*)a.proj.rect)[row];
            const float2 xy = ((const float2*)a.proj.xy)[row];
            const float4 co = ((const float4*)a.proj.conic_opacity)[row];
            const int x0 = max(rc.x - tx0, 0), x1 = min(rc.z - tx0, 8);
            const int y0 = max(rc.y - ty0, 0), y1 = min(rc.w - ty0, 4);
            if (x0 < x1 && y0 < y1) {
                float4 g0, g1;
                if (a.cull) footprint(xy, co, g0, g1);
                // the saturation bound needs a*c - b^2 >= 1e-3 a c: the relative
                // rounding of the power stays far below its size
                const bool sat_ok = a.cull && co.x > 0.f && co.z > 0.f &&
                                    co.x * co.z - co.y * co.y >= 1e-3f * co.x * co.z && co.w <= 1.f && co.w > 0.f;
                for (int r = y0; r < y1; ++r) {
                    const float vlo = (float)((ty0 + r) * kTile), vhi = fminf(vlo + (float)(kTile - 1), ymax_img);
                    const uint32_t cols = row_columns(x0, x1, tx0, vlo, g0, g1, a.cull);
                    m |= cols << (8 * r);
                    uint32_t left = sat_ok ? cols & inner_columns(g0, g1, vlo, vhi, tx0, xmax_img) : 0u;
                    if (left) {
                        const SatRow sr = sat_row(co, xy.x, xy.y, vlo, vhi);
                        for (; left; left &= left - 1) {
                            const int c = __ffs(left) - 1;
                            const float xlo = (float)((tx0 + c) * kTile);
                            const uint32_t wt = sat_weight(sr, xlo, fminf(xlo + (float)(kTile - 1), xmax_img));
                            if (wt) atomicAdd(&s_sum[g][8 * r + c], wt);
                        }
                    }
                }
            }
        }
        __syncwarp();
        const uint32_t word = warp_transpose(m, lane);
        s_word[g][lane] = word;
        __syncthreads();
        if (g == 0) {
            int cut = ended ? -1 : kGroups;
#pragma unroll
            for (int q = 0; q < kGroups; ++q) {
                if (q <= cut) {
                    cnt += __popc(s_word[q][lane]);
                    sum += s_sum[q][lane];
                    if (sum >= kSatThreshold) cut = min(cut, q);  // the list ends after this group
                }
                s_sum[q][lane] = 0u;
            }
            s_cut[lane] = cut;
            ended = cut < kGroups;
            // on its way: a quarter above the threshold by the end of the reach, at the mean rate so far (weights
            // fall with the depth)
            const bool good = ended || 4ull * sum * (unsigned)reach >= 5ull * kSatThreshold * (unsigned)(w0 + n);
            const bool open = __any_sync(0xffffffffu, !ended), all_good = __all_sync(0xffffffffu, good);
            if (lane == 0) s_on = open && all_good;
        }
        __syncthreads();
        if (32 * g < n) {  // warp-uniform
            const bool open = g <= s_cut[lane];
            const uint32_t allowed = __ballot_sync(0xffffffffu, open);
            uint32_t* out = reinterpret_cast<uint32_t*>(a.mask + rgs.x + w0 + 32 * g);
            if (32 * g + 32 <= n) out[32 * half + lane] = open ? word : 0u;
            else if (tid < n) out[2 * lane + half] = m & allowed;
        }
        w0 += n;
        if (w0 >= reach || !s_on) break;  // block-uniform
        __syncthreads();  // s_on, s_cut and s_word are rewritten by the next window
    }
    if (g == 0) {
        if (in) a.tile_total[a.tile_base[v] + ty * TX + tx] = cnt;
        const uint32_t sat = __ballot_sync(0xffffffffu, ended);
        if (lane == 0) {
            reinterpret_cast<uint32_t*>(a.sat_head + gs)[half] = sat;
            reinterpret_cast<uint32_t*>(a.n_head + gs)[half] = (uint32_t)w0;
        }
        __syncwarp();
    }
    __syncthreads();
    if (tid == 0) {  // the last CTA to finish plans the tail from every CTA's results
        __threadfence();
        s_last = atomicAdd(a.ticket + 2, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        seg_plan(a, s_tmp);
    }
}

// Tail pass, counting: what the head pass left of the lists of super-tiles with
// an open tile, in segments of kFilterSeg entries taken from a ticket counter
// (their costs differ).  As in the head, a lane finds its entry's tiles (64-bit
// mask, the tiles whose lists ended in the head taken out), the warp transposes
// the masks of its group and counts by population counts.  A queue of entries
// per tile row and a warp reduction per pair of columns took 312 us on 1M
// Gaussians at 4 x 2704x2028.
template <int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_tail_count(TileArgs a)
{
    wait_for_previous_kernel();
    __shared__ uint32_t s_cnt[WARPS][64];
    __shared__ uint32_t s_g;
    __shared__ int s_gs;
    if (status_failed(a.status)) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t nseg = a.seg_base[a.total_super];
    for (;;) {
        if (tid == 0) {
            s_g = atomicAdd(a.ticket + 1, 1u);
            if (s_g < nseg) s_gs = (int)a.seg_super[s_g];
        }
        __syncthreads();
        const uint32_t g = s_g;
        if (g >= nseg) break;
        const int gs = s_gs;
        int v = 0;
        for (int w = 1; w < a.V; ++w)
            if (gs >= a.super_base[w]) v = w;
        const int ls = gs - a.super_base[v];
        const int sy = ls / a.STX[v], sx = ls - sy * a.STX[v];
        const int ty0 = sy * 8, tx0 = sx * 8;
        const uint2 rgs = a.sranges[gs], sat = a.sat_head[gs], nh = a.n_head[gs];
        const uint32_t r0 = tail_start(sat, nh) + (g - a.seg_base[gs]) * kFilterSeg, b0 = rgs.x + r0;
        const int n = (int)min((uint32_t)kFilterSeg, rgs.y - b0);
        uint32_t c0 = 0u, c1 = 0u;  // entries listed in tiles lane and lane + 32
        for (int q = 32 * warp; q < n; q += 32 * WARPS) {  // warp-uniform
            const int e = q + lane;
            // (warp-uniform) whether each half is open and past its head: the words of a half's head stay as they are
            const bool h0 = sat.x != 0xffffffffu && r0 + q >= nh.x, h1 = sat.y != 0xffffffffu && r0 + q >= nh.y;
            uint32_t m0 = 0u, m1 = 0u;
            if (e < n) {
                const uint32_t row = a.list[b0 + e];
                const int4 rc = ((const int4*)a.proj.rect)[row];
                const float2 xy = ((const float2*)a.proj.xy)[row];
                const float4 co = ((const float4*)a.proj.conic_opacity)[row];
                const int x0 = max(rc.x - tx0, 0), x1 = min(rc.z - tx0, 8);
                const int y0 = max(rc.y - ty0, h0 ? 0 : 4), y1 = min(rc.w - ty0, h1 ? 8 : 4);
                if (x0 < x1 && y0 < y1) {
                    float4 g0, g1;
                    if (a.cull) footprint(xy, co, g0, g1);
                    for (int r = y0; r < y1; ++r) {
                        const uint32_t cols = row_columns(x0, x1, tx0, (float)((ty0 + r) * kTile), g0, g1, a.cull);
                        if (r < 4) m0 |= cols << (8 * r);
                        else m1 |= cols << (8 * r - 32);
                    }
                    m0 &= ~sat.x;
                    m1 &= ~sat.y;
                }
            }
            __syncwarp();
            const uint32_t t0 = warp_transpose(m0, lane), t1 = warp_transpose(m1, lane);
            c0 += __popc(t0);
            c1 += __popc(t1);
            if (q + 32 <= n) {
                uint32_t* out = reinterpret_cast<uint32_t*>(a.mask + b0 + q);
                if (h0) out[lane] = t0;
                if (h1) out[32 + lane] = t1;
            } else if (e < n) {
                if (h0) a.mask[b0 + e].x = m0;
                if (h1) a.mask[b0 + e].y = m1;
            }
        }
        s_cnt[warp][lane] = c0;
        s_cnt[warp][32 + lane] = c1;
        __syncthreads();
        if (tid < 64) {
            uint32_t c = 0u;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) c += s_cnt[w][tid];
            a.seg_cnt[(size_t)g * 64 + tid] = c;
        }
        __syncthreads();
    }
}

// Writing pass: the heads (one ticket per super-tile), then the tail segments,
// one CTA each, 8 / COLS warps per tile row; driven by the coverage words alone.
// Lane j holds group j's words of the row's eight tiles.  Tile by tile, the
// prefix over the groups' counts gives every listed entry its slot.  Where the
// groups list few entries (a mean of at most kSparse), each lane goes through
// its own group's bits, all groups at once, into a shared buffer that the warp
// copies out; else the warp goes through the groups one after the other, lane e
// taking entry e.  (A ballot per tile column and 32 queued entries of the row
// took 2.4 warp instructions per instance, 243 us for the 87M instances of 1M
// Gaussians at 4 x 2704x2028.)
constexpr int kSparse = 6;

// COLS columns of the row per warp: 8 / COLS warps share it.
template <int COLS>
__global__ void __launch_bounds__(32 * 64 / COLS) k_tile_write(TileArgs a)
{
    wait_for_previous_kernel();
    __shared__ uint32_t s_row[kFilterSeg];
    constexpr int kThreads = 32 * 64 / COLS;
    __shared__ uint32_t s_buf[64 / COLS][32 * kSparse];
    __shared__ uint32_t s_tk;
    __shared__ int s_gs;
    if (status_failed(a.status)) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tr = warp / (8 / COLS), tc = warp % (8 / COLS) * COLS;  // the warp's tile row and first column
    const unsigned lt = lanemask_lt();
    const uint32_t nseg = a.seg_base[a.total_super], nhead = (uint32_t)a.total_super;
    for (;;) {
        if (tid == 0) {
            const uint32_t tk = atomicAdd(a.ticket, 1u);
            s_tk = tk;
            if (tk < nhead) s_gs = (int)tk;
            else if (tk < nhead + nseg) s_gs = (int)a.seg_super[tk - nhead];
        }
        __syncthreads();
        const uint32_t tk = s_tk;
        if (tk >= nhead + nseg) break;
        const int gs = s_gs;
        const bool head = tk < nhead;
        int v = 0;
        for (int w = 1; w < a.V; ++w)
            if (gs >= a.super_base[w]) v = w;
        const int ls = gs - a.super_base[v];
        const int sy = ls / a.STX[v], sx = ls - sy * a.STX[v];
        const int TX = a.TX[v], TY = a.TY[v];
        const int ty = sy * 8 + tr, tx0 = sx * 8 + tc;
        const uint2 rgs = a.sranges[gs], sat = a.sat_head[gs], nh = a.n_head[gs];
        const bool open = (tr < 4 ? sat.x : sat.y) != 0xffffffffu;  // this warp's half has a tail
        const uint32_t my_head = tr < 4 ? nh.x : nh.y;
        uint32_t b0 = rgs.x, b1, from, to;  // the item's entries [b0, b1), of which this warp's are [from, to)
        if (head) {  // each half of the super-tile up to where its head stopped
            b1 = b0 + max(nh.x, nh.y);
            from = b0;
            to = b0 + my_head;
        } else {
            b0 += tail_start(sat, nh) + (tk - nhead - a.seg_base[gs]) * kFilterSeg;
            b1 = min(b0 + (uint32_t)kFilterSeg, rgs.y);
            from = max(b0, rgs.x + my_head);  // (whole groups: heads stop at multiples of kHeadEntries)
            to = open ? b1 : b0;
        }
        uint32_t first[COLS];  // next slot of each tile's list
#pragma unroll
        for (int k = 0; k < COLS; ++k) {
            first[k] = 0u;
            if (ty < TY && tx0 + k < TX) {
                const int tile = a.tile_base[v] + ty * TX + tx0 + k;
                first[k] = head ? a.ranges[tile].x
                                : a.tile_total[tile] + a.seg_cnt[(size_t)(tk - nhead) * 64 + 8 * tr + tc + k];
            }
        }
        for (; b0 < b1; b0 += kFilterSeg) {
            const int rows = (int)min((uint32_t)kFilterSeg, b1 - b0);
            for (int i = tid; i < rows; i += kThreads) s_row[i] = a.list[b0 + i];
            __syncthreads();
            const int n = to > max(b0, from) ? (int)min((uint32_t)kFilterSeg, to - b0) : 0;
            const int skip = from > b0 ? (int)(from - b0) >> 5 : 0;  // groups of the half's head
            if (ty < TY && n > 0) {  // warp-uniform
                const int full = n >> 5, part = n & 31, groups = full + (part ? 1 : 0);
                uint32_t word[COLS];
#pragma unroll
                for (int k = 0; k < COLS; ++k) word[k] = 0u;
                if (lane >= skip && lane < full) {
                    const uint2* p = a.mask + b0 + 32 * lane + 4 * tr + tc / 2;
#pragma unroll
                    for (int k = 0; k < COLS / 2; ++k) {
                        const uint2 t = p[k];
                        word[2 * k] = t.x;
                        word[2 * k + 1] = t.y;
                    }
                }
                if (part && full >= skip) {  // the last group keeps a word pair per entry
                    uint32_t byte = 0u;
                    if (lane < part) {
                        const uint2 t = a.mask[b0 + 32 * full + lane];
                        byte = (tr < 4 ? t.x >> (8 * tr) : t.y >> (8 * (tr - 4))) >> tc & 0xffu;
                    }
#pragma unroll
                    for (int k = 0; k < COLS; ++k) {
                        const uint32_t bal = __ballot_sync(0xffffffffu, (byte >> k) & 1u);
                        if (lane == full) word[k] = bal;
                    }
                }
#pragma unroll
                for (int k = 0; k < COLS; ++k) {
                    uint32_t w = word[k];
                    const uint32_t c = __popc(w);
                    uint32_t at = c;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, at, o);
                        if (lane >= o) at += y;
                    }
                    const uint32_t total = __shfl_sync(0xffffffffu, at, 31);
                    at -= c;
                    if (total == 0u) continue;  // warp-uniform
                    uint32_t* out = a.vals_out + first[k];
                    if (total <= (uint32_t)(kSparse * groups)) {
                        while (w) {
                            const int e = __ffs(w) - 1;
                            w &= w - 1;
                            s_buf[warp][at++] = s_row[32 * lane + e];
                        }
                        __syncwarp();
                        for (uint32_t i = lane; i < total; i += 32) out[i] = s_buf[warp][i];
                        __syncwarp();
                    } else {
                        for (int q = 0; q < groups; ++q) {
                            const uint32_t gw = __shfl_sync(0xffffffffu, w, q), ga = __shfl_sync(0xffffffffu, at, q);
                            if ((gw >> lane) & 1u) out[ga + __popc(gw & lt)] = s_row[32 * q + lane];
                        }
                    }
                    if (a.keys_out) {
                        const uint32_t tile = (uint32_t)(a.tile_base[v] + ty * TX + tx0 + k);
                        for (uint32_t i = lane; i < total; i += 32) a.keys_out[first[k] + i] = tile;
                    }
                    first[k] += total;
                }
            }
            if (b0 + kFilterSeg < b1) __syncthreads();  // (block-uniform) s_row is rewritten
        }
        __syncthreads();  // s_tk, s_gs and s_row are rewritten, also after an item without entries
    }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------


struct SortLayout {
    int64_t n_rows, capacity;
    int V;
    bool binned;
    int64_t parts_d, parts_t, parts_scan, n_chunks;
    int64_t total_tiles, total_super, max_segs;
    // radix path
    size_t off_dkeys[2], off_dvals[2], off_offsets, off_chunk, off_scan_lb, off_dlb[2], off_tlb[2], off_tkeys,
        off_tvals, off_hist;
    // binned path
    int bin_bits, copies;
    int64_t queue_cap;
    size_t off_rec, off_range, off_split, off_cell, off_cell_lb, off_queue, off_nqueue, off_rlb, off_total, off_vals1, off_sranges,
        off_ninst1, off_segbase, off_segcnt, off_segsuper, off_sathead, off_nhead, off_mask;
    // both
    size_t off_tord, off_tickets, zero_begin, zero_end;
    size_t bytes;
};

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

constexpr int kSuperShift = 3;  // super-tiles of 8 x 8 tiles

// Bytes of the workspace's first layout, in which both paths sorted the rows by
// depth with radix passes; none of its buffers is laid out so any more.  The sum
// stays the least that is asked for, and the cells keep within it, so that the
// sizes callers hold and the limit of splat_bin_sort_noalloc are what they were.
static size_t legacy_bytes(const SortLayout& L, int64_t n_rows, int64_t capacity, int V, int smax)
{
    size_t o = 0;
    auto take = [&](size_t bytes) { o = align256(o + std::max<size_t>(bytes, 4)); };
    const size_t rows = (size_t)n_rows, cap = (size_t)capacity, S = (size_t)L.total_super;
    const size_t parts_d = V > 0 ? (size_t)(V * ((n_rows / V + 4095) / 4096)) : 0, parts_c = (cap + 4095) / 4096;
    for (int b = 0; b < 5; ++b) take(4 * rows);
    take(L.binned ? 4 : 4 * ((cap + kDupChunk - 1) / kDupChunk + 1));
    take(8 * std::max<size_t>((rows + 4095) / 4096, 1));
    for (int b = 0; b < 2; ++b) take(1024 * std::max<size_t>(parts_d, 1));
    for (int b = 0; b < 2; ++b) take(1024 * std::max<size_t>(L.binned ? 0 : parts_c, 1));
    for (int b = 0; b < 2; ++b) take(L.binned ? 4 : 4 * cap);
    take(1024 * 9);
    take(4096 * (size_t)std::max(V, 1));
    take(L.binned ? 4 * S : 4);
    take(8 * (size_t)((L.total_tiles + 255) / 256 + 1));
    take(2 * kOrderClasses * 4);
    take(64);
    take(L.binned ? 8 * (size_t)smax * std::max<size_t>(parts_c + (size_t)V, 1) : 4);
    take(L.binned ? 4 * (size_t)L.total_tiles : 4);
    take(L.binned ? 4 * cap : 4);
    take(L.binned ? 8 * S : 4);
    take(8);
    take(4 * (S + 1));
    take(L.binned ? 256 * (size_t)L.max_segs : 4);
    take(L.binned ? 4 * (size_t)L.max_segs : 4);
    take(4 * std::max<size_t>(S, 1));
    take(8 * std::max<size_t>(S, 1));
    take(32 * std::max<size_t>(S, 1));
    take(L.binned ? 8 * cap : 4);
    return o;
}

SortLayout sort_layout(int64_t n_rows, int64_t capacity, int V, const int* TX, const int* TY, int tile_sort)
{
    SortLayout L{};
    L.n_rows = n_rows;
    L.capacity = capacity;
    L.V = V;
    int tmax = 1, smax = 1;
    for (int v = 0; v < V; ++v) {
        tmax = std::max(tmax, TX[v] * TY[v]);
        const int sx = (TX[v] + 7) >> kSuperShift, sy = (TY[v] + 7) >> kSuperShift;
        smax = std::max(smax, sx * sy);
        L.total_tiles += (int64_t)TX[v] * TY[v];
        L.total_super += (int64_t)sx * sy;
    }
    smax = (smax + 3) & ~3;
    // views of up to kBinMaxTiles tiles, or (forced) those whose super-tile grids fit the split's former
    // shared-memory counters
    int sdiff = 0;
    for (int v = 0; v < V; ++v)
        sdiff = std::max(sdiff, (((TX[v] + 7) >> kSuperShift) + 1) * (((TY[v] + 7) >> kSuperShift) + 1));
    const bool split_ok = 4 * (9 * (int64_t)smax + 8 * (int64_t)sdiff) <= kSplitMaxSmem;
    L.binned = split_ok && (tile_sort == 2 || (tile_sort == 0 && tmax <= kBinMaxTiles));
    L.max_segs = L.binned ? (capacity + kFilterSeg - 1) / kFilterSeg + L.total_super : 1;
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t r = o; o = align256(o + std::max<size_t>(bytes, 4)); return r; };
    if (!L.binned) {
        L.parts_d = (n_rows + kSortPart - 1) / kSortPart;
        L.parts_t = (capacity + kSortPart - 1) / kSortPart;
        L.parts_scan = (n_rows + kScanPart - 1) / kScanPart;
        L.n_chunks = (capacity + kDupChunk - 1) / kDupChunk + 1;
        for (int b = 0; b < 2; ++b) L.off_dkeys[b] = take(4 * (size_t)n_rows);
        for (int b = 0; b < 2; ++b) L.off_dvals[b] = take(4 * (size_t)n_rows);
        L.off_offsets = take(4 * (size_t)n_rows);
        L.off_chunk = take(4 * (size_t)L.n_chunks);
        L.off_scan_lb = take(8 * (size_t)std::max<int64_t>(L.parts_scan, 1));
        for (int b = 0; b < 2; ++b) L.off_dlb[b] = take(4 * (size_t)kRadix * std::max<int64_t>(L.parts_d, 1));
        for (int b = 0; b < 2; ++b) L.off_tlb[b] = take(4 * (size_t)kRadix * std::max<int64_t>(L.parts_t, 1));
        L.off_tkeys = take(4 * (size_t)capacity);
        L.off_tvals = take(4 * (size_t)capacity);
        L.zero_begin = L.off_hist = take(4 * (size_t)kRadix * 9);
        L.off_tickets = take(4 * 16);
        L.zero_end = o;
        L.off_tord = take(2 * kOrderClasses * 4);  // tile-order class counts and cursors
    }
    const size_t legacy = legacy_bytes(L, n_rows, capacity, V, smax);
    if (L.binned) {
        L.off_total = take(4 * (size_t)L.total_tiles);
        L.off_vals1 = take(4 * (size_t)capacity);
        L.off_sranges = take(8 * (size_t)L.total_super);
        L.off_ninst1 = take(8);
        L.off_segbase = take(4 * (size_t)(L.total_super + 1));
        L.off_segcnt = take(4 * 64 * (size_t)L.max_segs);
        L.off_segsuper = take(4 * (size_t)L.max_segs);
        L.off_sathead = take(8 * (size_t)std::max<int64_t>(L.total_super, 1));
        L.off_nhead = take(8 * (size_t)std::max<int64_t>(L.total_super, 1));
        L.off_mask = take(8 * (size_t)capacity);  // the unsorted entries, then the coverage words
        L.off_rec = take(8 * (size_t)n_rows);
        L.off_range = take(8 * (size_t)std::max(V, 1));
        L.off_split = take(8 * (size_t)kSplits * std::max(V, 1));
        // units of lists of more than kUnit entries: at most 2 n / kUnitStep + 1 of a list of n
        const int64_t per_view = V > 0 ? n_rows / V : 0;
        const int64_t most = std::min<int64_t>(capacity, per_view * L.total_super);
        L.queue_cap = 5 * (most / kUnit) + 8;
        L.off_queue = take(16 * (size_t)L.queue_cap);
        L.zero_begin = L.off_nqueue = take(8);
        L.off_tickets = take(4 * 16);
        L.off_cell_lb = take(8 * (size_t)L.total_super);
        L.off_rlb = take(8 * (size_t)((L.total_tiles + kRangeTiles - 1) / kRangeTiles + 1));
        L.off_tord = take(2 * kOrderClasses * 4);
        // depth bins: 1024 where lists are long (their cells then hold a few entries), 64 where a list is
        // about one unit; fewer where the cells would not fit the workspace
        L.bin_bits = n_rows >= 512 * L.total_super ? 10 : 6;
        while (L.bin_bits > 0 && align256(o + (4 * (size_t)L.total_super << L.bin_bits)) > legacy) L.bin_bits -= 2;
        const size_t cell_bytes = 4 * (size_t)L.total_super << L.bin_bits;
        // copies while they stay within 4 MB (8 for a view of 1352x1014, 1 for four of 2704x2028): 1M Gaussians
        // seen in a 128x128 view sort in 432 us with one copy, 337 with two, 270 with eight; the scan's extra
        // reads cost a view of 300k about 1 us
        for (L.copies = 1; L.copies < 8 && 2 * L.copies * cell_bytes <= (4u << 20) &&
                           align256(o + 2 * L.copies * cell_bytes) <= legacy;)
            L.copies *= 2;
        L.off_cell = take(L.copies * cell_bytes);
        L.zero_end = o;
    }
    L.bytes = std::max(o, legacy);
    return L;
}

// resident CTAs per SM of a kernel (grid-stride kernels launch one wave of them)
template <typename Kernel>
static int ctas_per_sm(Kernel kernel, int threads)
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, 0) != cudaSuccess || n < 1) n = 1;
    return n;
}

static int sort_ctas_per_sm()
{
    static int cached = 0;
    if (!cached) {
        int n0 = 0, n1 = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n0, k_onesweep<false>, kSortThreads, 0) != cudaSuccess) n0 = 1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n1, k_onesweep<true>, kSortThreads, 0) != cudaSuccess) n1 = 1;
        cached = std::max(1, std::min(n0, n1));
    }
    return cached;
}


// Tail segments and writing items, one wave of CTAs at most.  A segment's time is
// what few of them take, so they get as many warps as fill the chip: 32 up to 8
// segments per SM (capacity / 1024 of them), 16 up to 48, else 8, whose small CTAs
// pack best.  Bin sort us with 32 / 16 / 8 warps:
//   128x128, 4k            32 / 34 / 36       677x507, 101k        60 / 63 / 69
//   857x479, 60k, 2 views  70 / 75 / 84       857x479, 120k, 3     76 / 75 / 83
//   1352x1014, 300k       109 / 106 / 118     2704x2028, 1M       233 / 230 / 237
//   1352x1014, 300k, 4    264 / 260 / 260     676x507, 200k, 16   391 / 348 / 320
template <int WARPS>
static void tail_count(const TileArgs& t, int64_t segs, const LaunchCtx& ctx)
{
    static const int per_sm = ctas_per_sm(k_tail_count<WARPS>, 32 * WARPS);
    const int blocks = (int)std::min<int64_t>(segs, (int64_t)ctx.num_sms * per_sm);
    launch_kernel(k_tail_count<WARPS>, blocks, 32 * WARPS, 0, ctx.stream, t);
}

template <int COLS>
static void tile_write(const TileArgs& t, int64_t items, const LaunchCtx& ctx)
{
    static const int per_sm = ctas_per_sm(k_tile_write<COLS>, 32 * 64 / COLS);
    const int blocks = (int)std::min<int64_t>(items, (int64_t)ctx.num_sms * per_sm);
    launch_kernel(k_tile_write<COLS>, blocks, 32 * 64 / COLS, 0, ctx.stream, t);
}

// Whether a call takes k_small_lists: a list may hold every row of its view, and
// its blocks, which fill an SM, run in one wave.  A block also reads the rows of
// the views before its own, up to four times 8192 in all: 4 views of 8000 rows at
// 400x300 take 50 us instead of 53, 8 of 4000 at 300x200 48 instead of 52, but 16
// of 8000 at 200x150 70 instead of 60.
static bool small_lists(int64_t n, int64_t n_rows, int64_t total_super, int num_sms)
{
    return n <= kSmallRows && n_rows <= 4 * kSmallRows && total_super <= num_sms;
}

static cudaError_t run_pass(const PassArgs& a, int64_t parts, int resident, cudaStream_t s)
{
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(parts, resident));
    count_launch();
    if (a.ballot_rank)
        k_onesweep<true><<<blocks, kSortThreads, 0, s>>>(a);
    else
        k_onesweep<false><<<blocks, kSortThreads, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_bin_sort(const splat_proj& proj, const ViewBatch& vb, const splat_bins& bins, int32_t* status,
                            void* ws, const LaunchCtx& ctx)
{
    const int64_t n_rows = proj.n * vb.V;
    int TXs[SPLAT_MAX_VIEWS], TYs[SPLAT_MAX_VIEWS];
    for (int v = 0; v < vb.V; ++v) {
        TXs[v] = vb.v[v].TX;
        TYs[v] = vb.v[v].TY;
    }
    const SortLayout L = sort_layout(n_rows, bins.capacity, vb.V, TXs, TYs, ctx.tile_sort);
    if (!L.binned && bins.capacity > 0 && !bins.keys) return cudaErrorInvalidValue;
    char* w = (char*)ws;
    auto U = [&](size_t off) { return (uint32_t*)(w + off); };
    cudaStream_t s = ctx.stream;
    cudaError_t err;
    // (k_small_lists clears what its call needs)
    const bool small = L.binned && n_rows > 0 && small_lists(proj.n, n_rows, L.total_super, ctx.num_sms);
    if (!small && (err = cudaMemsetAsync(w + L.zero_begin, 0, L.zero_end - L.zero_begin, s)) != cudaSuccess) return err;
    if (n_rows == 0 || !L.binned) {  // (k_cell_count clears them otherwise)
        if ((err = cudaMemsetAsync(bins.ranges, 0, sizeof(uint32_t) * 2 * (size_t)vb.total_tiles, s)) != cudaSuccess)
            return err;
        if ((err = cudaMemsetAsync(bins.n_instances, 0, sizeof(int64_t), s)) != cudaSuccess) return err;
        if (bins.n_needed && (err = cudaMemsetAsync(bins.n_needed, 0, sizeof(int64_t), s)) != cudaSuccess) return err;
    }
    if (n_rows == 0) return cudaSuccess;
    uint32_t* tickets = U(L.off_tickets);
    if (L.binned) {
        // super-tile grids
        int super_base[SPLAT_MAX_VIEWS + 1], STX[SPLAT_MAX_VIEWS];
        int sb = 0;
        for (int v = 0; v < vb.V; ++v) {
            super_base[v] = sb;
            STX[v] = (vb.v[v].TX + 7) >> kSuperShift;
            sb += STX[v] * ((vb.v[v].TY + 7) >> kSuperShift);
        }
        super_base[vb.V] = sb;
        // 1. the super-tile lists, unsorted inside their cells.  The lists (K1 entries) live in a
        // capacity-sized buffer, so K1 is checked by the scan, before anything is written (K itself is
        // checked by the tile ranges once the tile lists are counted)
        const int long_heads = sb >= 2 * ctx.num_sms;  // (see k_head_count)
        CellArgs c{};
        c.proj = proj;
        c.V = vb.V;
        c.bin_bits = L.bin_bits;
        c.copies = L.copies;
        c.nbins = 1 << L.bin_bits;
        c.n = proj.n;
        c.range = (uint2*)(w + L.off_range);
        c.split = (unsigned long long*)(w + L.off_split);
        for (int v = 0; v < vb.V; ++v) c.STX[v] = STX[v];
        for (int v = 0; v <= vb.V; ++v) c.super_base[v] = super_base[v];
        c.rec = (uint2*)(w + L.off_rec);
        c.cell = U(L.off_cell);
        c.entries = (uint2*)(w + L.off_mask);
        c.capacity = bins.capacity;
        c.lb = (unsigned long long*)(w + L.off_cell_lb);
        c.ticket = tickets;
        c.sranges = (uint2*)(w + L.off_sranges);
        c.K1 = (int64_t*)(w + L.off_ninst1);
        c.queue = (uint4*)(w + L.off_queue);
        c.n_queue = U(L.off_nqueue);
        c.queue_cap = L.queue_cap;
        c.total_super = sb;
        c.long_heads = long_heads;
        c.status = status;
        c.spin_limit = ctx.spin_limit;
        c.ranges = (uint2*)bins.ranges;
        c.total_tiles = vb.total_tiles;
        c.n_instances = bins.n_instances;
        c.n_needed = bins.n_needed;
        auto row_grid = [&](int rows) { return dim3((unsigned)((proj.n + rows - 1) / rows), (unsigned)vb.V); };
        if (small) {
            SmallArgs sm{c, U(L.off_vals1), (uint32_t*)(w + L.zero_begin), (int)((L.off_cell - L.zero_begin) / 4)};
            constexpr int smem = (int)sizeof(SortSmem<kSmallThreads>);
            err = cudaFuncSetAttribute(k_small_lists, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (err != cudaSuccess) return err;  // (set for the current device)
            count_launch();
            launch_kernel(k_small_lists, sb, kSmallThreads, smem, s, sm);
        } else {
            count_launch(3);
            launch_kernel(k_cell_count, row_grid(256 * kRowsPerThread), 256, 0, s, c);
            launch_kernel(k_cell_scan, sb, 256, 0, s, c);
            launch_kernel(k_cell_scatter, row_grid(256), 256, 0, s, c);
        }
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
        // 2. the units of each list that the head pass takes, in order
        SortArgs u{};
        u.sranges = (const uint2*)(w + L.off_sranges);
        u.total_super = sb;
        u.entries = (const unsigned long long*)(w + L.off_mask);
        u.list = U(L.off_vals1);
        u.queue = (const uint4*)(w + L.off_queue);
        u.n_queue = U(L.off_nqueue);
        u.queue_cap = L.queue_cap;
        u.sat_head = (const uint2*)(w + L.off_sathead);
        u.status = status;
        static const int per_sm_u[2] = {ctas_per_sm(k_unit_sort<false>, kUnitThreads),
                                          ctas_per_sm(k_unit_sort<true>, kUnitThreads)};
        auto blocks_u = [&](int rest) {
            return (int)std::min<int64_t>(L.queue_cap + (rest ? 0 : sb), (int64_t)ctx.num_sms * per_sm_u[rest]);
        };
        // 3. tile level: per-super-tile lists filtered into per-tile lists (see above)
        TileArgs t{};
        t.proj = proj;
        t.V = vb.V;
        t.n_rows = n_rows;
        t.total_tiles = vb.total_tiles;
        for (int v = 0; v < vb.V; ++v) {
            t.tile_base[v] = vb.v[v].tile_base;
            t.TX[v] = vb.v[v].TX;
            t.TY[v] = vb.v[v].TY;
            t.W[v] = vb.v[v].W;
            t.H[v] = vb.v[v].H;
            t.super_base[v] = super_base[v];
            t.STX[v] = STX[v];
        }
        t.tile_base[vb.V] = vb.total_tiles;
        t.super_base[vb.V] = sb;
        t.total_super = sb;
        t.tile_total = U(L.off_total);
        t.list = U(L.off_vals1);
        t.sranges = (const uint2*)(w + L.off_sranges);
        t.ranges = (const uint2*)bins.ranges;
        t.vals_out = bins.vals;
        t.keys_out = bins.keys;
        t.status = status;
        t.stats = ctx.stats;
        t.cull = ctx.tile_cull;
        t.seg_base = U(L.off_segbase);
        t.seg_cnt = U(L.off_segcnt);
        t.seg_super = U(L.off_segsuper);
        t.sat_head = (uint2*)(w + L.off_sathead);
        t.n_head = (uint2*)(w + L.off_nhead);
        t.long_heads = long_heads;
        t.mask = (uint2*)(w + L.off_mask);
        t.ticket = tickets + 1;
        TileRangeArgs tr{};
        tr.lb = (unsigned long long*)(w + L.off_rlb);
        tr.ticket = tickets + 4;
        tr.ranges = (uint2*)bins.ranges;
        tr.K_out = bins.n_instances;
        tr.capacity = bins.capacity;
        tr.K_super = (const int64_t*)(w + L.off_ninst1);
        tr.needed = bins.n_needed;
        tr.cls = bins.tile_order ? U(L.off_tord) : nullptr;
        tr.order = vb.total_tiles <= kRangeTiles ? bins.tile_order : nullptr;
        tr.spin_limit = ctx.spin_limit;
        // the head of each super-tile list in order (each tile's list up to its
        // saturation), the rest of the units and the tail in parallel segments, the
        // prefix over head and segments with the ranges, K and the capacity check,
        // then the heads' and segments' writes in one pass
        // warps per segment by the segments per SM (see tail_count)
        const int64_t segs = L.max_segs + sb;
        const int tier = segs <= 8 * (int64_t)ctx.num_sms ? 0 : (segs <= 48 * (int64_t)ctx.num_sms ? 1 : 2);
        count_launch(small ? 4 : 6);
        if (!small) launch_kernel(k_unit_sort<false>, blocks_u(0), kUnitThreads, 0, s, u);
        launch_kernel(k_head_count, 2 * sb, kHeadEntries, 0, s, t);
        if (!small) launch_kernel(k_unit_sort<true>, blocks_u(1), kUnitThreads, 0, s, u);
        if (tier == 0) tail_count<32>(t, L.max_segs, ctx);
        else if (tier == 1) tail_count<16>(t, L.max_segs, ctx);
        else tail_count<8>(t, L.max_segs, ctx);
        launch_kernel(k_tile_ranges, (int)((vb.total_tiles + kRangeTiles - 1) / kRangeTiles), 256, 0, s, t, tr);
        if (tier == 0) tile_write<2>(t, segs, ctx);
        else if (tier == 1) tile_write<4>(t, segs, ctx);
        else tile_write<8>(t, segs, ctx);
        if ((err = cudaGetLastError()) != cudaSuccess || tr.order) return err;
        return launch_tile_order(bins, L.total_tiles, U(L.off_tord), status, ctx, true);
    }
    // radix path: 1. depth keys + digit counts; zero the first depth look-back buffer and the scan's
    uint32_t* hist = U(L.off_hist);
    const int resident = ctx.num_sms * sort_ctas_per_sm();
    {
        DepthArgs a{};
        a.proj = proj;
        a.n_rows = n_rows;
        a.keys = U(L.off_dkeys[0]);
        a.vals = U(L.off_dvals[0]);
        a.dhist = hist;
        a.zero_a = U(L.off_dlb[0]);
        a.n_zero_a = L.parts_d * kRadix;
        a.zero_b = (unsigned long long*)(w + L.off_scan_lb);
        a.n_zero_b = L.parts_scan;
        const int blocks = (int)std::min<int64_t>((n_rows + 255) / 256, (int64_t)ctx.num_sms * 8);
        count_launch();
        k_depth_keys<<<blocks, 256, 0, s>>>(a);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    // 2. depth passes (buffers 0 -> 1 -> 0 -> 1 -> 0): all rows by depth, those without tiles last (the
    // duplication's chunks assume no such row between listed ones)
    const int passes = 4;
    for (int p = 0; p < passes; ++p) {
        PassArgs a{};
        a.keys_in = U(L.off_dkeys[p & 1]);
        a.vals_in = U(L.off_dvals[p & 1]);
        a.keys_out = p + 1 < passes ? U(L.off_dkeys[(p + 1) & 1]) : nullptr;
        a.vals_out = U(L.off_dvals[(p + 1) & 1]);
        a.n_dev = nullptr;
        a.n_host = n_rows;
        a.cap = n_rows;
        a.hist = hist + p * kRadix;
        a.lb = U(L.off_dlb[p & 1]);
        a.lb_next = p + 1 < passes ? U(L.off_dlb[(p + 1) & 1]) : nullptr;
        a.ticket = tickets + p;
        a.status = status;
        a.stage = SPLAT_STAGE_DEPTH_SORT;
        a.shift = 8 * p;
        a.spin_limit = ctx.spin_limit;
        a.ballot_rank = p < 3;  // the low depth digits take many values in a warp, the top one few
        if ((err = run_pass(a, L.parts_d, resident, s)) != cudaSuccess) return err;
    }
    const uint32_t* rows = U(L.off_dvals[passes & 1]);
    // 3. scan of the per-row tile counts in depth order
    {
        ScanArgs a{};
        a.rows = rows;
        a.n_tiles = proj.n_tiles;
        a.n_rows = n_rows;
        a.offsets = U(L.off_offsets);
        a.chunk_row = U(L.off_chunk);
        a.n_chunks_max = L.n_chunks;
        a.lb = (unsigned long long*)(w + L.off_scan_lb);
        a.ticket = tickets + 4;
        a.n_instances = bins.n_instances;
        a.n_needed = bins.n_needed;
        a.capacity = bins.capacity;
        a.status = status;
        a.spin_limit = ctx.spin_limit;
        const int blocks = (int)std::min<int64_t>(L.parts_scan, (int64_t)ctx.num_sms * 4);
        count_launch();
        k_scan_tiles<<<blocks, kScanThreads, 0, s>>>(a);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    // 4. duplicate, tile-digit passes, ranges
    int bits = 1;
    while ((1ll << bits) < (int64_t)vb.total_tiles) ++bits;
    const int tile_passes = (bits + 7) / 8;
    uint32_t* tk[2] = {U(L.off_tkeys), bins.keys};
    uint32_t* tv[2] = {U(L.off_tvals), bins.vals};
    // the last pass must land in bins: start in the workspace when the pass count is odd
    int cur = (tile_passes & 1) ? 0 : 1;
    {
        DupArgs a{};
        a.proj = proj;
        a.rows = rows;
        a.offsets = U(L.off_offsets);
        a.chunk_row = U(L.off_chunk);
        a.n_rows = n_rows;
        a.n_instances = bins.n_instances;
        a.capacity = bins.capacity;
        a.keys_out = tk[cur];
        a.vals_out = tv[cur];
        a.hist = hist + 4 * kRadix;
        a.tile_passes = tile_passes;
        a.zero = U(L.off_tlb[0]);
        a.status = status;
        for (int v = 0; v < vb.V; ++v) {
            a.tile_base[v] = vb.v[v].tile_base;
            a.TX[v] = vb.v[v].TX;
        }
        const int blocks = ctx.num_sms * 4;
        count_launch();
        k_duplicate<<<blocks, kDupThreads, 0, s>>>(a);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    for (int p = 0; p < tile_passes; ++p) {
        PassArgs a{};
        a.keys_in = tk[cur];
        a.vals_in = tv[cur];
        a.keys_out = tk[cur ^ 1];
        a.vals_out = tv[cur ^ 1];
        a.n_dev = bins.n_instances;
        a.n_host = 0;
        a.cap = bins.capacity;
        a.hist = hist + (4 + p) * kRadix;
        a.lb = U(L.off_tlb[p & 1]);
        a.lb_next = p + 1 < tile_passes ? U(L.off_tlb[(p + 1) & 1]) : nullptr;
        a.ticket = tickets + 5 + p;
        a.status = status;
        a.stage = SPLAT_STAGE_TILE_SORT;
        a.shift = 8 * p;
        a.spin_limit = ctx.spin_limit;
        if ((err = run_pass(a, L.parts_t, resident, s)) != cudaSuccess) return err;
        cur ^= 1;
    }
    {
        const int blocks = ctx.num_sms * 8;
        count_launch();
        k_ranges<<<blocks, 256, 0, s>>>(bins.keys, bins.n_instances, bins.capacity, (uint2*)bins.ranges, status);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    return launch_tile_order(bins, L.total_tiles, U(L.off_tord), status, ctx);
}

size_t bin_sort_workspace(int64_t n_rows, int64_t capacity, int V, const int* TX, const int* TY, int tile_sort)
{
    return sort_layout(n_rows, capacity, V, TX, TY, tile_sort).bytes;
}

}  // namespace splat
