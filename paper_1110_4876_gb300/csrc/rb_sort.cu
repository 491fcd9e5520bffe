// rb_sort.cu -- stable LSD radix sort of (64-bit key, 32-bit value) pairs,
// sized on the device.
//
// The sort replaces the insertion/reconstruction of the paper's tree
// (Sect. 4.2): particles are put in Morton order so that every cell is a
// contiguous range.  One launch counts the digits of every pass; then each
// 8-bit digit pass is one launch that ranks keys within a tile with warp
// ballots and finds the tile's place among the earlier tiles by a
// bounded decoupled look-back over per-tile status words.
#include <algorithm>

#include "rb_internal.cuh"

namespace rb {

namespace {
constexpr int kThreads = 256;
constexpr int kItems = 8;
constexpr int kTile = kThreads * kItems;   // 2048 keys per block
constexpr int kBins = 256;

__device__ __forceinline__ int read_n(const int* d_n, int ncap) {
    if (!d_n) return ncap;
    int n = *d_n;
    return n < ncap ? n : ncap;
}

// Status words of the decoupled look-back: a tile's count of one digit with
// a two-bit flag (0: not yet published, aggregate: this tile's own count,
// prefix: this tile's count plus every earlier tile's).  Flag and count
// share one 32-bit word, so a single store publishes both.
constexpr uint32_t kFlagAgg = 1u << 30;
constexpr uint32_t kFlagPre = 2u << 30;
constexpr uint32_t kCountMask = (1u << 30) - 1u;
constexpr int kMaxPasses = 12;   // 64-bit keys: 8 digits; 32-bit box digits: 4
constexpr int kLongCount = (kMaxPasses - 1) * kBins;   // word of hist that counts long runs (no pass's total)
constexpr int kLook = 16;   // predecessors read per look-back step
constexpr unsigned long long kLookLimitNs = 500000000ull;   // half a second

__device__ __forceinline__ unsigned long long sort_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The lanes of act whose 8-bit digit equals this lane's: one ballot per
// digit bit (a match-any vote through eight ballots; a pass with them took
// 21 us at 1M keys against 23 us with the match instruction).  Every lane of
// the warp must call it.
__device__ __forceinline__ unsigned digit_peers(unsigned act, uint32_t d) {
    unsigned peers = act;
#pragma unroll
    for (int b = 0; b < 8; b++) {
        const bool bit = (d >> b) & 1u;
        const unsigned m = __ballot_sync(0xffffffffu, bit);
        peers &= bit ? m : ~m;
    }
    return peers;
}

// Digit counts of every pass in one read of the keys (the digit multiset of
// a pass does not depend on the order the earlier passes leave), plus the
// zeroing of both status banks for the tiles in use.  A thread counts
// kItems consecutive keys and adds each run of equal digits with one shared
// atomic: nearly sorted keys share their high digits over long runs.
// hist[p * 256 + d] must be zero on entry (the caller clears it).
template <bool kHasBox>
__global__ void __launch_bounds__(kThreads) k_rs_hist(const uint64_t* __restrict__ key,
                                                      const uint32_t* __restrict__ val,
                                                      const int32_t* __restrict__ box,
                                                      const int* d_n, int ncap, int low_bit,
                                                      int passes_key, int passes_box,
                                                      uint32_t* __restrict__ hist,
                                                      uint32_t* __restrict__ status, int tiles_cap,
                                                      Ctl* pairs, unsigned long long* long_keys) {
    __shared__ uint32_t h[kMaxPasses][kBins];
    const int P = passes_key + passes_box;
    for (int i = threadIdx.x; i < P * kBins; i += kThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    int n;
    if (pairs) {
        const int c = pairs->pair_count;
        n = c <= ncap ? c : 0;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            pairs->pair_n = n;
            pairs->resolved = 0;
        }
    } else {
        n = read_n(d_n, ncap);
    }
    if (low_bit > 0 && blockIdx.x == 0 && threadIdx.x == 0) {
        hist[kLongCount] = 0u;
        if (long_keys) *long_keys = 0;
    }
    const int nt = (n + kTile - 1) / kTile;
    const size_t rows = (size_t)nt * kBins;
    const size_t stride = (size_t)gridDim.x * kThreads;
    for (size_t w = (size_t)blockIdx.x * kThreads + threadIdx.x; w < 2 * rows; w += stride) {
        const size_t bank = w >= rows ? 1 : 0;
        status[bank * (size_t)tiles_cap * kBins + (w - bank * rows)] = 0u;
    }
    for (long long i0 = ((long long)blockIdx.x * kThreads + threadIdx.x) * kItems; i0 < n;
         i0 += (long long)stride * kItems) {
        const int c = (int)min((long long)kItems, (long long)n - i0);
        uint64_t k[kItems];
        uint32_t bd[kItems];
#pragma unroll
        for (int r = 0; r < kItems; r++) {
            k[r] = r < c ? key[i0 + r] : 0ull;
            bd[r] = kHasBox && r < c ? (uint32_t)box[val[i0 + r]] : 0u;
        }
        for (int p = 0; p < P; p++) {
            const bool bp = kHasBox && p >= passes_key;
            const int sh = bp ? 8 * (p - passes_key) : low_bit + 8 * p;
            uint32_t run_d = bp ? (bd[0] >> sh) & 255u : (uint32_t)(k[0] >> sh) & 255u;
            uint32_t run_c = 1;
#pragma unroll
            for (int r = 1; r < kItems; r++) {
                if (r < c) {
                    const uint32_t dg = bp ? (bd[r] >> sh) & 255u : (uint32_t)(k[r] >> sh) & 255u;
                    if (dg == run_d) {
                        run_c++;
                    } else {
                        atomicAdd(&h[p][run_d], run_c);
                        run_d = dg;
                        run_c = 1;
                    }
                }
            }
            atomicAdd(&h[p][run_d], run_c);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < P * kBins; i += kThreads) {
        const uint32_t c = (&h[0][0])[i];
        if (c) atomicAdd(&hist[i], c);
    }
}

// One digit pass, one launch: block b takes tile b (2048 keys).  It ranks
// the tile's keys with warp ballots, publishes its per-digit counts, finds
// the counts of all earlier tiles by looking back over their status words
// (decoupled look-back: sum aggregates until a prefix is met), and writes
// the tile in digit order.  A tile waits only on smaller tiles, whose blocks
// the GPU dispatched before it (blocks start in index order) and which
// publish before they wait themselves, so the waits end whether or not the
// whole grid is resident, also beside other kernels; each wait is bounded
// all the same (half a second, or at once when another wait gave up) and
// reports kErrSortStall when it gives up.  Stable: within a tile keys keep
// their order, and the tiles are in key order.
template <bool kBoxDigit>
__global__ void __launch_bounds__(kThreads, 4) k_rs_pass(const uint64_t* __restrict__ kin,
                                                      const uint32_t* __restrict__ vin,
                                                      uint64_t* __restrict__ kout,
                                                      uint32_t* __restrict__ vout,
                                                      const int32_t* __restrict__ box,
                                                      const int* d_n, int ncap, int shift, int pass,
                                                      const uint32_t* __restrict__ hist,
                                                      uint32_t* __restrict__ status, int tiles_cap,
                                                      int* __restrict__ err, bool hold) {
    __shared__ uint32_t wcnt[kThreads / 32][kBins];
    __shared__ uint32_t gstart[kBins];   // where digit d of this tile starts in the output
    __shared__ uint32_t lstart[kBins];   // where digit d starts inside the tile
    __shared__ uint32_t wsum[kThreads / 32];
    __shared__ uint64_t sk[kTile];
    __shared__ uint32_t sv[kTile];
    const int n = read_n(d_n, ncap);
    if ((long long)blockIdx.x * kTile >= n) return;   // past the keys in use
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int d = threadIdx.x;   // the digit this thread counts and looks back for
    uint32_t* mine = status + (size_t)(pass & 1) * tiles_cap * kBins;
    uint32_t* other = status + (size_t)((pass & 1) ^ 1) * tiles_cap * kBins;
    uint32_t digit_base;
    {
        // exclusive scan of this pass's digit totals: where digit d starts
        const uint32_t tot = hist[pass * kBins + d];
        uint32_t v = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += t;
        }
        if (lane == 31) wsum[warp] = v;
        __syncthreads();
        uint32_t before = 0;
        for (int w = 0; w < warp; w++) before += wsum[w];
        digit_base = before + v - tot;
    }
    const unsigned lt = (1u << lane) - 1u;
    const int tile = blockIdx.x;
    if (tile * kTile < n) {
        const int base = tile * kTile;
        const int tn = min(kTile, n - base);
        // the other bank held the previous pass's words; clear this tile's
        // row of it for the next pass
        other[(size_t)tile * kBins + d] = 0u;
        for (int q = threadIdx.x; q < (kThreads / 32) * kBins; q += kThreads) (&wcnt[0][0])[q] = 0;
        __syncthreads();
        uint64_t k[kItems];
        uint32_t v[kItems];
        uint32_t pos[kItems];
        int dig[kItems];
        const int wbase = base + warp * (kTile / (kThreads / 32));
        // all loads first: the ranking below orders shared-memory updates
        // with __syncwarp, which would otherwise keep each item's loads
        // behind the previous item's
#pragma unroll
        for (int r = 0; r < kItems; r++) {
            const int i = wbase + r * 32 + lane;
            const bool ok = i < n;
            k[r] = ok ? kin[i] : 0ull;
            v[r] = ok ? vin[i] : 0u;
        }
#pragma unroll
        for (int r = 0; r < kItems; r++) {
            const bool ok = wbase + r * 32 + lane < n;
            int dd = 0;
            if (ok) dd = kBoxDigit ? (int)((box[v[r]] >> shift) & 255) : (int)((k[r] >> shift) & 255ull);
            dig[r] = ok ? dd : -1;
        }
#pragma unroll
        for (int r = 0; r < kItems; r++) {
            const bool ok = dig[r] >= 0;
            const int dd = ok ? dig[r] : 0;
            const unsigned act = __ballot_sync(0xffffffffu, ok);
            const unsigned peers = digit_peers(act, (uint32_t)dd);
            pos[r] = 0;
            if (ok) {
                const int rank = __popc(peers & lt);
                const uint32_t c = wcnt[warp][dd];
                pos[r] = c + rank;
                __syncwarp(act);
                if (rank == 0) wcnt[warp][dd] = c + __popc(peers);
                __syncwarp(act);
            }
        }
        __syncthreads();
        uint32_t cnt = 0;   // this tile's keys of digit d
#pragma unroll
        for (int w = 0; w < kThreads / 32; w++) {
            const uint32_t x = wcnt[w][d];
            wcnt[w][d] = cnt;
            cnt += x;
        }
        volatile uint32_t* row = mine + (size_t)tile * kBins;
        if (!hold || tile > 0) row[d] = (tile == 0 ? kFlagPre : kFlagAgg) | cnt;
        {
            // where digit d starts inside the tile (block scan of the counts)
            uint32_t x = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += t;
            }
            if (lane == 31) wsum[warp] = x;
            __syncthreads();
            uint32_t before = 0;
            for (int w = 0; w < warp; w++) before += wsum[w];
            lstart[d] = before + x - cnt;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kItems; r++) {
            if (dig[r] >= 0) {
                const uint32_t lp = lstart[dig[r]] + wcnt[warp][dig[r]] + pos[r];
                sk[lp] = k[r];
                sv[lp] = v[r];
            }
        }
        // look back: keys of digit d in all earlier tiles.  The tiles of a
        // pass start together, so a walk that read one predecessor per L2
        // round trip would take about sqrt(2 tile) trips; each step reads a
        // window of kLook predecessors at once and sums them from the nearest
        // down to the first prefix, or up to the first tile that has not
        // published yet (read again next step).
        uint32_t excl = 0;
        if (tile > 0) {
            const volatile uint32_t* col = mine + d;
            int j = tile - 1;   // nearest tile not yet counted
            unsigned long long t0 = 0;
            for (;;) {
                uint32_t w[kLook];
#pragma unroll
                for (int q = 0; q < kLook; q++) w[q] = j - q >= 0 ? col[(size_t)(j - q) * kBins] : kFlagPre;
                int used = 0;
                bool done = false;
#pragma unroll
                for (int q = 0; q < kLook; q++) {
                    if (!done && used == q && (w[q] & (kFlagAgg | kFlagPre))) {
                        excl += w[q] & kCountMask;
                        used++;
                        done = (w[q] & kFlagPre) != 0;
                    }
                }
                if (done) break;
                j -= used;
                if (used == kLook) continue;
                // tile j has not published yet
                if (t0 == 0) {
                    t0 = sort_ns();
                } else if ((*(volatile int*)err & kErrSortStall) || sort_ns() - t0 > kLookLimitNs) {
                    atomicOr(err, kErrSortStall);
                    break;
                }
                __nanosleep(32);
            }
            row[d] = kFlagPre | ((excl + cnt) & kCountMask);
        }
        gstart[d] = digit_base + excl;
        __syncthreads();
        for (int j = threadIdx.x; j < tn; j += kThreads) {
            const uint64_t kk = sk[j];
            const uint32_t vv = sv[j];
            const int dd = kBoxDigit ? (int)((box[vv] >> shift) & 255) : (int)((kk >> shift) & 255ull);
            const uint32_t p = gstart[dd] + ((uint32_t)j - lstart[dd]);
            if (p < (uint32_t)n) {   // always true unless a look-back gave up
                kout[p] = kk;
                vout[p] = vv;
            }
        }
    }
}

// ---- runs of keys that agree in the sorted bits ----
//
// A sort by the high bits of the keys leaves each run of keys that agree there
// in input order.  Where such runs are short (Morton keys cut at depth 13,
// pairs sorted by one particle), putting them in order afterwards costs less
// than the passes over the low bits: particles by 40 of 64 bits 209 -> 168 us
// at 1M (with the gather) and 64 -> 48 us at 20k, pairs by the lower id alone
// 125 -> 76 and 52 -> 28 us.
constexpr int kShortRun = 16;   // runs up to this length: by one thread, in place
constexpr int kSlowRun = 2048;  // runs above this length take a block longer than the passes they save

// Do neighbours a, b (a = b - 1) belong to one run?
__device__ __forceinline__ bool same_run(const uint64_t* key, const uint32_t* val, const int32_t* box, int low_bit,
                                         int a, int b) {
    return ((key[a] ^ key[b]) >> low_bit) == 0ull && (!box || box[val[a]] == box[val[b]]);
}

// Insertion sort (stable) of every run of up to kShortRun keys by the thread
// of its first key; the first keys of longer runs are listed.  Keys of all
// ones (removed particles) are equal and stay as they are, and so do all keys
// after a pass whose look-back gave up: there the runs are not together, and
// blocks at parts of one would write over each other's.
__global__ void __launch_bounds__(256) k_rs_runs(uint64_t* __restrict__ key, uint32_t* __restrict__ val,
                                                 const int32_t* __restrict__ box, const int* d_n, int ncap,
                                                 int low_bit, uint32_t* __restrict__ hist,
                                                 uint32_t* __restrict__ list, const int* __restrict__ err) {
    const int gave_up = *err & kErrSortStall, keys = read_n(d_n, ncap);
    const int n = gave_up ? 0 : keys;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    // the digit totals are done with: zero for the next sort
    for (int k = i; k < kLongCount; k += gridDim.x * blockDim.x) hist[k] = 0u;
    bool many = false;
    if (i + 1 < n && key[i] != ~0ull && same_run(key, val, box, low_bit, i, i + 1) &&
        (i == 0 || !same_run(key, val, box, low_bit, i - 1, i))) {
        int len = 2;
        while (len <= kShortRun && i + len < n && same_run(key, val, box, low_bit, i + len - 1, i + len)) len++;
        many = len > kShortRun;
        for (int a = 1; a < len && !many; a++) {
            const uint64_t k = key[i + a];
            int b = a;
            if (key[i + b - 1] > k) {
                const uint32_t v = val[i + a];
                do {
                    key[i + b] = key[i + b - 1];
                    val[i + b] = val[i + b - 1];
                    b--;
                } while (b > 0 && key[i + b - 1] > k);
                key[i + b] = k;
                val[i + b] = v;
            }
        }
    }
    if (many) list[atomicAdd(&hist[kLongCount], 1u)] = (uint32_t)i;
}

// The listed runs, a block each: nothing to do if in order already (equal
// keys), else LSD passes over the low bits, 8 at a time, by one block through
// the other buffers.
__global__ void __launch_bounds__(kThreads) k_rs_long(uint64_t* __restrict__ k0, uint32_t* __restrict__ v0,
                                                      uint64_t* __restrict__ k1, uint32_t* __restrict__ v1,
                                                      const int32_t* __restrict__ box, const int* d_n, int ncap,
                                                      int low_bit, const uint32_t* __restrict__ nlong,
                                                      const uint32_t* __restrict__ list,
                                                      unsigned long long* long_keys) {
    __shared__ uint32_t wcnt[kThreads / 32][kBins], base[kBins], wsum[kThreads / 32];
    __shared__ int end_s;
    const int n = read_n(d_n, ncap), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t runs = *nlong;
    for (uint32_t r = blockIdx.x; r < runs; r += gridDim.x) {
        const int i0 = (int)list[r];
        if (tid == 0) {
            // the run's end: doubling steps, then halving
            int good = i0 + kShortRun, bad = n, step = kShortRun;
            auto in = [&](int j) {
                return ((k0[i0] ^ k0[j]) >> low_bit) == 0ull && (!box || box[v0[i0]] == box[v0[j]]);
            };
            for (;;) {
                const int j = good + step;
                if (j >= n) break;
                if (!in(j)) {
                    bad = j;
                    break;
                }
                good = j;
                step <<= 1;
            }
            while (bad - good > 1) {
                const int mid = good + (bad - good) / 2;
                if (in(mid)) good = mid; else bad = mid;
            }
            end_s = bad;
            // what the run costs: its keys, and as much as all keys if one block is long at it
            if (long_keys) atomicAdd(long_keys, (unsigned long long)(bad - i0 > kSlowRun ? n : bad - i0));
        }
        __syncthreads();
        const int i1 = end_s;
        bool unordered = false;
        for (int j = i0 + 1 + tid; j < i1; j += kThreads) unordered = unordered || k0[j - 1] > k0[j];
        if (!__syncthreads_or(unordered)) continue;
        uint64_t *ki = k0, *ko = k1;
        uint32_t *vi = v0, *vo = v1;
        for (int sh = 0; sh < low_bit; sh += 8) {
            const uint64_t mask = low_bit - sh >= 8 ? 255ull : (1ull << (low_bit - sh)) - 1ull;
            for (int q = tid; q < (kThreads / 32) * kBins; q += kThreads) (&wcnt[0][0])[q] = 0;
            __syncthreads();
            for (int j = i0 + tid; j < i1; j += kThreads) atomicAdd(&wcnt[0][(ki[j] >> sh) & mask], 1u);
            __syncthreads();
            {
                const uint32_t c = wcnt[0][tid];
                uint32_t x = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += t;
                }
                if (lane == 31) wsum[warp] = x;
                __syncthreads();
                uint32_t before = 0;
                for (int w = 0; w < warp; w++) before += wsum[w];
                base[tid] = (uint32_t)i0 + before + x - c;
                wcnt[0][tid] = 0;
            }
            __syncthreads();
            for (int c0 = i0; c0 < i1; c0 += kThreads) {
                const int j = c0 + tid;
                const bool ok = j < i1;
                const uint64_t k = ok ? ki[j] : 0ull;
                const uint32_t v = ok ? vi[j] : 0u;
                const uint32_t d = ok ? (uint32_t)((k >> sh) & mask) : 0u;
                const unsigned peers = digit_peers(__ballot_sync(0xffffffffu, ok), d);
                const int rank = __popc(peers & ((1u << lane) - 1u));
                if (ok && rank == 0) wcnt[warp][d] = __popc(peers);
                __syncthreads();
                // per digit: where each warp's keys go, then the next chunk's start
                uint32_t at = base[tid];
#pragma unroll
                for (int w = 0; w < kThreads / 32; w++) {
                    const uint32_t x = wcnt[w][tid];
                    wcnt[w][tid] = at;
                    at += x;
                }
                base[tid] = at;
                __syncthreads();
                if (ok) {
                    const uint32_t p = wcnt[warp][d] + rank;
                    ko[p] = k;
                    vo[p] = v;
                }
                __syncthreads();
#pragma unroll
                for (int w = 0; w < kThreads / 32; w++) wcnt[w][tid] = 0;
                __syncthreads();
            }
            uint64_t* tk = ki; ki = ko; ko = tk;
            uint32_t* tv = vi; vi = vo; vo = tv;
        }
        if (ki != k0)
            for (int j = i0 + tid; j < i1; j += kThreads) {
                k0[j] = ki[j];
                v0[j] = vi[j];
            }
        __syncthreads();
    }
}

}  // namespace

// Digit totals of every pass, then two banks of per-tile status words.
size_t radix_hist_words(int ncap) {
    return (size_t)kMaxPasses * kBins +
           2 * (size_t)kBins * (size_t)ceil_div(ncap > 0 ? ncap : 1, kTile);
}

size_t radix_digit_words() { return (size_t)kMaxPasses * kBins; }

int radix_sort(uint64_t* k0, uint32_t* v0, uint64_t* k1, uint32_t* v1, int ncap, const int* d_n,
               int key_bits, const int32_t* box_digits, int box_bits, uint32_t* hist, int* err,
               cudaStream_t s, int low_bit, Ctl* pairs, unsigned long long* long_keys, bool hold) {
    if (ncap <= 0) return 0;
    const int tiles_cap = ceil_div(ncap, kTile);
    uint32_t* status = hist + kMaxPasses * kBins;
    const int passes_key = ceil_div(key_bits - low_bit, 8);
    const int passes_box = box_digits ? ceil_div(box_bits, 8) : 0;
    // digit totals start at zero (k_rs_runs leaves them so); the status banks
    // are cleared by the kernels, for the tiles in use only
    if (low_bit == 0) cudaMemsetAsync(hist, 0, sizeof(uint32_t) * kMaxPasses * kBins, s);
    const int hgrid = std::max(1, std::min(ceil_div(ncap, 8 * kThreads), 1024));
    if (box_digits)
        k_rs_hist<true><<<hgrid, kThreads, 0, s>>>(k0, v0, box_digits, d_n, ncap, low_bit,
                                                   passes_key, passes_box, hist, status, tiles_cap, pairs,
                                                   long_keys);
    else
        k_rs_hist<false><<<hgrid, kThreads, 0, s>>>(k0, v0, nullptr, d_n, ncap, low_bit, passes_key, 0, hist,
                                                    status, tiles_cap, pairs, long_keys);
    int cur = 0;
    uint64_t* K[2] = {k0, k1};
    uint32_t* V[2] = {v0, v1};
    for (int p = 0; p < passes_key + passes_box; p++) {
        const bool boxp = p >= passes_key;
        const int sh = boxp ? 8 * (p - passes_key) : low_bit + 8 * p;
        if (boxp)
            k_rs_pass<true><<<tiles_cap, kThreads, 0, s>>>(K[cur], V[cur], K[cur ^ 1], V[cur ^ 1],
                                                           box_digits, d_n, ncap, sh, p, hist,
                                                           status, tiles_cap, err, hold);
        else
            k_rs_pass<false><<<tiles_cap, kThreads, 0, s>>>(K[cur], V[cur], K[cur ^ 1], V[cur ^ 1],
                                                            nullptr, d_n, ncap, sh, p, hist, status,
                                                            tiles_cap, err, hold);
        cur ^= 1;
    }
    if (low_bit > 0) {
        // the list of long runs takes the status words, which the passes are
        // done with (at most one run per kShortRun + 1 keys)
        const uint32_t* nlong = hist + kLongCount;
        k_rs_runs<<<ceil_div(ncap, 256), 256, 0, s>>>(K[cur], V[cur], box_digits, d_n, ncap, low_bit, hist, status,
                                                        err);
        k_rs_long<<<std::min(ceil_div(ncap, kShortRun), 152), kThreads, 0, s>>>(
            K[cur], V[cur], K[cur ^ 1], V[cur ^ 1], box_digits, d_n, ncap, low_bit, nlong, status, long_keys);
    }
    return cur;
}

}  // namespace rb
