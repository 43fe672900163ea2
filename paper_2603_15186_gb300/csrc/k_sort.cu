// K5: stable least-significant-digit radix sort of (key, value) pairs in the
// "onesweep" arrangement: one upsweep kernel builds the digit histograms of
// every pass from a single read of the keys, then each 8-bit digit pass is one
// kernel that ranks a 4096-key partition in shared memory and finds, for each
// of the 256 digits, the partition's global offset by decoupled look-back over
// the preceding partitions (no separate scan kernel per pass).
//
// Stability: keys are loaded warp-striped (item i of lane l is key
// base + 32 ITEMS w + 32 i + l), each warp ranks its items in that order (peers
// = lanes holding the same digit, from one shared-memory OR of lane bits per
// item), warps are offset in order, and partitions in ticket order; equal
// digits therefore keep their input order, which is what the two-stage binning
// needs.
//
// Forward progress: partition ids come from an atomic ticket, so every
// partition a look-back waits on is held by a CTA that is already running.
// Every wait is bounded (kSpinLimit) and latches kErrTimeout if it runs out.
//
// Depth keys of a scene within 13 km (every camera's means' bounds are checked on the
// host) are sorted by three digits of 9 bits instead of four of 8: the 118.8 M records of
// 256 mixed views in 2.17 ms instead of 2.72 ms, a 13k-node scene's 1269 in 16 us instead of
// 25 us, and a launch less. A thread per digit leaves no thread idle in the look-back.
//
// HBM per pass: read key + value, write key + value (16 B/pair for 32-bit
// keys, 24 B for 64-bit), plus the upsweep's one read of the keys.
// Partitions are 8192 keys (32-bit) or 4096 (64-bit) over 512 threads: long
// runs per digit keep the scattered writes close to whole sectors, and values
// are read only once the keys are ranked, which keeps two CTAs resident.
#include <algorithm>

#include "ngs_internal.cuh"

namespace ngs {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kRadix = 256;
constexpr int kMaxPasses = 8;

int sort_passes(int begin_bit, int end_bit) { return (end_bit - begin_bit + 7) / 8; }

template <typename K>
__device__ __forceinline__ uint32_t digit_of(K key, int shift, uint32_t mask) {
    return (uint32_t)(key >> shift) & mask;
}

// kUp keys per thread are requested at once, eight CTAs per SM: 12.3M 32-bit keys in
// 28 us (84 us with one key at a time and two CTAs per SM, a chain of memory round
// trips). The CTA that is done last scans the digits.
constexpr int kUp = 8;

template <typename K>
__global__ void __launch_bounds__(kSortThreads)
k_upsweep(const K *__restrict__ keys, const uint32_t *n_dev, int64_t n_host, int begin_bit,
          int end_bit, uint32_t *hist, uint32_t *done, const int *err) {
    __shared__ uint32_t s_h[kMaxPasses][kRadix];
    __shared__ uint32_t s_last, s_warp[kSortWarps];
    if (*err) return;
    const int passes = (end_bit - begin_bit + 7) / 8;
    for (int i = threadIdx.x; i < passes * kRadix; i += kSortThreads) (&s_h[0][0])[i] = 0;
    __syncthreads();
    const int64_t n = n_dev ? (int64_t)*n_dev : n_host;
    for (int64_t i0 = (int64_t)blockIdx.x * kSortThreads * kUp + threadIdx.x; i0 < n;
         i0 += (int64_t)gridDim.x * kSortThreads * kUp) {
        K k[kUp];
#pragma unroll
        for (int u = 0; u < kUp; ++u) {
            const int64_t i = i0 + u * kSortThreads;
            k[u] = i < n ? keys[i] : (K)0;
        }
#pragma unroll
        for (int u = 0; u < kUp; ++u) {
            if (i0 + u * kSortThreads >= n) break;
            for (int p = 0; p < passes; ++p) {
                const int sh = begin_bit + 8 * p;
                const int bits = min(8, end_bit - sh);
                atomicAdd(&s_h[p][digit_of(k[u], sh, (1u << bits) - 1u)], 1u);
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * kRadix; i += kSortThreads) {
        const uint32_t v = (&s_h[0][0])[i];
        if (v) atomicAdd(&hist[i], v);
    }
    digit_scan_by_last<kRadix>(hist, passes, done, &s_last, s_warp);
}

constexpr int kOsWarps = kOsThreads / 32;

// BITS: digit width, 8 or (depth keys) 9 bits.
template <typename K, int BITS>
struct SortSmem {
    static constexpr int kPart = kOsPart<K>;
    static constexpr int kDigits = 1 << BITS;
    uint32_t whist[kOsWarps][kDigits];    // per-warp digit counts, then warp offsets
    // per-warp lane masks of one item's digits (kept 0); 512 digits' share the values'
    // place, which are staged after the ranking, so that two CTAs fit an SM
    uint32_t match[BITS == 8 ? kOsWarps : 1][BITS == 8 ? kDigits : 1];
    uint32_t gstart[kDigits];             // global output position of staged slot 0 of each digit's run
    uint32_t wtot[kDigits / 32];
    K keys[kPart];
    uint32_t vals[kPart];
    uint32_t part;
};

// kOut: 0 writes keys and values; 1 values only (last pass of a sort whose
// keys are not needed afterwards); 2 values only, plus the [first, end) range
// of every key in the sorted output (last pass of the tile sort, 32-bit keys):
// within a partition equal keys are adjacent in the staged order and land on
// consecutive output positions, so each run of equal keys contributes its
// first and end position with one atomicMax each (first stored as ~first), and
// the runs a key has in several partitions combine to its global range.
template <typename K, int kOut, int BITS>
__global__ void __launch_bounds__(kOsThreads, 2)
k_onesweep(const K *__restrict__ kin, const uint32_t *__restrict__ vin, K *__restrict__ kout,
           uint32_t *__restrict__ vout, const uint32_t *n_dev, int64_t n_host, int shift,
           uint32_t mask, const uint32_t *__restrict__ digit_base, uint64_t *status,
           uint32_t *ticket, const uint32_t *epoch_ptr, uint32_t epoch_off, int *err,
           uint2 *__restrict__ ranges) {
    constexpr int ITEMS = SortShape<K>::kItems;
    using Smem = SortSmem<K, BITS>;
    constexpr int PART = Smem::kPart, kRadix = Smem::kDigits;
    static_assert(kRadix <= kOsThreads, "a thread per digit");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem &S = *reinterpret_cast<Smem *>(smem_raw);
    after_previous();
    if (*err) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t n = n_dev ? (int64_t)*n_dev : n_host;
    const int64_t nparts = (n + PART - 1) / PART;
    const uint32_t epoch = *epoch_ptr + epoch_off;
    const uint32_t lt = lanemask_lt();
    static_assert(BITS == 8 || kOsWarps * kRadix <= PART, "masks in the values' place");
    uint32_t *match9 = S.vals + warp * kRadix;
    auto match = [&](uint32_t d) -> uint32_t & {
        if constexpr (BITS == 8) return S.match[warp][d];
        else return match9[d];
    };
    if constexpr (BITS == 8)
        for (int i = tid; i < kOsWarps * kRadix; i += kOsThreads) (&S.match[0][0])[i] = 0;
    for (;;) {
        if (tid == 0) S.part = atomicAdd(ticket, 1u);
        for (int i = tid; i < kOsWarps * kRadix; i += kOsThreads) {
            (&S.whist[0][0])[i] = 0;
            if (BITS != 8) S.vals[i] = 0;
        }
        __syncthreads();
        const int64_t part = S.part;
        if (part >= nparts) break;
        const int64_t base = part * PART + (int64_t)warp * (ITEMS * 32);
        // keys first; values are loaded only after ranking, to keep few live registers
        K key[ITEMS];
        uint32_t rank[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int64_t idx = base + i * 32 + lane;
            key[i] = idx < n ? kin[idx] : (K)0;
        }
        // kOut == 2: the keys come in the order of their lower digits. Where the partition
        // has one value of them (nearly all of a large sort's), a digit's run is one key's
        // and the digit's owner records it; else every key looks at its neighbours in the
        // write-out. 431 M pairs: 2496 us with the look at the neighbours everywhere, 2326 us.
        K low = 0;
        bool one_low = false;
        if (kOut == 2) {
            const K lows = ((K)1 << shift) - 1;
            low = kin[part * PART] & lows;
            one_low = low == (kin[min(n, (part + 1) * PART) - 1] & lows);
        }
        // rank of each item among the warp's earlier items with its digit:
        // the lanes sharing a digit (peers) are found by one shared-memory OR
        // of the lane bits into the warp's mask of that digit (the lowest
        // peer clears it again). (A shortcut for warps whose lanes all share
        // one digit cost more in its test than it saved, even on depth keys.)
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const bool valid = base + i * 32 + lane < n;
            const uint32_t d = digit_of(key[i], shift, mask);
            if (valid) atomicOr(&match(d), 1u << lane);
            __syncwarp();
            const uint32_t peers = valid ? match(d) : 0u;
            uint32_t before = 0;
            if (valid) before = S.whist[warp][d];
            __syncwarp();
            if (valid && (peers & lt) == 0) {
                S.whist[warp][d] = before + __popc(peers);
                match(d) = 0u;
            }
            __syncwarp();
            rank[i] = before + __popc(peers & lt);
        }
        __syncthreads();
        // threads 0..kRadix - 1 own one digit each: warp offsets and the partition's
        // total (published at once for the successors' look-back), then the
        // block-local scan of the totals
        uint32_t run = 0, incl = 0, ds = 0;
        uint64_t *slot = status + part * kRadix + tid;
        if (tid < kRadix) {
            const int d = tid;
#pragma unroll
            for (int w = 0; w < kOsWarps; ++w) {
                const uint32_t t = S.whist[w][d];
                S.whist[w][d] = run;
                run += t;
            }
            publish(slot, pack_status(part == 0 ? kFlagPrefix : kFlagAgg, epoch, run));
            incl = run;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) S.wtot[warp] = incl;
        }
        __syncthreads();
        if (tid < kRadix) {
            // block-local start of digit d, folded into every warp's offset of
            // d (one lookup per item when staging)
            uint32_t wbase = 0;
            for (int w = 0; w < warp; ++w) wbase += S.wtot[w];
            ds = wbase + incl - run;
#pragma unroll
            for (int w = 0; w < kOsWarps; ++w) S.whist[w][tid] += ds;
        }
        __syncthreads();
        // stage the keys in digit order, then request the values (they arrive
        // while the digit owners look back)
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if (base + i * 32 + lane < n) {
                const uint32_t d = digit_of(key[i], shift, mask);
                rank[i] += S.whist[warp][d];
                S.keys[rank[i]] = key[i];
            }
        }
        uint32_t val[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int64_t idx = base + i * 32 + lane;
            val[i] = idx < n ? vin[idx] : 0u;
        }
        if (tid < kRadix) {
            // the partition's exclusive prefix of digit d by decoupled look-back;
            // output position = gstart[d] + staged position (modulo 2^32)
            uint32_t prev = 0;
            if (part > 0) {
                look_back(status + tid, part, kRadix, epoch, &prev, err);
                publish(slot, pack_status(kFlagPrefix, epoch, prev + run));
            }
            S.gstart[tid] = digit_base[tid] + prev - ds;
            if (kOut == 2 && one_low && run) {
                const uint32_t g0 = digit_base[tid] + prev;
                const uint32_t t = (uint32_t)(low | (K)tid << shift);
                if (g0 < n) {
                    atomicMax(&ranges[t].x, ~g0);
                    atomicMax(&ranges[t].y, g0 + min(run, (uint32_t)n - g0));
                }
            }
        }
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            if (base + i * 32 + lane < n) S.vals[rank[i]] = val[i];
        __syncthreads();
        const int64_t rem = n - part * PART;
        const int cnt = rem < PART ? (int)rem : PART;
        for (int j = tid; j < cnt; j += kOsThreads) {
            const K k = S.keys[j];
            const uint32_t d = digit_of(k, shift, mask);
            const int64_t g = (int64_t)(S.gstart[d] + (uint32_t)j);
            // digit counts that disagree with the keys (a caller's histogram)
            // would place a key outside [0, n): never written there
            if (g >= n) continue;
            if (kOut == 0) kout[g] = k;
            vout[g] = S.vals[j];
            if (kOut == 2 && !one_low) {
                const uint32_t t = (uint32_t)k;
                if (j == 0 || S.keys[j - 1] != k) atomicMax(&ranges[t].x, ~(uint32_t)g);
                if (j + 1 == cnt || S.keys[j + 1] != k) atomicMax(&ranges[t].y, (uint32_t)g + 1u);
            }
        }
        __syncthreads();
    }
}

template <typename K, int kOut, int BITS>
static void set_sort_attr() {
    cudaFuncSetAttribute(k_onesweep<K, kOut, BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(SortSmem<K, BITS>));
}

void sort_init_attributes() {
    set_sort_attr<uint32_t, 0, 8>();
    set_sort_attr<uint32_t, 1, 8>();
    set_sort_attr<uint32_t, 2, 8>();
    set_sort_attr<uint32_t, 0, 9>();
    set_sort_attr<uint32_t, 1, 9>();
    set_sort_attr<uint64_t, 0, 8>();
    set_sort_attr<uint64_t, 1, 8>();
}

template <typename K, int kOut, int BITS>
static void launch_pass(int grid, const SortArgs &a, int p, uint32_t mask, const LaunchOn &st) {
    const int src = p & 1, dst = src ^ 1;
    launch_on(st, k_onesweep<K, kOut, BITS>, grid, kOsThreads, sizeof(SortSmem<K, BITS>),
        (const K *)a.keys[src], a.vals[src], (K *)a.keys[dst], a.vals[dst], a.n_dev, a.n_host,
        a.begin_bit + BITS * p, mask, a.hist + (p << BITS), a.status, a.tickets + p, a.epoch,
        a.epoch_off + p, a.err, a.ranges);
}

template <typename K, int BITS>
static void launch_sort_t(const SortArgs &a, int grid, const LaunchOn &st) {
    const int passes = (a.end_bit - a.begin_bit + BITS - 1) / BITS;
    if (!a.hist_ready) {
        cudaMemsetAsync(a.hist, 0, sizeof(uint32_t) * kRadix * passes, st.st);
        const int ugrid = (int)std::max<int64_t>(
            1, std::min<int64_t>(parts_of(a.n_max, kSortThreads * kUp), 8 * a.num_sms));
        k_upsweep<K><<<ugrid, kSortThreads, 0, st.st>>>((const K *)a.keys[0], a.n_dev, a.n_host,
                                                     a.begin_bit, a.end_bit, a.hist,
                                                     a.tickets + kMaxPasses, a.err);
    }
    if (a.hook) a.hook(a.hook_user, 0);
    for (int p = 0; p < passes; ++p) {
        const int bits = std::min(BITS, a.end_bit - a.begin_bit - BITS * p);
        const uint32_t mask = (1u << bits) - 1u;
        const bool last = p == passes - 1;
        if constexpr (sizeof(K) == 4 && BITS == 8) {
            if (last && a.ranges) {
                launch_pass<K, 2, BITS>(grid, a, p, mask, st);
                if (a.hook) a.hook(a.hook_user, p + 1);
                continue;
            }
        }
        if (last && a.skip_last_keys) launch_pass<K, 1, BITS>(grid, a, p, mask, st);
        else launch_pass<K, 0, BITS>(grid, a, p, mask, st);
        if (a.hook) a.hook(a.hook_user, p + 1);
    }
}

void launch_sort(const SortArgs &a, int grid, const LaunchOn &st) {
    if (a.key_bytes == 8) launch_sort_t<uint64_t, 8>(a, grid, st);
    else if (a.digit_bits == 9) launch_sort_t<uint32_t, 9>(a, grid, st);
    else launch_sort_t<uint32_t, 8>(a, grid, st);
}

}  // namespace ngs
