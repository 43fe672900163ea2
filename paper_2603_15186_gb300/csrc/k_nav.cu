// Navigable map and shortest paths on the GS-slice occupancy (NavGSim
// Sec. III-C: the slices give the navigable area for collision checks and path
// planning; Sec. IV-A: expert trajectories come from a shortest-path planner).
//
//  - blocked(i, j): some plane k in [k_lo, k_hi] (the robot's height range) is
//    occupied at a cell within Chebyshev distance `inflate` of (i, j).
//  - One distance field per goal: 4-connected breadth-first steps over free
//    cells, UINT32_MAX where unreachable, level by level: on the map's bits, one
//    cluster of CTAs per goal (k_nav_bfs), or, for large maps and many goals, on a
//    frontier queue, one CTA per goal (k_nav_bfs_queue: its threads expand the
//    frontier's cells and admit each unreached free neighbour once, by an
//    atomicCAS from UINT32_MAX to L + 1). Every cell enters a frontier at most
//    once, so the loop ends after at most one level per cell; the only waits are
//    the barriers of a CTA and of its cluster.
//  - A path descends a field from its start, taking the first neighbour in the
//    order (+x, -x, +y, -y) whose distance is one less, one CTA per agent, or, of
//    thousands of agents, one thread each.
#include <cooperative_groups.h>

#include "ngs_internal.cuh"
#include "nav.h"

namespace ngs {

constexpr uint32_t kNavUnreached = 0xFFFFFFFFu;
constexpr size_t kNavSmemMax = 96 * 1024;   // of k_nav_bfs

__global__ void k_nav_any(const uint8_t *__restrict__ occ, int64_t plane, int k_lo, int k_hi,
                          uint8_t *__restrict__ any) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < plane;
         c += (int64_t)gridDim.x * blockDim.x) {
        uint8_t a = 0;
        for (int k = k_lo; k <= k_hi; ++k) a |= occ[(int64_t)k * plane + c];
        any[c] = a ? 1 : 0;
    }
}

// One warp per 32-cell word of a row: blocked bytes, and the row's free cells as
// bits (free_bits[j * wpr + i / 32], bit i & 31; bits past the row's end are 0).
__global__ void __launch_bounds__(256)
k_nav_dilate(const uint8_t *__restrict__ any, int nx, int ny, int r, int wpr,
             uint8_t *__restrict__ blocked, uint32_t *__restrict__ free_bits) {
    const int lane = threadIdx.x & 31;
    const int64_t words = (int64_t)wpr * ny;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < words; w += nw) {
        const int j = (int)(w / wpr), i = (int)(w - (int64_t)j * wpr) * 32 + lane;
        uint8_t b = 1;
        if (i < nx) {
            b = 0;
            for (int y = max(j - r, 0); y <= min(j + r, ny - 1) && !b; ++y)
                for (int x = max(i - r, 0); x <= min(i + r, nx - 1); ++x)
                    if (any[(int64_t)y * nx + x]) { b = 1; break; }
            blocked[(int64_t)j * nx + i] = b;
        }
        const uint32_t bits = __ballot_sync(0xffffffffu, b == 0);
        if (lane == 0) free_bits[w] = bits;
    }
}

// Maps of more words than k_nav_bfs is built for (about a million cells), and many goals
// (nav_words_per_thread).
__global__ void __launch_bounds__(1024)
k_nav_bfs_queue(const uint8_t *__restrict__ blocked, int nx, int ny, const int2 *__restrict__ goals,
          uint32_t *dist, uint32_t *queues) {
    __shared__ uint32_t s_next, s_cur;
    const int g = blockIdx.x, tid = threadIdx.x;
    const int64_t plane = (int64_t)nx * ny;
    uint32_t *dg = dist + (int64_t)g * plane;
    uint32_t *cur = queues + (int64_t)g * 2 * plane, *nxt = cur + plane;
    const int2 q = goals[g];
    if (tid == 0) {
        const bool ok = q.x >= 0 && q.x < nx && q.y >= 0 && q.y < ny &&
                        !blocked[(int64_t)q.y * nx + q.x];
        if (ok) {
            cur[0] = (uint32_t)((int64_t)q.y * nx + q.x);
            dg[cur[0]] = 0u;
        }
        s_cur = ok ? 1u : 0u;
        s_next = 0;
    }
    __syncthreads();
    for (uint32_t level = 0; s_cur > 0; ++level) {
        const uint32_t ncur = s_cur;
        for (uint32_t k = tid; k < ncur; k += blockDim.x) {
            const uint32_t c = cur[k];
            const int i = (int)(c % (uint32_t)nx), j = (int)(c / (uint32_t)nx);
            const int ni[4] = {i + 1, i - 1, i, i}, nj[4] = {j, j, j + 1, j - 1};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (ni[e] < 0 || ni[e] >= nx || nj[e] < 0 || nj[e] >= ny) continue;
                const uint32_t n = (uint32_t)nj[e] * (uint32_t)nx + (uint32_t)ni[e];
                if (blocked[n] || dg[n] != kNavUnreached) continue;
                if (atomicCAS(&dg[n], kNavUnreached, level + 1u) == kNavUnreached)
                    nxt[atomicAdd(&s_next, 1u)] = n;
            }
        }
        __syncthreads();
        if (tid == 0) {
            s_cur = s_next;
            s_next = 0;
        }
        uint32_t *t = cur;
        cur = nxt;
        nxt = t;
        __syncthreads();
    }
}

// The search on bits: the map's rows are split over a cluster of kNavCtas CTAs, each
// with kNavHalo further rows above and below its own, kWords words of 32 cells per
// thread. A thread keeps its words' unreached free cells and frontier in registers;
// the frontier also goes to shared memory (two buffers, a row of zeros above and
// below) for the neighbours:
//   next = (left | right | up | down of the frontier) & unreached
// A level is one CTA barrier. After kNavHalo levels the halo rows are out of date by
// as many rows, the own rows are not: then every CTA sends its first and last
// kNavHalo rows (frontier and unreached cells) to its neighbours' mailboxes and
// whether it has a frontier to all, by distributed shared memory, with one cluster
// barrier; the search ends when none has. The mailboxes alternate, so a CTA's next
// writes cannot meet a neighbour still reading. Rows are nav_row_words(nx) words with
// at least one 0 bit past the row's end, so bits that a shift carries into another row
// fall on a cell that is never free.
// The level of a cell is kept in bit planes (levels_: kPlanes of them, the word's
// cells found in the last 2^kPlanes levels), unpacked 32 cells at a time every
// 2^kPlanes levels and at the end.
//
// A search is a serial chain of levels (about 650 of some 200 cells each on a 528 x
// 276 map of rooms), so the time of a level bounds it. Measured for 9 goals on that
// map: 2252 us with the queue in global memory (k_nav_bfs_queue: three round trips
// there and two barriers per level); 471 us with the map's bits and the queue in
// one CTA's shared memory (atomics on its bits and on its length); 1100 us with all
// the map's words in one CTA each level; 166 us here.
constexpr int kNavThreads = 1024;
constexpr int kNavCtas = 8;
constexpr int kNavHalo = 8;
constexpr int kPlanes = 8;
static_assert(kNavHalo == 8, "three bits of a level come from its place in a period");

// rows of a CTA (its halos lie within its neighbours' rows), its words, and its
// shared memory: two frontiers, then the mailboxes [parity][above, below][frontier,
// unreached][kNavHalo rows]
__host__ __device__ inline int nav_cta_rows(int ny) {
    const int r = (ny + kNavCtas - 1) / kNavCtas;
    return r < kNavHalo ? kNavHalo : r;
}
static int64_t nav_cta_words(int ny, int wpr) {
    return (int64_t)(nav_cta_rows(ny) + 2 * kNavHalo) * wpr;
}
static size_t nav_smem_bytes(int ny, int wpr) {
    return sizeof(uint32_t) * (size_t)(2 * (nav_cta_words(ny, wpr) + 2 * wpr) + 8 * kNavHalo * wpr);
}

template <int kWords>
__global__ void __cluster_dims__(kNavCtas, 1, 1) __launch_bounds__(kNavThreads)
k_nav_bfs(const uint32_t *__restrict__ free_bits, int nx, int ny, int wpr,
          const int2 *__restrict__ goals, uint32_t *__restrict__ dist) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ uint32_t s_dyn[];
    __shared__ uint32_t s_alive[2][kNavCtas];
    const int tid = threadIdx.x, lane = tid & 31;
    const int rank = (int)cluster.block_rank(), goal = blockIdx.x / kNavCtas;
    const int rows = nav_cta_rows(ny), words = (rows + 2 * kNavHalo) * wpr;
    const int stride = words + 2 * wpr, hw = kNavHalo * wpr;
    uint32_t *s_box = s_dyn + 2 * stride;
    uint32_t *dg = dist + (int64_t)goal * nx * ny;
    for (int i = tid; i < 2 * stride; i += kNavThreads) s_dyn[i] = 0;
    uint32_t todo[kWords], f[kWords], found[kWords], levels_[kWords][kPlanes];
    const int2 q = goals[goal];
#pragma unroll
    for (int k = 0; k < kWords; ++k) {
        const int w = k * kNavThreads + tid;
        const int y = rank * rows - kNavHalo + w / wpr, c = w % wpr;
        const bool in = w < words && y >= 0 && y < ny;
        todo[k] = in ? free_bits[(int64_t)y * wpr + c] : 0u;
        f[k] = 0;
        if (in && y == q.y && q.x >= 0 && q.x < nx && c == q.x >> 5) f[k] = todo[k] & 1u << (q.x & 31);
        todo[k] &= ~f[k];
        found[k] = 0;
#pragma unroll
        for (int p = 0; p < kPlanes; ++p) levels_[k][p] = 0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kWords; ++k) {
        const int w = k * kNavThreads + tid;
        if (f[k]) {
            s_dyn[wpr + w] = f[k];
            if (w >= hw && w < hw + rows * wpr) dg[(int64_t)q.y * nx + q.x] = 0u;
        }
    }
    // writes the levels base + 1 .. of the own cells found since `base`
    auto unpack = [&](uint32_t base) {
#pragma unroll
        for (int k = 0; k < kWords; ++k) {
            const int w0 = k * kNavThreads + (tid & ~31);
            for (uint32_t any = __ballot_sync(0xffffffffu, found[k] != 0); any; any &= any - 1) {
                const int src = __ffs(any) - 1, w = w0 + src;
                const uint32_t m = __shfl_sync(0xffffffffu, found[k], src);
                uint32_t lv = 0;
#pragma unroll
                for (int p = 0; p < kPlanes; ++p)
                    lv |= (__shfl_sync(0xffffffffu, levels_[k][p], src) >> lane & 1u) << p;
                const int y = rank * rows - kNavHalo + w / wpr, c = w % wpr;
                if (m >> lane & 1u) dg[(int64_t)y * nx + c * 32 + lane] = base + lv + 1u;
            }
            found[k] = 0;
#pragma unroll
            for (int p = 0; p < kPlanes; ++p) levels_[k][p] = 0;
        }
    };
    uint32_t base = 0;
    cluster.sync();   // every CTA of the cluster runs: its shared memory may be written
    for (uint32_t period = 0;; ++period, base += kNavHalo) {
        // the own rows at the edges to the neighbours, and whether there is a frontier
        const uint32_t par = period & 1u;
        uint32_t *up = rank > 0 ? cluster.map_shared_rank(s_box, rank - 1) : nullptr;
        uint32_t *down = rank + 1 < kNavCtas ? cluster.map_shared_rank(s_box, rank + 1) : nullptr;
        bool mine = false;
#pragma unroll
        for (int k = 0; k < kWords; ++k) {
            const int w = k * kNavThreads + tid;
            if (w >= hw && w < hw + rows * wpr) {
                mine = mine || f[k] != 0;
                if (up && w < 2 * hw) {                       // its rows below
                    up[(par * 4 + 2) * hw + w - hw] = f[k];
                    up[(par * 4 + 3) * hw + w - hw] = todo[k];
                }
                if (down && w >= rows * wpr) {                // its rows above
                    down[par * 4 * hw + w - rows * wpr] = f[k];
                    down[(par * 4 + 1) * hw + w - rows * wpr] = todo[k];
                }
            }
        }
        const int alive = __syncthreads_or(mine);
        if (tid < kNavCtas) cluster.map_shared_rank(&s_alive[0][0], tid)[par * kNavCtas + rank] = alive;
        cluster.sync();
        uint32_t any = 0;
#pragma unroll
        for (int r = 0; r < kNavCtas; ++r) any |= s_alive[par][r];
        if (!any) break;   // the same words in every CTA
        bool here = false;
#pragma unroll
        for (int k = 0; k < kWords; ++k) {
            const int w = k * kNavThreads + tid, below = w - hw - rows * wpr;
            if (w < hw && rank > 0) {
                f[k] = s_box[par * 4 * hw + w];
                todo[k] = s_box[(par * 4 + 1) * hw + w];
                s_dyn[wpr + w] = f[k];
            } else if (below >= 0 && below < hw && rank + 1 < kNavCtas) {
                f[k] = s_box[(par * 4 + 2) * hw + below];
                todo[k] = s_box[(par * 4 + 3) * hw + below];
                s_dyn[wpr + w] = f[k];
            }
            here = here || f[k] != 0;
        }
        if (__syncthreads_or(here)) {   // else nothing can reach this CTA's rows yet
            uint32_t fresh[kWords];
#pragma unroll
            for (int k = 0; k < kWords; ++k) fresh[k] = 0;
#pragma unroll
            for (int s = 0; s < kNavHalo; ++s) {
                const uint32_t *cur = s_dyn + (s & 1) * stride + wpr + tid;
                uint32_t *nxt = s_dyn + ((s & 1) ^ 1) * stride + wpr + tid;
#pragma unroll
                for (int k = 0; k < kWords; ++k) {
                    const int at = k * kNavThreads;
                    if (at + tid < words) {
                        uint32_t n = f[k] << 1 | f[k] >> 1 | cur[at - 1] >> 31 | cur[at + 1] << 31 |
                                     cur[at - wpr] | cur[at + wpr];
                        n &= todo[k];
                        todo[k] &= ~n;
                        nxt[at] = n;
                        f[k] = n;
                        fresh[k] |= n;
#pragma unroll
                        for (int p = 0; p < 3; ++p)
                            if (s >> p & 1) levels_[k][p] |= n;
                    }
                }
                __syncthreads();
            }
#pragma unroll
            for (int k = 0; k < kWords; ++k) {
                const int w = k * kNavThreads + tid;
                if (w < hw || w >= hw + rows * wpr) fresh[k] = 0;   // the neighbours' rows
                found[k] |= fresh[k];
#pragma unroll
                for (int p = 3; p < kPlanes; ++p)
                    if (base >> p & 1u) levels_[k][p] |= fresh[k];
            }
        }
        if ((base & ((1u << kPlanes) - 1u)) == (1u << kPlanes) - kNavHalo)
            unpack(base & ~((1u << kPlanes) - 1u));
    }
    unpack(base & ~((1u << kPlanes) - 1u));
}

// A path is a serial chain too: one step needs the distances around the cell that
// the step before chose. One CTA per agent keeps a kNavWin x kNavWin window of the
// field around the agent in shared memory (one memory round trip per 31 steps or
// more, instead of two per step) and finds every cell's
// next one at once; a warp then walks, one shared-memory load per step, and the cells
// go out 32 at a time. 64 paths of 373 cells on average: 319 us with one thread per
// agent reading the field in global memory, 88 us with one warp, a 32 x 32 window and
// the neighbours compared at each step, 59 us here.
constexpr int kNavWin = 64;
constexpr int kNavPathThreads = 512;
constexpr uint32_t kNavEdge = 0xfffeu;    // the window's outermost cells
constexpr uint32_t kNavNone = 0xffffu;    // no neighbour is one step nearer

__global__ void __launch_bounds__(kNavPathThreads)
k_nav_paths(const uint32_t *__restrict__ dist, int nx, int ny, int n_goals,
            const int3 *__restrict__ starts, int n, int max_len, int2 *__restrict__ paths,
            int32_t *__restrict__ lens) {
    __shared__ uint32_t s_win[kNavWin * kNavWin];
    __shared__ uint16_t s_to[kNavWin * kNavWin];
    __shared__ int s_state[6];   // x, y, length, distance, on a distance field, done
    const int a = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const int3 s = starts[a];
    if (!(s.z >= 0 && s.z < n_goals && s.x >= 0 && s.x < nx && s.y >= 0 && s.y < ny && max_len > 0)) {
        if (tid == 0) lens[a] = 0;
        return;
    }
    const uint32_t *dg = dist + (int64_t)s.z * nx * ny;
    int2 *out = paths + (int64_t)a * max_len;
    uint32_t d = dg[(int64_t)s.y * nx + s.x];
    int i = s.x, j = s.y, len = 0;
    if (d == kNavUnreached) {
        if (tid == 0) lens[a] = 0;
        return;
    }
    int2 mine = make_int2(0, 0);   // this lane's cell of the next 32 to go out
    // whether the distance counted so far is the one at the cell: always on a distance
    // field; other fields are followed by comparing the neighbours at each step
    bool good = true;
    for (;;) {
        const int x0 = i - kNavWin / 2, y0 = j - kNavWin / 2;
#pragma unroll
        for (int r = 0; r < kNavWin * kNavWin / kNavPathThreads; ++r) {
            const int c = r * kNavPathThreads + tid, x = x0 + c % kNavWin, y = y0 + c / kNavWin;
            // a cell outside the map never holds d - 1
            s_win[c] = x >= 0 && x < nx && y >= 0 && y < ny ? dg[(int64_t)y * nx + x] : kNavUnreached;
        }
        __syncthreads();
#pragma unroll 4
        for (int c = tid; c < kNavWin * kNavWin; c += kNavPathThreads) {
            const int x = c % kNavWin, y = c / kNavWin;
            uint32_t to = kNavEdge;
            if (x > 0 && x < kNavWin - 1 && y > 0 && y < kNavWin - 1) {
                const uint32_t at = s_win[c], w = at - 1u;
                to = kNavNone;
                if (s_win[c - kNavWin] == w) to = c - kNavWin;
                if (s_win[c + kNavWin] == w) to = c + kNavWin;
                if (s_win[c - 1] == w) to = c - 1;
                if (s_win[c + 1] == w) to = c + 1;
                if (at == 0) to = c;   // a path ends there
            }
            s_to[c] = (uint16_t)to;
        }
        __syncthreads();
        if (tid < 32) {
            uint32_t c = (uint32_t)((j - y0) * kNavWin + (i - x0));
            bool done = false;
            for (;;) {
                // the next cells, from c on, until 32 go out or the path ends
                const uint32_t left = min((uint32_t)(max_len - len), d + 1u);
                const uint32_t room = good ? min(left, 32u - (uint32_t)(len & 31)) : 1u;
                uint32_t k = 0, to = 0;
                for (; k < room; ++k) {
                    to = s_to[c];
                    if (to == kNavEdge || (good && to == kNavNone)) break;
                    if (lane == ((len + (int)k) & 31))
                        mine = make_int2(x0 + (int)(c % kNavWin), y0 + (int)(c / kNavWin));
                    if (good) c = to;
                }
                len += (int)k;
                done = k == left;
                if (done || (k > 0 && (len & 31) == 0)) {
                    const int b = (len - 1) & ~31;
                    if (b + lane < len) out[b + lane] = mine;
                }
                if (done) break;
                d -= k;
                if (k < room && to == kNavEdge) break;   // the next window counts this cell
                if (good) {
                    good = k == room;
                } else {
                    if (s_win[c + 1] == d) c += 1;
                    else if (s_win[c - 1] == d) c -= 1;
                    else if (s_win[c + kNavWin] == d) c += kNavWin;
                    else if (s_win[c - kNavWin] == d) c -= kNavWin;
                }
            }
            if (lane == 0) {
                s_state[0] = x0 + (int)(c % kNavWin);
                s_state[1] = y0 + (int)(c / kNavWin);
                s_state[2] = len;
                s_state[3] = (int)d;
                s_state[4] = good;
                s_state[5] = done;
            }
        }
        __syncthreads();
        i = s_state[0]; j = s_state[1]; len = s_state[2]; d = (uint32_t)s_state[3];
        good = s_state[4] != 0;
        if (s_state[5]) break;
    }
    if (tid == 0) lens[a] = len;
}

// A thread per agent, reading the field in global memory: two memory round trips a
// step, hidden by nothing but the other agents.
__global__ void __launch_bounds__(128)
k_nav_paths_each(const uint32_t *__restrict__ dist, int nx, int ny, int n_goals,
                 const int3 *__restrict__ starts, int n, int max_len, int2 *__restrict__ paths,
                 int32_t *__restrict__ lens) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= n) return;
    const int3 s = starts[a];
    int len = 0;
    if (s.z >= 0 && s.z < n_goals && s.x >= 0 && s.x < nx && s.y >= 0 && s.y < ny && max_len > 0) {
        const uint32_t *dg = dist + (int64_t)s.z * nx * ny;
        uint32_t d = dg[(int64_t)s.y * nx + s.x];
        int i = s.x, j = s.y;
        if (d != kNavUnreached) {
            for (;;) {
                paths[(int64_t)a * max_len + len] = make_int2(i, j);
                ++len;
                if (d == 0 || len >= max_len) break;
                const int ni[4] = {i + 1, i - 1, i, i}, nj[4] = {j, j, j + 1, j - 1};
                for (int e = 0; e < 4; ++e) {
                    if (ni[e] < 0 || ni[e] >= nx || nj[e] < 0 || nj[e] >= ny) continue;
                    if (dg[(int64_t)nj[e] * nx + ni[e]] == d - 1u) { i = ni[e]; j = nj[e]; break; }
                }
                --d;
            }
        }
    }
    lens[a] = len;
}

static int nav_grid(int64_t work, int num_sms) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, (int64_t)num_sms * 16));
}

// Words per thread of k_nav_bfs, 0 where the queue searches: maps too large for the
// bits, and more goals than the bits are faster for. A search on bits is the faster
// one, but it holds eight CTAs that look at every word on every level, so that a few
// dozen run at once; the queue's CTA looks at its frontier alone, and two run on each
// SM. Bits / queue on open maps, us: 64 x 64 cells (1 word a thread) 128 goals 283 / 380,
// 256 goals 484 / 388; 528 x 276 (1 word) 200 goals 2208 / 2401, 256 goals 2737 / 2418; 511 x 896
// (2 words) 128 goals 4145 / 4727, 256 goals 8008 / 5692; 511 x 1920 (4 words) 64 goals 8023 /
// 9280, 128 goals 13789 / 9510.
static int nav_words_per_thread(int ny, int wpr, int n_goals, int num_sms) {
    const int64_t k = (nav_cta_words(ny, wpr) + kNavThreads - 1) / kNavThreads;
    if (k > 4 || nav_smem_bytes(ny, wpr) > kNavSmemMax) return 0;
    const int words = k <= 2 ? (int)k : 4;
    const int most = words == 4 ? num_sms / 2 : words == 2 ? num_sms
                     : ny * wpr < 512 ? num_sms * 5 / 4 : num_sms * 3 / 2;
    return n_goals <= most ? words : 0;
}

template <int kWords>
static void launch_bfs(const uint32_t *free_bits, int nx, int ny, int wpr, const int2 *goals,
                       int n_goals, uint32_t *dist, cudaStream_t st) {
    cudaFuncSetAttribute(k_nav_bfs<kWords>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)kNavSmemMax);
    k_nav_bfs<kWords><<<n_goals * kNavCtas, kNavThreads, nav_smem_bytes(ny, wpr), st>>>(
        free_bits, nx, ny, wpr, goals, dist);
}

size_t nav_queue_words(int nx, int ny, int n_goals, int num_sms) {
    return nav_words_per_thread(ny, nav_row_words(nx), n_goals, num_sms)
               ? 0 : (size_t)n_goals * 2 * nx * ny;
}

// scratch: any [ny * nx] bytes, free_bits [ny * nav_row_words(nx)], queues
// [nav_queue_words()] u32; returns 0 or a cudaError_t (synchronises the stream)
int launch_nav_fields(const uint8_t *occ, int nx, int ny, int k_lo, int k_hi, int inflate,
                      const int2 *d_goals, int n_goals, uint8_t *any, uint32_t *free_bits,
                      uint32_t *queues, uint8_t *blocked, uint32_t *dist, int num_sms,
                      cudaStream_t st) {
    const int64_t plane = (int64_t)nx * ny;
    const int wpr = nav_row_words(nx);
    const int64_t words = (int64_t)wpr * ny;
    k_nav_any<<<nav_grid(plane, num_sms), 256, 0, st>>>(occ, plane, k_lo, k_hi, any);
    k_nav_dilate<<<nav_grid(32 * words, num_sms), 256, 0, st>>>(any, nx, ny, inflate, wpr, blocked,
                                                                free_bits);
    cudaMemsetAsync(dist, 0xff, (size_t)plane * n_goals * sizeof(uint32_t), st);   // kNavUnreached
    switch (nav_words_per_thread(ny, wpr, n_goals, num_sms)) {
    case 1: launch_bfs<1>(free_bits, nx, ny, wpr, d_goals, n_goals, dist, st); break;
    case 2: launch_bfs<2>(free_bits, nx, ny, wpr, d_goals, n_goals, dist, st); break;
    case 4: launch_bfs<4>(free_bits, nx, ny, wpr, d_goals, n_goals, dist, st); break;
    default:
        k_nav_bfs_queue<<<n_goals, 1024, 0, st>>>(blocked, nx, ny, d_goals, dist, queues);
        break;
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return (int)e;
}

// Above this many agents a thread each: four CTAs run on an SM, and from the seventh
// round of them on the windows take longer. CTAs / threads, us, on a 528 x 276 map: 64
// paths of 286 cells on average 72 / 438, 4096 of 251 cells 284 / 437, 16384 981 / 466,
// 131072 7453 / 605; of 53 cells 64 paths 22 / 65, 4096 72 / 70, 16384 232 / 71.
static int nav_paths_few(int num_sms) { return 7 * 4 * num_sms; }

void launch_nav_paths(const uint32_t *dist, int nx, int ny, int n_goals, const int3 *starts,
                      int n, int max_len, int2 *paths, int32_t *lens, int num_sms,
                      cudaStream_t st) {
    if (n > nav_paths_few(num_sms))
        k_nav_paths_each<<<(n + 127) / 128, 128, 0, st>>>(dist, nx, ny, n_goals, starts, n, max_len,
                                                          paths, lens);
    else if (n > 0)
        k_nav_paths<<<n, kNavPathThreads, 0, st>>>(dist, nx, ny, n_goals, starts, n, max_len, paths,
                                                   lens);
}

}  // namespace ngs
