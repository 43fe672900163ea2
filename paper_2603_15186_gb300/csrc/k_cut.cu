// K1: level-of-detail cut of the Gaussian hierarchy (NavGSim Sec. III-B:
// per view, Gaussians are taken from the level of the tree whose granularity
// matches the requested one).
//
// Node n is selected for camera c iff
//     (n is a leaf or s_c(n) <= tau_c) and (n is the root or s_c(parent(n)) > tau_c)
// with s_c(n) = fx * (longest side of box(n)) / (distance from the camera
// centre to box(n)), s = +inf when the centre lies inside the box. Boxes nest,
// so s never decreases towards the root and every root-to-leaf path holds
// exactly one selected node.
//
// Variants (Sec. III-B's per-view, dynamic selection of levels): a frustum
// cull drops the nodes whose box lies wholly outside one of the five planes of
// a camera's view volume (near plane 0.2, image rectangle widened by a guard
// band), and a group of cameras can share one cut, in which a node is fine
// enough when it is for every member that does not cull it. Boxes nest and the
// float32 tests below are monotone in the box bounds (each step rounds
// monotonically), so both the cull and "fine enough" spread from a node to its
// whole subtree and the result stays an antichain of the tree.
//
// One pass, order preserving: partitions are (camera or group, block of 2048
// nodes) in camera-major order, taken from an atomic ticket so every
// predecessor of a partition is already running; each partition counts its
// selected nodes, finds its output offset by decoupled look-back and writes
// the ids in ascending order. HBM traffic per node and camera: the node's two box words
// (32 B) plus its parent's (mostly L1/L2 hits: siblings share a parent), and
// 4 B per selected node.
#include "ngs_internal.cuh"
#include "cut.h"

namespace ngs {

constexpr int kCutThreads = 256;
constexpr int kCutItems = 8;
constexpr int kCutPart = kCutThreads * kCutItems;

int cut_partition_nodes() { return kCutPart; }

// Selection of the plain cut: one camera per unit.
struct PlainSelect {
    const float4 *box_lo, *box_hi;
    const DevCamera *cams;
    float px, py, pz, fx, tau;
    __device__ __forceinline__ void begin(int c) {
        px = cams[c].pos[0]; py = cams[c].pos[1]; pz = cams[c].pos[2];
        fx = cams[c].fx; tau = cams[c].tau;
    }
    __device__ __forceinline__ bool operator()(int64_t node) const {
        return cut_selects(box_lo, box_hi, node, px, py, pz, fx, tau);
    }
};

// True when the box lies wholly outside one of the camera's five half-spaces:
// the largest value of a_k . (x - pos) + b_k over the box (per axis the larger
// of the two faces' terms) is negative.
__device__ __forceinline__ bool frustum_culled(const CutCam &k, const float4 lo, const float4 hi) {
    const float dl0 = __fsub_rn(lo.x, k.pos[0]), dh0 = __fsub_rn(hi.x, k.pos[0]);
    const float dl1 = __fsub_rn(lo.y, k.pos[1]), dh1 = __fsub_rn(hi.y, k.pos[1]);
    const float dl2 = __fsub_rn(lo.z, k.pos[2]), dh2 = __fsub_rn(hi.z, k.pos[2]);
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const float t0 = fmaxf(__fmul_rn(k.a[j][0], dl0), __fmul_rn(k.a[j][0], dh0));
        const float t1 = fmaxf(__fmul_rn(k.a[j][1], dl1), __fmul_rn(k.a[j][1], dh1));
        const float t2 = fmaxf(__fmul_rn(k.a[j][2], dl2), __fmul_rn(k.a[j][2], dh2));
        const float m = __fadd_rn(__fadd_rn(__fadd_rn(t0, t1), t2), j == 0 ? k.b0 : 0.0f);
        if (m < 0.0f) return true;
    }
    return false;
}

// Selection of a shared cut: one group of cameras per unit. n is fine enough
// for the group when every member culls it (kFrustum) or has s(n) <= tau; n is
// selected iff (leaf or fine(n)) and (root or not fine(parent)) and, with
// kFrustum, some member keeps it.
template <bool kFrustum>
struct SharedSelect {
    const float4 *box_lo, *box_hi;
    const CutCam *cams;
    const int32_t *group_begin;
    int c0, c1;
    __device__ __forceinline__ void begin(int g) {
        c0 = group_begin[g];
        c1 = group_begin[g + 1];
    }
    __device__ __forceinline__ bool operator()(int64_t node) const {
        const float4 lo = box_lo[node], hi = box_hi[node];
        const int parent = __float_as_int(lo.w);
        const bool leaf = __float_as_int(hi.w) == 0;
        float4 plo = lo, phi = hi;
        if (parent >= 0) {
            plo = box_lo[parent];
            phi = box_hi[parent];
        }
        bool fine_p = true, seen = !kFrustum;
        for (int c = c0; c < c1; ++c) {
            const CutCam &k = cams[c];
            bool vis_n = true, vis_p = true;
            if (kFrustum) {
                vis_n = !frustum_culled(k, lo, hi);
                // a culled parent culls the node, so a kept node's parent is kept
                vis_p = vis_n || (parent >= 0 && !frustum_culled(k, plo, phi));
                seen = seen || vis_n;
            }
            // neither a leaf nor fine enough for this member: not selected
            if (!leaf && vis_n &&
                !fine_enough(lo, hi, k.pos[0], k.pos[1], k.pos[2], k.fx, k.tau))
                return false;
            if (parent >= 0 && fine_p && vis_p &&
                !fine_enough(plo, phi, k.pos[0], k.pos[1], k.pos[2], k.fx, k.tau))
                fine_p = false;
        }
        return (parent < 0 || !fine_p) && seen;
    }
};

// Persistent loop over (unit, node block) partitions: count the selected
// nodes of the block, find the output offset by decoupled look-back, write
// the ids in ascending order.
template <class Select>
__device__ __forceinline__ void cut_partitions(Select sel, int64_t n_nodes, int n_units,
                                               uint32_t *__restrict__ ids, int64_t cap,
                                               uint32_t *__restrict__ offsets,
                                               uint32_t *__restrict__ counters, uint32_t *ticket,
                                               uint64_t *status, const uint32_t *epoch_ptr,
                                               uint32_t epoch_off, int *err) {
    __shared__ uint32_t s_part;
    __shared__ uint32_t s_cnt[kCutItems * 8];   // per (item row, warp), then exclusive
    __shared__ uint32_t s_excl;
    if (*err) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t nblk = (n_nodes + kCutPart - 1) / kCutPart;
    const int64_t nparts = nblk * n_units;
    const uint32_t epoch = *epoch_ptr + epoch_off;
    for (;;) {
        if (tid == 0) s_part = atomicAdd(ticket, 1u);
        __syncthreads();
        const int64_t part = s_part;
        if (part >= nparts) break;
        const int c = (int)(part / nblk);
        const int64_t b = part - (int64_t)c * nblk;
        sel.begin(c);
        uint32_t bal[kCutItems];
#pragma unroll
        for (int k = 0; k < kCutItems; ++k) {
            const int64_t node = b * kCutPart + k * kCutThreads + tid;
            const bool on = node < n_nodes && sel(node);
            bal[k] = __ballot_sync(0xffffffffu, on);
            if (lane == 0) s_cnt[k * 8 + warp] = __popc(bal[k]);
        }
        __syncthreads();
        if (warp == 0) {
            // exclusive scan of the 64 (row, warp) counts in node order
            const uint32_t v0 = s_cnt[2 * lane], v1 = s_cnt[2 * lane + 1];
            uint32_t incl = v0 + v1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            const uint32_t excl = incl - (v0 + v1);
            s_cnt[2 * lane] = excl;
            s_cnt[2 * lane + 1] = excl + v0;
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
            if (lane == 0) {
                uint64_t *slot = status + part;
                uint32_t prev = 0;
                if (part == 0) {
                    publish(slot, pack_status(kFlagPrefix, epoch, total));
                } else {
                    publish(slot, pack_status(kFlagAgg, epoch, total));
                    look_back(status, part, 1, epoch, &prev, err);
                    publish(slot, pack_status(kFlagPrefix, epoch, prev + total));
                }
                s_excl = prev;
                if (b == 0) offsets[c] = prev;
                if (part == nparts - 1) {
                    offsets[n_units] = prev + total;
                    counters[CNT_CUT] = prev + total;
                    if ((int64_t)prev + total > cap) latch_error(err, kErrCapacity);
                }
            }
        }
        __syncthreads();
        const uint32_t base = s_excl;
#pragma unroll
        for (int k = 0; k < kCutItems; ++k) {
            if ((bal[k] >> lane) & 1u) {
                const uint32_t pos = base + s_cnt[k * 8 + warp] + __popc(bal[k] & lanemask_lt());
                if (pos < cap) ids[pos] = (uint32_t)(b * kCutPart + k * kCutThreads + tid);
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kCutThreads)
k_cut(const float4 *__restrict__ box_lo, const float4 *__restrict__ box_hi, int64_t n_nodes,
      const DevCamera *__restrict__ cams, int n_cams, uint32_t *__restrict__ ids, int64_t cap,
      uint32_t *__restrict__ offsets, uint32_t *__restrict__ counters, uint32_t *ticket,
      uint64_t *status, const uint32_t *epoch_ptr, uint32_t epoch_off, int *err) {
    PlainSelect sel{box_lo, box_hi, cams, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    cut_partitions(sel, n_nodes, n_cams, ids, cap, offsets, counters, ticket, status, epoch_ptr,
                   epoch_off, err);
}

template <bool kFrustum>
__global__ void __launch_bounds__(kCutThreads)
k_cut_shared(const float4 *__restrict__ box_lo, const float4 *__restrict__ box_hi,
             int64_t n_nodes, const CutCam *__restrict__ cams,
             const int32_t *__restrict__ group_begin, int n_groups, uint32_t *__restrict__ ids,
             int64_t cap, uint32_t *__restrict__ offsets, uint32_t *__restrict__ counters,
             uint32_t *ticket, uint64_t *status, const uint32_t *epoch_ptr, uint32_t epoch_off,
             int *err) {
    SharedSelect<kFrustum> sel{box_lo, box_hi, cams, group_begin, 0, 0};
    cut_partitions(sel, n_nodes, n_groups, ids, cap, offsets, counters, ticket, status,
                   epoch_ptr, epoch_off, err);
}

// Cuts of many cameras or groups ("units"), in four steps: k_cut_nodes tests every
// interior node for every camera; k_cut_masks decides every (node, unit) from that and
// keeps one bit each, 32 nodes to a word, and each unit's count per node block; a scan
// of the counts in unit-major order gives the output offsets (k_cut_unit_offsets: those
// of the units); k_cut_write turns the words into ids, a pure stream.
//
// Both of the first run one CTA per (block of kCutPart nodes, chunk of up to C cameras)
// and use bit masks over the chunk's cameras: N (the camera keeps the node's box and it
// is not fine enough) and, with kFrustum, V (the camera keeps it).
//   k_cut_nodes: one lane per camera, 32 / C boxes at a time, so that a ballot is a box's
//     mask. With kFrustum the union of 32 nodes' boxes is tested first, a lane per camera:
//     those that cull it cull them all (a box outside a half-space has every box it
//     contains outside too, also in float32: the tests are monotone in the bounds). With
//     chunks of 32 cameras the others are put side by side, W of them, 32 / W boxes at a
//     time, where that saves two rounds (with 16 or 8 cameras it cost what it saved).
//   k_cut_masks: a node's own masks and its parent's. A leaf has N = 0; its V is tested
//     only for the cameras whose unit wants its parent refined and that keep the parent,
//     one lane per leaf: with groups each lane takes its own cameras, until one of a unit
//     keeps the leaf, else the word's cameras in turn. A unit's decision is bits: (leaf or
//     no N_n) and (root or some N_p) and some V_n over the unit's cameras; without kGroups
//     (units of one camera) that is the same formula on whole masks, and a 32 x 32 bit
//     transpose turns 32 nodes' masks into the cameras' words.
//
// Bound by the issue of the tests (about 14 instructions for a granularity, 75 for
// five planes). A test per (node, camera) on the node and on its parent, once to count
// and once to write, took 683 + 1016 us for 64 plain cuts of 5.25 M nodes, and one
// thread per node over its group's members 1557 us for 8 frustum-culled cuts of 8
// cameras each; with the parents tested again for the children of each word 228 us (+ 159
// us to write 850 MB of ids) and 530 us, with their masks read 172 us (108 + 64) and 433 us
// (228 + 205). With live cameras side by side and each lane at its own cameras 253 us (139 +
// 113), and the call of 8 shared cuts takes 390 - 447 us (by where the cameras are; 515 - 645
// before), that of 64 culled cuts of one camera each 505 - 588 us (555 - 675).
constexpr int kCutWords = kCutPart / 32;

template <bool kFrustum, int C>
__global__ void __launch_bounds__(kCutThreads, kFrustum ? 4 : 1)
k_cut_nodes(const float4 *__restrict__ box_lo, const float4 *__restrict__ box_hi,
            int64_t n_nodes, const CutCam *__restrict__ cams, const CutChunk *__restrict__ chunks,
            int n_chunks, uint2 *__restrict__ masks, const int *err) {
    constexpr int kWarps = kCutThreads / 32;
    __shared__ float4 s_lo[kWarps][32], s_hi[kWarps][32];   // the boxes under test, per warp
    constexpr bool kNarrow = kFrustum && C == 32;
    constexpr int kCamWords = 21;   // the planes, b0, pos, fx, tau
    __shared__ float s_cam[kNarrow ? kCamWords : 1][C];
    __shared__ int s_from[kNarrow ? kWarps : 1][32];       // lanes of the cameras under test
    if (*err) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t b = blockIdx.x / n_chunks;
    const int k = (int)(blockIdx.x - b * n_chunks);
    const CutChunk ch = chunks[k];
    uint2 *out = masks + k * n_nodes;
    // this lane's camera, and which of the boxes taken at once it tests
    const int cl = lane % C, grp = lane / C;
    CutCam cam = cams[ch.cam0 + min(cl, ch.n_cams - 1)];
    float tau2 = __fmul_rn(cam.tau, cam.tau);
    if (kNarrow) {
        if (tid < C) {
            const float *from = reinterpret_cast<const float *>(&cam);
#pragma unroll
            for (int k = 0; k < kCamWords; ++k) s_cam[k][tid] = from[k];
        }
        __syncthreads();
    }
    // camera c of the chunk becomes this lane's
    auto take = [&](int c) {
        float *to = reinterpret_cast<float *>(&cam);
#pragma unroll
        for (int k = 0; k < kCamWords; ++k) to[k] = s_cam[k][c];
        tau2 = __fmul_rn(cam.tau, cam.tau);
    };
    bool moved = false;   // `cam` is another than cl's
    for (int j = warp; j < kCutWords; j += kWarps) {
        const int64_t node = b * kCutPart + 32 * j + lane;
        const bool valid = node < n_nodes;
        float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
        if (valid) {
            lo = box_lo[node];
            hi = box_hi[node];
        }
        const bool inner = valid && __float_as_int(hi.w) != 0;
        const uint32_t inners = __ballot_sync(0xffffffffu, inner);
        if (inners == 0) continue;
        uint32_t N = 0, V = 0;
        // the lanes of one camera set that have a box to test
        uint32_t live = C == 32 ? 0xffffffffu : (1u << C) - 1u;
        if (kFrustum) {
            const float inf = __int_as_float(0x7f800000);
            float4 ulo = inner ? lo : make_float4(inf, inf, inf, 0.f);
            float4 uhi = inner ? hi : make_float4(-inf, -inf, -inf, 0.f);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                ulo.x = fminf(ulo.x, __shfl_xor_sync(0xffffffffu, ulo.x, o));
                ulo.y = fminf(ulo.y, __shfl_xor_sync(0xffffffffu, ulo.y, o));
                ulo.z = fminf(ulo.z, __shfl_xor_sync(0xffffffffu, ulo.z, o));
                uhi.x = fmaxf(uhi.x, __shfl_xor_sync(0xffffffffu, uhi.x, o));
                uhi.y = fmaxf(uhi.y, __shfl_xor_sync(0xffffffffu, uhi.y, o));
                uhi.z = fmaxf(uhi.z, __shfl_xor_sync(0xffffffffu, uhi.z, o));
            }
            if (kNarrow && moved) {
                take(cl);
                moved = false;
            }
            live &= __ballot_sync(0xffffffffu, cl < ch.n_cams && !frustum_culled(cam, ulo, uhi));
        }
        if (live) {
            const int n = __popc(inners), rank = inner ? __popc(inners & lanemask_lt()) : -1;
            if (inner) {
                s_lo[warp][rank] = lo;
                s_hi[warp][rank] = hi;
            }
            __syncwarp();
            // the cameras that do not cull all of these boxes, W of them (a power of two)
            // side by side: 32 / W boxes at a time
            int W = C, box = grp;
            if (kNarrow) {
                const int n_live = __popc(live);
                const int w = n_live == 1 ? 1 : 1 << (32 - __clz(n_live - 1));
                if ((n * C + 31) / 32 - (n * w + 31) / 32 >= 2) {   // rounds saved
                    W = w;
                    if (live >> lane & 1u) s_from[warp][__popc(live & lanemask_lt())] = lane;
                    __syncwarp();
                    box = lane / W;
                    moved = true;
                    take(s_from[warp][min(lane & (W - 1), n_live - 1)]);
                }
            }
            const int boxes = 32 / W;
#pragma unroll 2
            for (int t = 0; t < n; t += boxes) {
                const int q = min(t + box, n - 1);
                const float4 l = s_lo[warp][q], h = s_hi[warp][q];
                const bool keep = !kFrustum || !frustum_culled(cam, l, h);
                const bool fine = fine_enough_pre(l, h, box_extent(l, h), cam.pos[0], cam.pos[1],
                                                  cam.pos[2], cam.fx, tau2);
                const uint32_t nm = __ballot_sync(0xffffffffu, keep && !fine);
                const uint32_t vm = kFrustum ? __ballot_sync(0xffffffffu, keep) : 0xffffffffu;
                const int at = rank - t;   // a lane whose box is among these takes its masks
                if (at >= 0 && at < boxes) {
                    N = nm >> (W * at % 32);
                    V = vm >> (W * at % 32);
                }
            }
            if (kNarrow && W < C) {   // from the cameras side by side to the chunk's
                uint32_t n_all = 0, v_all = 0;
                int k = 0;
                for (uint32_t m = live; m; m &= m - 1, ++k) {
                    const int to = __ffs(m) - 1;
                    n_all |= (N >> k & 1u) << to;
                    v_all |= (V >> k & 1u) << to;
                }
                N = n_all;
                V = v_all;
            }
            __syncwarp();
        }
        if (inner) out[node] = make_uint2(N, V);
    }
}

template <bool kFrustum, bool kGroups, int C>
__global__ void __launch_bounds__(kCutThreads)
k_cut_masks(const float4 *__restrict__ box_lo, const float4 *__restrict__ box_hi,
            int64_t n_nodes, const CutCam *__restrict__ cams,
            const int32_t *__restrict__ group_begin, const CutChunk *__restrict__ chunks,
            int n_chunks, const uint2 *__restrict__ masks, uint32_t *__restrict__ words,
            uint32_t *__restrict__ counts, const int *err) {
    constexpr int kWarps = kCutThreads / 32;
    static_assert(kCutWords % kWarps == 0 && kCutWords == 64, "two words per lane");
    __shared__ uint32_t s_word[C][kCutWords + 1];
    // with groups every lane reads the camera that it is at (no bank conflicts by fields)
    constexpr int kCamWords = 19;   // the planes, b0, pos
    __shared__ float s_field[kFrustum && kGroups ? kCamWords : 1][C];
    __shared__ CutCam s_cam[kFrustum && !kGroups ? C : 1];
    __shared__ uint32_t s_peers[kFrustum && kGroups ? C : 1];   // each camera's unit
    __shared__ uint32_t s_unit[kGroups ? C : 1];   // each unit's cameras of the chunk
    if (*err) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t nblk = (n_nodes + kCutPart - 1) / kCutPart;
    const int64_t b = blockIdx.x / n_chunks;
    const int k = (int)(blockIdx.x - b * n_chunks);
    const CutChunk ch = chunks[k];
    const uint2 *mask = masks + k * n_nodes;
    const uint32_t live = ch.n_cams == 32 ? 0xffffffffu : (1u << ch.n_cams) - 1u;
    if (kFrustum && tid < ch.n_cams) {
        if (kGroups) {
            const float *from = reinterpret_cast<const float *>(cams + ch.cam0 + tid);
#pragma unroll
            for (int w = 0; w < kCamWords; ++w) s_field[w][tid] = from[w];
        } else {
            s_cam[tid] = cams[ch.cam0 + tid];
        }
    }
    if (kGroups && tid < ch.n_units) {
        const int g0 = group_begin[ch.unit0 + tid] - ch.cam0, g1 = group_begin[ch.unit0 + tid + 1] - ch.cam0;
        s_unit[tid] = (g1 == 32 ? 0xffffffffu : (1u << g1) - 1u) & ~((1u << g0) - 1u);
        if (kFrustum)
            for (int c = g0; c < g1; ++c) s_peers[c] = s_unit[tid];
    }
    __syncthreads();
#pragma unroll 2
    for (int j = warp; j < kCutWords; j += kWarps) {
        const int64_t node = b * kCutPart + 32 * j + lane;
        const bool valid = node < n_nodes;
        int parent = -1;
        bool leaf = true;
        if (valid) {
            parent = __float_as_int(box_lo[node].w);
            leaf = __float_as_int(box_hi[node].w) == 0;
        }
        // the parent's N (the root: as if one were refined) and, with groups, V (a unit of
        // one camera that wants the parent refined keeps it)
        uint32_t Np, Vp = 0xffffffffu;
        if (kFrustum && kGroups) {
            const uint2 up = parent >= 0 ? mask[parent] : make_uint2(valid ? 0xffffffffu : 0u, Vp);
            Np = up.x;
            Vp = up.y;
        } else {
            Np = !valid ? 0u : parent < 0 ? 0xffffffffu : mask[parent].x;
        }
        Np &= live;
        // the cameras whose units want the parent refined
        uint32_t want = Np;
        if (kGroups) {
            want = 0;
            for (int u = 0; u < ch.n_units; ++u)
                if (Np & s_unit[u]) want |= s_unit[u];
        }
        uint32_t sel = 0;     // bit u: unit u (camera, without kGroups) selects the node
        if (__any_sync(0xffffffffu, want != 0)) {
            uint2 own = make_uint2(0u, kFrustum ? 0u : 0xffffffffu);   // N, V
            if (!leaf && want) own = mask[node];
            if (kFrustum) {
                // the leaves: a lane each, but for the cameras that cull its parent (they
                // cull it too). With groups every lane takes its own cameras, as one that
                // keeps the leaf ends its unit's; else all have to look, each camera of the
                // word at a time
                uint32_t need = leaf ? want & Vp : 0u;
                float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
                if (need) {
                    lo = box_lo[node];
                    hi = box_hi[node];
                }
                if (kGroups) {
                    while (need) {
                        const int q = __ffs(need) - 1;
                        need &= need - 1;
                        CutCam cam;
                        float *to = reinterpret_cast<float *>(&cam);
#pragma unroll
                        for (int w = 0; w < kCamWords; ++w) to[w] = s_field[w][q];
                        if (!frustum_culled(cam, lo, hi)) {
                            own.y |= 1u << q;
                            need &= ~s_peers[q];   // its unit's others need not look
                        }
                    }
                } else {
                    for (uint32_t c = __reduce_or_sync(0xffffffffu, need); c; c &= c - 1) {
                        const int q = __ffs(c) - 1;
                        if ((need >> q & 1u) && !frustum_culled(s_cam[q], lo, hi)) own.y |= 1u << q;
                    }
                }
            }
            if (kGroups) {
                for (int u = 0; u < ch.n_units; ++u) {
                    const uint32_t m = s_unit[u];
                    if ((leaf || !(own.x & m)) && (Np & m) && (own.y & m)) sel |= 1u << u;
                }
            } else {
                sel = (leaf ? 0xffffffffu : ~own.x) & Np & own.y;
            }
        }
        // rows of nodes to rows of units
        uint32_t x = sel, m = 0x0000ffffu;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const uint32_t y = __shfl_xor_sync(0xffffffffu, x, o);
            x = lane & o ? (x & ~m) | (y & ~m) >> o : (x & m) | (y & m) << o;
            m ^= m << (o >> 1);
        }
        if (lane < C) s_word[lane][j] = x;
    }
    __syncthreads();
    for (int u = warp; u < ch.n_units; u += kWarps) {
        const uint32_t x = s_word[u][2 * lane], y = s_word[u][2 * lane + 1];
        const uint32_t n = __reduce_add_sync(0xffffffffu, (uint32_t)(__popc(x) + __popc(y)));
        const int64_t at = (int64_t)(ch.unit0 + u) * nblk + b;
        reinterpret_cast<uint2 *>(words)[at * (kCutWords / 2) + lane] = make_uint2(x, y);
        if (lane == 0) counts[at] = n;
    }
}

// The ids of one (unit, block) per warp, in unit-major order: two words per lane,
// then 64 nodes at a time, every lane a node.
__global__ void __launch_bounds__(256)
k_cut_write(const uint32_t *__restrict__ words, const uint32_t *__restrict__ part_off,
            const int64_t *__restrict__ offsets, int64_t nblk, int64_t n_parts,
            uint32_t *__restrict__ ids, int64_t cap, const int *err) {
    if (*err) return;
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= n_parts) return;
    const uint2 two = reinterpret_cast<const uint2 *>(words)[w * (kCutWords / 2) + lane];
    const uint32_t n0 = __popc(two.x), n = n0 + __popc(two.y);
    uint32_t incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (total == 0) return;
    const int64_t base = offsets[0] + part_off[w];
    const uint32_t excl = incl - n, lt = lanemask_lt();
    // nothing past the caller's capacity (an earlier slice of a call that exceeds it)
    const uint32_t room = (uint32_t)min(max(cap - base, (int64_t)0), (int64_t)total);
    uint32_t *out = ids + base;
    const uint32_t node0 = (uint32_t)(w % nblk) * kCutPart + lane;
#pragma unroll 4
    for (int j = 0; j < 32; ++j) {
        const uint32_t x = __shfl_sync(0xffffffffu, two.x, j), y = __shfl_sync(0xffffffffu, two.y, j);
        const uint32_t e = __shfl_sync(0xffffffffu, excl, j);
        const uint32_t px = e + __popc(x & lt), py = e + __popc(x) + __popc(y & lt);
        if ((x >> lane & 1u) && px < room) out[px] = node0 + 64 * j;
        if ((y >> lane & 1u) && py < room) out[py] = node0 + 64 * j + 32;
    }
}

// offsets[i] of the units of one call's slice (int64, offsets[0] being where the
// slice begins, 0 for the first one), and after the last slice the total.
__global__ void k_cut_unit_offsets(const uint32_t *__restrict__ part_off,
                                   const uint32_t *__restrict__ total, int64_t nblk, int n_units,
                                   int first, int last, int64_t cap, int64_t *offsets,
                                   uint32_t *__restrict__ counters, int *err) {
    const int64_t base = first ? 0 : offsets[0];
    __syncthreads();
    for (int i = threadIdx.x; i <= n_units; i += blockDim.x) {
        const int64_t v = base + (i < n_units ? part_off[(int64_t)i * nblk] : *total);
        offsets[i] = v;
        if (i == n_units && last) {
            counters[CNT_CUT] = (uint32_t)v;
            if (v > cap) latch_error(err, kErrCapacity);
        }
    }
}

int64_t cut_words_per_unit(int64_t n_nodes) {
    return (n_nodes + kCutPart - 1) / kCutPart * kCutWords;
}

template <bool kFrustum, bool kGroups, int C>
static void launch_masks_c(const float4 *box_lo, const float4 *box_hi, int64_t n_nodes,
                           const CutCam *cams, const int32_t *group_begin, const CutChunk *chunks,
                           int n_chunks, uint2 *masks, uint32_t *words, uint32_t *counts,
                           const int *err, cudaStream_t st) {
    const unsigned grid = (unsigned)((n_nodes + kCutPart - 1) / kCutPart * n_chunks);
    k_cut_nodes<kFrustum, C><<<grid, kCutThreads, 0, st>>>(box_lo, box_hi, n_nodes, cams, chunks,
                                                           n_chunks, masks, err);
    k_cut_masks<kFrustum, kGroups, C><<<grid, kCutThreads, 0, st>>>(
        box_lo, box_hi, n_nodes, cams, group_begin, chunks, n_chunks, masks, words, counts, err);
}

template <bool kFrustum, bool kGroups>
static void launch_masks(int c, const float4 *box_lo, const float4 *box_hi, int64_t n_nodes,
                         const CutCam *cams, const int32_t *group_begin, const CutChunk *chunks,
                         int n_chunks, uint2 *masks, uint32_t *words, uint32_t *counts,
                         const int *err, cudaStream_t st) {
    auto go = [&](auto f) {
        f(box_lo, box_hi, n_nodes, cams, group_begin, chunks, n_chunks, masks, words, counts, err, st);
    };
    if (c <= 8) go(launch_masks_c<kFrustum, kGroups, 8>);
    else if (c <= 16) go(launch_masks_c<kFrustum, kGroups, 16>);
    else go(launch_masks_c<kFrustum, kGroups, 32>);
}

void launch_cut_masks(bool frustum, bool groups, int c, const float4 *box_lo,
                      const float4 *box_hi, int64_t n_nodes, const CutCam *cams,
                      const int32_t *group_begin, const CutChunk *chunks, int n_chunks,
                      uint2 *masks, uint32_t *words, uint32_t *counts, const int *err,
                      cudaStream_t st) {
    auto go = [&](auto f) {
        f(c, box_lo, box_hi, n_nodes, cams, group_begin, chunks, n_chunks, masks, words, counts, err,
          st);
    };
    if (frustum) groups ? go(launch_masks<true, true>) : go(launch_masks<true, false>);
    else groups ? go(launch_masks<false, true>) : go(launch_masks<false, false>);
}

void launch_cut_write(const uint32_t *words, const uint32_t *part_off, const uint32_t *total,
                      int64_t n_nodes, int n_units, bool first, bool last, int64_t cap,
                      uint32_t *ids, int64_t *offsets, uint32_t *counters, int *err,
                      cudaStream_t st) {
    const int64_t nblk = (n_nodes + kCutPart - 1) / kCutPart, n_parts = nblk * n_units;
    k_cut_unit_offsets<<<1, 256, 0, st>>>(part_off, total, nblk, n_units, first, last, cap,
                                          offsets, counters, err);
    // writes nothing once the capacity is exceeded (latched above)
    k_cut_write<<<(unsigned)((n_parts + 7) / 8), 256, 0, st>>>(words, part_off, offsets, nblk,
                                                               n_parts, ids, cap, err);
}

void launch_cut(const SceneDev &sc, const DevCamera *cams, int n_cams, uint32_t *ids, int64_t cap,
                uint32_t *offsets, uint32_t *counters, uint32_t *ticket, uint64_t *status,
                const uint32_t *epoch, uint32_t epoch_off, int *err, int grid, cudaStream_t st) {
    k_cut<<<grid, kCutThreads, 0, st>>>(sc.box_lo, sc.box_hi, sc.n, cams, n_cams, ids, cap,
                                        offsets, counters, ticket, status, epoch, epoch_off, err);
}

void launch_cut_shared(bool frustum, const float4 *box_lo, const float4 *box_hi, int64_t n_nodes,
                       const CutCam *cams, const int32_t *group_begin, int n_groups,
                       uint32_t *ids, int64_t cap, uint32_t *offsets, uint32_t *counters,
                       uint32_t *ticket, uint64_t *status, const uint32_t *epoch,
                       uint32_t epoch_off, int *err, int grid, cudaStream_t st) {
    if (frustum)
        k_cut_shared<true><<<grid, kCutThreads, 0, st>>>(box_lo, box_hi, n_nodes, cams,
                                                         group_begin, n_groups, ids, cap, offsets,
                                                         counters, ticket, status, epoch,
                                                         epoch_off, err);
    else
        k_cut_shared<false><<<grid, kCutThreads, 0, st>>>(box_lo, box_hi, n_nodes, cams,
                                                          group_begin, n_groups, ids, cap,
                                                          offsets, counters, ticket, status,
                                                          epoch, epoch_off, err);
}

}  // namespace ngs
