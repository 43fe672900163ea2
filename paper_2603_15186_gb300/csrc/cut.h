// Frustum-culled and shared level-of-detail cuts (k_cut.cu), used by the C ABI.
#ifndef NGS_CUT_H
#define NGS_CUT_H

#include <cuda_runtime.h>
#include <stdint.h>

#include "cut_plan.h"

namespace ngs {

struct DevCamera;

// One camera of a shared cut: the five planes of its view volume in world
// terms, P_k(x) = a[k] . (x - pos) + (k == 0 ? b0 : 0), in the order near,
// left, right, top, bottom (a node whose box has P_k < 0 everywhere for some k
// is culled), and the inputs of its granularity test.
struct CutCam {
    float a[5][3];
    float b0;
    float pos[3];
    float fx, tau;
    float pad[3];
};
static_assert(sizeof(CutCam) == 96, "CutCam layout");

// Group g of the cameras is cams[group_begin[g] .. group_begin[g + 1]); its
// cut goes to ids[offsets[g] .. offsets[g + 1]) (ascending node ids), the
// total to counters[CNT_CUT]. The status words, ticket and epoch follow the
// plain cut's conventions.
void launch_cut_shared(bool frustum, const float4 *box_lo, const float4 *box_hi, int64_t n_nodes,
                       const CutCam *cams, const int32_t *group_begin, int n_groups,
                       uint32_t *ids, int64_t cap, uint32_t *offsets, uint32_t *counters,
                       uint32_t *ticket, uint64_t *status, const uint32_t *epoch,
                       uint32_t epoch_off, int *err, int grid, cudaStream_t st);

// Cuts of many units, one slice of them at a time (cut_plan.h): launch_cut_masks
// decides, for chunks of at most c <= 32 cameras, every (node, unit) into words[unit *
// cut_words_per_unit() ...] and counts[unit * blocks + block] (blocks of
// cut_partition_nodes() nodes), with masks[n_chunks][n_nodes] as scratch; after all
// chunks of the slice and an exclusive scan of the counts into part_off (its sum in
// *total), launch_cut_write writes the units' offsets (offsets[0] ..
// offsets[n_units], continuing from offsets[0] unless `first`) and ids; with `last`
// also counters[CNT_CUT], and it latches the capacity error when the ids exceed cap.
// group_begin (with groups): the slice's entries. Without groups a unit is a camera.
// frustum: the cameras' planes cull.
void launch_cut_masks(bool frustum, bool groups, int c, const float4 *box_lo,
                      const float4 *box_hi, int64_t n_nodes, const CutCam *cams,
                      const int32_t *group_begin, const CutChunk *chunks, int n_chunks,
                      uint2 *masks, uint32_t *words, uint32_t *counts, const int *err,
                      cudaStream_t st);
void launch_cut_write(const uint32_t *words, const uint32_t *part_off, const uint32_t *total,
                      int64_t n_nodes, int n_units, bool first, bool last, int64_t cap,
                      uint32_t *ids, int64_t *offsets, uint32_t *counters, int *err,
                      cudaStream_t st);
int64_t cut_words_per_unit(int64_t n_nodes);

}  // namespace ngs

#endif
