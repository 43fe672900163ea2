// How the cameras of a cut by masks are split: slices of units whose words fit the
// scratch at once, in each of them chunks of up to 32 cameras with an array of node
// masks, as many arrays side by side as fit beside the words. Host arithmetic only.
#ifndef NGS_CUT_PLAN_H
#define NGS_CUT_PLAN_H

#include <algorithm>
#include <cstdint>
#include <vector>

namespace ngs {

// A chunk of a call's cameras, cams[cam0 .. cam0 + n_cams) (at most 32), and its
// units (cameras or whole groups), unit0 counted within the slice.
struct CutChunk {
    int32_t cam0, n_cams, unit0, n_units;
};

// Units [unit0, unit0 + n_units), of chunks [chunk0, chunk0 + n_chunks), decided n_masks
// chunks at a time.
struct CutSlice {
    int unit0, n_units, chunk0, n_chunks, n_masks;
};

struct CutPlan {
    int lanes;      // most cameras of a chunk: 8, 16 or 32
    std::vector<CutChunk> chunks;
    std::vector<CutSlice> slices;
};

// The least scratch: one array of masks and 32 units' words. mask_bytes: of a chunk's
// array, word_bytes: of a unit's words.
inline int64_t cut_least_bytes(int64_t mask_bytes, int64_t word_bytes) {
    return mask_bytes + 32 * word_bytes;
}

// group_begin null: units of one camera each; groups of up to 32 cameras otherwise.
// room: the scratch, at least cut_least_bytes. A slice has its own scan of counts and its
// own write, a further pass of chunks only its two launches: so the words come first.
inline void plan_cuts(int n_cams, const int32_t *group_begin, int n_units, int64_t mask_bytes,
                      int64_t word_bytes, int64_t room, CutPlan *p) {
    auto begin = [&](int u) { return group_begin ? group_begin[u] : u; };
    p->lanes = n_cams <= 8 ? 8 : n_cams <= 16 ? 16 : 32;
    p->chunks.clear();
    p->slices.clear();
    const int units = (int)std::min<int64_t>(n_units, (room - mask_bytes) / word_bytes);
    for (int u0 = 0; u0 < n_units; u0 += units) {
        CutSlice s{u0, std::min(units, n_units - u0), (int)p->chunks.size(), 0, 0};
        for (int u = u0; u < u0 + s.n_units;) {
            CutChunk ch{begin(u), 0, u - u0, 0};
            while (u < u0 + s.n_units && begin(u + 1) - ch.cam0 <= p->lanes) {
                ch.n_cams = begin(u + 1) - ch.cam0;
                ++ch.n_units;
                ++u;
            }
            p->chunks.push_back(ch);
        }
        s.n_chunks = (int)p->chunks.size() - s.chunk0;
        s.n_masks = (int)std::min<int64_t>(s.n_chunks, (room - s.n_units * word_bytes) / mask_bytes);
        p->slices.push_back(s);
    }
}

// Whether the plan's masks take less time than the single-pass kernels, by estimates in
// us. blocks: of nodes; largest: cameras of the largest group; resident: CTAs of the
// single-pass grid.
//   The single-pass kernel goes in rounds of `resident` (unit, block) partitions; a
// partition's time grows with its group, most under a frustum, where each member's five
// planes are tested one after the other. The masks' two kernels are a chain of several
// launches whose first CTAs take long (a CTA tests 2048 boxes for all cameras of a chunk),
// but then the chunk's cameras cost little more than one; a pass of chunks takes another
// launch of both.
//   Measured, masks / single pass, us: 64 plain cuts of 2.6k nodes 68 / 48, 26k 81 / 68,
// 79k 85 / 102, 1.31M 149 / 853; frustum-culled groups of 4 (64 cameras) 109 / 71, 142 / 83,
// 148 / 94, 216 / 535, of 12 104 / 97, 129 / 122, 126 / 127, 196 / 485; one group of 4 cameras,
// 1.31M nodes 77 / 68, with the frustum 97 / 96. On 945 such calls the choice is at most 8%
// slower than the better of the two.
inline bool cut_masks_pay(const CutPlan &p, int64_t blocks, int n_cams, int n_units, int largest,
                          bool frustum, int64_t resident) {
    // a last round of an eighth or less is hidden behind the others' ends
    const int64_t parts = blocks * n_units - resident / 8;
    const double rounds = (double)std::max<int64_t>(1, (parts + resident - 1) / resident);
    const double mean = (double)n_cams / n_units;
    const double cams = largest + (rounds - 1.0) * mean;   // one after the other
    const double single = frustum ? 52.0 + 9.0 * rounds + 5.0 * cams
                                  : 46.0 + 12.0 * rounds + 0.625 * cams;
    const int k = p.lanes == 8 ? 0 : p.lanes == 16 ? 1 : 2;
    constexpr double kPlain[3] = {70.0, 76.0, 86.0};
    constexpr double kCulled[3] = {88.0, 100.0, 134.0}, kOfUnits[3] = {5.0, 20.0, 35.0};
    double masks = frustum ? kCulled[k] + kOfUnits[k] / mean : kPlain[k];
    int passes = 0;
    for (const CutSlice &s : p.slices) passes += (s.n_chunks + s.n_masks - 1) / s.n_masks;
    masks += 44.0 * (passes - 1);
    return masks < single;
}

}  // namespace ngs

#endif
