// Launchers of the navigation kernels (k_nav.cu), used by the C ABI.
#ifndef NGS_NAV_H
#define NGS_NAV_H

#include <cuda_runtime.h>
#include <stdint.h>

namespace ngs {

// navigable map and breadth-first distance fields (synchronises `st`; returns
// 0 or a cudaError_t), and shortest paths by descent
int launch_nav_fields(const uint8_t *occ, int nx, int ny, int k_lo, int k_hi, int inflate,
                      const int2 *d_goals, int n_goals, uint8_t *any, uint32_t *free_bits,
                      uint32_t *queues, uint8_t *blocked, uint32_t *dist, int num_sms,
                      cudaStream_t st);
// 32-bit words of a row of the free-cell map: at least one bit past the row's end
inline int nav_row_words(int nx) { return nx / 32 + 1; }
// words of the queues that launch_nav_fields takes for such a map (0: none)
size_t nav_queue_words(int nx, int ny, int n_goals, int num_sms);
void launch_nav_paths(const uint32_t *dist, int nx, int ny, int n_goals, const int3 *starts,
                      int n, int max_len, int2 *paths, int32_t *lens, int num_sms,
                      cudaStream_t st);

}  // namespace ngs

#endif
