// Partitions of the chained kernels (decoupled look-back: the offset scan in
// k_binning.cu, the radix sort in k_sort.cu), and the status words that a context
// holds for them. Host arithmetic only.
#ifndef NGS_LOOKBACK_H
#define NGS_LOOKBACK_H

#include <algorithm>
#include <cstdint>

namespace ngs {

// The scan's partitions: kScanPart elements; of pair offsets, up to kScanFew records go
// in partitions of kScanPartFew, which spread the rects that are slow to count. Other
// scans have no such elements: a million in 49 us by 2048, in 66 us by 256.
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8, kScanItemsFew = 1;      // elements per thread
constexpr int kScanPart = kScanThreads * kScanItems, kScanPartFew = kScanThreads * kScanItemsFew;
constexpr int64_t kScanFew = 1 << 20;

// The sort's: 8192 32-bit or 4096 64-bit keys, a status word per digit in each.
constexpr int kOsThreads = 512;
template <typename K> struct SortShape;
template <> struct SortShape<uint32_t> { static constexpr int kItems = 16; };
template <> struct SortShape<uint64_t> { static constexpr int kItems = 8; };
template <typename K>
constexpr int kOsPart = kOsThreads * SortShape<K>::kItems;
constexpr int kSortPart = kOsPart<uint64_t>;          // the smaller of the two

inline int64_t parts_of(int64_t n, int64_t part) { return (n + part - 1) / part; }

// partitions, and status words, of a scan of n elements, and of n records' pair offsets
inline int64_t scan_parts(int64_t n) { return parts_of(n, kScanPart); }
inline int64_t offset_parts(int64_t n) {
    return n <= kScanFew ? parts_of(n, kScanPartFew) : scan_parts(n);
}
// the most that the pair offsets of up to n records have
inline int64_t offset_status_words(int64_t n) {
    return std::max(offset_parts(n), offset_parts(std::min(n, kScanFew)));
}

struct LookBack {
    int64_t limit;   // bounds the standalone sort and scan: they are refused beyond it
    int64_t words;   // what the buffer holds
};

// For renders of up to rec_cap records and pair_cap pairs, cuts of max_units units of
// cut_blocks node blocks each (a partition per unit and block, or a scan of their
// counts), and every standalone sort and scan within the limit: a word for each partition
// that the limit counts.
inline LookBack look_back_words(int64_t cut_blocks, int64_t max_units, int64_t rec_cap,
                                int64_t pair_cap) {
    LookBack b;
    b.limit = std::max<int64_t>(cut_blocks * max_units, 1);
    b.limit = std::max(b.limit, parts_of(std::max(rec_cap, pair_cap), kSortPart) * 256);
    b.limit = std::max(b.limit, scan_parts(rec_cap));
    b.words = std::max(b.limit, offset_status_words(rec_cap));
    b.words = std::max(b.words, parts_of(rec_cap, kOsPart<uint32_t>) * 512);   // depth sort, 512 digits
    return b;
}

inline bool scan_accepted(int64_t n, int64_t limit) { return scan_parts(n) <= limit; }
inline bool sort_accepted(int64_t n, int64_t limit) { return parts_of(n, kSortPart) * 256 <= limit; }

}  // namespace ngs

#endif
