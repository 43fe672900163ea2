// Partitions of the chained kernels (decoupled look-back: the offset scan in
// k_binning.cu, the radix sort in k_sort.cu), and the status words that a context
// holds for them. Host arithmetic only.
#ifndef NGS_LOOKBACK_H
#define NGS_LOOKBACK_H

#include <algorithm>
#include <cstdint>

namespace ngs {

// The scan's partitions: kScanPart elements, or kScanPartFew for inputs of up to kScanFew.
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

// partitions, and status words, of a scan of n elements
inline int64_t scan_parts(int64_t n) { return parts_of(n, n <= kScanFew ? kScanPartFew : kScanPart); }
// the most that a scan of up to n elements has
inline int64_t scan_status_words(int64_t n) {
    return std::max(scan_parts(n), scan_parts(std::min(n, kScanFew)));
}

struct LookBack {
    int64_t limit;   // bounds the standalone sort and scan: they are refused beyond it
    int64_t words;   // what the buffer holds
};

// For renders of up to rec_cap records and pair_cap pairs, cuts of max_units units of
// cut_blocks node blocks each (a partition per unit and block, or a scan of their
// counts), and every standalone sort and scan within the limit.
inline LookBack look_back_words(int64_t cut_blocks, int64_t max_units, int64_t rec_cap,
                                int64_t pair_cap) {
    LookBack b;
    b.limit = std::max<int64_t>(cut_blocks * max_units, 1);
    b.limit = std::max(b.limit, parts_of(std::max(rec_cap, pair_cap), kSortPart) * 256);
    b.limit = std::max(b.limit, parts_of(rec_cap, kScanPart));
    // the limit counts partitions of kScanPart: a scan of kScanFew elements within it has
    // eight times as many
    b.words = scan_status_words(b.limit * kScanPart);
    b.words = std::max(b.words, scan_status_words(rec_cap));
    b.words = std::max(b.words, scan_status_words(cut_blocks * max_units));
    b.words = std::max(b.words, parts_of(rec_cap, kOsPart<uint32_t>) * 512);   // depth sort, 512 digits
    return b;
}

inline bool scan_accepted(int64_t n, int64_t limit) { return parts_of(n, kScanPart) <= limit; }
inline bool sort_accepted(int64_t n, int64_t limit) { return parts_of(n, kSortPart) * 256 <= limit; }

}  // namespace ngs

#endif
