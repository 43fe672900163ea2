"""The host arithmetic that sizes shared work buffers. CPU only."""
import os
import subprocess


def run_host(tmp_path, source):
    """stdout words of a C++ program that includes the library's host-only headers."""
    from paper_2603_15186_gb300 import build
    prog, exe = tmp_path / "prog.cpp", tmp_path / "prog"
    prog.write_text(source)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-I", build.CSRC, str(prog), "-o",
                    str(exe)], check=True)
    return [int(x) for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()]


def test_status_words_hold_every_accepted_scan_and_sort(tmp_path):
    """Over capacities from one element to the default and scenes from one node block up:
    the status words that a standalone scan or sort within the limit uses, a render's
    and a cut's, are all in the buffer, whatever the partitions that the header's constants
    give them. What the limit accepts is one partition of 2048 elements a word."""
    n, refused, accepted, short = run_host(tmp_path, r"""
#include <cstdio>
#include <vector>
#include "lookback.h"
using namespace ngs;
int main() {
  long n = 0, refused = 0, accepted = 0, lacking = 0;
  std::vector<int64_t> caps;
  for (int k = 0; k <= 26; ++k) for (int64_t d : {-1, 0, 1}) if ((1ll << k) + d > 0) caps.push_back((1ll << k) + d);
  for (int64_t blocks : {1, 2, 3, 4, 5, 70, 2600}) for (int64_t rec : caps) for (int64_t pairs : caps) {
    const LookBack b = look_back_words(blocks, 1024, rec, pairs);
    const int64_t old = std::max({blocks * 1024, (std::max(rec, pairs) + 4095) / 4096 * 256, (rec + 2047) / 2048});
    auto need = [&](int64_t words) { ++n; lacking += words > b.words; };
    // scans: every power of two and the largest accepted, one less and one more
    for (int k = 0; k <= 31; ++k) for (int64_t d : {-1, 0, 1}) for (int64_t s : {(int64_t)1 << k, b.limit * 2048}) {
      const int64_t m = s + d;
      if (m <= 0) continue;
      if (scan_accepted(m, b.limit) != ((m + 2047) / 2048 <= old)) return 1;
      if (!scan_accepted(m, b.limit)) { ++refused; continue; }
      ++accepted;
      need(scan_parts(m));
    }
    // sorts: 4096 keys a partition (64 bits), 256 words each
    const int64_t most = b.limit / 256 * 4096;
    if (!sort_accepted(most, b.limit) || sort_accepted(most + 1, b.limit)) return 2;
    need((most + 4095) / 4096 * 256);
    // a render's scan of any number of records, its sorts; a cut's partitions and scan of counts
    need((std::min<int64_t>(rec, 1 << 20) + 255) / 256);
    need((rec + 2047) / 2048);
    need((rec + 8191) / 8192 * 512);
    need((pairs + 8191) / 8192 * 256);
    need(blocks * 1024);
    need(scan_parts(blocks * 1024));
  }
  std::printf("%ld %ld %ld %ld\n", n, refused, accepted, lacking);
  return 0;
}
""")
    assert n > 100_000 and refused > 1000 and accepted > 1000
    assert short == 0


def test_cut_plans_fill_their_slices(tmp_path):
    """Every unit is in one chunk of one slice, in order; masks and words of a slice fit
    the room; a slice holds as many units as words fit beside one array of masks (32 at the
    least room, so that a call of n units takes at most n / 32 slices however small the
    record buffer is), and its chunks as many arrays as fit then."""
    calls, slices, bad = run_host(tmp_path, r"""
#include <cstdio>
#include <random>
#include "cut_plan.h"
using namespace ngs;
int main() {
  std::mt19937 rng(1);
  long calls = 0, slices = 0, bad = 0;
  for (int64_t nodes : {1, 2049, 1'310'000, 50'000'000}) for (int n_cams : {4, 8, 9, 16, 17, 64, 1023, 1024})
    for (int most : {1, 3, 20, 32}) for (double scale : {1.0, 1.5, 3.0, 7.9, 40.0, 1e4}) {
      std::vector<int32_t> begin{0};
      while (begin.back() < n_cams)
        begin.push_back(std::min<int>(n_cams, begin.back() + (most == 1 ? 1 : 1 + rng() % most)));
      const int units = (int)begin.size() - 1;
      const int64_t mask = 8 * nodes, word = (nodes + 2047) / 2048 * 256;
      const int64_t room = (int64_t)(cut_least_bytes(mask, word) * scale);
      CutPlan p;
      plan_cuts(n_cams, most == 1 ? nullptr : begin.data(), units, mask, word, room, &p);
      ++calls;
      slices += (long)p.slices.size();
      const int64_t full = (room - mask) / word;
      bad += full < 32 || (int64_t)p.slices.size() != (units + full - 1) / full;
      int u = 0, chunk = 0;
      for (const CutSlice &s : p.slices) {
        bad += s.unit0 != u || s.chunk0 != chunk || s.n_masks < 1 || s.n_masks > s.n_chunks;
        bad += s.n_masks * mask + s.n_units * word > room;
        bad += s.n_masks < s.n_chunks && (s.n_masks + 1) * mask + s.n_units * word <= room;
        for (int k = 0; k < s.n_chunks; ++k, ++chunk) {
          const CutChunk &c = p.chunks.at(chunk);
          bad += c.cam0 != begin[u] || c.unit0 != u - s.unit0 || c.n_units < 1 || c.n_cams > p.lanes;
          bad += c.n_cams != begin[u + c.n_units] - begin[u];
          u += c.n_units;
          // no unit of the slice would have fitted too
          bad += u < s.unit0 + s.n_units && c.n_cams + begin[u + 1] - begin[u] <= p.lanes;
        }
        bad += u != s.unit0 + s.n_units;
      }
      bad += u != units || chunk != (int)p.chunks.size() || p.lanes > 32 || (p.lanes < n_cams && p.lanes < 32);
    }
  std::printf("%ld %ld %ld\n", calls, slices, bad);
  return 0;
}
""")
    assert calls > 500 and slices > calls and bad == 0


# (blocks of 2048 nodes, group sizes, frustum, masks pay)
CUT_ROUTES = [
    # small scenes and few groups: the single-pass kernels, measured 1.1 to 2.2 times as fast
    (2, [1] * 64, False, False), (13, [1] * 64, False, False), (39, [1] * 16, False, False),
    (2, [4] * 16, True, False), (13, [2] * 32, True, False), (39, [4] * 16, True, False),
    (39, [1] * 24, True, False), (97, [2] * 12, True, False), (97, [8] * 3, True, False),
    (39, [4] * 8, False, False), (194, [8], False, False), (643, [4], False, False), (643, [12], False, False),
    # large ones: the masks, 1.1 to 5 times as fast
    (39, [1] * 128, False, True), (194, [1] * 6, False, True), (643, [1] * 4, False, True),
    (643, [4] * 4, False, True), (2564, [4], False, True), (643, [1] * 4, True, True), (643, [8], True, True),
    (13, [12], True, True), (39, [32], True, True), (39, [4] * 64, True, True), (194, [1] * 64, True, True),
    (643, [4] * 16, True, True), (643, [12] * 5 + [4], True, True),
    # the calls of test_cuts_by_masks_of_a_larger_scene
    (381, [1] * 4, False, True), (381, [3, 5], False, True), (381, [32, 1, 31], False, True),
    (381, [1] * 4, True, True), (381, [1] * 16, True, True), (381, [3, 5], True, True),
    (381, [3, 12, 1], True, True), (381, [20, 30, 7], True, True)]


def test_cuts_go_by_masks_where_they_pay(tmp_path):
    calls = "".join("{%d, %d, {%s}},\n" % (b, f, ",".join(map(str, g))) for b, g, f, _ in CUT_ROUTES)
    got = run_host(tmp_path, r"""
#include <cstdio>
#include "cut_plan.h"
using namespace ngs;
struct Call { int64_t blocks; int frustum; std::vector<int> groups; };
int main() {
  for (const Call &c : std::vector<Call>{""" + calls + r"""}) {
    std::vector<int32_t> begin{0};
    int largest = 0;
    for (int g : c.groups) { begin.push_back(begin.back() + g); largest = std::max(largest, g); }
    CutPlan p;
    plan_cuts(begin.back(), begin.data(), (int)c.groups.size(), c.blocks * 16384, c.blocks * 256,
              (int64_t)1 << 33, &p);
    std::printf("%d\n", (int)cut_masks_pay(p, c.blocks, begin.back(), (int)c.groups.size(), largest,
                                           c.frustum != 0, 608));
  }
  return 0;
}
""")
    assert [bool(x) for x in got] == [pays for *_, pays in CUT_ROUTES]
