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
    and a cut's, are all in the buffer. What the limit accepts is what it accepted when
    every scan had partitions of 2048 elements."""
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
      need((m + (m <= 1 << 20 ? 255 : 2047)) / (m <= 1 << 20 ? 256 : 2048));
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
    need((std::min<int64_t>(blocks * 1024, 1 << 20) + 255) / 256);
  }
  std::printf("%ld %ld %ld %ld\n", n, refused, accepted, lacking);
  return 0;
}
""")
    assert n > 100_000 and refused > 1000 and accepted > 1000
    assert short == 0
