"""Which rows of a store the dense epilogue stages in shared memory, and which tiles the different-sample weight gradient copies
there: the rules of csrc/store.cuh, run on the host."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2007_10412_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "store.cuh"
using namespace rad;
int main() {
  std::mt19937 rng(5);
  const uint32_t top = 0xffffffffu;
  const uint32_t at[] = {0u, 1u, 7u, 8u, 9u, 1791u, 1792u, 1793u, 4096u, 0x7fffffffu, 0x80000000u, top - 1800u, top - 128u, top - 7u, top};
  long long outside = 0, refused = 0, taken = 0;
  // whatever an index holds, a row that is let in stays inside the buffer
  auto row = [&](uint32_t first, uint32_t pos, uint32_t kept) {
    const uint32_t end = pos + kept;
    if (!row_fits_stage(first, pos, end)) return;
    ++taken;
    for (uint32_t i = 0; i < kept; ++i) {
      const uint32_t byte = 2u * (pos + i - (first & ~7u));
      if (byte + 2u > (uint32_t)kFillBytes || pos + i < first) ++outside;
    }
  };
  for (uint32_t first : at)
    for (uint32_t pos : at)
      for (uint32_t kept = 0; kept <= 128; ++kept) row(first, pos, kept);
  for (int i = 0; i < 2000000; ++i) {
    const uint32_t first = rng() >> (rng() % 32), pos = (rng() & 1) ? first + (uint32_t)(rng() % 4096) - 2048u : rng();
    row(first, pos, rng() % 129);
  }
  // a drawn index (rows one behind the other) is in order, and staged exactly when the 32 rows fit
  for (int i = 0; i < 20000; ++i) {
    const uint32_t first = rng() >> (1 + rng() % 31), most = rng() % 129;
    uint32_t pos = first, last = 0;
    bool all = true;
    for (int r = 0; r < 32; ++r) {
      const uint32_t end = pos + (most > 0 ? rng() % (most + 1) : 0);
      if (!row_in_order(first, pos, end)) ++refused;
      all = all && row_fits_stage(first, pos, end);
      pos = last = end;
    }
    if (all != (last - (first & ~7u) <= kFillValues)) ++refused;
  }
  // a tile that is let in is a copy of whole 16-byte pieces from inside the buffer, no longer than its room
  long long bad = 0, copied = 0;
  for (int i = 0; i < 2000000; ++i) {
    const uint32_t near = rng() >> (rng() % 32), begin = (rng() & 1) ? near & ~7u : near;
    const uint32_t end = (rng() & 3) ? begin + (rng() % 1025) * ((rng() & 3) ? 8u : 1u) : (uint32_t)rng();
    const int64_t capacity = (rng() & 1) ? (int64_t)end + (int64_t)(rng() % 33) - 16 : (int64_t)rng();
    const uint32_t room = 128u * (1u + rng() % 128u);
    if (!tile_in_order(begin, end) || !tile_fits(begin, end, capacity, room)) continue;
    ++copied;
    const uint64_t bytes = ((uint64_t)end - begin) * 2u;
    if (begin % 8 != 0 || bytes % 16 != 0 || end < begin || (int64_t)end > capacity || bytes > room) ++bad;
  }
  for (uint32_t begin : at)
    for (uint32_t end : at)
      if (tile_in_order(begin, end) && tile_fits(begin, end, 0xffffffffll, 16384u) && (end < begin || end - begin > 8192u)) ++bad;
  // every tile of a store that its buffer holds is copied
  for (uint32_t kept = 0; kept <= 8192; kept += 8)
    if (!tile_in_order(1u << 30, (1u << 30) + kept) || !tile_fits(1u << 30, (1u << 30) + kept, (1ll << 30) + kept, 16384u)) ++bad;
  outside += bad;
  taken = taken > 100000 && copied > 100000 ? taken : 0;
  printf("%lld %lld %d\n", outside, refused, taken > 100000 ? 1 : 0);
  return 0;
}
"""


def test_staged_rows_and_tiles_lie_in_their_buffers_whatever_the_index_holds(tmp_path):
    src, exe = tmp_path / "rows.cu", tmp_path / "rows"
    src.write_text(PROGRAM)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_100a,code=sm_100a", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["0", "0", "1"]
