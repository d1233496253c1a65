// Checks the packed sweeps' gather tables (window_rows_host,
// window_chunks_host) against the orbit tables: for slabs of nk sets, every
// (set, orbit) item once, with its orbit's class and string addresses.
#include <cstdio>
#include <cstdlib>
#include <map>

#include "fs_internal.h"

using namespace fs;

int main(int argc, char** argv) {
  const int N = std::atoi(argv[1]), n = std::atoi(argv[2]), W = 6, nk = std::atoi(argv[3]);
  std::vector<uint32_t> orbits;
  std::vector<int> off, coff;
  std::vector<uint16_t> offs, rows;
  std::vector<uint8_t> okey;
  std::vector<uint2> cls;
  std::vector<uint4> chunk;
  window_tables_host(N, n, W, orbits, off, offs, okey);
  window_rows_host(n, W, orbits, off, offs, cls, rows);
  window_chunks_host(W, nk, cls, coff, chunk);
  if (coff.size() != off.size()) return std::puts("positions"), 1;
  for (size_t a = 0; a + 1 < off.size(); ++a) {
    // wanted: (class, strings' addresses) -> times
    std::map<std::vector<int>, int> want, got;
    for (int i = off[a]; i < off[a + 1]; ++i) {
      const int m = orbits[i] >> 24;
      if (!m) continue;
      std::vector<int> key{m};
      for (int S = 0; S < (1 << W); ++S)
        if (__builtin_popcount(S) == m)
          key.push_back((int)(orbits[i] & 0xFFFF) +
                        offs[((a * (n + 1) + ((orbits[i] >> 16) & 0xFF)) << W) + S]);
      for (int k = 0; k < nk; ++k) {
        key.push_back(k);
        ++want[key];
        key.pop_back();
      }
    }
    for (int c = coff[a]; c < coff[a + 1]; ++c)
      for (int lane = 0; lane < 32; ++lane) {
        const uint4 e = chunk[c];
        const uint32_t cnt = e.y & 0xFFFF, us = e.y >> 16, m = e.x >> 24;
        uint32_t o = (e.z & 0xFFFF) + lane;
        const uint32_t t = (uint32_t)(((uint64_t)(2 * o) * e.w) >> 32);
        if (t != o / cnt) return std::puts("division"), 1;
        const uint32_t k = (e.z >> 16) + t;
        o -= t * cnt;
        if (k >= (uint32_t)nk) continue;
        std::vector<int> key{(int)m};
        int s = 0;
        for (int S = 0; S < (1 << W); ++S)
          if (__builtin_popcount(S) == (int)m) {
            const size_t at = ((size_t)(e.x & 0xFFFFFF) + (s / 8) * us + o) * 8 + s % 8;
            if (at >= rows.size()) return std::puts("range"), 1;
            key.push_back(rows[at]);
            ++s;
          }
        key.push_back((int)k);
        ++got[key];
      }
    if (want != got) return std::printf("items at %zu\n", a), 1;
  }
  std::puts("ok");
  return 0;
}
