// The pulls of a standalone commit + pull call that decide its replicas.
#ifndef AGN_LAST_PULLS_H
#define AGN_LAST_PULLS_H

#include <cstdint>

namespace agn {

// Workers up to which a call finds its superseded pulls in a table on the stack
// (16 KB): agn_commit_pull_noalloc takes no memory from the heap.
constexpr int32_t kStackPullWorkers = 4096;

// Each worker's last pull of a call.  Nothing reads a replica between two pulls
// of one call, so the earlier ones would only write bytes that a later one
// overwrites (four pulls after each of 64 commits, 64 workers, 2^24 parameters:
// 4327 us a call with every pull written, 2602 with the last ones).  pw
// [n_pulls] as in agn_commit_pull (validated, workers < n); last: n entries, or
// null, where every pull counts.
class LastPulls {
 public:
  LastPulls(const int32_t* pw, int32_t n_pulls, int32_t* last) : pw_(pw), last_(last) {
    if (last)
      for (int32_t p = 0; p < n_pulls; ++p) last[pw[p]] = p;
  }
  bool writes(int32_t p) const { return !last_ || last_[pw_[p]] == p; }
  // how many of the pulls [p0, p1) write
  int32_t count(int32_t p0, int32_t p1) const {
    if (!last_) return p1 - p0;
    int32_t k = 0;
    for (int32_t p = p0; p < p1; ++p) k += writes(p);
    return k;
  }

 private:
  const int32_t* pw_;
  const int32_t* last_;
};

}  // namespace agn

#endif  // AGN_LAST_PULLS_H
