// Host-side rules that need no GPU.
#ifndef SBG_HOST_H
#define SBG_HOST_H

#include <cstddef>
#include <thread>

namespace sbg {

// Host threads (the caller's among them) that copy `bytes` of results out of pinned
// staging, at most `cores` of them.  Starting threads right after the wait for the GPU
// costs a call about 50 us for three and 370 us for seven (a call of 0.1 MB: 138 / 203 /
// 511 us on 1 / 4 / 8), and one thread copies into a fresh array, page faults with it,
// at about 11 GB/s.  Whole projected calls into fresh arrays, us, on 1 / 3 / 4 / 8:
// 1.1 MB 216 / 245 / 251 / 567, 1.6 MB 246 / 254 / 256 / 588, 1.85 MB 270 / 267 / 268 /
// 602, 2.5 MB 330 / 294 / 296 / 613, 4.1 MB 445 / 349 / 339 / 663, 15 MB 1288 / 763 /
// 699 / 840, 27 MB 2312 / 1242 / 1127 / 1183, 35 MB 3442 / 1753 / 1533 / 1387, 54 MB
// 5042 / 2501 / 2139 / 1814; into kept arrays the lines lie at the same sizes.
inline int copy_threads(size_t bytes, unsigned cores) {
  if (bytes < (7u << 18) || cores < 2) return 1;
  const size_t most = bytes < (32u << 20) ? (bytes >> 19 < 4 ? bytes >> 19 : 4) : 8;
  return (int)(most < cores ? most : cores);
}
// The same on this machine.  Its cores are counted once, by the first call that needs
// them: the count takes 15 to 20 us after a wait for the GPU.
inline int copy_threads(size_t bytes) {
  if (copy_threads(bytes, 8) == 1) return 1;
  static const unsigned cores = std::thread::hardware_concurrency();
  return copy_threads(bytes, cores);
}

}  // namespace sbg

#endif  // SBG_HOST_H
