// The rules of the persistent kernel's grid barrier, apart from the kernel so that the CPU can
// run them too.
#pragma once

#ifdef __CUDACC__
#define KCMG_HD __host__ __device__
#else
#define KCMG_HD
#endif

namespace kcmg {

// Whether a counter of arrivals has reached target.  Both run modulo 2^32 and at most one barrier
// apart, so the sign of their difference tells, also when the counter has wrapped: after 28 million
// barriers of 152 blocks, which a whole solve with an iteration cap of some 100,000 gets to.
KCMG_HD inline bool count_reached(unsigned int count, unsigned int target) { return (int)(count - target) >= 0; }

// Whether a block that waits gives up: after so many polls (a few seconds) without a sign of block 0.
// That block leaves its clock after every phase on the levels that it runs alone, which can take as
// long as their iteration caps allow.
constexpr unsigned int kMaxPolls = 1u << 23;
KCMG_HD inline bool give_up(unsigned int& polls, unsigned int& seen, unsigned int progress) {
  if (progress != seen) {
    seen = progress;
    polls = 0;
  }
  return polls > kMaxPolls;
}

}  // namespace kcmg
