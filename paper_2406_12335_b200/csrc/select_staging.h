// Layout of a unit's staged keys in the selection kernel's shared memory (plain C++: the host sizes the launch with it, the
// kernel indexes with it, a CPU test walks it).
//
// Key i of the middle range sits at word pad + i, pad in 0 .. 3, so that 16-byte loads from global memory pair with 16-byte
// stores; the passes then read whole groups of four words, the last of which may reach beyond the last key.
#pragma once

namespace vatp {

#ifdef __CUDACC__
#define VATP_HD __host__ __device__
#else
#define VATP_HD
#endif

// groups of four words that hold n keys from word `pad` on
VATP_HD constexpr int staged_groups(int pad, int n) { return (pad + n + 3) >> 2; }

// words of shared memory for n keys, whatever the padding
VATP_HD constexpr int staged_words(int n) { return 4 * staged_groups(3, n); }

#undef VATP_HD

}  // namespace vatp
