// Work split and shared-memory layout of the row transforms (Toeplitz / 2-D-mask
// passes, gridding adjoint, Cartesian row adjoint).
#pragma once
#include "common.cuh"
#include "kernels.cuh"

namespace pico {

// Row passes.  A block owns kRowLines image rows of one image and walks the
// coils in steps of CS at once, so that the b-jobs (one per coil, row and
// frequency group k2) fill all NT threads; the a-jobs (one per row and n1) of
// GA coil subgroups fill up to NT threads too, each thread working through
// CA = CS / GA coils of a step.  kRowLines divides every supported side.
//
// Before, a block's one coil at a time left half of its threads without a b-job,
// the strided twiddle look-ups made up most of the shared-memory wavefronts, and
// every coil waited for its own global loads (ncu: issue 30-36 %, barrier and
// load stalls 6 of 8 warps): 32 images at L = 480, forward 176 -> 138 us,
// inverse 221 -> 171 us, now at half of the DRAM rate.
//
// Exchange layout: a line of each (coil, image row) holds P1 rows of P2 values,
// row n1 the P2 values of that n1, with the 16-byte chunk of value k at
// (k >> 1) ^ (n1 & 7) (64-byte rows: ^ ((n1 >> 1) & 3)) -- the TMA swizzle of
// that row width, lines padded to the pattern's period.  a-jobs (consecutive
// lanes, consecutive n1) move two values per 16-byte access, b-jobs
// (consecutive lanes, consecutive k2) one value per 8-byte access, both without
// bank conflicts, and the inverse pass's rows arrive in it directly.  The
// twiddles of the a-jobs are stored [k][n1] for the same reason: the strided
// look-ups W^(n1 k) of the plain table cost more shared-memory wavefronts than
// the data.

template <int P1, int P2, int NT_>
struct RowPass {
  static constexpr int RL = kRowLines;
  static constexpr int NT = NT_;
  static constexpr int CS = NT / (RL * P2);          // coils per step
  static constexpr int ga(int nin) {
    int g = CS;
    while (RL * P1 * g > NT || g > nin) g /= 2;
    return g;
  }
  static constexpr int GA = ga(P2 / 2);               // coil subgroups of the a-jobs
  static constexpr int CA = CS / GA;                  // coils per a-thread and step
  static constexpr int AT = RL * P1 * GA;             // a-threads
  static constexpr int RB = P2 * 8;                   // bytes of an exchange row
  static constexpr int period = P2 == 16 ? 1024 : 512;  // of the swizzle pattern
  static constexpr int line = (P1 * RB + period - 1) / period * period;  // bytes of a line
  static constexpr size_t slot = (size_t)RL * line;
  static constexpr size_t tw = (size_t)P1 * P2 * sizeof(float2);
  // exchange slots, sensitivity rows, twiddles, two mbarriers, alignment slack
  static constexpr size_t smem(int n) { return 1024 + CS * slot + (size_t)CS * RL * n * 8 + tw + 16; }
  // byte offset of value k of row n1 in a line (the XOR is on bits 4 ..)
  static __device__ __forceinline__ uint32_t at(int n1, int k) {
    const uint32_t sw = P2 == 16 ? (n1 & 7) : ((n1 >> 1) & 3);
    return (uint32_t)(n1 * RB) + ((((uint32_t)(k >> 1) ^ sw) << 4) | ((k & 1) << 3));
  }
};

}  // namespace pico
