// Where the beams of a path are worked out, and with how much shared memory.  Plain arithmetic, host and device.
#pragma once

#ifdef __CUDACC__
#define SDMS_HD __host__ __device__ __forceinline__
#else
#define SDMS_HD inline
#endif

namespace sdms {

// log2 of the slots of one layer's node table (beams): a power of two above 5/4 of the matches.
SDMS_HD int beam_lcap(int M) {
  int l = 6;
  while ((1ll << l) < (long long)M + (M >> 2) + 1) ++l;
  return l;
}

struct BeamPlan { int cap, stride; bool lists; };    // slots per layer's table (0: does not fit), items per row, lists in shared memory
SDMS_HD BeamPlan beam_plan(int M, int D, int B, unsigned bytes) {
  BeamPlan w;
  w.cap = 1 << beam_lcap(M < (1 << 20) ? M : 1 << 20);
  w.stride = (M + 31) & ~31;
  const long long tables = (long long)D * (w.cap * 16ll + w.stride * 2ll) + w.cap * 6ll + w.stride * 2ll;
  w.lists = tables + (long long)D * w.cap * B * 16 <= (long long)bytes;
  if (tables > (long long)bytes || M >= 0xffff) w.cap = 0;
  return w;
}

// Shared memory of a CTA (one per SM).  Tables and lists want as much as there is, the form over the table area wants L1, and one
// launch has both (a launch for each form, side by side or not: the SMs keep the split of the launch before, 320 us for 203 on 32
// prompts of 16 x 1024, k = 1).  An SM splits its 256 KB at 164, 196 and 228 KB, so 160 and 192 KB are what just fits below a step;
// the smallest size is taken with which every pool has the same plan as with 200 KB.  Both sides, 8 prompts of 16 x 1024 tokens
// of small alphabets, k = 1, sdms_get_beams:
//   tables that only fit the larger size: D = 10, one beam, up to 674 matches, 66 us with 200 KB, 174 with 160; D = 11, four beams,
//     119 with 200, 610 with 192
//   lists: D = 16, two beams, up to 146 matches, 66 us with 200, 109 with 192; D = 20, one beam, up to 176, 72 with 200, 122 with 160
//   pools beyond every table: D = 16, up to 667 matches, one beam 319 us with 200, 267 with 160; four beams 1067 with 200, 893 with 192;
//     what takes 200 for its smaller pools pays for it here (two beams: 543 for 462 with 192)
constexpr int kBeamSizes[3] = {160 * 1024, 192 * 1024, 200 * 1024};

inline bool beam_same_plans(int D, int B, int bytes) {
  for (int M = 1;; ++M) {
    const BeamPlan a = beam_plan(M, D, B, (unsigned)kBeamSizes[2]), b = beam_plan(M, D, B, (unsigned)bytes);
    if (a.cap != b.cap || a.lists != b.lists) return false;
    if (!a.cap) return true;                           // more matches need more still
  }
}

// Shared memory for B beams of D tokens.  All are worked out by the first call (when a context is created).
inline int beam_bytes(int D, int B) {
  constexpr int kD = 32, kB = 8;
  struct Sizes {
    int of[kD + 1][kB + 1];
    Sizes() {
      for (int d = 0; d <= kD; ++d)
        for (int b = 0; b <= kB; ++b) {
          int x = 0;
          while (d && b && x < 2 && !beam_same_plans(d, b, kBeamSizes[x])) ++x;
          of[d][b] = kBeamSizes[x];
        }
    }
  };
  static const Sizes sizes;
  return D <= kD && B <= kB ? sizes.of[D][B] : kBeamSizes[2];
}

}  // namespace sdms
