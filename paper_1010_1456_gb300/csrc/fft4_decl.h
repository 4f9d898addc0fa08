// Entry points of the four-step FFT kernels (fft4_launch.cuh), one
// specialisation per list of lengths (fourstep_part): 1 launched, 0 no kernel
// for this length, < 0 minus an error code.
#pragma once

#include "common.h"

namespace aim {

struct StridedArgs4;
struct XArgs4;

#define AIM_FFT4_DECLARE(pol, S)                                                                                  \
  template <int PART>                                                                                             \
  int fft4_strided_##pol(aim_ctx*, const char*, bool, const S*, S*, const StridedArgs4&, int, int, const S*); \
  template <int PART>                                                                                             \
  int fft4_x_##pol(aim_ctx*, const char*, S*, const XArgs4&, int, const S*, const S*, int);
AIM_FFT4_DECLARE(p32, float2)
AIM_FFT4_DECLARE(p64, double2)
AIM_FFT4_DECLARE(pff, float4)
#undef AIM_FFT4_DECLARE

#define AIM_FFT4_PART_DECLARE(pol, S, PART)                                                                        \
  template <>                                                                                                     \
  int fft4_strided_##pol<PART>(aim_ctx*, const char*, bool, const S*, S*, const StridedArgs4&, int, int, const S*); \
  template <>                                                                                                     \
  int fft4_x_##pol<PART>(aim_ctx*, const char*, S*, const XArgs4&, int, const S*, const S*, int);
#define AIM_FFT4_PARTS_DECLARE(pol, S)                                                 \
  AIM_FFT4_PART_DECLARE(pol, S, 0) AIM_FFT4_PART_DECLARE(pol, S, 1)                    \
  AIM_FFT4_PART_DECLARE(pol, S, 2) AIM_FFT4_PART_DECLARE(pol, S, 3)                    \
  AIM_FFT4_PART_DECLARE(pol, S, 4) AIM_FFT4_PART_DECLARE(pol, S, 5)
AIM_FFT4_PARTS_DECLARE(p32, float2)
AIM_FFT4_PARTS_DECLARE(p64, double2)
AIM_FFT4_PARTS_DECLARE(pff, float4)
#undef AIM_FFT4_PARTS_DECLARE
#undef AIM_FFT4_PART_DECLARE

}  // namespace aim
