// Float-float FFT pass launchers for L = 16, 32, 48, 64, 96, 128, 256 (see fft_passes.cuh).
#include "fft_passes.cuh"

namespace ls {

LS_PASS_INST(, ffp, 16)
LS_PASS_INST(, ffp, 32)
LS_PASS_INST(, ffp, 48)
LS_PASS_INST(, ffp, 64)
LS_PASS_INST(, ffp, 96)
LS_PASS_INST(, ffp, 128)
LS_PASS_INST(, ffp, 256)

}  // namespace ls
