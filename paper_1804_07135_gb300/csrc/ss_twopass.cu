// The two-pass kernels of one length: compiled once per length of SS_T2_LENGTHS with SS_T2_P defined.
#include "ss_twopass.cuh"

namespace ss {
SS_T2_INSTANTIATE(float, SS_T2_P)
}  // namespace ss
