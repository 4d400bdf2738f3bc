// The two-pass kernels of one length and type: compiled for every length of SS_T2_LENGTHS in float and double,
// with SS_T2_P and SS_T2_T defined.
#include "ss_twopass.cuh"

namespace ss {
SS_T2_INSTANTIATE(SS_T2_T, SS_T2_P)
}  // namespace ss
