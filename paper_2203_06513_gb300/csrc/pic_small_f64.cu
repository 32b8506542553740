// pic_small_f64.cu -- the one-kernel steps of small plasmas, double form (pic_small.cuh).
#include "pic_small.cuh"

namespace pic {
int launch_small_f64(const SmallArgs &a, int num_sms, cudaStream_t s) { return launch_small_r<double>(a, num_sms, s); }
}  // namespace pic
