// pic_small_f32.cu -- the one-kernel steps of small plasmas, float form (pic_small.cuh).
#include "pic_small.cuh"

namespace pic {
int launch_small_f32(const SmallArgs &a, int num_sms, cudaStream_t s) { return launch_small_r<float>(a, num_sms, s); }
}  // namespace pic
