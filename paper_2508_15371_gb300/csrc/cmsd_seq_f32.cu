// float32 instantiations of the cluster-per-sequence kernel.
#include "cmsd_seq_impl.cuh"

namespace cmsd {

cudaError_t launch_seq_f32(int mode, bool sampled, bool second, const StreamArgs& a, int nc, int threads,
                            cudaStream_t s) {
  return threads == 512 ? launch_seq_t<float, 512>(mode, sampled, second, a, nc, s)
                        : launch_seq_t<float, 256>(mode, sampled, second, a, nc, s);
}

int seq_clusters_f32(int nc, int threads) {
  return threads == 512 ? seq_clusters_t<float, 512>(nc) : seq_clusters_t<float, 256>(nc);
}

bool seq_draw_fits_bf16(int V);
bool seq_draw_fits(int dtype, int V) { return dtype == 0 ? seq_draw_fits_t<float>(V) : seq_draw_fits_bf16(V); }

}  // namespace cmsd
