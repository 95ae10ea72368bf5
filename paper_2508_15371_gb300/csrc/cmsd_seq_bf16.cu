// bfloat16 instantiations of the cluster-per-sequence kernel.
#include "cmsd_seq_impl.cuh"

namespace cmsd {

cudaError_t launch_seq_bf16(int mode, bool sampled, bool second, const StreamArgs& a, int nc, int threads,
                            cudaStream_t s) {
  return threads == 512 ? launch_seq_t<uint16_t, 512>(mode, sampled, second, a, nc, s)
                        : launch_seq_t<uint16_t, 256>(mode, sampled, second, a, nc, s);
}

int seq_clusters_bf16(int nc, int threads) {
  return threads == 512 ? seq_clusters_t<uint16_t, 512>(nc) : seq_clusters_t<uint16_t, 256>(nc);
}

bool seq_draw_fits_bf16(int V) { return seq_draw_fits_t<uint16_t>(V); }

}  // namespace cmsd
