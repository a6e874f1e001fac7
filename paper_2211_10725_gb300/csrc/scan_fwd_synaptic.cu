// Forward scan launchers of the Synaptic neuron.
#include "scan_dispatch.cuh"

namespace snn {

cudaError_t launch_scan_fwd_synaptic(ScanArgs a, int in_dt, int io_dt, bool staged, cudaStream_t stream) {
  SNN_DTYPE_DISPATCH(in_dt, io_dt, return (fwd_t<true, TI, TO>(a, staged, stream)));
}

}  // namespace snn
