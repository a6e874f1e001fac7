// Forward scan launchers (Leaky; the Synaptic neuron's in a translation unit
// of its own, so that the two compile in parallel).
#include "scan_dispatch.cuh"

namespace snn {

cudaError_t launch_scan_fwd(ScanArgs a, bool synaptic, int in_dt, int io_dt, bool staged,
                            cudaStream_t stream) {
  if (synaptic) return launch_scan_fwd_synaptic(a, in_dt, io_dt, staged, stream);
  SNN_DTYPE_DISPATCH(in_dt, io_dt, return (fwd_t<false, TI, TO>(a, staged, stream)));
}

}  // namespace snn
