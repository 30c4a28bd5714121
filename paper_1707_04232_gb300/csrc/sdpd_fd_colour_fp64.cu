// sdpd_fd_colour_fp64.cu -- the colour kernels of the float64 state, every
// block-schedule variant, with float64 or float32 pair arithmetic (kept apart
// from the mixed state so that the variants compile in parallel).
#include "sdpd_fd_team64.cuh"

namespace sdpd {

template void fd_prepare<Fp64, Fp64>();
template void fd_prepare<Fp64, Mixed>();
template void launch_stage_geometry<Fp64, Fp64>(const Consts&, const Workspace&, cudaStream_t);
template void launch_stage_geometry<Fp64, Mixed>(const Consts&, const Workspace&, cudaStream_t);
template void launch_fd_colours<Fp64, Fp64>(const Consts&, const Workspace&, int, double, uint64_t, int,
                                          cudaStream_t);
// float64 state, float32 pair arithmetic
template void launch_fd_colours<Fp64, Mixed>(const Consts&, const Workspace&, int, double, uint64_t, int,
                                           cudaStream_t);

int fd_round_width(const Consts& c, bool float_arith, bool large) {
  return float_arith ? (large ? 32 : 32 / kFdOpw[fd_launch_variant(c)]) : kTeamPairs;
}

}  // namespace sdpd
