// Plain (one field per launch) shoot kernel.
#include "rs_internal.h"

namespace {

using namespace rsdev;

// MINB resident CTAs per SM as the occupancy floor: two let the compiler keep a small CTA's eight rays
// per thread, their two-float accumulators and a deep instruction window in up to 255 registers;
// three (168 registers) hide more latency with twelve warps per SM; eight-warp CTAs take one.
template <int WARPS, int RPT, int TILE, int MASS, int MINB>
__global__ void __launch_bounds__(WARPS * 32, MINB) shoot_kernel(const ShootDesc d) {
  extern __shared__ __align__(128) unsigned char rs_smem[];
  auto& ss = *reinterpret_cast<ShootSmem<WARPS, RPT, TILE>*>(rs_smem);
  PipeState ps;
  pipe_init(ss.lens.bar, ps);
  (void)shoot_tile<WARPS, RPT, TILE, MASS>(d, (int64_t)blockIdx.x, ss, ps);
}

template <int WARPS, int RPT, int TILE, int MASS, int MINB>
cudaError_t launch_shoot_m(const ShootDesc& d, int64_t grid, cudaStream_t s) {
  constexpr size_t smem = sizeof(ShootSmem<WARPS, RPT, TILE>);
  cudaError_t e = rsint::smem_opt_in<shoot_kernel<WARPS, RPT, TILE, MASS, MINB>>(smem);
  if (e != cudaSuccess) return e;
  shoot_kernel<WARPS, RPT, TILE, MASS, MINB><<<(unsigned)grid, WARPS * 32, smem, s>>>(d);
  return cudaGetLastError();
}

template <int WARPS, int RPT, int TILE, int MINB>
cudaError_t launch_shoot_t(const ShootDesc& d, cudaStream_t s) {
  const int64_t grid = shoot_tiles<WARPS, RPT>(d.n_rows, d.n0);
  if (grid <= 0) return cudaSuccess;
  if (grid >= ((int64_t)1 << 31)) return cudaErrorInvalidValue;
  return d.f.has_mass ? launch_shoot_m<WARPS, RPT, TILE, kMass, MINB>(d, grid, s)
                      : launch_shoot_m<WARPS, RPT, TILE, kUnitMass, MINB>(d, grid, s);
}

template <int WARPS, int RPT, int TILE, int MASS, int MINB>
cudaError_t occupancy_m(int* blocks) {
  constexpr size_t smem = sizeof(ShootSmem<WARPS, RPT, TILE>);
  cudaError_t e = rsint::smem_opt_in<shoot_kernel<WARPS, RPT, TILE, MASS, MINB>>(smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, shoot_kernel<WARPS, RPT, TILE, MASS, MINB>,
                                                       WARPS * 32, smem);
}

template <int WARPS, int RPT, int TILE, int MINB>
cudaError_t occupancy_t(bool mass, int* blocks) {
  return mass ? occupancy_m<WARPS, RPT, TILE, kMass, MINB>(blocks)
              : occupancy_m<WARPS, RPT, TILE, kUnitMass, MINB>(blocks);
}

}  // namespace

namespace rsint {

cudaError_t shoot_blocks_per_sm(int cfg, bool mass, int* blocks) {
  switch (cfg) {
#define RS_CASE(i, w, r, t, m) \
  case i:                       \
    return occupancy_t<w, r, t, m>(mass, blocks);
    RS_LAUNCH_SHAPES(RS_CASE)
#undef RS_CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_shoot(int cfg, const rsdev::ShootDesc& d, cudaStream_t s) {
  if (d.f.has_mass == rsdev::kWideMass) {  // built for the default shape only
    const int64_t grid = rsdev::shoot_tiles<kWideWarps, kWideRpt>(d.n_rows, d.n0);
    if (grid <= 0) return cudaSuccess;
    if (grid >= ((int64_t)1 << 31)) return cudaErrorInvalidValue;
    return launch_shoot_m<kWideWarps, kWideRpt, kWideTile, rsdev::kWideMass, 2>(d, grid, s);
  }
  switch (cfg) {
#define RS_CASE(i, w, r, t, m) \
  case i:                       \
    return launch_shoot_t<w, r, t, m>(d, s);
    RS_LAUNCH_SHAPES(RS_CASE)
#undef RS_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace rsint
