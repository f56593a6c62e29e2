// gs_small_inst.cu -- the small-grid kernels (gs_small.cuh) for every grid of
// power-of-two sides 32 ... 256 with at most kSmallMaxPixels pixels, and their
// host-side launch.
#include "gs_small.cuh"

namespace gsk {

namespace {

struct SmallEntry {
  const void* fn;
  int (*smem)(int lc);
  int (*lanes)(int lc);
};

template <int LX, int LY>
SmallEntry entry() {
  using Gm = SmallGeom<LX, LY>;
  return {reinterpret_cast<const void*>(&gs_small<LX, LY>), [](int lc) { return Gm::smem(lc); },
          [](int lc) { return Gm::lanes(lc); }};
}

int log2_of(int n) {
  int l = 0;
  while ((1 << l) < n) ++l;
  return l;
}

bool lookup(int nx, int ny, SmallEntry* e) {
  if (!small_grid(nx, ny)) return false;
  switch (log2_of(nx) * 16 + log2_of(ny)) {
    case 5 * 16 + 5: *e = entry<5, 5>(); return true;
    case 5 * 16 + 6: *e = entry<5, 6>(); return true;
    case 5 * 16 + 7: *e = entry<5, 7>(); return true;
    case 5 * 16 + 8: *e = entry<5, 8>(); return true;
    case 6 * 16 + 5: *e = entry<6, 5>(); return true;
    case 6 * 16 + 6: *e = entry<6, 6>(); return true;
    case 6 * 16 + 7: *e = entry<6, 7>(); return true;
    case 6 * 16 + 8: *e = entry<6, 8>(); return true;
    case 7 * 16 + 5: *e = entry<7, 5>(); return true;
    case 7 * 16 + 6: *e = entry<7, 6>(); return true;
    case 7 * 16 + 7: *e = entry<7, 7>(); return true;
    case 7 * 16 + 8: *e = entry<7, 8>(); return true;
    case 8 * 16 + 5: *e = entry<8, 5>(); return true;
    case 8 * 16 + 6: *e = entry<8, 6>(); return true;
    case 8 * 16 + 7: *e = entry<8, 7>(); return true;
    default: return false;
  }
}

cudaLaunchConfig_t config(const SmallEntry& e, int batch, int lc, cudaLaunchAttribute* attr, cudaStream_t s) {
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = 1u << lc;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(batch) << lc);
  cfg.blockDim = dim3(4 * e.lanes(lc));
  cfg.dynamicSmemBytes = e.smem(lc);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

}  // namespace

cudaError_t small_prepare(int nx, int ny, int clusters[kSmallMaxLogC + 1]) {
  for (int lc = 0; lc <= kSmallMaxLogC; ++lc) clusters[lc] = 0;
  SmallEntry e;
  if (!lookup(nx, ny, &e)) return cudaErrorInvalidValue;
  const int lo = small_min_logc(nx, ny), hi = small_max_logc(nx, ny);
  cudaError_t rc = cudaFuncSetAttribute(e.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, e.smem(lo));
  for (int lc = lo; lc <= hi && rc == cudaSuccess; ++lc) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = config(e, 1, lc, &attr, nullptr);
    rc = cudaOccupancyMaxActiveClusters(&clusters[lc], e.fn, &cfg);
  }
  return rc;
}

cudaError_t launch_small(const Params& p, cudaStream_t s) {
  SmallEntry e;
  if (!lookup(p.nx, p.ny, &e)) return cudaErrorInvalidValue;
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg = config(e, p.batch, p.small_logc, &attr, s);
  void* args[] = {const_cast<Params*>(&p)};
  return cudaLaunchKernelExC(&cfg, e.fn, args);
}

}  // namespace gsk
