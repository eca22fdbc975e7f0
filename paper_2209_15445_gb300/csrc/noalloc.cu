// adept_build_tables_noalloc: the physics-table build for callers that cannot allocate
// device memory. The kernels of adept_build_tables' rows (tables.cuh), with their working rows
// in a file-scope __device__ array instead of a caller-provided arena.
#include <cuda_runtime.h>

#include <mutex>

#include "../../include/adept.h"
#include "device.cuh"
#include "layout.h"
#include "tables.cuh"

namespace adept {
namespace {

constexpr int kRows = V_NROW + B_NROW;
constexpr int kNoAllocMat = ADEPT_NOALLOC_MAX_MATERIALS;

// Working rows (kNoAllocMat x 17 x 289 doubles) and material constants of every call, 158 KB on
// every device that loads the library (held until exit). Calls share it; each call writes every
// word it reads before reading it, so nothing needs clearing, but calls that overlap on the GPU
// race on it.
struct Scratch {
  double rows[kNoAllocMat * kRows * kNNode];
  MatDev mats[kNoAllocMat];
};
static __device__ __align__(256) Scratch g_noalloc_scratch;

struct MatIn {
  double v[kNoAllocMat][kMatRec];  // material records (elements only), passed by value
  __device__ const double* record(int m) const { return v[m]; }
};

std::mutex g_mu;
Scratch* g_ptr[256] = {};

}  // namespace
}  // namespace adept

using namespace adept;

extern "C" int adept_build_tables_noalloc(const adept_material* materials, int32_t n_materials, double range_cut_mm,
                                          double* dev_tables, double* dev_cuts, void* stream) {
  if (!materials || !dev_tables || !dev_cuts) return ADEPT_EINVAL;
  if (n_materials < 1 || n_materials > kNoAllocMat) return ADEPT_EINVAL;  // beyond the static scratch
  if (!(range_cut_mm > 0.0)) return ADEPT_EINVAL;
  MatIn in{};
  for (int m = 0; m < n_materials; ++m) {
    const adept_material& t = materials[m];
    if (t.n_elements != 0) return ADEPT_EINVAL;  // single elements only
    if (t.Z < 0 || t.Z > 100 || (t.Z > 0 && !(t.A_g_mol > 0 && t.density_g_cm3 > 0 && t.I_eV > 0))) return ADEPT_EINVAL;
    in.v[m][0] = t.Z; in.v[m][1] = t.A_g_mol; in.v[m][2] = t.density_g_cm3; in.v[m][3] = t.I_eV; in.v[m][4] = 0.0;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return ADEPT_ECUDA;
  // held until the last of the call's four launches is queued: between two of them no call of
  // another thread on the same stream may queue its own, which write the same scratch
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_ptr[dev]) {
    // the array's device address, once per device with that device current; host code
    // cannot use the symbol itself (it names a host-side stand-in)
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return ADEPT_ECUDA;
    g_ptr[dev] = static_cast<Scratch*>(p);
  }
  Scratch* const scratch = g_ptr[dev];
  const TableRows r{scratch->rows, (size_t)kRows * kNNode, scratch->rows + V_NROW * kNNode, (size_t)kRows * kNNode,
                    dev_cuts, dev_cuts + 1, 2, dev_tables};
  return launch_table_rows(in, n_materials, range_cut_mm, scratch->mats, r, static_cast<cudaStream_t>(stream)) == cudaSuccess
             ? ADEPT_OK : ADEPT_ECUDA;
}
