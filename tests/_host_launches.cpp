// The host side of the chi launches on a machine without a GPU: the launch code
// linked against a CUDA runtime that only records.  Devices have 152 SMs; a
// kernel's occupancy is what its shared memory and its launch bounds allow.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

#include <cuda_runtime.h>
template <class T>
T atomicAdd(T* p, T x);  // named by an inline device function
#include "chi_lane.h"

namespace {

std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> m;
  return m;
}
bool record = false;  // print and count launches
uint32_t launched = 0;

// The template arguments of a sum-tree kernel.
bool lane_args(const std::string& n, int a[5]) {
  const size_t at = n.find("k_chi_laneI");
  return at != std::string::npos &&
         std::sscanf(n.c_str() + at, "k_chi_laneILi%dELi%dELi%dELi%dELi%dE", a, a + 1, a + 2, a + 3,
                     a + 4) == 5;
}

}  // namespace

extern "C" {
void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*,
                            dim3*, dim3*, int*) {
  names()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* k,
                                                                   int threads, size_t smem,
                                                                   unsigned) {
  int a[5];
  int by_regs = 2048 / threads / 4;
  if (lane_args(names()[k], a))
    by_regs = a[4] ? a[4] : a[2] == tsg::kLeafShared ? 12 : a[3] > 1 ? 14 : a[1] == 5 ? 4 : 7;
  const int by_smem = static_cast<int>(228 * 1024 / (smem + 1024));
  *n = by_regs < by_smem ? by_regs : by_smem;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* k, void**) {
  if (!record) return cudaSuccess;
  ++launched;
  int early = 0, priority = 0;
  for (unsigned i = 0; i < c->numAttrs; ++i) {
    if (c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization)
      early = c->attrs[i].val.programmaticStreamSerializationAllowed;
    if (c->attrs[i].id == cudaLaunchAttributePriority) priority = c->attrs[i].val.priority;
  }
  const std::string& n = names()[k];
  std::printf("%s early %d priority %d\n",
              n.find("k_chi_lane") != std::string::npos ? "tree" : "segmented", early, priority);
  return cudaSuccess;
}
}

// The launches of one chi phase whose cells are packed, so that there is a pass
// over those past the packed range; then one without.
static int launches(int priority, bool early) {
  record = true;
  for (const uint32_t cells : {30u * 152u, 152u}) {
    const tsg::LanePlan pl = tsg::lane_plan(1024, cells, 0);
    if (pl.G == 0 || (pl.leaf == tsg::kLeafShared) != (cells == 152u)) return 1;
    launched = 0;
    if (tsg::launch_chi_lane(pl, 0, nullptr, nullptr, cells, nullptr, nullptr,
                             tsg::ChiRedo{nullptr, nullptr}, 1024, 32, 0, 0.1, nullptr, priority,
                             early) != cudaSuccess ||
        launched != tsg::lane_info(pl).launches)
      return 1;
  }
  return 0;
}

// Every class a batch may hold, behind up to a chip full of other warps: the
// plans that have no kernel, and those whose blocks do not hold all cells.
static int plans() {
  for (uint32_t n = 2; n <= 32; ++n)
    for (int model = 0; model < 3; ++model)
      for (uint64_t cells = 1; cells < 200000; cells += 1 + cells / 4)
        for (uint64_t beside : {0, 100, 152 * 5, 152 * 6, 152 * 7, 152 * 8 - 1, 152 * 8, 152 * 16, 40000}) {
          const tsg::LanePlan pl = tsg::lane_plan(n * n, cells, model, beside);
          if (pl.G == 0 || pl.blocks == 0 || pl.smem > tsg::kMaxSmem)
            std::printf("V %u model %d cells %llu beside %llu: G %u\n", n * n, model,
                        (unsigned long long)cells, (unsigned long long)beside, pl.G);
        }
  return 0;
}

int main(int argc, char** argv) {
  if (argc == 2 && !std::strcmp(argv[1], "plans")) return plans();
  if (argc == 4 && !std::strcmp(argv[1], "launches"))
    return launches(std::atoi(argv[2]), std::atoi(argv[3]) != 0);
  return 2;
}
