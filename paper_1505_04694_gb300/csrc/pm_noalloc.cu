// pm_quality_arrays_noalloc_dev: the quality sum and its gradient on plain
// device arrays (same computation as pm_quality_arrays_dev) without any
// device allocation during the call.
//
// Some callers cannot allocate device memory when they call in: a framework
// that has already reserved the device's memory for its own caching
// allocator, a latency-bound loop that cannot afford an allocation (or the
// synchronisation one may imply), or a program that forbids allocation after
// start-up.  For them every temporary lives in one fixed array compiled into
// this library (kScratchBytes below, about 6.5 MB): each GPU that loads the
// library keeps it until the process exits.  The sizes it admits are
// kMaxElements elements and kMaxVertices vertices; larger inputs are refused.
//
// All calls share the array and it keeps the last call's contents, so the
// parts that must start at zero are cleared by each call.  Two calls that
// overlap on the GPU (for example on two streams) race on the array; order
// them on one stream or synchronise between them.
#include <mutex>

#include "pm_internal.cuh"

namespace pm {

namespace {

constexpr int kMaxElements = 65536;
constexpr int kMaxVertices = 65536;
// byte offsets inside the array (each a multiple of 256)
constexpr size_t round256(size_t x) { return (x + 255) & ~size_t(255); }
constexpr size_t kScanTiles = (kMaxVertices + 1 + 2047) / 2048;
constexpr size_t kOffHead = 0;  // head and scan state first: cleared together
constexpr size_t kOffScan = round256(kOffHead + sizeof(QHead));
constexpr size_t kOffCnt = round256(kOffScan + sizeof(unsigned long long) * kScanTiles);
constexpr size_t kOffGrad = round256(kOffCnt + sizeof(int) * 2 * (kMaxVertices + 1));
constexpr size_t kOffPart = round256(kOffGrad + sizeof(EGrad) * kMaxElements);
constexpr size_t kOffOff = round256(kOffPart + sizeof(double) * kQualityBlocks);
constexpr size_t kOffCol = round256(kOffOff + sizeof(int) * (kMaxVertices + 1));
constexpr size_t kOffPos = round256(kOffCol + sizeof(int) * 3 * kMaxElements);
constexpr size_t kScratchBytes = round256(kOffPos + 3 * kMaxElements);

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

// Host side: the array's device address, looked up once per device.
std::mutex g_mu;
unsigned char* g_base[64];

}  // namespace

}  // namespace pm

using namespace pm;

extern "C" pm_status pm_quality_arrays_noalloc_dev(const double* xy, const double* M, int32_t nv,
                                                   const int32_t* tri, int32_t ne, double* q_sum,
                                                   double* dxy, double* dm, void* stream) {
  if (!xy || !M || (!tri && ne > 0) || !q_sum || nv < 1 || ne < 0) {
    set_last_error("need xy, m, tri, q_sum, nv >= 1, ne >= 0");
    return PM_ERR_INVALID_ARG;
  }
  if (ne > kMaxElements || nv > kMaxVertices) {
    set_last_error("pm_quality_arrays_noalloc_dev handles at most 65536 elements and 65536 "
                   "vertices; use pm_quality_arrays_dev for larger meshes");
    return PM_ERR_CAPACITY;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    set_last_error("no current CUDA device");
    return PM_ERR_CUDA;
  }
  unsigned char* base = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_base[dev]) {
      // one-time set-up on this device (the device is current here)
      void* p = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
      if (e != cudaSuccess || !p) {
        set_last_error(std::string("locating the scratch array: ") + cudaGetErrorString(e));
        return PM_ERR_CUDA;
      }
      g_base[dev] = (unsigned char*)p;
    }
    base = g_base[dev];
  }
  cudaStream_t s = (cudaStream_t)stream;
  QualityWork w;
  w.head = (QHead*)(base + kOffHead);
  w.state = (unsigned long long*)(base + kOffScan);
  w.cnt = (int*)(base + kOffCnt);
  w.eg = (EGrad*)(base + kOffGrad);
  w.part = (double*)(base + kOffPart);
  w.off = (int*)(base + kOffOff);
  w.col = (int*)(base + kOffCol);
  w.pos = (uint8_t*)(base + kOffPos);
  const DevStatus* st = &w.head->st;
  // head, scan state and the counters of nv vertices are adjacent
  cudaError_t e = cudaMemsetAsync(base, 0, kOffCnt + sizeof(int) * 2 * ((size_t)nv + 1), s);
  if (e == cudaSuccess) e = quality_launch(w, xy, M, nv, tri, ne, q_sum, dxy, dm, nullptr, s);
  // the status word of this call (a copy into pageable host memory returns
  // once the stream has reached it)
  DevStatus h{};
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, st, sizeof(DevStatus), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    set_last_error(std::string("CUDA: ") + cudaGetErrorString(e));
    return PM_ERR_CUDA;
  }
  if (h.err == PM_ERR_INVALID_MESH) set_last_error("vertex id outside [0, nv) in tri");
  if (h.err == PM_ERR_TIMEOUT) set_last_error("the gradient's scan gave up waiting");
  return (pm_status)h.err;
}
