// Element quality functional (Sec. 2.2, Vasilevskii et al.) summed over a
// mesh, and its gradient with respect to vertex coordinates and metric
// entries (hand-written reverse mode, see quality_grad_c).
//
// Two passes: one thread per element writes q and the 15 partial derivatives
// of its three vertices; one thread per vertex then sums its elements'
// contributions in ascending element id, so the result does not depend on
// thread timing.  The sum of q is a fixed-shape two-level reduction.
//
// The FP64 pipe bounds both element passes (85% active at 4M elements, DRAM 4%).
// Forward and backward on 2.1M elements took 2.87 ms with a gradient evaluated in
// both, a corner list built by a pass of its own and pageable status copies; 2.16 ms
// as it is (418 -> 357 us on 6.8k elements, most of it launches and the two waits).
#include <algorithm>

#include "pm_internal.cuh"

namespace pm {

namespace {

constexpr int RED_BLOCKS = 256;
constexpr int RED_THREADS = 256;

__device__ __forceinline__ EGrad pack_grad(const double g[3][5]) {
  EGrad out;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    out.xy[2 * k] = g[k][0];
    out.xy[2 * k + 1] = g[k][1];
    out.m[k] = g[0][2 + k];
  }
  return out;
}

// acc += the derivatives of corner i of an element
__device__ __forceinline__ void add_corner(double acc[5], const EGrad& e, int i) {
  acc[0] = acc[0] + e.xy[2 * i];
  acc[1] = acc[1] + e.xy[2 * i + 1];
  acc[2] = acc[2] + e.m[0];
  acc[3] = acc[3] + e.m[1];
  acc[4] = acc[4] + e.m[2];
}

__global__ void k_elem_qgrad_store(Store S, int mesh, double* qel, EGrad* eg) {
  int vb = S.tab.vbase[mesh], eb = S.tab.ebase[mesh], ne = S.tab.ne[mesh];
  for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < ne; l += gridDim.x * blockDim.x) {
    int4 e = S.EN[eb + l];
    if (!e.w) {
      qel[l] = 0.0;
      continue;
    }
    const VD a = load_vd(S, vb + e.x), b = load_vd(S, vb + e.y), c = load_vd(S, vb + e.z);
    if (!eg) {
      qel[l] = quality_c(e.x, e.y, e.z, a, b, c);
      continue;
    }
    double g[3][5];
    qel[l] = quality_grad_c(e.x, e.y, e.z, a, b, c, g);
    eg[l] = pack_grad(g);
  }
}

__global__ void k_vgather_store(Store S, int mesh, const EGrad* eg, double* dxy, double* dm) {
  int vb = S.tab.vbase[mesh], eb = S.tab.ebase[mesh], nv = S.tab.nv[mesh];
  for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < nv; l += gridDim.x * blockDim.x) {
    int s = vb + l;
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (S.vflag[s] & VF_ALIVE) {
      const int* ne = S.NE + (size_t)s * S.W;
      int nel = S.NElen[s];
      for (int k = 0; k < nel; ++k) {
        int K = ne[k];
        int4 e = S.EN[eb + K];
        int i = (e.x == l) ? 0 : (e.y == l) ? 1 : 2;
        add_corner(acc, eg[K], i);
      }
    }
    if (dxy) {
      dxy[2 * l] = acc[0];
      dxy[2 * l + 1] = acc[1];
    }
    if (dm) {
      dm[3 * l] = acc[2];
      dm[3 * l + 1] = acc[3];
      dm[3 * l + 2] = acc[4];
    }
  }
}

// ---- arrays (no mesh handle) ----------------------------------------------------

__device__ __forceinline__ VD arr_vd(const double* xy, const double* m, int v) {
  return VD{xy[2 * v], xy[2 * v + 1], m[3 * v], m[3 * v + 1], m[3 * v + 2]};
}

// Sum over the block in a fixed order (blockDim.x: a power of two of at most
// RED_THREADS); thread 0 gets it.
__device__ __forceinline__ double block_sum(double x) {
  __shared__ double sh[RED_THREADS];
  sh[threadIdx.x] = x;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] = sh[threadIdx.x] + sh[threadIdx.x + o];
    __syncthreads();
  }
  const double r = sh[0];
  __syncthreads();
  return r;
}

// Quality (and, with GRAD, the derivatives) of every element, and the sum over
// all of them: block b sums elements b T + t, b T + t + G T, ... (T threads, G
// blocks), the last block to finish adds the blocks' sums; the shape of the sum
// depends on the element count alone.  With GRAD each corner also takes its
// place in its vertex's list (`pos`), under the FP64 work that bounds this
// kernel; without it only the quality itself is evaluated (77 operations instead
// of about 230).  An element with a vertex id outside [0, nv) records
// PM_ERR_INVALID_MESH and contributes NaN (nothing is read through a bad id).
// The status goes to `out_st` (pinned host memory) with the sum.
constexpr int QT = 128;
template <bool GRAD>
__global__ void __launch_bounds__(QT)
k_elem_quality_arr(const double* xy, const double* m, const int* tri, int ne, int nv, EGrad* eg,
                   int* cnt, uint8_t* pos, double* part, double* qsum, QHead* head,
                   DevStatus* out_st) {
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  double sum = 0.0;
  for (int K = blockIdx.x * QT + threadIdx.x; K < ne; K += gridDim.x * QT) {
    const int t[3] = {tri[3 * K], tri[3 * K + 1], tri[3 * K + 2]};
    if ((unsigned)t[0] >= (unsigned)nv || (unsigned)t[1] >= (unsigned)nv ||
        (unsigned)t[2] >= (unsigned)nv) {
      set_err(&head->st, PM_ERR_INVALID_MESH);
      sum = sum + nan;
      continue;
    }
    const VD a = arr_vd(xy, m, t[0]), b = arr_vd(xy, m, t[1]), c = arr_vd(xy, m, t[2]);
    if (GRAD) {
      // (a vertex in more than 255 elements marks its later corners 255: the
      // fill pass then takes places from the counter)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const int p = atomicAdd(cnt + t[i], 1);
        pos[3 * (size_t)K + i] = (uint8_t)(p < 255 ? p : 255);
      }
      double g[3][5];
      sum = sum + quality_grad_c(t[0], t[1], t[2], a, b, c, g);
      eg[K] = pack_grad(g);
    } else {
      sum = sum + quality_c(t[0], t[1], t[2], a, b, c);
    }
  }
  const double bs = block_sum(sum);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    part[blockIdx.x] = bs;
    __threadfence();
    last = atomicAdd(&head->done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double s = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += QT) s = s + __ldcg(part + i);
  s = block_sum(s);
  if (threadIdx.x == 0) {
    *qsum = s;
    if (out_st) {
      DevStatus r = head->st;
      r.err = atomicAdd(&head->st.err, 0);
      *out_st = r;
    }
  }
}

// Corner list per vertex: entry = 3 * element + corner position; nothing is
// written after a device error (the offsets may be unwritten) and no entry
// leaves its vertex's range.  `more` counts the corners beyond a vertex's 255th.
__global__ void k_corner_fill(const int* tri, int ne, int nv, const int* off, const uint8_t* pos,
                              int* more, int* col, const DevStatus* st) {
  if (st->err) return;
  for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < ne; K += gridDim.x * blockDim.x) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int v = tri[3 * K + i];
      if ((unsigned)v >= (unsigned)nv) continue;
      int p = pos[3 * (size_t)K + i];
      if (p == 255) p += atomicAdd(more + v, 1);
      if (off[v] + p < off[v + 1]) col[off[v] + p] = 3 * K + i;
    }
  }
}

// Per vertex: its corners in ascending element id, contributions summed in
// that order.  After a device error every output entry is NaN.  Up to 12
// corners are sorted in registers (rank by comparison, all loads in flight);
// more are sorted in place.  The status goes to `out_st` (pinned host memory).
constexpr int kCornerFast = 12;
__global__ void k_vgather_arr(const int* off, int* col, const EGrad* eg, int nv, double* dxy,
                              double* dm, const DevStatus* st, DevStatus* out_st) {
  const bool bad = st->err != 0;
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  if (out_st && blockIdx.x == 0 && threadIdx.x == 0) *out_st = *st;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x) {
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (bad) {
#pragma unroll
      for (int j = 0; j < 5; ++j) acc[j] = nan;
    } else {
      const int a = off[v], b = off[v + 1];
      if (b - a <= kCornerFast) {
        int x[kCornerFast], o[kCornerFast];
#pragma unroll
        for (int k = 0; k < kCornerFast; ++k) {
          x[k] = a + k < b ? col[a + k] : 0x7fffffff;
          o[k] = 0x7fffffff;
        }
        // insertion through a minimum-maximum network keeps o sorted
#pragma unroll
        for (int k = 0; k < kCornerFast; ++k) {
#pragma unroll
          for (int j = kCornerFast - 1; j > 0; --j) o[j] = max(o[j - 1], min(o[j], x[k]));
          o[0] = min(o[0], x[k]);
        }
#pragma unroll
        for (int k = 0; k < kCornerFast; ++k)
          if (a + k < b) add_corner(acc, eg[o[k] / 3], o[k] % 3);
      } else {
        for (int k = a + 1; k < b; ++k) {  // ascending element id
          int x = col[k];
          int j = k - 1;
          while (j >= a && col[j] > x) {
            col[j + 1] = col[j];
            --j;
          }
          col[j + 1] = x;
        }
        for (int k = a; k < b; ++k) add_corner(acc, eg[col[k] / 3], col[k] % 3);
      }
    }
    if (dxy) {
      dxy[2 * v] = acc[0];
      dxy[2 * v + 1] = acc[1];
    }
    if (dm) {
      dm[3 * v] = acc[2];
      dm[3 * v + 1] = acc[3];
      dm[3 * v + 2] = acc[4];
    }
  }
}

// ---- deterministic sum -------------------------------------------------------------

__global__ void k_sum_stage1(const double* x, int n, double* part) {
  __shared__ double sh[RED_THREADS];
  long long chunk = ((long long)n + gridDim.x - 1) / gridDim.x;
  long long a = chunk * blockIdx.x, b = a + chunk < n ? a + chunk : n;
  double s = 0.0;
  for (long long i = a + threadIdx.x; i < b; i += blockDim.x) s = s + x[i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] = sh[threadIdx.x] + sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void k_sum_stage2(const double* part, int n, double* out) {
  __shared__ double sh[RED_BLOCKS];
  sh[threadIdx.x] = threadIdx.x < n ? part[threadIdx.x] : 0.0;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] = sh[threadIdx.x] + sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

void dsum(const double* x, int n, double* part, double* out, cudaStream_t s) {
  PM_LAUNCH(k_sum_stage1, RED_BLOCKS, RED_THREADS, 0, s, x, n, part);
  PM_LAUNCH(k_sum_stage2, 1, RED_BLOCKS, 0, s, part, RED_BLOCKS, out);
}

int gridn(long long n) {
  long long g = (n + 127) / 128;
  return (int)std::max<long long>(1, std::min<long long>(g, 152 * 16));
}

}  // namespace

// Quality sum and gradient of mesh 0 of the set, written to host arrays
// indexed by vertex slot (dxy[2*nv], dm[3*nv]; each may be null).
int quality_mesh(MeshSet& m, double* qsum_host, double* dxy_host, double* dm_host) {
  cudaStream_t s = m.stream;
  int ne = m.ne[0], nv = m.nv[0];
  bool grad = dxy_host || dm_host;
  double *qel = nullptr, *part = nullptr, *out = nullptr, *dxy = nullptr, *dm = nullptr;
  EGrad* eg = nullptr;
  cudaError_t e = device_alloc(&qel, std::max(ne, 1) * sizeof(double), s);
  if (!e) e = device_alloc(&part, (RED_BLOCKS + 1) * sizeof(double), s);
  if (!e && grad) e = device_alloc(&eg, std::max(ne, 1) * sizeof(EGrad), s);
  if (!e && grad) e = device_alloc(&dxy, std::max(nv, 1) * 2 * sizeof(double), s);
  if (!e && grad) e = device_alloc(&dm, std::max(nv, 1) * 3 * sizeof(double), s);
  int status = PM_OK;
  if (e) {
    set_last_error(std::string("quality workspace: ") + cudaGetErrorString(e));
    status = PM_ERR_OOM;
  } else {
    out = part + RED_BLOCKS;
    PM_LAUNCH(k_elem_qgrad_store, gridn(ne), 128, 0, s, m.S, 0, qel, eg);
    dsum(qel, ne, part, out, s);
    if (grad) PM_LAUNCH(k_vgather_store, gridn(nv), 128, 0, s, m.S, 0, eg, dxy, dm);
    cudaMemcpyAsync(qsum_host, out, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (dxy_host)
      cudaMemcpyAsync(dxy_host, dxy, nv * 2 * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (dm_host) cudaMemcpyAsync(dm_host, dm, nv * 3 * sizeof(double), cudaMemcpyDeviceToHost, s);
  }
  for (void* p : {(void*)qel, (void*)part, (void*)eg, (void*)dxy, (void*)dm})
    if (p) cudaFreeAsync(p, s);
  int err = sync_status(m);
  return status ? status : err;
}

// Blocks of the element pass: 8 of 128 threads on each of the 152 SMs hide the
// latency of the FP64 chains; the shape of the sum follows from the block count.
int quality_blocks(int ne) {
  return (int)std::max<long long>(1, std::min<long long>((ne + QT - 1LL) / QT, kQualityBlocks));
}

// The kernels of one call on a workspace whose head, counters and scan state
// the caller has cleared.
cudaError_t quality_launch(const QualityWork& w, const double* xy, const double* mt, int nv,
                           const int* tri, int ne, double* qsum, double* dxy, double* dm,
                           DevStatus* out_st, cudaStream_t s) {
  const int blocks = quality_blocks(ne);
  if (!dxy && !dm) {
    PM_LAUNCH(k_elem_quality_arr<false>, blocks, QT, 0, s, xy, mt, tri, ne, nv, w.eg, w.cnt, w.pos,
              w.part, qsum, w.head, out_st);
    return cudaGetLastError();
  }
  PM_LAUNCH(k_elem_quality_arr<true>, blocks, QT, 0, s, xy, mt, tri, ne, nv, w.eg, w.cnt, w.pos,
            w.part, qsum, w.head, (DevStatus*)nullptr);
  ScanWork sw;
  sw.state = w.state;
  sw.ticket = &w.head->ticket;
  sw.tiles_cap = scan_tiles(nv + 1);
  scan_exclusive(w.cnt, w.off, nv, sw, &w.head->st, s);
  PM_LAUNCH(k_corner_fill, gridn(ne), 128, 0, s, tri, ne, nv, (const int*)w.off,
            (const uint8_t*)w.pos, w.cnt + (nv + 1), w.col, (const DevStatus*)&w.head->st);
  PM_LAUNCH(k_vgather_arr, gridn(nv), 128, 0, s, (const int*)w.off, w.col, (const EGrad*)w.eg, nv,
            dxy, dm, (const DevStatus*)&w.head->st, out_st);
  return cudaGetLastError();
}

// Quality sum (and gradient) on plain device arrays.  Temporaries come from
// one stream-ordered allocation, of which one memset clears the part that starts
// at zero; the kernels write the status straight into pinned host memory (a copy
// into pageable memory cost 30 us a call); the call waits for its stream and
// returns it (PM_ERR_INVALID_MESH for a vertex id outside [0, nv),
// PM_ERR_TIMEOUT when the scan's bounded wait gave up; the outputs then hold
// NaN).
int quality_arrays(const double* xy, const double* mt, int nv, const int* tri, int ne,
                   double* qsum, double* dxy, double* dm, cudaStream_t s) {
  const bool grad = dxy || dm;
  const int tiles = scan_tiles(nv + 1), blocks = quality_blocks(ne);
  auto r256 = [](size_t x) { return (x + 255) & ~size_t(255); };
  const size_t b_head = r256(sizeof(QHead));
  const size_t b_cnt = grad ? r256(2 * ((size_t)nv + 1) * sizeof(int)) : 0;
  const size_t b_state = grad ? r256((size_t)tiles * sizeof(unsigned long long)) : 0;
  const size_t b_part = r256(blocks * sizeof(double));
  const size_t b_eg = grad ? r256(std::max(ne, 1) * sizeof(EGrad)) : 0;
  const size_t b_off = grad ? r256(((size_t)nv + 1) * sizeof(int)) : 0;
  const size_t b_col = grad ? r256(std::max(3LL * ne, 1LL) * sizeof(int)) : 0;
  const size_t b_pos = grad ? r256(std::max(3LL * ne, 1LL)) : 0;
  DevStatus* h = (DevStatus*)pinned_slot();
  if (!h) {
    set_last_error("pinned status word");
    return PM_ERR_OOM;
  }
  h->err = PM_ERR_CUDA;  // overwritten by the last kernel
  char* base = nullptr;
  cudaError_t e = device_alloc(&base, b_head + b_cnt + b_state + b_part + b_eg + b_off +
                                                     b_col + b_pos, s);
  if (e != cudaSuccess) {
    set_last_error(std::string("quality workspace: ") + cudaGetErrorString(e));
    pinned_slot_free(h);
    return e == cudaErrorMemoryAllocation ? PM_ERR_OOM : PM_ERR_CUDA;
  }
  char* p = base;
  QualityWork w;
  w.head = (QHead*)p; p += b_head;
  w.cnt = (int*)p; p += b_cnt;
  w.state = (unsigned long long*)p; p += b_state;
  w.part = (double*)p; p += b_part;
  w.eg = (EGrad*)p; p += b_eg;
  w.off = (int*)p; p += b_off;
  w.col = (int*)p; p += b_col;
  w.pos = (uint8_t*)p;
  e = cudaMemsetAsync(base, 0, b_head + b_cnt + b_state, s);
  if (!e) e = quality_launch(w, xy, mt, nv, tri, ne, qsum, dxy, dm, h, s);
  cudaFreeAsync(base, s);
  // (waits also after an error: the status slot goes back)
  const cudaError_t es = cudaStreamSynchronize(s);
  if (!e) e = es;
  const int err = h->err;
  pinned_slot_free(h);
  if (e != cudaSuccess) {
    set_last_error(std::string("CUDA: ") + cudaGetErrorString(e));
    return PM_ERR_CUDA;
  }
  if (err == PM_ERR_INVALID_MESH) set_last_error("vertex id outside [0, nv) in tri");
  if (err == PM_ERR_TIMEOUT) set_last_error("the gradient's scan gave up waiting");
  return err;
}

}  // namespace pm
