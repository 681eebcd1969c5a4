// Host-side structures of the library (one translation unit per subsystem
// shares these declarations).
#pragma once

#include <cuda_runtime.h>

#include <string>
#include <vector>

#include "pm_common.cuh"

namespace pm {

constexpr int MAXW = 128;         // largest supported adjacency row (a vertex's degree)
constexpr int BLOCK = 128;        // threads per block of the round kernels

struct ScanWork {
  unsigned long long* state = nullptr;  // one word per tile
  int* ticket = nullptr;
  unsigned epoch = 0;
  int tiles_cap = 0;
};

int scan_tiles(int n);
void scan_exclusive(const int* in, int* out, int n, ScanWork& w, DevStatus* st, cudaStream_t s,
                    const int* go = nullptr);
void scan_alive_vertices(const Store& S, int* out, int n, ScanWork& w, DevStatus* st,
                         cudaStream_t s);
void scan_alive_elements(const Store& S, int* out, int n, ScanWork& w, DevStatus* st,
                         cudaStream_t s);

// Per-round worklists and marks (slot-indexed scratch, sized with the store).
struct Work {
  int* D[2] = {nullptr, nullptr};  // dirty / pending lists (ping-pong)
  int* C = nullptr;                // candidates
  int* Sl = nullptr;               // independent set
  int* A = nullptr;                // vertices whose rows change (commit owners)
  int* P = nullptr;                // next-sweep list (smoothing)
  int* target = nullptr;           // collapse target (local id) per vertex
  int4* opA = nullptr;             // flip record (w, c, d, K1) per vertex
  int* opK2 = nullptr;
  double2* mvxy = nullptr;         // smoothing move per vertex (shares its place with items)
  double4* mvM = nullptr;
  int* dmark = nullptr;            // per-round stamps
  int* amark = nullptr;
  int* cmark = nullptr;
  int* smark = nullptr;
  int* pmark = nullptr;
  int* vcnt = nullptr;             // per-vertex counts (refine / renumber), vslots + 1
  int* vscan = nullptr;            // vslots + 1
  RowMask* vmask = nullptr;        // refine: marked NN entries
  int* ecnt = nullptr;             // per-element counts, eslots + 1
  int* escan = nullptr;
  int4* emid = nullptr;            // refine: midpoint ids per element edge
  int* elist = nullptr;            // refine: elements split this round, eslots
  int* clist = nullptr;            // refine: their children's slots, eslots
  int* E = nullptr;                // vertices evaluated in full this round
  int2* items = nullptr;           // flip candidates (vertex, edge slots) of this round
  double* gains = nullptr;         // gain of each (vertex, ball-element slot), vslots * W (in the
                                   // spare rows)
  int* cand = nullptr;             // collapse candidates of each vertex (see kCandRest), vslots * W
  int* counts = nullptr;           // device counters (see CountIdx)
  int* cprop = nullptr;            // colouring: proposed colour per vertex slot
  int* cstamp = nullptr;           // colouring: round in which the slot was uncoloured
};

// The per-round counters sit between the two dirty-list counts so that one
// memset clears them together with the next round's list (zero_round).
enum CountIdx {
  CN_D0 = 0, CN_C = 1, CN_S = 2, CN_A = 3, CN_E = 4, CN_I = 5, CN_D1 = 7,
  CN_P = 8, CN_EL = 9, CN_CL = 10, CN_DONE = 11,
  CN_RES = 12,  // persistent rounds: rounds run, list index after, pass complete; smoothing:
                // see SmoothRes (8)
  CN_BAR = 20,  // persistent rounds: grid barrier arrivals
  CN_C2 = 21,   // persistent rounds: candidates of odd rounds
  CN_RENUM = 22,  // renumbering: 1 when some mesh's compaction is not the identity
  CN_NUM = 23
};
// Words per mesh after the counters: live counts (vertices, elements; two per
// mesh), the new vertices of a refinement round, the sizes after it.
constexpr int kMeshWords = 5;
constexpr int cn_newv(int n) { return CN_NUM + 2 * n; }
constexpr int cn_sizes(int n) { return CN_NUM + 3 * n; }
// A second set of counters behind them, for flips queued behind collapses.
constexpr int cn_second(int n) { return CN_NUM + kMeshWords * n; }
// What a persistent smoothing launch leaves at CN_RES: rounds with candidates,
// sweeps finished, 1 when the sweeps are over, 1 when the current sweep has
// moved a vertex, the buffers holding the current, the next and the pending list
// (0, 1: D, 2: P; two bits each), tags used, the stamp of the pending list.
enum SmoothRes { SR_ROUNDS = 0, SR_SWEEPS, SR_OVER, SR_MOVED, SR_PERM, SR_TAGS, SR_PTAG };
constexpr int cn_list(int i) { return i == 0 ? CN_D0 : CN_D1; }

// Everything the library keeps on the device for a set of meshes.
struct MeshSet {
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  int nmesh = 0;
  // host mirror of the per-mesh table
  std::vector<int> vbase, vcap, ebase, ecap, nv, ne;
  std::vector<uint32_t> seed;
  std::vector<double> L_low, L_up, q_thresh;
  std::vector<int> select;  // PM_SELECT_* per mesh
  Store S{};          // device arrays (S.tab points into tabmem)
  Store B{};          // second buffer set for renumbering
  Work w{};
  ScanWork scan{};
  DevStatus* st = nullptr;     // device
  DevStatus* hst = nullptr;    // pinned host
  int* hcounts = nullptr;      // pinned host copy of w.counts
  unsigned long long* hops = nullptr;  // pinned: operation counts (see OpSlot, OS_NUM * nmesh)
  uint32_t* hr = nullptr;              // pinned: round counters
  unsigned long long* ops = nullptr;   // device: operation counts of the call
  std::vector<long long> edead;        // dead element slots of each mesh
  std::vector<long long> seen_dead;    // those of the current call counted so far
  bool dense = false;  // no dead slot: ids are the slot offsets and the sizes are nv, ne
  std::vector<int> hpre;               // source of upload_prefix
  char* hup = nullptr;                 // pinned: staging of the per-mesh table for upload_tab
  cudaEvent_t upev = nullptr;          // the last table upload has left the staging
  void* pinned = nullptr;      // slot of the process-wide pinned arena (hst, hcounts)
  bool pinned_own = false;     // slot too small: a private pinned allocation
  void* tabmem = nullptr;      // device block holding MeshTab arrays
  void* rowmem = nullptr;      // device block holding the adjacency rows of both buffer sets
  int* lidbuf = nullptr;       // S.lid and S.voff when in use (vslots, nmesh)
  int* voffbuf = nullptr;
  int tag = 0;                 // per-round tag (even); the round's change stamp is tag + 1
  // evaluations with tags at or below these are stale for that operator
  int lo_coarsen = 0, lo_swap = 0, lo_refine = 0;
  int num_sms = 152;
  bool qvalid = false;         // the element quality cache matches the current metric
  bool mesh_index_ok = false;  // S.tab.vmesh / emesh describe the current layout
  std::vector<void*> allocs;   // device allocations owned by the set
};

// Stream-ordered allocation.  A failure is the caller's to report: it does not stay
// behind as the thread's last error, which the next check after a launch would take for
// that launch's.
template <class T>
cudaError_t device_alloc(T** p, size_t bytes, cudaStream_t s) {
  const cudaError_t e = cudaMallocAsync((void**)p, bytes, s);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

// ---- mesh storage (pm_mesh.cu) ----
cudaError_t set_alloc(MeshSet& m, const std::vector<int>& vcap, const std::vector<int>& ecap,
                      int W);
void set_free(MeshSet& m);
// Release the status word and the pinned read-back slot of a set.
void set_release(MeshSet& m);
// A slot of the process-wide pinned arena (16 KB; null when none can be had).
void* pinned_slot();
void pinned_slot_free(void* p);
cudaError_t upload_tab(MeshSet& m);
void set_used(MeshSet& m);
cudaError_t grow(MeshSet& m, const std::vector<int>& vcap, const std::vector<int>& ecap, int W);
int rebuild_adjacency(MeshSet& m, bool derive_flags, bool corners_given);
int presize(MeshSet& m);
int spare_slots(long long need, int most, int nmesh);
// The part of a renumbering inside the outer loop that runs before its
// read-back (sync_call); `renumber` does it unless it has been queued.
// The scan of the live vertices goes to `vscan` (vslots + 1), which has to be
// Work::vscan when `renumber` runs.
void renumber_queue(MeshSet& m, int* vscan);
int renumber(MeshSet& m, bool final, bool queued = false);
int compact_out(MeshSet& m, int mesh, double* xy, int32_t* tri, double* mt, int* nv_out,
                int* ne_out);
int compact_out_set(MeshSet& m, double* xy, int32_t* tri, double* mt, int* nv_out, int* ne_out);
int sync_status(MeshSet& m);
// The status, the counters and the per-mesh words after them (`extra` ints) in
// one copy; then the whole call state (operation counts and rounds too).
int sync_counts(MeshSet& m, int extra);
int sync_call(MeshSet& m);
void validate_mesh(MeshSet& m);
int refresh_quality(MeshSet& m);
// The quality cache of every element, computed now when it is stale (a mesh
// whose metric was never set gets it at its first operator call).
int ensure_quality(MeshSet& m);

// ---- operators (pm_ops.cu) ----
// What ops_ahead has done of an iteration: collapse rounds, flip rounds (0: none
// run, 1: the pass is complete, 2: to be continued) and the first split marks.
struct Ahead {
  int coarsen = 0, swap = 0, mark_tag = 0;
  int cur_c = 0, cur_s = 0;        // list the next round of a pass reads
  int pass0_c = 0, pass0_s = 0;    // tag at the start of each pass
};
// Collapse rounds, flip rounds and the first split marks of an iteration queued one
// behind the other with one read-back; each starts on the device only when the one
// before is complete.
int ops_ahead(MeshSet& m, Ahead& h);
int op_coarsen(MeshSet& m, int max_rounds, const Ahead& h = Ahead());
int op_swap(MeshSet& m, int max_rounds, const Ahead& h = Ahead());
int op_refine(MeshSet& m, int max_rounds, const Ahead& h = Ahead(),
              bool* renumber_queued = nullptr);
int op_smooth(MeshSet& m, int max_sweeps, int max_rounds);
int op_opt_smooth(MeshSet& m, int nrounds, int max_rounds);
// Operation counters of a call: one set per operator, selected before it runs.
// OS_BND counts the collapses that kill one element (a boundary edge) instead of
// two, so that the host knows the dead elements without a pass over them.
enum OpSlot { OS_COARSEN = 0, OS_SWAP, OS_REFINE, OS_SMOOTH, OS_BND, OS_NUM };
inline void select_ops(MeshSet& m, OpSlot k) { m.S.tab.ops = m.ops + (size_t)k * m.nmesh; }

// ---- quality (pm_quality.cu) ----
int quality_mesh(MeshSet& m, double* qsum_host, double* dxy_host, double* dm_host);
int quality_arrays(const double* xy, const double* mt, int nv, const int* tri, int ne,
                   double* qsum, double* dxy, double* dm, cudaStream_t s);

// Partial derivatives of an element's quality: d/d(x, y) of its three
// vertices, then the metric's three, which are the same for each vertex (the
// element metric is their mean).
struct EGrad {
  double xy[6];
  double m[3];
};
// Status, block counter and scan ticket of a call.
struct QHead {
  DevStatus st;
  unsigned done;
  int ticket;
};
// Workspace of one call on plain arrays; head, cnt and state start at zero.
struct QualityWork {
  QHead* head;
  int* cnt;                   // 2 (nv + 1): corners per vertex, and beyond its 255th
  unsigned long long* state;  // scan_tiles(nv + 1)
  double* part;               // quality_blocks(ne)
  EGrad* eg;                  // ne
  int* off;                   // nv + 1
  int* col;                   // 3 ne
  uint8_t* pos;               // 3 ne
};
constexpr int kQualityBlocks = 152 * 8;
int quality_blocks(int ne);
cudaError_t quality_launch(const QualityWork& w, const double* xy, const double* mt, int nv,
                           const int* tri, int ne, double* qsum, double* dxy, double* dm,
                           DevStatus* out_st, cudaStream_t s);

// ---- errors (pm_capi.cu) ----
void set_last_error(const std::string& msg);

// ---- launches (pm_prof.cu) ----
// Every kernel of the library is launched through PM_LAUNCH: it counts the
// launch and, while profiling is on for a matching kernel name, brackets it
// with CUDA events on its own stream.
extern unsigned long long g_launches;
extern bool g_prof_on;
int prof_begin(const char* name, cudaStream_t s);
void prof_end(int slot, cudaStream_t s);
// Device counter of algorithmic work (FP64 operations) for the kernel being
// profiled, or null when `name` is not being profiled.
unsigned long long* prof_work(const char* name);

template <class K, class... A>
inline void launch(const char* name, K kern, dim3 g, dim3 b, size_t sh, cudaStream_t s,
                   A... args) {
  __atomic_fetch_add(&g_launches, 1ull, __ATOMIC_RELAXED);
  int slot = g_prof_on ? prof_begin(name, s) : -1;
  kern<<<g, b, sh, s>>>(args...);
  if (slot >= 0) prof_end(slot, s);
}

#define PM_LAUNCH(k, g, b, sh, s, ...) ::pm::launch(#k, k, g, b, sh, s, __VA_ARGS__)

// ---- launch shapes (pm_tune.cu) ----
// Per operator (collapse, flip, split, smoothing): threads per block and the
// cap on blocks per SM of the one-kernel-per-phase grids; per operator
// (collapse, flip, smoothing): the largest list whose rounds run in one
// persistent launch, the blocks per SM of that launch, and (flips,
// smoothing) the list size up to which its rounds evaluate in one phase.
// No choice changes a result.
enum TuneOp { TO_COARSEN = 0, TO_SWAP = 1, TO_REFINE = 2, TO_SMOOTH = 3 };
struct Tuning {
  int block[4];
  int blocks_per_sm[4];
  int rounds_limit[3];
  int rounds_blocks_per_sm[3];  // resident blocks per SM of the persistent round kernels
  int fuse_limit[2];            // flips, smoothing: one-phase evaluation up to this list size
};
Tuning tuning();
void tuning_autoload();

// Blocks of `block` threads for n items, at most per_sm blocks per SM.
inline int grid_tuned(const MeshSet& m, long long n, int block, int per_sm) {
  long long want = (n + block - 1) / block;
  long long cap = (long long)m.num_sms * per_sm;
  if (want < 1) want = 1;
  return (int)(want < cap ? want : cap);
}

inline int grid_for(const MeshSet& m, long long n, int per_sm = 16) {
  long long want = (n + BLOCK - 1) / BLOCK;
  long long cap = (long long)m.num_sms * per_sm;
  if (want < 1) want = 1;
  return (int)(want < cap ? want : cap);
}

}  // namespace pm
