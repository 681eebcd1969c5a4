// The adaptation operators (Sec. 2.4) run in rounds of independent sets
// (Sec. 3.2).  One round of coarsening, swapping or smoothing is:
//
//   evaluate  every dirty vertex decides its operation on the current mesh and
//             joins the candidate list (warp-aggregated atomic append, the
//             worklist scheme of Sec. 3.4);
//   select    candidates that beat every candidate neighbour by hash priority
//             form the independent set S; the others stay dirty;
//   apply     each member of S rewrites only its own ball (disjoint between
//             members) and records which vertices' adjacency changes;
//   commit    the deferred update of Sec. 3.3: after the whole set has been
//             applied, every affected vertex rebuilds its own NN/NE rows from
//             the operations of its S neighbours, so exactly one thread writes
//             each list.
//
// Every kernel walks its list with a grid-stride loop over a count that lives
// in device memory, so a round needs no host round trip until the candidate
// count is read to decide termination.
#include <algorithm>
#include <mutex>
#include <string>

#include "pm_internal.cuh"

namespace pm {

namespace {

// ---- shared device helpers ---------------------------------------------------

struct MeshCtx {
  int mi, vb, eb;
};

__device__ __forceinline__ MeshCtx ctx_of(const Store& S, int slot) {
  MeshCtx c{0, 0, 0};  // the regions of a single mesh start at 0: no loads
  if (S.nmesh > 1) {
    c.mi = mesh_of_vslot(S, slot);
    c.vb = S.tab.vbase[c.mi];
    c.eb = S.tab.ebase[c.mi];
  }
  return c;
}

// Which thread takes list entry i.  Contiguous: consecutive entries to
// consecutive threads of a block (coalesced list reads, for long lists).
// Interleaved (`il`): entry i to block i mod gridDim.x, so that a short list
// spreads over every SM instead of the first few blocks; that matters when
// an entry's work is FP64, whose issue cost per warp is the same for one
// active lane as for 32.
__device__ __forceinline__ int grank(bool il) {
  return il ? threadIdx.x * gridDim.x + blockIdx.x : blockIdx.x * blockDim.x + threadIdx.x;
}
__device__ __forceinline__ int gsize() { return gridDim.x * blockDim.x; }

// The list entry of a thread's first turn, loaded together with the list's
// length instead of after it (any position below the list's capacity may be
// read; the value is used only below the length).
__device__ __forceinline__ int first_entry(const int* list, int i, int cap) {
  return i < cap ? list[i] : 0;
}

__device__ __forceinline__ const int* nn_row(const Store& S, int slot) {
  return S.NN + (size_t)slot * S.W;
}
__device__ __forceinline__ const int* ne_row(const Store& S, int slot) {
  return S.NE + (size_t)slot * S.W;
}

// Per-mesh operation counter, aggregated over the lanes of a warp that share a
// mesh (all lanes must call).
__device__ __forceinline__ void count_op(const Store& S, bool pred, int mi) {
  unsigned act = __ballot_sync(0xffffffffu, pred);
  if (!act) return;
  unsigned grp = __match_any_sync(0xffffffffu, pred ? mi : -1);
  int lane = threadIdx.x & 31;
  if (pred && (__ffs(grp) - 1) == lane) atomicAdd(S.tab.ops + mi, (unsigned long long)__popc(grp));
}

// Advance the per-mesh round counter of every mesh that formed candidates in
// the round whose set was just selected (run by one block before the apply).
__device__ __forceinline__ void advance_rounds(const Store& S) {
  if (blockIdx.x != 0) return;
  for (int i = threadIdx.x; i < S.nmesh; i += blockDim.x) {
    if (S.tab.had[i]) {
      S.tab.r[i] += 1;
      S.tab.had[i] = 0;
    }
  }
}

__device__ __forceinline__ int count_elems_with(const Store& S, const int* ne, int nel, int eb,
                                                int lw) {
  int c = 0;
  for (int b = 0; b < nel; b += 8) {
    const Row8 r = row8(ne, b);
    int4 e[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      e[k] = b + k < nel ? S.EN[eb + r.a[k]] : make_int4(-1, -1, -1, 0);
#pragma unroll
    for (int k = 0; k < 8; ++k) c += (e[k].x == lw || e[k].y == lw || e[k].z == lw) ? 1 : 0;
  }
  return c;
}


// Inputs of v's evaluation unchanged since tag `et`?  Evaluations read v's
// rows, the elements and vertices of its ball and the rows and positions of
// its neighbours; every change to those stamps v (touch) or, for a change of
// a neighbour x, every vertex adjacent to x after the change (ntouch).  An
// edge (v, x) that exists now existed at x's last change (adding it would
// have changed x again), so ntouch[v] covers every current neighbour.  Only
// evaluations newer than `lo` count.
__device__ __forceinline__ bool unchanged(const Store& S, int v, int vb, int et, int lo) {
  return et > lo && S.touch[v] <= et && S.ntouch[v] <= et;
}

// Measurement only: adds every lane's count of FP64 operations to *work
// (one atomic per warp).  All 32 lanes must call it.  The counts follow the
// arithmetic as written: a metric length 17 operations, an orientation 8, a
// quality 77, a square root or a division 1.
constexpr unsigned kOpsLen2 = 17, kOpsOrient = 8, kOpsQuality = 77;

// Warps per block that own a per-warp shared-memory queue or array in the
// scan phases (blocks hold at most 256 threads).
constexpr int kScanWarps = 8;

__device__ __forceinline__ void add_work(unsigned long long* work, unsigned ops) {
  if (!work) return;
  unsigned tot = __reduce_add_sync(0xffffffffu, ops);
  if ((threadIdx.x & 31) == 0 && tot) atomicAdd(work, (unsigned long long)tot);
}

// qK of every listed element slot, one element per thread.
// 77 FP64 operations on 32 lanes: the FP64 pipe bounds it (83% active); 114 bytes
// gathered per element are a tenth of the memory's rate beside that.
__device__ __forceinline__ void elem_quality_phase(const Store& S, const int* list, const int* np,
                                                   unsigned long long* work, bool il = false) {
  // in the persistent rounds from the last warp of every block backwards: the
  // commit that shares the phase fills the blocks from their first warp
  const int r0 = il ? (blockDim.x - 1 - threadIdx.x) * gridDim.x + blockIdx.x : grank(false);
  const int first = first_entry(list, r0, S.eslots);
  const int n = *np;
  for (int i0 = 0; i0 < n; i0 += gsize()) {
    const int i = i0 + r0;
    unsigned ops = 0;
    if (i < n) {
      const int slot = i0 == 0 ? first : list[i];
      const int vb = S.nmesh > 1 ? S.tab.vbase[mesh_of_eslot(S, slot)] : 0;
      int4 e = S.EN[slot];
      S.qK[slot] = quality_c(e.x, e.y, e.z, load_vd(S, vb + e.x), load_vd(S, vb + e.y),
                             load_vd(S, vb + e.z));
      ops = kOpsQuality;
    }
    add_work(work, ops);
  }
}

// Stamps the neighbours in `row` (local ids, whole chunks of 8 readable) after a
// change of their vertex.
__device__ __forceinline__ void stamp_neighbours(const Store& S, const int* row, int len, int vb,
                                                 int stamp) {
  for (int b = 0; b < len; b += 8) {
    const Row8 r = row8(row, b);
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (b + k < len) S.ntouch[vb + r.a[k]] = stamp;
  }
}

// ---- worklist initialisation ---------------------------------------------------

// mode 0: every live vertex of an active mesh; mode 1: live interior vertices.
// With `ev`, vertices whose last evaluation (newer than `lo`) found nothing
// and whose inputs are unchanged since are left out: they would find
// nothing again.
// A pass queued behind another's persistent rounds, whose results are `before`
// (rounds run, list, complete): it does nothing unless those are complete and no
// row has outgrown its width, and its tags follow theirs.
__device__ __forceinline__ bool may_go(const int* before, const DevStatus* st) {
  return !before || (before[2] != 0 && *(volatile const int*)&st->overflow == 0 &&
                     *(volatile const int*)&st->err == 0);
}
__device__ __forceinline__ int tags_of(const int* before) {
  return before ? 2 * before[0] : 0;
}

__global__ void k_init_list(Store S, int mode, int* list, int* count, const int* ev, int lo,
                            const int* before, const DevStatus* st) {
  if (!may_go(before, st)) return;
  for (int i0 = blockIdx.x * blockDim.x; i0 < S.vused; i0 += gridDim.x * blockDim.x) {
    int s = i0 + threadIdx.x;
    bool take = false;
    if (s < S.vused) {
      int mi = mesh_of_vslot(S, s);
      int vb = S.tab.vbase[mi];
      if (s - vb < S.tab.nv[mi] && S.tab.active[mi]) {
        uint8_t f = S.vflag[s];
        take = (f & VF_ALIVE) && (mode == 0 || !(f & VF_BND));
        if (take && ev) take = !unchanged(S, s, vb, ev[s], lo);
      }
    }
    warp_append(take, s, list, count);
  }
}

// ---- independent set (Sec. 3.2) -------------------------------------------------
// v joins S when prio(v) exceeds the priority of every neighbour that is a
// candidate of the same round.  Losers go to `keep` (still dirty / pending).
__global__ void k_select(Store S, const int* C, const int* nCp, const int* cmark, int* smark,
                         int tag, int* Sl, int* nS, int* keep, int* nkeep, int* kmark) {
  const int n = *nCp;
  for (int i0 = blockIdx.x * blockDim.x; i0 < n; i0 += gridDim.x * blockDim.x) {
    int i = i0 + threadIdx.x;
    bool win = false, lose = false;
    int v = 0;
    if (i < n) {
      v = C[i];
      MeshCtx c = ctx_of(S, v);
      uint32_t seed = S.tab.seed[c.mi], r = S.tab.r[c.mi];
      uint32_t pv = prio(vid_of(S, v, c.vb), seed, r);
      const int* nn = nn_row(S, v);
      int nnl = S.NNlen[v];
      win = true;
#pragma unroll 4
      for (int k = 0; k < nnl; ++k) {
        int u = c.vb + nn[k];
        int cu = cmark[u];
        uint32_t iu = vid_of(S, u, c.vb);
        win &= !(cu == tag && prio(iu, seed, r) > pv);
      }
      if (win) smark[v] = tag;
      else if (keep) lose = stamp_first(kmark, v, tag);
    }
    warp_append(win, v, Sl, nS);
    if (keep) warp_append(lose, v, keep, nkeep);
  }
}

// Whether candidate v is a local maximum of the priority among this round's
// candidates (cmark == tag) in its neighbourhood.
__device__ __forceinline__ bool local_max(const Store& S, int v, const int* cmark, int tag) {
  MeshCtx c = ctx_of(S, v);
  uint32_t seed = S.tab.seed[c.mi], r = S.tab.r[c.mi];
  // colour-class sets: only the candidates of colour r mod ncol compete
  const bool by_colour = S.tab.select[c.mi] == PM_SELECT_COLOUR;
  const int cls = by_colour ? (int)(r % (uint32_t)S.tab.ncol[c.mi]) : 0;
  if (by_colour && S.tab.col[v] != cls) return false;
  uint32_t pv = prio(vid_of(S, v, c.vb), seed, r);
  const int* nn = nn_row(S, v);
  Row8 nb = row8(nn, 0);
  const int nnl = S.NNlen[v];
  bool win = true;
  for (int b = 0;;) {
    int cu[8];
    uint32_t iu[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const bool in = b + k < nnl;
      cu[k] = in ? cmark[c.vb + nb.a[k]] : tag - 1;
      iu[k] = in ? vid_of(S, c.vb + nb.a[k], c.vb) : 0u;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (cu[k] != tag) continue;
      win &= !((!by_colour || S.tab.col[c.vb + nb.a[k]] == cls) && prio(iu[k], seed, r) > pv);
    }
    b += 8;
    if (b >= nnl) break;
    nb = row8(nn, b);
  }
  return win;
}

// ---- colouring of the vertex graph (Sec. 3.2, colour-class sets) --------------
// Speculative rounds on a snapshot, the same as the oracle's: every uncoloured
// live vertex of a mesh in colour mode proposes the smallest colour no
// coloured neighbour holds; of two uncoloured neighbours proposing the same
// colour the one of lower priority (prio with the mesh's round counter at the
// start of the pass) withdraws; the others keep their proposals.  The
// proposals of a round are stamped with the round, so the resolve pass reads
// only stamps and proposals while it writes colours.
__global__ void k_colour_init(Store S, int* U, int* nU) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < S.nmesh; i += gridDim.x * blockDim.x)
    S.tab.ncol[i] = 1;
  for (int i0 = blockIdx.x * blockDim.x; i0 < S.vused; i0 += gridDim.x * blockDim.x) {
    const int s = i0 + threadIdx.x;
    bool take = false;
    if (s < S.vused) {
      S.tab.col[s] = -1;
      const int mi = mesh_of_vslot(S, s);
      take = s - S.tab.vbase[mi] < S.tab.nv[mi] && S.tab.active[mi] &&
             S.tab.select[mi] == PM_SELECT_COLOUR && (S.vflag[s] & VF_ALIVE);
    }
    warp_append(take, s, U, nU);
  }
}

__device__ __forceinline__ void colour_propose_phase(const Store& S, const int* U, const int* nUp,
                                                     int* prop, int* stamp, int rt, bool il) {
  const int n = *nUp;
  for (int i = grank(il); i < n; i += gsize()) {
    const int v = U[i];
    const int vb = ctx_of(S, v).vb;
    const int* nn = nn_row(S, v);
    Row8 r = row8(nn, 0);
    const int nnl = S.NNlen[v];
    RowMask used;  // colours 0..127 held by coloured neighbours
    for (int b = 0;;) {
      int c[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) c[k] = b + k < nnl ? S.tab.col[vb + r.a[k]] : -1;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (c[k] >= 0 && c[k] < MAXW) used.set(c[k]);
      b += 8;
      if (b >= nnl) break;
      r = row8(nn, b);
    }
    int c = 0;
    if (~used.lo) c = __ffsll((long long)~used.lo) - 1;
    else if (~used.hi) c = 64 + __ffsll((long long)~used.hi) - 1;
    else c = MAXW;  // a vertex of degree MAXW whose neighbours hold 0..MAXW-1
    prop[v] = c;
    stamp[v] = rt;
  }
}

__device__ __forceinline__ void colour_resolve_phase(const Store& S, const int* U, const int* nUp,
                                                     const int* prop, const int* stamp, int rt,
                                                     int* Un, int* nUn, bool il) {
  const int n = *nUp;
  for (int i0 = 0; i0 < n; i0 += gsize()) {
    const int i = i0 + grank(il);
    bool again = false;
    int v = 0;
    if (i < n) {
      v = U[i];
      const MeshCtx c = ctx_of(S, v);
      const uint32_t seed = S.tab.seed[c.mi], r = S.tab.r[c.mi];
      const uint32_t pv = prio(vid_of(S, v, c.vb), seed, r);
      const int pc = prop[v];
      const int* nn = nn_row(S, v);
      Row8 nb = row8(nn, 0);
      const int nnl = S.NNlen[v];
      bool keep = true;
      for (int b = 0;;) {
        int su[8], pu[8];
        uint32_t iu[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const bool in = b + k < nnl;
          const int u = c.vb + nb.a[k];
          su[k] = in ? stamp[u] : rt - 1;
          pu[k] = in ? prop[u] : -1;
          iu[k] = in ? vid_of(S, u, c.vb) : 0u;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
          keep &= !(su[k] == rt && pu[k] == pc && prio(iu[k], seed, r) > pv);
        b += 8;
        if (b >= nnl) break;
        nb = row8(nn, b);
      }
      if (keep) {
        S.tab.col[v] = pc;
        atomicMax(S.tab.ncol + c.mi, pc + 1);
      }
      again = !keep;
    }
    warp_append(again, v, Un, nUn);
  }
}

__global__ void k_colour_propose(Store S, const int* U, const int* nUp, int* prop, int* stamp,
                                 int rt) {
  colour_propose_phase(S, U, nUp, prop, stamp, rt, false);
}

__global__ void k_colour_resolve(Store S, const int* U, const int* nUp, const int* prop,
                                 const int* stamp, int rt, int* Un, int* nUn) {
  colour_resolve_phase(S, U, nUp, prop, stamp, rt, Un, nUn, false);
}


// End of a fused select-and-apply launch: the last block to finish advances
// the round counter of every mesh that formed candidates (every block has
// read the counters by then) and re-arms the block counter.
__device__ __forceinline__ void round_done(const Store& S, unsigned* done) {
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int i = threadIdx.x; i < S.nmesh; i += blockDim.x) {
    if (S.tab.had[i]) {
      S.tab.r[i] += 1;
      S.tab.had[i] = 0;
    }
  }
  if (threadIdx.x == 0) *done = 0;
}

// ---- tile-parallel evaluation: 8 lanes per vertex, one ball element each ----
// Sums keep the ascending order of the definition (every lane accumulates the
// lanes' terms in order through shuffles); minima and all-of votes do not
// depend on order.  All lanes of a tile end with the same result.

constexpr int TW = 8;
constexpr int kTileMax = 32;  // tiles per block (blocks hold at most 256 threads)

struct Tile {
  int tl;          // lane within the tile
  unsigned mask;   // the tile's lanes in the warp
  int shift;       // bit offset of the tile in a warp ballot
};

__device__ __forceinline__ Tile tile_of() {
  int lane = threadIdx.x & 31;
  Tile t;
  t.tl = lane & (TW - 1);
  t.shift = lane & ~(TW - 1);
  t.mask = 0xFFu << t.shift;
  return t;
}

__device__ __forceinline__ double tshfl(const Tile& t, double x, int src) {
  return __shfl_sync(t.mask, x, src, TW);
}

__device__ __forceinline__ double tmin(const Tile& t, double x) {
#pragma unroll
  for (int o = TW / 2; o > 0; o >>= 1) {
    double y = __shfl_xor_sync(t.mask, x, o, TW);
    x = dlt(y, x) ? y : x;
  }
  return x;
}

__device__ __forceinline__ bool tall(const Tile& t, bool p) {
  return ((__ballot_sync(t.mask, !p) >> t.shift) & 0xFFu) == 0u;
}

__device__ __forceinline__ int tsum(const Tile& t, int x) {
  return __reduce_add_sync(t.mask, x);
}

// Position of tile `tid` and the number of tiles of the grid.  Interleaved
// (`il`): tile i to block i mod gridDim.x (see grank).
__device__ __forceinline__ int trank(bool il) {
  const int tpb = blockDim.x / TW, tib = threadIdx.x / TW;
  return il ? tib * gridDim.x + blockIdx.x : blockIdx.x * tpb + tib;
}
__device__ __forceinline__ int tcount() { return gridDim.x * (blockDim.x / TW); }

// ---- coarsening (Sec. 2.4.1) ---------------------------------------------------

struct CoarsenCtx {
  const Store* S;
  MeshCtx c;
  int v, lv;
  const int* nn;
  int nnl;
  const int* ne;
  int nel;
  bool bnd;
};

// Is edge (a, b) certainly longer (+1) or shorter (-1) than a bound, or is
// that for the exact length to say (0)?
__device__ __forceinline__ int edge_cmp(const VF& a, const VF& b, float lo2, float hi2) {
  return f_len_cmp(f_edge2(a, b), lo2, hi2);
}

// Edge (va, vb) longer than L_up, shorter than L_low: the FP32 filter first.
__device__ __forceinline__ bool edge_longer(const Store& S, int mi, const VF& fa, const VF& fb,
                                            int va, int vb, unsigned& ops) {
  const float4 bf = S.tab.bandf[mi];
  const int r = edge_cmp(fa, fb, bf.z, bf.w);
  if (r != 0) return r > 0;
  const double4 band = S.tab.band[mi];
  ops += kOpsLen2;
  return len_gt(metric_len2(load_vd(S, va), load_vd(S, vb)), band.z, band.w, S.tab.L_up[mi]);
}
__device__ __forceinline__ bool edge_shorter(const Store& S, int mi, const VF& fa, const VF& fb,
                                             int va, int vb, unsigned& ops) {
  const float4 bf = S.tab.bandf[mi];
  const int r = edge_cmp(fa, fb, bf.x, bf.y);
  if (r != 0) return r < 0;
  const double4 band = S.tab.band[mi];
  ops += kOpsLen2;
  return len_lt(metric_len2(load_vd(S, va), load_vd(S, vb)), band.x, band.y, S.tab.L_low[mi]);
}

// collapse_valid with the lanes of a tile splitting v's ball elements (the
// element count of the edge and the orientations with v on u) and v's
// neighbours (the link condition and the new edge lengths): the same
// conjunction of the same tests.  Every lane returns the tile's answer.
__device__ bool tile_collapse_valid(const Tile& t, const CoarsenCtx& x, int u, unsigned& ops) {
  const Store& S = *x.S;
  int cnt = 0;
  for (int k = t.tl; k < x.nel; k += TW) {
    int4 e = S.EN[x.c.eb + x.ne[k]];
    cnt += (e.x == u || e.y == u || e.z == u) ? 1 : 0;
  }
  const bool bedge = tsum(t, cnt) == 1;
  if (x.bnd && !bedge) return false;
  const int ws = x.c.vb + u;
  const int* nnw = nn_row(S, ws);
  const int nnwl = S.NNlen[ws];
  int common = 0;
  for (int k = t.tl; k < x.nnl; k += TW) common += row_has(nnw, nnwl, x.nn[k]) ? 1 : 0;
  if (tsum(t, common) != (bedge ? 1 : 2)) return false;
  const VF fw = load_vf(S, ws);
  bool ok = true;
  for (int k = t.tl; k < x.nel; k += TW) {
    int4 e = S.EN[x.c.eb + x.ne[k]];
    if (e.x == u || e.y == u || e.z == u) continue;
    const int s0 = (e.x == x.lv) ? ws : x.c.vb + e.x, s1 = (e.y == x.lv) ? ws : x.c.vb + e.y,
              s2 = (e.z == x.lv) ? ws : x.c.vb + e.z;
    int o = f_orient(load_vf(S, s0), load_vf(S, s1), load_vf(S, s2));
    if (o == 0) {
      o = orient_sign(load_vd(S, s0), load_vd(S, s1), load_vd(S, s2)) > 0 ? 1 : -1;
      ops += kOpsOrient;
    }
    ok &= o > 0;
  }
  if (!tall(t, ok)) return false;
  for (int k = t.tl; k < x.nnl; k += TW) {
    int y = x.nn[k];
    if (y == u || row_has(nnw, nnwl, y)) continue;
    ok &= !edge_longer(S, x.c.mi, fw, load_vf(S, x.c.vb + y), ws, x.c.vb + y, ops);
  }
  return tall(t, ok);
}

// Collapse candidates of v: neighbours with metric length below L_low (a
// boundary vertex: only along boundary edges), sorted by (length, id) into
// out[0..n); corners and dead vertices have none.  The lanes of a tile split
// v's neighbours: lane tl holds neighbours tl, tl + 8, ...; each candidate's
// place in the order is the number of candidates before it (a neighbour of
// lower index has the lower id: rows are sorted), which is the stable order
// by length the definition asks for.  Returns the candidate count (every
// lane).
__device__ int tile_coarsen_candidates(const Tile& t, const Store& S, int v, MeshCtx c, int* out,
                                       unsigned& ops) {
  uint8_t f = S.vflag[v];
  if (!(f & VF_ALIVE) || (f & VF_CORNER)) return 0;
  const bool bnd = (f & VF_BND) != 0;
  const int* nn = nn_row(S, v);
  const int nnl = S.NNlen[v];
  const int* ne = ne_row(S, v);
  const int nel = S.NElen[v];
  const VF fv = load_vf(S, v);
  constexpr int kPer = MAXW / TW;
  double L[kPer];
  bool is[kPer];
  int mine = 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int k = j * TW + t.tl;
    is[j] = false;
    L[j] = 0.0;
    if (k < nnl) {
      const int u = nn[k];
      bool cand = edge_shorter(S, c.mi, fv, load_vf(S, c.vb + u), v, c.vb + u, ops);
      if (cand && bnd) cand = count_elems_with(S, ne, nel, c.eb, u) == 1;
      if (cand) {
        is[j] = true;
        ++mine;
      }
    }
  }
  const int total = tsum(t, mine);
  if (total == 0) return 0;
  // the exact lengths, for the order of several candidates
  if (total > 1) {
    const VD dv = load_vd(S, v);
#pragma unroll
    for (int j = 0; j < kPer; ++j)
      if (is[j]) {
        L[j] = sqrt(metric_len2(dv, load_vd(S, c.vb + nn[j * TW + t.tl])));
        ops += kOpsLen2 + 1;
      }
  }
  const int steps = (nnl + TW - 1) / TW;
  for (int j = 0; j < steps; ++j) {
    int rank = 0;
    for (int j2 = 0; j2 < steps; ++j2) {
#pragma unroll
      for (int src = 0; src < TW; ++src) {
        const double Lo = tshfl(t, L[j2], src);
        const bool co = __shfl_sync(t.mask, is[j2] ? 1 : 0, src, TW) != 0;
        const int ko = j2 * TW + src, k = j * TW + t.tl;
        if (co && (dlt(Lo, L[j]) || (dbits(Lo) == dbits(L[j]) && ko < k))) ++rank;
      }
    }
    if (is[j]) out[rank] = nn[j * TW + t.tl];
  }
  return total;
}

__device__ __forceinline__ CoarsenCtx coarsen_ctx(const Store& S, int v, MeshCtx c) {
  CoarsenCtx x;
  x.S = &S;
  x.c = c;
  x.v = v;
  x.lv = v - c.vb;
  x.nn = nn_row(S, v);
  x.nnl = S.NNlen[v];
  x.ne = ne_row(S, v);
  x.nel = S.NElen[v];
  x.bnd = (S.vflag[v] & VF_BND) != 0;
  return x;
}

// Collapse evaluation.  The target of v is the first candidate, by (metric
// length, id), whose collapse is valid.  Pass 1 (per dirty vertex) reuses an
// unchanged earlier result or finds v's first candidate; a dense pass then
// checks every listed vertex's first candidate (one work item each), and a
// last pass checks all other candidates of the vertices whose first one failed
// and takes the first of the valid ones.  A vertex's row of `cand` holds its first
// candidate and, from kCandRest on, the others as bits over its neighbours.
constexpr int kCandRest = 4;

__device__ __forceinline__ ulonglong2* cand_rest(int* cand, const Store& S, int v) {
  return reinterpret_cast<ulonglong2*>(cand + (size_t)v * S.W + kCandRest);
}

// The first of the neighbours `cm` (not empty) of v by (metric length, position in
// the row, hence id).  It is mostly plain from the FP32 lengths: only neighbours
// whose error intervals overlap that of the shortest (equal lengths on regular
// grids) are compared by their exact lengths.  `first` is the smallest upper
// bound of the squared lengths (a NaN bound leaves it as it is, and passes here).
__device__ __forceinline__ int first_by_length(const Store& S, int v, int vb, const int* nn,
                                               const VF& fv, RowMask cm, float first,
                                               unsigned& ops) {
  int best = cm.pop();
  if (!cm.any()) return best;
  cm.set(best);
  RowMask near;
  while (cm.any()) {
    const int k = cm.pop();
    const FLen l = f_edge2(fv, load_vf(S, vb + nn[k]));
    if (!(l.L2 - l.err > first)) near.set(k);
  }
  best = near.pop();
  if (!near.any()) return best;
  const VD dv = load_vd(S, v);
  double Lb = sqrt(metric_len2(dv, load_vd(S, vb + nn[best])));
  ops += kOpsLen2 + 1;
  while (near.any()) {  // ascending position
    const int k = near.pop();
    const double L = sqrt(metric_len2(dv, load_vd(S, vb + nn[k])));
    ops += kOpsLen2 + 1;
    if (dlt(L, Lb)) {
      Lb = L;
      best = k;
    }
  }
  return best;
}

// Pass 1 of the large rounds, one dirty vertex per thread.  Which neighbours
// are candidates is a length against L_low, and which of them comes first is
// mostly plain from the FP32 lengths too.  A length that is certainly above
// another's stays above it after rounding, so the order is the exact one.
// Dependent gathers bound it (DRAM 21-27%, FP64 pipe below 10%, on regular grids whose
// equal lengths are compared exactly 39-63%; with all lengths exact it was 80%): 36
// ms of a 512-mesh batch's collapses, 12.1 with the FP32 lengths, 11.5 held to 80
// registers (24 warps an SM instead of 16; at 64 it spills: 12.3).  These times are
// sums over CUDA events around each launch of one adaptation of 512 jittered grids; the
// benchmark's, whose grids are regular, takes 13.0.
__device__ __forceinline__ void coarsen_scan_phase(Store S, const int* D, const int* nDp,
                                                   int* target, int* cand, int* C, int* nC,
                                                   int* cmark, int tag, int pass0, int* W0,
                                                   int* nW0) {
  const int n = *nDp;
  unsigned ops = 0;
  for (int i0 = blockIdx.x * blockDim.x; i0 < n; i0 += gridDim.x * blockDim.x) {
    const int i = i0 + threadIdx.x;
    int v = 0, nc = 0;
    bool reuse_cand = false, eval = false;
    if (i < n) {
      v = D[i];
      const MeshCtx c = ctx_of(S, v);
      if (unchanged(S, v, c.vb, S.evc[v], pass0)) {
        reuse_cand = target[v] >= 0;
        if (reuse_cand) {
          cmark[v] = tag;
          S.tab.had[c.mi] = 1;
        }
      } else {
        S.evc[v] = tag;
        eval = true;
        const uint8_t f = S.vflag[v];
        // corners and dead vertices have no candidates
        const int nnl = ((f & VF_ALIVE) && !(f & VF_CORNER)) ? S.NNlen[v] : 0;
        const int* nn = nn_row(S, v);
        const VF fv = load_vf(S, v);
        const float4 bf = S.tab.bandf[c.mi];
        float first = INFINITY;  // the smallest upper bound
        RowMask cm;
        for (int b = 0; b < nnl; b += 4) {
          const int4 r4 = *reinterpret_cast<const int4*>(nn + b);
          const int u4[4] = {r4.x, r4.y, r4.z, r4.w};
          VF fu[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) fu[j] = b + j < nnl ? load_vf(S, c.vb + u4[j]) : VF{};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int k = b + j;
            if (k >= nnl) continue;
            const FLen l = f_edge2(fv, fu[j]);
            const int r = f_len_cmp(l, bf.x, bf.y);
            bool is = r < 0;
            if (r == 0) is = edge_shorter(S, c.mi, fv, fu[j], v, c.vb + u4[j], ops);
            // a boundary vertex collapses only along a boundary edge
            if (is && (f & VF_BND))
              is = count_elems_with(S, ne_row(S, v), S.NElen[v], c.eb, u4[j]) == 1;
            if (is) {
              cm.set(k);
              first = l.L2 + l.err < first ? l.L2 + l.err : first;
            }
          }
        }
        nc = cm.count();
        if (nc > 0) {
          const int best = first_by_length(S, v, c.vb, nn, fv, cm, first, ops);
          cand[(size_t)v * S.W] = nn[best];
          cm.clear(best);
          *cand_rest(cand, S, v) = make_ulonglong2(cm.lo, cm.hi);
        }
        if (nc == 0) target[v] = -1;
      }
    }
    warp_append(reuse_cand, v, C, nC);
    warp_append(eval && nc > 0, v, W0, nW0);
  }
}

__global__ void __launch_bounds__(256, 3)
k_coarsen_scan(Store S, const int* D, const int* nDp, int* target, int* cand, int* C, int* nC,
               int* cmark, int tag, int pass0, int* W0, int* nW0) {
  coarsen_scan_phase(S, D, nDp, target, cand, C, nC, cmark, tag, pass0, W0, nW0);
}

// The check passes, one candidate per thread: is collapsing v onto it valid?
// Validity is the conjunction of the link condition (|NN(v) & NN(u)| = 2 for
// an interior edge, 1 for a boundary edge; a boundary vertex only along a
// boundary edge) and, for the collapse with v on u, every remaining ball
// element counter-clockwise and no new edge longer than L_up (the tile form
// above).  The FP32 filters decide most tests; what they leave open of an
// item that has not failed (collinear points of regular grids above all) is
// queued in shared memory per warp, orientations and lengths apart, and
// evaluated in FP64 32 at a time.  Any failed test clears the owner's flag;
// the conjunction does not depend on the order of its tests.
constexpr int kCheckWarps = 8;

struct CheckQueues {
  int4* qo;  // orientations: (owner lane, element's local vertex ids)
  int2* ql;  // lengths: (owner lane, neighbour's local id)
  int* ok;   // per lane of the warp: its item's conjunction so far
};

// Evaluate the first `cnt` (<= 32) queued orientations; all lanes call.
__device__ __forceinline__ void check_orient_chunk(const Store& S, const CheckQueues& Q, int cnt,
                                                   int vb, int lv, int ws, unsigned& ops) {
  const int lane = threadIdx.x & 31;
  const int4 r = lane < cnt ? Q.qo[lane] : make_int4(lane, 0, 0, 0);
  const int o_vb = __shfl_sync(0xffffffffu, vb, r.x);
  const int o_lv = __shfl_sync(0xffffffffu, lv, r.x);
  const int o_ws = __shfl_sync(0xffffffffu, ws, r.x);
  if (lane < cnt) {
    const VD dw = load_vd(S, o_ws);
    const VD d0 = (r.y == o_lv) ? dw : load_vd(S, o_vb + r.y);
    const VD d1 = (r.z == o_lv) ? dw : load_vd(S, o_vb + r.z);
    const VD d2 = (r.w == o_lv) ? dw : load_vd(S, o_vb + r.w);
    if (orient_sign(d0, d1, d2) <= 0) Q.ok[r.x] = 0;
    ops += kOpsOrient;
  }
}

// Evaluate the first `cnt` (<= 32) queued new-edge lengths; all lanes call.
__device__ __forceinline__ void check_len_chunk(const Store& S, const CheckQueues& Q, int cnt,
                                                int vb, int ws, int mi, unsigned& ops) {
  const int lane = threadIdx.x & 31;
  const int2 r = lane < cnt ? Q.ql[lane] : make_int2(lane, 0);
  const int o_vb = __shfl_sync(0xffffffffu, vb, r.x);
  const int o_ws = __shfl_sync(0xffffffffu, ws, r.x);
  const int o_mi = __shfl_sync(0xffffffffu, mi, r.x);
  if (lane < cnt) {
    const double4 band = S.tab.band[o_mi];
    const double L_up = S.tab.L_up[o_mi];
    if (len_gt(metric_len2(load_vd(S, o_ws), load_vd(S, o_vb + r.y)), band.z, band.w, L_up))
      Q.ok[r.x] = 0;
    ops += kOpsLen2;
  }
}

// The integer part and the FP32 filters for collapsing x.v onto u: false when
// it is certainly invalid; else the tests left open, as bits over the ball's
// elements and v's neighbours.
// All its loads run in chunks whose addresses do not wait on one another.
__device__ __forceinline__ bool check_filter(const Store& S, const CoarsenCtx& x, int u,
                                             RowMask& oo, RowMask& ol) {
  const int ws = x.c.vb + u;
  const int* nnw = nn_row(S, ws);
  const int nnwl = S.NNlen[ws];
  const VF fw = load_vf(S, ws);
  const bool bedge = count_elems_with(S, x.ne, x.nel, x.c.eb, u) == 1;
  if (x.bnd && !bedge) return false;
  // v's neighbours in u's row
  RowMask common;
  for (int b = 0; b < nnwl; b += 8) {
    const Row8 w8 = row8(nnw, b);
    for (int a = 0; a < x.nnl; a += 8) {
      const Row8 v8 = row8(x.nn, a);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        bool in = false;
#pragma unroll
        for (int j = 0; j < 8; ++j) in |= b + j < nnwl && w8.a[j] == v8.a[k];
        if (in && a + k < x.nnl) common.set(a + k);
      }
    }
  }
  if (common.count() != (bedge ? 1 : 2)) return false;
  bool ok = true;
  for (int b = 0; b < x.nel; b += 4) {
    const int4 r4 = *reinterpret_cast<const int4*>(x.ne + b);
    const int K4[4] = {r4.x, r4.y, r4.z, r4.w};
    int4 e[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      e[j] = b + j < x.nel ? S.EN[x.c.eb + K4[j]] : make_int4(u, u, u, 0);
    VF p[4], q[4];
    bool test[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      test[j] = e[j].x != u && e[j].y != u && e[j].z != u;
      // the element in the order (u in place of v, next, before)
      const int n1 = (e[j].x == x.lv) ? e[j].y : (e[j].y == x.lv) ? e[j].z : e[j].x;
      const int n2 = (e[j].x == x.lv) ? e[j].z : (e[j].y == x.lv) ? e[j].x : e[j].y;
      p[j] = test[j] ? load_vf(S, x.c.vb + n1) : VF{};
      q[j] = test[j] ? load_vf(S, x.c.vb + n2) : VF{};
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (!test[j]) continue;
      const int o = f_orient(fw, p[j], q[j]);
      ok &= o >= 0;
      if (o == 0) oo.set(b + j);
    }
  }
  if (!ok) return false;
  const float4 bf = S.tab.bandf[x.c.mi];
  for (int b = 0; b < x.nnl; b += 4) {
    const int4 r4 = *reinterpret_cast<const int4*>(x.nn + b);
    const int y4[4] = {r4.x, r4.y, r4.z, r4.w};
    VF p[4];
    bool test[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      test[j] = b + j < x.nnl && y4[j] != u && !common.test(b + j);
      p[j] = test[j] ? load_vf(S, x.c.vb + y4[j]) : VF{};
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (!test[j]) continue;
      const int r = edge_cmp(fw, p[j], bf.z, bf.w);
      ok &= r <= 0;
      if (r == 0) ol.set(b + j);
    }
  }
  return ok;
}

// The warp's candidates, one per lane (`have` lanes): u for x.v.  Whole warps call.
__device__ __forceinline__ bool check_candidates(const Store& S, const CheckQueues& Q,
                                                 const CoarsenCtx& x, int u, bool have,
                                                 unsigned& ops) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  RowMask oo, ol;
  const bool may = have && check_filter(S, x, u, oo, ol);
  Q.ok[lane] = may ? 1 : 0;
  if (!may) oo = ol = RowMask();
  const int ws = x.c.vb + u;
  int no = 0, nl = 0;  // queue lengths, the same in every lane
  __syncwarp();
  while (__ballot_sync(0xffffffffu, oo.any() || ol.any())) {
    const bool po = oo.any(), pl = ol.any();
    const unsigned mo = __ballot_sync(0xffffffffu, po);
    const unsigned ml = __ballot_sync(0xffffffffu, pl);
    if (po) {
      const int4 e = S.EN[x.c.eb + x.ne[oo.pop()]];
      Q.qo[no + __popc(mo & lt)] = make_int4(lane, e.x, e.y, e.z);
    }
    if (pl) Q.ql[nl + __popc(ml & lt)] = make_int2(lane, x.nn[ol.pop()]);
    no += __popc(mo);
    nl += __popc(ml);
    __syncwarp();
    if (no >= 32) {
      check_orient_chunk(S, Q, 32, x.c.vb, x.lv, ws, ops);
      __syncwarp();
      if (lane < no - 32) Q.qo[lane] = Q.qo[32 + lane];
      no -= 32;
      __syncwarp();
    }
    if (nl >= 32) {
      check_len_chunk(S, Q, 32, x.c.vb, ws, x.c.mi, ops);
      __syncwarp();
      if (lane < nl - 32) Q.ql[lane] = Q.ql[32 + lane];
      nl -= 32;
      __syncwarp();
    }
  }
  if (no > 0) check_orient_chunk(S, Q, no, x.c.vb, x.lv, ws, ops);
  if (nl > 0) check_len_chunk(S, Q, nl, x.c.vb, ws, x.c.mi, ops);
  __syncwarp();
  const bool ok = Q.ok[lane] != 0;
  __syncwarp();
  return ok;
}

// Pass 2: every listed vertex's first candidate.  Gathers bound it (L1 50-65%, DRAM
// 31-48%, FP64 pipe below 1%, on regular grids 33%); with every test in FP64 the
// two check passes took 47 ms of a 512-mesh batch, 26.4 with the filters, 21.3 (15.0 and
// 6.3) with pass 3 as it is (jittered grids; on the benchmark's regular ones, whose
// collinear points are decided exactly, 15.2 and 12.7).
__device__ __forceinline__ void coarsen_check_phase(Store S, const int* Win, const int* nWin,
                                                    int* Wout, int* nWout, int* target, int* cand,
                                                    int* C, int* nC, int* cmark, int tag,
                                                    unsigned long long* work) {
  __shared__ int4 sqo[kCheckWarps][64];
  __shared__ int2 sql[kCheckWarps][64];
  __shared__ int sok[kCheckWarps][32];
  const int wq = (threadIdx.x >> 5) % kCheckWarps;
  const CheckQueues Q{sqo[wq], sql[wq], sok[wq]};
  unsigned ops = 0;
  const int n = *nWin;
  for (int i0 = blockIdx.x * blockDim.x; i0 < n; i0 += gridDim.x * blockDim.x) {
    const int i = i0 + threadIdx.x;
    const bool have = i < n;
    int v = 0, u = 0;
    CoarsenCtx x{};
    if (have) {
      v = Win[i];
      x = coarsen_ctx(S, v, ctx_of(S, v));
      u = cand[(size_t)v * S.W];
    }
    const bool found = check_candidates(S, Q, x, u, have, ops);
    bool next = false;
    if (found) {
      target[v] = u;
      cmark[v] = tag;
      S.tab.had[x.c.mi] = 1;
    } else if (have) {
      const ulonglong2 rest = *cand_rest(cand, S, v);
      next = (rest.x | rest.y) != 0;
      if (!next) target[v] = -1;
    }
    warp_append(found, v, C, nC);
    warp_append(next, v, Wout, nWout);
  }
  add_work(work, ops);
}

__global__ void k_coarsen_check(Store S, const int* Win, const int* nWin, int* Wout, int* nWout,
                                int* target, int* cand, int* C, int* nC, int* cmark, int tag,
                                unsigned long long* work) {
  coarsen_check_phase(S, Win, nWin, Wout, nWout, target, cand, C, nC, cmark, tag, work);
}

// Pass 3: all other candidates of the vertices whose first one failed, one per lane.
// Most of these vertices have no valid candidate at all, so checking one after
// the other by length (a thread per vertex) was a chain of up to six checks in a
// few warps (9-16% of the warp slots held); eight vertices a warp fill its lanes
// once, and lengths are compared only where several candidates are valid.
constexpr int kRestOwners = 8;

__device__ __forceinline__ void coarsen_rest_phase(Store S, const int* Win, const int* nWin,
                                                   int* target, int* cand, int* C, int* nC,
                                                   int* cmark, int tag,
                                                   unsigned long long* work) {
  __shared__ int4 sqo[kCheckWarps][64];
  __shared__ int2 sql[kCheckWarps][64];
  __shared__ int sok[kCheckWarps][32];
  __shared__ unsigned long long svalid[kCheckWarps][kRestOwners][2];
  const int lane = threadIdx.x & 31, wq = (threadIdx.x >> 5) % kCheckWarps;
  const CheckQueues Q{sqo[wq], sql[wq], sok[wq]};
  unsigned long long (*valid)[2] = svalid[wq];
  unsigned ops = 0;
  const int n = *nWin;
  const int warps = gridDim.x * (blockDim.x >> 5);
  for (int i0 = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kRestOwners; i0 < n;
       i0 += warps * kRestOwners) {
    const bool own = lane < kRestOwners && i0 + lane < n;
    int v = 0;
    RowMask rest;
    if (own) {
      v = Win[i0 + lane];
      const ulonglong2 r = *cand_rest(cand, S, v);
      rest.lo = r.x;
      rest.hi = r.y;
    }
    if (lane < kRestOwners) valid[lane][0] = valid[lane][1] = 0ull;
    int end = rest.count();  // of the owner's candidates in the warp's sequence
#pragma unroll
    for (int o = 1; o < kRestOwners; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += y;
    }
    const int total = __shfl_sync(0xffffffffu, end, kRestOwners - 1);
    __syncwarp();
    for (int p0 = 0; p0 < total; p0 += 32) {
      const int p = p0 + lane;
      const bool have = p < total;
      int o = 0, start = 0;  // the owner of candidate p, its first candidate
#pragma unroll
      for (int q = 0; q < kRestOwners - 1; ++q) {
        const int e = __shfl_sync(0xffffffffu, end, q);
        if (p >= e) {
          o = q + 1;
          start = e;
        }
      }
      const int ov = __shfl_sync(0xffffffffu, v, o);
      RowMask r;
      r.lo = __shfl_sync(0xffffffffu, rest.lo, o);
      r.hi = __shfl_sync(0xffffffffu, rest.hi, o);
      int k = 0, u = 0;
      CoarsenCtx x{};
      if (have) {
        for (int j = p - start; j >= 0; --j) k = r.pop();
        x = coarsen_ctx(S, ov, ctx_of(S, ov));
        u = x.nn[k];
      }
      if (check_candidates(S, Q, x, u, have, ops)) atomicOr(&valid[o][k >> 6], 1ull << (k & 63));
    }
    __syncwarp();
    bool found = false;
    if (own) {
      RowMask ok;
      ok.lo = valid[lane][0];
      ok.hi = valid[lane][1];
      found = ok.any();
      if (found) {
        const MeshCtx c = ctx_of(S, v);
        const int* nn = nn_row(S, v);
        const VF fv = load_vf(S, v);
        float first = INFINITY;
        RowMask a = ok;
        while (a.any()) {
          const FLen l = f_edge2(fv, load_vf(S, c.vb + nn[a.pop()]));
          first = l.L2 + l.err < first ? l.L2 + l.err : first;
        }
        target[v] = nn[first_by_length(S, v, c.vb, nn, fv, ok, first, ops)];
        cmark[v] = tag;
        S.tab.had[c.mi] = 1;
      } else {
        target[v] = -1;
      }
    }
    warp_append(found, v, C, nC);
    __syncwarp();
  }
  add_work(work, ops);
}

__global__ void k_coarsen_rest(Store S, const int* Win, const int* nWin, int* target, int* cand,
                               int* C, int* nC, int* cmark, int tag, unsigned long long* work) {
  coarsen_rest_phase(S, Win, nWin, target, cand, C, nC, cmark, tag, work);
}

// One tile per listed vertex, listing and checking at once (persistent
// rounds): reuse or re-evaluate, then the candidates in order until one is a
// valid collapse.  Same results as coarsen_scan_phase and the two check passes.
__device__ __forceinline__ void coarsen_eval_phase(Store S, const int* D, const int* nDp,
                                                   int* target, int* cand, int* C, int* nC,
                                                   int* cmark, int tag, int pass0,
                                                   unsigned long long* work, bool il = false) {
  const Tile t = tile_of();
  const int first = first_entry(D, trank(il), S.vslots);
  const int n = *nDp;
  unsigned ops = 0;
  for (int i0 = 0; i0 < n; i0 += tcount()) {
    const int i = i0 + trank(il);
    int v = 0;
    bool found = false;
    if (i < n) {
      v = i0 == 0 ? first : D[i];
      MeshCtx c = ctx_of(S, v);
      const int et = __shfl_sync(t.mask, S.evc[v], 0, TW);
      if (unchanged(S, v, c.vb, et, pass0)) {
        found = target[v] >= 0;
      } else {
        if (t.tl == 0) S.evc[v] = tag;
        int* cv = cand + (size_t)v * S.W;
        int nc = tile_coarsen_candidates(t, S, v, c, cv, ops);
        __syncwarp(t.mask);  // the candidates written by every lane
        if (nc > 0) {
          CoarsenCtx x = coarsen_ctx(S, v, c);
          for (int k = 0; k < nc && !found; ++k)
            if (tile_collapse_valid(t, x, cv[k], ops)) {
              found = true;
              if (t.tl == 0) target[v] = cv[k];
            }
        }
        if (!found && t.tl == 0) target[v] = -1;
      }
      if (found && t.tl == 0) {
        cmark[v] = tag;
        S.tab.had[c.mi] = 1;
      }
    }
    warp_append(found && t.tl == 0, v, C, nC);
  }
  add_work(work, ops);
}

// One round's independent set and its collapses: a winner applies its
// collapse at once (no other vertex of the round reads what a collapse
// writes); losers stay dirty for the next round.  Elements containing edge
// (v, w) die, the other ball elements take w in v's place (slot and
// orientation kept), v dies.
// Neighbours of v are affected (rows change) and dirty for the next round.
// The qualities of the elements that change are not computed here: their
// slots join list Q and a dense pass computes them (one element per thread
// instead of a serial chain of qualities per collapse).
__device__ __forceinline__ void coarsen_select_apply_phase(Store S, const int* C, const int* nCp,
                                                           const int* cmark, int* smark, int tag,
                                                           const int* target, int* A, int* nA,
                                                           int* amark, int* Dn, int* nDn,
                                                           int* dmark,
                                                           int* Q, int* nQ,
                                                           bool il = false) {
  const int first = first_entry(C, grank(il), S.vslots);
  const int n = *nCp;
  for (int i0 = 0; i0 < n; i0 += gsize()) {
    int i = i0 + grank(il);
    bool win = false, lose = false;
    int v = 0, nnl = 0, mi = 0, vb = 0, eb = 0;
    const int* nn = nullptr;
    const int* ne = nullptr;
    RowMask qbits, fa, fd;
    if (i < n) {
      v = i0 == 0 ? first : C[i];
      win = local_max(S, v, cmark, tag);
      if (win) smark[v] = tag;
      else lose = stamp_first(dmark, v, tag);
    }
    if (win) {
      const MeshCtx c = ctx_of(S, v);
      mi = c.mi;
      vb = c.vb;
      eb = c.eb;
      const int lv = v - c.vb;
      const int w = target[v];
      ne = ne_row(S, v);
      nn = nn_row(S, v);
      nnl = S.NNlen[v];
      const int nel = S.NElen[v];
      // the ball is read first (all loads in flight), then only the words that
      // change are written: v's slot takes w, or the alive word is cleared in
      // the elements that hold w
      int dead = 0;
      for (int b = 0; b < nel; b += 8) {
        const Row8 r = row8(ne, b);
        int4 e[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
          e[k] = b + k < nel ? S.EN[c.eb + r.a[k]] : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (b + k >= nel) continue;
          const bool dies = e[k].x == w || e[k].y == w || e[k].z == w;
          const int f = dies ? 3 : (e[k].x == lv ? 0 : (e[k].y == lv ? 1 : 2));
          reinterpret_cast<int*>(S.EN + c.eb + r.a[k])[f] = dies ? 0 : w;
          if (!dies) qbits.set(b + k);
          else ++dead;
        }
      }
      if (dead == 1) atomicAdd(S.tab.bnd + mi, 1ull);
      S.vflag[v] = (uint8_t)(S.vflag[v] & ~VF_ALIVE);
      for (int b = 0; b < nnl; b += 8) {
        const Row8 r = row8(nn, b);
        int oa[8], od[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const bool in = b + k < nnl;
          oa[k] = in ? atomicExch(amark + vb + r.a[k], tag) : tag;
          od[k] = in ? atomicExch(dmark + vb + r.a[k], tag) : tag;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (oa[k] != tag) fa.set(b + k);
          if (od[k] != tag) fd.set(b + k);
        }
      }
    }
    count_op(S, win, mi);
    // a loser's one entry of the next list is itself
    const Room3 at = warp_reserve3(fa.count(), nA, lose ? 1 : fd.count(), nDn, qbits.count(), nQ);
    int pq = at.c;
    while (qbits.any()) Q[pq++] = eb + ne[qbits.pop()];
    write_row_bits(fa, nn, vb, A, at.a);
    if (lose) Dn[at.b] = v;
    else write_row_bits(fd, nn, vb, Dn, at.b);
  }
}

__global__ void k_coarsen_select_apply(Store S, const int* C, const int* nCp, const int* cmark,
                                       int* smark, int tag, const int* target, int* A, int* nA,
                                       int* amark, int* Dn, int* nDn, int* dmark, int* Q, int* nQ,
                                       unsigned* done) {
  coarsen_select_apply_phase(S, C, nCp, cmark, smark, tag, target, A, nA, amark, Dn, nDn, dmark,
                             Q, nQ);
  round_done(S, done);
}

// The commit below for rows of at most 16 entries that stay so: both rows in
// registers, edited in place (a row of dependent local-memory accesses per
// edit otherwise).  False, with nothing written, when a row grows past 16.
// A commit waits for its gathers (long-scoreboard stalls, DRAM 20-30%); with the rows
// in registers, one reservation for all lists and the qualities on the idle warps, a
// 317 x 317 grid coarsens in 11.9 instead of 13.7 ms, 16 small meshes adapt in 17.9
// instead of 20.6.
__device__ __forceinline__ bool coarsen_commit_short(const Store& S, int u, MeshCtx c, int lu,
                                                     const int* target, const int* smark,
                                                     int tag) {
  int* nn = S.NN + (size_t)u * S.W;
  int* ne = S.NE + (size_t)u * S.W;
  const int nnl = S.NNlen[u], nel = S.NElen[u];
  Row16 R, Q;
  R.load(nn, nnl);
  Q.load(ne, nel);
  if (nnl > kRowReg || nel > kRowReg) return false;
  unsigned dead = 0, sel = 0;
#pragma unroll
  for (int k = 0; k < kRowReg; ++k)
    if (k < nel && S.EN[c.eb + Q.a[k]].w == 0) dead |= 1u << k;
#pragma unroll
  for (int k = 0; k < kRowReg; ++k)
    if (k < nnl && smark[c.vb + R.a[k]] == tag) sel |= 1u << k;
  for (; dead; dead &= dead - 1u) Q.erase(ne[__ffs(dead) - 1]);
  bool ok = true;
  for (; sel && ok; sel &= sel - 1u) {
    const int x = nn[__ffs(sel) - 1], xs = c.vb + x;
    const int t = target[xs];
    R.erase(x);
    if (t != lu) {
      ok = R.insert(t);
      continue;
    }
    // the collapsed neighbour's rows join u's
    const int* nx = nn_row(S, xs);
    const int nxl = S.NNlen[xs];
    for (int j = 0; j < nxl && ok; ++j)
      if (nx[j] != lu) ok = R.insert(nx[j]);
    const int* ex = ne_row(S, xs);
    const int exl = S.NElen[xs];
    RowMask live;
#pragma unroll 4
    for (int j = 0; j < exl; ++j)
      if (S.EN[c.eb + ex[j]].w) live.set(j);
    while (live.any() && ok) ok = Q.insert(ex[live.pop()]);
  }
  if (!ok) return false;
  const int nn2 = R.len(), ne2 = Q.len();
  R.store(nn, nn2);
  Q.store(ne, ne2);
  S.NNlen[u] = nn2;
  S.NElen[u] = ne2;
#pragma unroll
  for (int k = 0; k < kRowReg; ++k)
    if (k < nn2) S.ntouch[c.vb + R.a[k]] = tag + 1;
  return true;
}

// Deferred-update commit of a coarsening round for affected vertex u:
//   NN(u) <- (NN(u) minus collapsed neighbours) + their targets, and when u is
//            the target of x: + NN(x) minus u;
//   NE(u) <- live elements of NE(u) + (when u is the target of x) NE(x).
__device__ __forceinline__ void coarsen_commit_phase(Store S, const int* A, const int* nAp,
                                                     const int* target, const int* smark, int tag,
                                                     DevStatus* st, bool il = false) {
  const int first = first_entry(A, grank(il), S.vslots);
  const int n = *nAp;
  for (int i = grank(il); i < n; i += gsize()) {
    const int u = i < gsize() ? first : A[i];
    S.touch[u] = tag + 1;
    MeshCtx c = ctx_of(S, u);
    int lu = u - c.vb;
    const int* nn = nn_row(S, u);
    const int* ne = ne_row(S, u);
    if (coarsen_commit_short(S, u, c, lu, target, smark, tag)) continue;
    int nnl = S.NNlen[u], nel = S.NElen[u];
    __align__(16) int nb[MAXW];  // read in chunks below
    int eb[MAXW];
    int nn2 = 0, ne2 = 0;
    bool ok = true;
    // gather the per-entry facts first so that their loads overlap
    RowMask alive, sel;
#pragma unroll 4
    for (int k = 0; k < nel; ++k)
      if (S.EN[c.eb + ne[k]].w) alive.set(k);
#pragma unroll 4
    for (int k = 0; k < nnl; ++k)
      if (smark[c.vb + nn[k]] == tag) sel.set(k);
    for (int k = 0; k < nel; ++k)
      if (alive.test(k)) ok &= sorted_insert(eb, ne2, MAXW, ne[k]);
    for (int k = 0; k < nnl; ++k) {
      int x = nn[k];
      int xs = c.vb + x;
      if (!sel.test(k)) {
        ok &= sorted_insert(nb, nn2, MAXW, x);
        continue;
      }
      int t = target[xs];
      if (t != lu) {
        ok &= sorted_insert(nb, nn2, MAXW, t);
        continue;
      }
      // the collapsed neighbour's rows, read in chunks; its elements'
      // liveness gathered before the merge so that those loads overlap
      int rb[MAXW];
      const int nnxl = S.NNlen[xs];
      load_row(nn_row(S, xs), nnxl, rb);
      for (int j = 0; j < nnxl; ++j)
        if (rb[j] != lu) ok &= sorted_insert(nb, nn2, MAXW, rb[j]);
      const int nexl = S.NElen[xs];
      load_row(ne_row(S, xs), nexl, rb);
      RowMask live;
#pragma unroll 4
      for (int j = 0; j < nexl; ++j)
        if (S.EN[c.eb + rb[j]].w) live.set(j);
      for (int j = 0; j < nexl; ++j)
        if (live.test(j)) ok &= sorted_insert(eb, ne2, MAXW, rb[j]);
    }
    if (!ok || nn2 > S.W || ne2 > S.W) {
      atomicExch(&st->overflow, 1);
      atomicMax(&st->maxdeg, max(nn2, ne2));
      continue;
    }
    int* wn = S.NN + (size_t)u * S.W;
    int* we = S.NE + (size_t)u * S.W;
    for (int k = 0; k < nn2; ++k) wn[k] = nb[k];
    for (int k = 0; k < ne2; ++k) we[k] = eb[k];
    S.NNlen[u] = nn2;
    S.NElen[u] = ne2;
    stamp_neighbours(S, nb, nn2, c.vb, tag + 1);
  }
}

__global__ void k_coarsen_commit(Store S, const int* A, const int* nAp, const int* target,
                                 const int* smark, int tag, DevStatus* st) {
  coarsen_commit_phase(S, A, nAp, target, smark, tag, st);
}

// ---- swapping (Sec. 2.4.3) ------------------------------------------------------

// Balls of at most this many elements take the register path of the flip
// scan (the ball's vertices gathered once); larger ones search the elements.
constexpr int kBallFast = 16;

// A vertex whose ball holds more than kBallFast elements, listed by the whole
// warp (all lanes call): lane l gathers elements l, l + 32, ... into the
// warp's shared arrays and then finds the partner elements of its own poor
// elements there; the same pairs, in the same order per poor element, as the
// register path below.  One such vertex used to hold up its round: one thread
// walked its whole ball for every poor element.

__device__ __forceinline__ void swap_scan_heavy(const Store& S, int v, int* sx, int* sp,
                                                int2* items, int* nI, int icap, double* gains,
                                                DevStatus* st) {
  const int lane = threadIdx.x & 31;
  const MeshCtx c = ctx_of(S, v);
  const int lv = v - c.vb;
  const int* ne = ne_row(S, v);
  const int nel = S.NElen[v];
  const double qt = S.tab.q_thresh[c.mi];
  unsigned pw[MAXW / 32];
#pragma unroll
  for (int j = 0; j < MAXW / 32; ++j) {
    const int k = 32 * j + lane;
    bool poor = false;
    if (k < nel) {
      const int K = ne[k];
      const int4 f = S.EN[c.eb + K];
      sx[k] = (f.x == lv) ? f.y : (f.y == lv) ? f.z : f.x;  // after v
      sp[k] = (f.x == lv) ? f.z : (f.y == lv) ? f.x : f.y;  // before v
      poor = dlt(S.qK[c.eb + K], qt);
      gains[(size_t)v * S.W + k] = -1.0;
    }
    pw[j] = __ballot_sync(0xffffffffu, poor);
  }
  __syncwarp();
  int at = 0;
  for (int pass = 0; pass < 2; ++pass) {  // count, reserve, write
    int cnt = 0;
#pragma unroll
    for (int j = 0; j < MAXW / 32; ++j) {
      const int kb = 32 * j + lane;
      if (kb >= nel || !((pw[j] >> lane) & 1u)) continue;
      const int w = sx[kb], cc = sp[kb];
      int k2 = -1, k1 = -1;
      for (int k = 0; k < nel && (k2 < 0 || k1 < 0); ++k) {  // the first match wins
        if (k == kb) continue;
        if (k2 < 0 && sp[k] == w) k2 = k;
        if (k1 < 0 && sx[k] == cc) k1 = k;
      }
      if (k2 >= 0) {
        if (pass == 1) {
          if (at < icap) items[at] = make_int2(v, kb | (k2 << 8));
          else set_err(st, PM_ERR_CAPACITY);
          ++at;
        }
        ++cnt;
      }
      bool k1poor = false;
#pragma unroll
      for (int jj = 0; jj < MAXW / 32; ++jj)
        if (k1 >= 0 && (k1 >> 5) == jj) k1poor = (pw[jj] >> (k1 & 31)) & 1u;
      if (k1 >= 0 && !k1poor) {
        if (pass == 1) {
          if (at < icap) items[at] = make_int2(v, k1 | (kb << 8));
          else set_err(st, PM_ERR_CAPACITY);
          ++at;
        }
        ++cnt;
      }
    }
    if (pass == 0) at = warp_reserve(cnt, nI);
  }
  __syncwarp();  // the shared arrays serve the next heavy vertex
}

// Flip evaluation in three passes so that the FP64 work runs on full warps.
// Pass 1 (per dirty vertex): reuse an unchanged earlier result, or list the
// vertex's interior edges whose two elements' cached minimum quality is below
// q_thresh and whose flip would not duplicate an edge.
__device__ __forceinline__ void swap_scan_phase(Store S, const int* D, const int* nDp,
                                                const int4* opA, int* C, int* nC, int* cmark,
                                                int tag, int pass0, int* E, int* nE, int2* items,
                                                int* nI, int icap, double* gains, DevStatus* st,
                                                bool il = false) {
  __shared__ int s_hx[kScanWarps][MAXW], s_hp[kScanWarps][MAXW];
  const int wq = (threadIdx.x >> 5) % kScanWarps;
  const int n = *nDp;
  for (int i0 = 0; i0 < n; i0 += gsize()) {
    int i = i0 + grank(il);
    int v = 0, nel = 0;
    bool reuse_cand = false, eval = false;
    MeshCtx c{0, 0, 0};
    const int* ne = nullptr;
    if (i < n) {
      v = D[i];
      c = ctx_of(S, v);
      if (unchanged(S, v, c.vb, S.evs[v], pass0)) {
        reuse_cand = opA[v].x >= 0;
        if (reuse_cand) {
          cmark[v] = tag;
          S.tab.had[c.mi] = 1;
        }
      } else if (S.vflag[v] & VF_ALIVE) {
        eval = true;
        S.evs[v] = tag;
        ne = ne_row(S, v);
        nel = S.NElen[v];
      }
    }
    warp_append(reuse_cand, v, C, nC);
    warp_append(eval, v, E, nE);
    const int lv = v - c.vb;
    const double qt = eval ? S.tab.q_thresh[c.mi] : 0.0;
    // An edge (v, w) qualifies only when one of its two elements has quality
    // below q_thresh, so the pairs are found from v's poor elements alone.
    // Each poor element kb = (v, w, c) gives the pair (kb, k2), k2 the
    // element (v, d, w) after it around v, and the pair (k1, kb), k1 the
    // element before it, when k1 is not poor itself (else that pair is found
    // from k1).  Whether the flipped edge (c, d) already exists is left to
    // the gain evaluation (gain -1): the scan reads no adjacency row, so its
    // loop over the poor elements is register arithmetic.  Items are counted
    // first, reserved with one atomic per warp, then written.
    // balls above kBallFast elements are listed by the whole warp after the
    // register path, which the other lanes take
    const bool heavy = nel > kBallFast;
    const int nfast = heavy ? 0 : nel;
    {
      // the ball's vertices after and before v and its poor elements,
      // gathered once into registers (unrolled: the loads of all elements
      // are in flight together)
      int nx[kBallFast], pv[kBallFast];
      RowMask poor0;
#pragma unroll
      for (int k = 0; k < kBallFast; ++k) {
        nx[k] = pv[k] = -1;
        if (k < nfast) {
          const int K = ne[k];
          const int4 f = S.EN[c.eb + K];
          nx[k] = (f.x == lv) ? f.y : (f.y == lv) ? f.z : f.x;
          pv[k] = (f.x == lv) ? f.z : (f.y == lv) ? f.x : f.y;
          if (dlt(S.qK[c.eb + K], qt)) poor0.set(k);
          gains[(size_t)v * S.W + k] = -1.0;
        }
      }
      // pass 0 counts the items, pass 1 writes them
      int at = 0;
      for (int pass = 0; pass < 2; ++pass) {
        RowMask pm = poor0;
        int cnt = 0;
        while (pm.any()) {
          const int kb = pm.pop();
          int w = -1, cc = -1;
#pragma unroll
          for (int k = 0; k < kBallFast; ++k)
            if (k == kb) {
              w = nx[k];
              cc = pv[k];
            }
          int k2 = -1, k1 = -1;
#pragma unroll
          for (int k = kBallFast - 1; k >= 0; --k) {  // the first match wins
            if (k == kb || k >= nfast) continue;
            if (pv[k] == w) k2 = k;
            if (nx[k] == cc) k1 = k;
          }
          if (k2 >= 0) {
            if (pass == 1) {
              if (at < icap) items[at] = make_int2(v, kb | (k2 << 8));
              else set_err(st, PM_ERR_CAPACITY);
              ++at;
            }
            ++cnt;
          }
          if (k1 >= 0 && !poor0.test(k1)) {
            if (pass == 1) {
              if (at < icap) items[at] = make_int2(v, k1 | (kb << 8));
              else set_err(st, PM_ERR_CAPACITY);
              ++at;
            }
            ++cnt;
          }
        }
        if (pass == 0) at = warp_reserve(cnt, nI);
      }
    }
    for (unsigned hb = __ballot_sync(0xffffffffu, heavy); hb; hb &= hb - 1u) {
      const int hv = __shfl_sync(0xffffffffu, v, __ffs(hb) - 1);
      swap_scan_heavy(S, hv, s_hx[wq], s_hp[wq], items, nI, icap, gains, st);
    }
  }
}

__global__ void k_swap_scan(Store S, const int* D, const int* nDp, const int4* opA, int* C, int* nC,
                            int* cmark, int tag, int pass0, int* E, int* nE, int2* items, int* nI,
                            int icap, double* gains, DevStatus* st) {
  swap_scan_phase(S, D, nDp, opA, C, nC, cmark, tag, pass0, E, nE, items, nI, icap, gains, st);
}

// An edge both of whose end points are evaluated this round is listed from
// both ends with the same two new elements: in canonical rotation their
// qualities and orientations, hence the gain, are bitwise equal from either
// side.  The end point with the smaller id evaluates it and writes the gain
// into both vertices' slots (the other's slot of the same element pair is
// found in its sorted element row); the other item does no arithmetic.
//
// The gain is -1, which the scan has left in its slot, unless both new
// elements are counter-clockwise and their qualities above the old minimum.
// Most items fail one of these, and the FP32 filters decide that (an
// orientation certainly negative, an upper bound of a quality below the old
// minimum) without an FP64 instruction.  What is left is collected in a
// per-warp queue in shared memory and evaluated in FP64, 16 flips at a time:
// two lanes a flip, one new element each, so that a warp's FP64 instructions
// run with all lanes and the two qualities of a flip side by side instead of
// one after the other.
// At most 8 warps per block.
constexpr int kEdgeQueueWarps = 8;

// A queued flip of edge (v, w) between v's ball elements K1 = (v, w, c) and
// K2 = (v, d, w): id = (v, k1 | k2 << 8 | both << 16 | open signs << 17,
// first vertex slot of the mesh, K2), vt = local ids (v, w, c, d).
struct FlipQueue {
  int4 *id, *vt;
  double *qold, *gain;
  int n;  // entries, the same in every lane
};

// One queue per warp, in the block's shared memory.  The callers leave at most
// 15 entries queued between turns and add at most 32 a turn.
__device__ __forceinline__ FlipQueue flip_queue() {
  __shared__ int4 s_id[kEdgeQueueWarps][48];
  __shared__ int4 s_vt[kEdgeQueueWarps][48];
  __shared__ double s_q[kEdgeQueueWarps][48];
  __shared__ double s_g[kEdgeQueueWarps][48];
  const int wq = (threadIdx.x >> 5) % kEdgeQueueWarps;
  return FlipQueue{s_id[wq], s_vt[wq], s_q[wq], s_g[wq], 0};
}

// The FP32 part of the gain of flipping (v, w), K1 = (v, w, c), K2 = (v, d, w)
// (slots and local ids): false when the flip certainly fails, else the queue
// entry of what is left to decide.
__device__ __forceinline__ bool flip_filter(const Store& S, MeshCtx c, int lv, int w, int cc, int d,
                                            int K2, double qold, int low, int4& id, int4& vt) {
  const VF fv = load_vf(S, c.vb + lv), fw = load_vf(S, c.vb + w), fc = load_vf(S, c.vb + cc),
           fd = load_vf(S, c.vb + d);
  // the flipped edge (c, d) must not exist already
  const bool dup = row_has(nn_row(S, c.vb + d), S.NNlen[c.vb + d], cc);
  const float floor = __double2float_rd(qold);
  int s1, s2;
  const float u1 = f_quality_up(fv, fd, fc, s1), u2 = f_quality_up(fd, fw, fc, s2);
  id = make_int4(c.vb + lv, low | ((s1 == 0 ? 1 : 0) << 17) | ((s2 == 0 ? 1 : 0) << 18), c.vb, K2);
  vt = make_int4(lv, w, cc, d);
  return !dup && s1 >= 0 && s2 >= 0 && !(u1 < floor) && !(u2 < floor);
}

// The exact gains of queued flips at..at + 15 (those below n) into Q.gain, -1
// for a flip that fails: flip j on lanes 2 j and 2 j + 1.  All lanes call.
__device__ __forceinline__ void flip_gains16(const Store& S, const FlipQueue& Q, int at, int n,
                                             unsigned& ops) {
  const int lane = threadIdx.x & 31, j = at + (lane >> 1);
  const bool second = lane & 1;  // element (d, w, c); else (v, d, c)
  bool ok = false;
  double q = 0.0;
  if (j < n) {
    const int4 id = Q.id[j], vt = Q.vt[j];
    const int i0 = second ? vt.w : vt.x, i1 = second ? vt.y : vt.w, i2 = vt.z;
    q = quality_c(i0, i1, i2, load_vd(S, id.z + i0), load_vd(S, id.z + i1),
                  load_vd(S, id.z + i2));
    ops += kOpsQuality;
    ok = dgt(q, Q.qold[j]);
    if (ok && ((id.y >> (second ? 18 : 17)) & 1)) {
      ops += kOpsOrient;
      ok = orient_sign(load_xy_again(S, id.z + i0), load_xy_again(S, id.z + i1),
                       load_xy_again(S, id.z + i2)) > 0;
    }
  }
  const unsigned okm = __ballot_sync(0xffffffffu, ok);
  const double q2 = __shfl_xor_sync(0xffffffffu, q, 1);
  if (!second && j < n) {
    const bool both = ((okm >> lane) & 3u) == 3u;
    Q.gain[j] = both ? (dlt(q, q2) ? q : q2) - Q.qold[j] : -1.0;
    ++ops;
  }
  __syncwarp();
}

// Evaluates the first `cnt` (<= 16) queued flips and stores the gains; all
// lanes call.
__device__ __forceinline__ void flip_run(const Store& S, FlipQueue& Q, int cnt, double* gains,
                                         unsigned& ops) {
  const int lane = threadIdx.x & 31;
  flip_gains16(S, Q, 0, cnt, ops);
  if (lane < cnt && dgt(Q.gain[lane], 0.0)) {
    const int4 id = Q.id[lane], vt = Q.vt[lane];
    const double g = Q.gain[lane];
    gains[(size_t)id.x * S.W + (id.y & 0xFF)] = g;
    if ((id.y >> 16) & 1) {
      // from w's side the pair is (K2, K1): w's slot of K2
      const int ws = id.z + vt.y;
      const int kk = row_find(ne_row(S, ws), S.NElen[ws], id.w);
      if (kk >= 0) gains[(size_t)ws * S.W + kk] = g;
    }
  }
  __syncwarp();
  int4 mid = make_int4(0, 0, 0, 0), mvt = mid;
  double mq = 0.0;
  const bool move = lane < Q.n - cnt;
  if (move) {
    mid = Q.id[cnt + lane];
    mvt = Q.vt[cnt + lane];
    mq = Q.qold[cnt + lane];
  }
  __syncwarp();
  if (move) {
    Q.id[lane] = mid;
    Q.vt[lane] = mvt;
    Q.qold[lane] = mq;
  }
  Q.n -= cnt;
  __syncwarp();
}

// Pass 2: the gains, by stages, full warps of items in each.  FP64 in full bound it
// (57 ms of a 512-mesh batch); the FP32 bounds end most items, and the exact rest
// runs at 64 registers, four blocks of 256 an SM (16.5 ms at three, 14.8 at four,
// 17.9 at five, which spill; jittered grids, on the benchmark's regular ones 17.7).
__device__ __forceinline__ void swap_edge_phase(Store S, const int2* items, const int* nIp,
                                                int icap, double* gains, int tag,
                                                unsigned long long* work, bool il = false) {
  const int n = min(*nIp, icap);
  const int lane = threadIdx.x & 31;
  FlipQueue Q = flip_queue();
  unsigned ops = 0;
  for (int i0 = 0; i0 < n; i0 += gsize()) {
    const int i = i0 + grank(il);
    bool need = false;
    int4 id = make_int4(0, 0, 0, 0), vt = make_int4(0, 0, 0, 0);
    double qold = 0.0;
    if (i < n) {
      const int2 it = items[i];
      const int v = it.x, k1 = it.y & 0xFF, k2 = it.y >> 8;
      const MeshCtx c = ctx_of(S, v);
      const int lv = v - c.vb;
      const int* ne = ne_row(S, v);
      const int K1 = ne[k1], K2 = ne[k2];
      const int4 e = S.EN[c.eb + K1], f = S.EN[c.eb + K2];
      const double qa = S.qK[c.eb + K1], qb = S.qK[c.eb + K2];
      const int w = (e.x == lv) ? e.y : (e.y == lv) ? e.z : e.x;
      const int cc = (e.x == lv) ? e.z : (e.y == lv) ? e.x : e.y;
      const int d = (f.x == lv) ? f.y : (f.y == lv) ? f.z : f.x;
      const bool both = S.evs[c.vb + w] == tag;
      if (!both || lv < w) {
        qold = dlt(qa, qb) ? qa : qb;
        need = flip_filter(S, c, lv, w, cc, d, K2, qold,
                           k1 | (k2 << 8) | ((both ? 1 : 0) << 16), id, vt);
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, need);
    if (need) {
      const int at = Q.n + __popc(m & ((1u << lane) - 1u));
      Q.id[at] = id;
      Q.vt[at] = vt;
      Q.qold[at] = qold;
    }
    Q.n += __popc(m);
    __syncwarp();
    while (Q.n >= 16) flip_run(S, Q, 16, gains, ops);
  }
  if (Q.n > 0) flip_run(S, Q, Q.n, gains, ops);
  add_work(work, ops);
}

__global__ void __launch_bounds__(256, 4)
k_swap_edge(Store S, const int2* items, const int* nIp, int icap, double* gains, int tag,
            unsigned long long* work) {
  swap_edge_phase(S, items, nIp, icap, gains, tag, work);
}

// Pass 3 (per evaluated vertex): largest strictly positive gain, ties to the
// smallest w; the flip record (w, c, d, K1, K2) of the winner.
__device__ __forceinline__ void swap_pick_phase(Store S, const int* E, const int* nEp,
                                                const double* gains, int4* opA, int* opK2, int* C,
                                                int* nC, int* cmark, int tag, bool il = false) {
  const int n = *nEp;
  for (int i0 = 0; i0 < n; i0 += gsize()) {
    int i = i0 + grank(il);
    int v = 0;
    bool found = false;
    if (i < n) {
      v = E[i];
      MeshCtx c = ctx_of(S, v);
      int lv = v - c.vb;
      const int* ne = ne_row(S, v);
      int nel = S.NElen[v];
      double best = 0.0;
      int bw = 0, bk = -1;
      if (nel <= kBallFast) {
        // gains, elements and the vertices after and before v gathered in
        // one unrolled pass (all loads in flight together), then decided in
        // registers
        int nx[kBallFast], pv[kBallFast], K[kBallFast];
        double g[kBallFast];
#pragma unroll
        for (int k = 0; k < kBallFast; ++k) {
          nx[k] = pv[k] = K[k] = -1;
          g[k] = -1.0;
          if (k < nel) {
            K[k] = ne[k];
            g[k] = gains[(size_t)v * S.W + k];
            const int4 f = S.EN[c.eb + K[k]];
            nx[k] = (f.x == lv) ? f.y : (f.y == lv) ? f.z : f.x;
            pv[k] = (f.x == lv) ? f.z : (f.y == lv) ? f.x : f.y;
          }
        }
        int bc = 0;
#pragma unroll
        for (int k = 0; k < kBallFast; ++k) {
          if (k < nel && dgt(g[k], 0.0) &&
              (!found || dgt(g[k], best) || (dbits(g[k]) == dbits(best) && nx[k] < bw))) {
            found = true;
            best = g[k];
            bw = nx[k];
            bk = k;
            bc = pv[k];
          }
        }
        if (found) {
          int k2 = -1;
#pragma unroll
          for (int k = kBallFast - 1; k >= 0; --k)  // the first match wins
            if (k < nel && pv[k] == bw) k2 = k;
          int K1 = -1, K2 = -1, d = -1;
#pragma unroll
          for (int k = 0; k < kBallFast; ++k) {
            if (k == bk) K1 = K[k];
            if (k == k2) {
              K2 = K[k];
              d = nx[k];
            }
          }
          opA[v] = make_int4(bw, bc, d, K1);
          opK2[v] = K2;
          cmark[v] = tag;
          S.tab.had[c.mi] = 1;
        } else {
          opA[v].x = -1;
        }
      } else {
#pragma unroll 8
        for (int k = 0; k < nel; ++k) {
          double g = gains[(size_t)v * S.W + k];
          if (!dgt(g, 0.0)) continue;
          int4 e = S.EN[c.eb + ne[k]];
          int w = (e.x == lv) ? e.y : (e.y == lv) ? e.z : e.x;
          if (!found || dgt(g, best) || (dbits(g) == dbits(best) && w < bw)) {
            found = true;
            best = g;
            bw = w;
            bk = k;
          }
        }
        if (found) {
          int4 e = S.EN[c.eb + ne[bk]];
          int cc = (e.x == lv) ? e.z : (e.y == lv) ? e.x : e.y;
          int k2 = -1;
#pragma unroll 8
          for (int k = nel - 1; k >= 0; --k) {  // the first match wins
            int4 f = S.EN[c.eb + ne[k]];
            int pv = (f.x == lv) ? f.z : (f.y == lv) ? f.x : f.y;
            if (pv == bw) k2 = k;
          }
          int4 f = S.EN[c.eb + ne[k2]];
          int d = (f.x == lv) ? f.y : (f.y == lv) ? f.z : f.x;
          opA[v] = make_int4(bw, cc, d, ne[bk]);
          opK2[v] = ne[k2];
          cmark[v] = tag;
          S.tab.had[c.mi] = 1;
        } else {
          opA[v].x = -1;
        }
      }
    }
    warp_append(found, v, C, nC);
  }
}

__global__ void k_swap_pick(Store S, const int* E, const int* nEp, const double* gains, int4* opA,
                            int* opK2, int* C, int* nC, int* cmark, int tag) {
  swap_pick_phase(S, E, nEp, gains, opA, opK2, C, nC, cmark, tag);
}

// Passes 1-3 in one, for persistent rounds whose list fits kFusePasses passes of
// the grid's tiles: lane j of v's tile takes v's ball elements j, j + 8, ... as
// K1 of the edge (v, w) that follows v in it, finds the element K2 = (v, d, w)
// that follows K1 around v among the tile's elements (shuffles), lists the edge
// by pass 1's rule (interior, one of the pair below q_thresh), filters it and,
// when something is left to decide, gets its gain from the warp's queue (pass
// 2); the tile keeps the largest positive gain, ties to the smallest w (pass
// 3's order: a total order, w differs between v's edges).  Each edge of v is
// the K1 edge of exactly one ball element, so the candidate edges are those
// pass 1 lists.  An edge between two listed vertices is evaluated from both
// ends; in exchange a round takes two barriers fewer and no trip of items and
// gains through memory.  A short round is a chain of latencies (about 5 us of this
// phase's 10 are two dependent gathers and the first FP64 stage): 15.8 -> 15.0 ms on
// the 201 x 201 mesh, 17.9 -> 16.4 on 16 small ones against five phases.
__device__ __forceinline__ bool flip_better(bool f2, double g2, int w2, bool f, double g, int w) {
  return f2 && (!f || dgt(g2, g) || (dbits(g2) == dbits(g) && w2 < w));
}

__device__ __forceinline__ void swap_scan_eval_phase(Store S, const int* D, const int* nDp,
                                                     int4* opA, int* opK2, int* C, int* nC,
                                                     int* cmark, int tag, int pass0,
                                                     unsigned long long* work) {
  const Tile t = tile_of();
  const int lane = threadIdx.x & 31;
  FlipQueue Q = flip_queue();
  const int first = first_entry(D, trank(true), S.vslots);
  const int n = *nDp;
  unsigned ops = 0;
  for (int i0 = 0; i0 < n; i0 += tcount()) {
    const int i = i0 + trank(true);
    int v = 0, lv = 0, nel = 0, K0 = 0;
    bool cand = false, eval = false;
    MeshCtx c{0, 0, 0};
    const int* ne = nullptr;
    double qt = 0.0;
    if (i < n) {
      v = i0 == 0 ? first : D[i];
      c = ctx_of(S, v);
      ne = ne_row(S, v);
      // everything the vertex itself holds, in flight together
      const int evs = S.evs[v], tch = S.touch[v], ntch = S.ntouch[v], old = opA[v].x;
      const int len = S.NElen[v];
      K0 = ne[t.tl];
      const bool alive = (S.vflag[v] & VF_ALIVE) != 0;
      const int et = __shfl_sync(t.mask, evs, 0, TW);
      if (et > pass0 && tch <= et && ntch <= et) {  // see unchanged()
        cand = old >= 0;
        if (cand && t.tl == 0) {
          cmark[v] = tag;
          S.tab.had[c.mi] = 1;
        }
      } else if (alive) {
        eval = true;
        lv = v - c.vb;
        nel = len;
        qt = S.tab.q_thresh[c.mi];
      }
    }
    if (eval && t.tl == 0) S.evs[v] = tag;
    const int nelw = __reduce_max_sync(0xffffffffu, nel);
    bool found = false;
    double best = 0.0;
    int bw = 0, bK1 = -1, bK2 = -1, bc = 0, bd = 0;
    for (int base = 0; base < nelw; base += TW) {
      const int k = base + t.tl;
      int K1 = -1, w = -1, cc = -2;
      double q1 = 0.0;
      if (k < nel) {
        K1 = base == 0 ? K0 : ne[k];
        const int4 e = S.EN[c.eb + K1];
        q1 = S.qK[c.eb + K1];
        w = (e.x == lv) ? e.y : (e.y == lv) ? e.z : e.x;   // after v
        cc = (e.x == lv) ? e.z : (e.y == lv) ? e.x : e.y;  // before v
      }
      // K2: the element whose vertex before v is w (one at most)
      int K2 = -1, d = 0;
      double q2 = 0.0;
      for (int other = 0; other < nelw; other += TW) {
        int oK = K1, onx = w, opv = cc;
        double oq = q1;
        if (other != base) {
          oK = -1;
          opv = -2;
          const int ko = other + t.tl;
          if (ko < nel) {
            oK = ne[ko];
            const int4 f = S.EN[c.eb + oK];
            oq = S.qK[c.eb + oK];
            onx = (f.x == lv) ? f.y : (f.y == lv) ? f.z : f.x;
            opv = (f.x == lv) ? f.z : (f.y == lv) ? f.x : f.y;
          }
        }
        int src = -1;
#pragma unroll
        for (int j = TW - 1; j >= 0; --j)
          if (__shfl_sync(0xffffffffu, opv, j, TW) == w) src = j;
        const int from = src >= 0 ? src : 0;
        const int sK = __shfl_sync(0xffffffffu, oK, from, TW);
        const int sd = __shfl_sync(0xffffffffu, onx, from, TW);
        const double sq = __shfl_sync(0xffffffffu, oq, from, TW);
        if (src >= 0 && K2 < 0) {
          K2 = sK;
          d = sd;
          q2 = sq;
        }
      }
      bool need = false;
      int4 id = make_int4(0, 0, 0, 0), vt = id;
      double qold = 0.0;
      if (k < nel && K2 >= 0 && K2 != K1 && (dlt(q1, qt) || dlt(q2, qt))) {
        qold = dlt(q1, q2) ? q1 : q2;
        need = flip_filter(S, c, lv, w, cc, d, K2, qold, 0, id, vt);
      }
      const unsigned m = __ballot_sync(0xffffffffu, need);
      const int at = __popc(m & ((1u << lane) - 1u)), cnt = __popc(m);
      if (need) {
        Q.id[at] = id;
        Q.vt[at] = vt;
        Q.qold[at] = qold;
      }
      __syncwarp();
      for (int b = 0; b < cnt; b += 16) flip_gains16(S, Q, b, cnt, ops);
      if (need) {
        const double g = Q.gain[at];
        if (dgt(g, 0.0) && flip_better(true, g, w, found, best, bw)) {
          found = true;
          best = g;
          bw = w;
          bK1 = K1;
          bK2 = K2;
          bc = cc;
          bd = d;
        }
      }
      __syncwarp();
    }
    // the tile's best: lane `src` holds it
    int src = t.tl;
#pragma unroll
    for (int o = TW / 2; o > 0; o >>= 1) {
      const bool f2 = __shfl_xor_sync(0xffffffffu, found ? 1 : 0, o, TW) != 0;
      const double g2 = __shfl_xor_sync(0xffffffffu, best, o, TW);
      const int w2 = __shfl_xor_sync(0xffffffffu, bw, o, TW);
      const int s2 = __shfl_xor_sync(0xffffffffu, src, o, TW);
      if (flip_better(f2, g2, w2, found, best, bw)) {
        found = true;
        best = g2;
        bw = w2;
        src = s2;
      }
    }
    if (eval) {
      if (found && src == t.tl) {
        opA[v] = make_int4(bw, bc, bd, bK1);
        opK2[v] = bK2;
        cmark[v] = tag;
        S.tab.had[c.mi] = 1;
      }
      if (!found && t.tl == 0) opA[v].x = -1;
      cand = found;
    }
    warp_append(cand && t.tl == 0, v, C, nC);
  }
  add_work(work, ops);
}

// One round's independent set and its flips (see k_coarsen_select_apply).
// The two new elements' qualities are left to a dense pass (their slots join
// list Q), as for collapses.
__device__ __forceinline__ void swap_select_apply_phase(Store S, const int* C, const int* nCp,
                                                        const int* cmark, int* smark, int tag,
                                                        const int4* opA, const int* opK2, int* A,
                                                        int* nA, int* amark, int* Dn, int* nDn,
                                                        int* dmark, int* Q, int* nQ,
                                                        bool il = false) {
  const int first = first_entry(C, grank(il), S.vslots);
  const int n = *nCp;
  for (int i0 = 0; i0 < n; i0 += gsize()) {
    int i = i0 + grank(il);
    bool win = false, lose = false;
    int v = 0, mi = 0, q1 = 0, q2 = 0;
    int t[4] = {0, 0, 0, 0};
    bool fa[4] = {false, false, false, false}, fd[4] = {false, false, false, false};
    if (i < n) {
      v = i0 == 0 ? first : C[i];
      const int4 op = opA[v];
      const int K2 = opK2[v];
      win = local_max(S, v, cmark, tag);
      if (win) {
        smark[v] = tag;
        const MeshCtx c = ctx_of(S, v);
        mi = c.mi;
        const int lv = v - c.vb;
        q1 = c.eb + op.w;
        q2 = c.eb + K2;
        S.EN[q1] = make_int4(lv, op.z, op.y, 1);    // K1 = (v, d, c)
        S.EN[q2] = make_int4(op.z, op.x, op.y, 1);  // K2 = (d, w, c)
        t[0] = v;
        t[1] = c.vb + op.x;
        t[2] = c.vb + op.y;
        t[3] = c.vb + op.z;
        int oa[4], od[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          oa[k] = atomicExch(amark + t[k], tag);
          od[k] = atomicExch(dmark + t[k], tag);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          fa[k] = oa[k] != tag;
          fd[k] = od[k] != tag;
        }
      } else {
        lose = stamp_first(dmark, v, tag);
      }
    }
    count_op(S, win, mi);
    int na = 0, nd = lose ? 1 : 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      na += fa[k];
      nd += fd[k];
    }
    Room3 at = warp_reserve3(na, nA, nd, nDn, win ? 2 : 0, nQ);
    if (lose) Dn[at.b] = v;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (fa[k]) A[at.a++] = t[k];
      if (fd[k]) Dn[at.b++] = t[k];
    }
    if (win) {
      Q[at.c] = q1;
      Q[at.c + 1] = q2;
    }
  }
}

__global__ void k_swap_select_apply(Store S, const int* C, const int* nCp, const int* cmark,
                                    int* smark, int tag, const int4* opA, const int* opK2, int* A,
                                    int* nA, int* amark, int* Dn, int* nDn, int* dmark, int* Q,
                                    int* nQ, unsigned* done) {
  swap_select_apply_phase(S, C, nCp, cmark, smark, tag, opA, opK2, A, nA, amark, Dn, nDn, dmark,
                          Q, nQ);
  round_done(S, done);
}

// The commit below for rows of at most 16 entries that stay so (see
// coarsen_commit_short).
__device__ __forceinline__ bool swap_commit_short(const Store& S, int u, MeshCtx c, int lu,
                                                  const int4* opA, const int* opK2,
                                                  const int* smark, int tag) {
  int* nn = S.NN + (size_t)u * S.W;
  int* ne = S.NE + (size_t)u * S.W;
  const int nnl = S.NNlen[u], nel = S.NElen[u], own = smark[u];
  Row16 R, Q;
  R.load(nn, nnl);
  Q.load(ne, nel);
  if (nnl > kRowReg || nel > kRowReg) return false;
  unsigned sel = own == tag ? 1u << kRowReg : 0u;
#pragma unroll
  for (int k = 0; k < kRowReg; ++k)
    if (k < nnl && smark[c.vb + R.a[k]] == tag) sel |= 1u << k;
  bool ok = true;
  for (; sel && ok; sel &= sel - 1u) {
    const int k = __ffs(sel) - 1;
    const int x = k == kRowReg ? lu : nn[k];
    const int4 op = opA[c.vb + x];
    const int K2 = opK2[c.vb + x];
    // u is v (x itself), w, c or d of the flip, or not in it
    if (x == lu || op.x == lu) {
      R.erase(x == lu ? op.x : x);
      Q.erase(x == lu ? K2 : op.w);
    } else if (op.y == lu || op.z == lu) {
      ok = R.insert(op.y == lu ? op.z : op.y);
      ok &= Q.insert(op.y == lu ? K2 : op.w);
    }
  }
  if (!ok) return false;
  const int nn2 = R.len(), ne2 = Q.len();
  R.store(nn, nn2);
  Q.store(ne, ne2);
  S.NNlen[u] = nn2;
  S.NElen[u] = ne2;
#pragma unroll
  for (int k = 0; k < kRowReg; ++k)
    if (k < nn2) S.ntouch[c.vb + R.a[k]] = tag + 1;
  return true;
}

// Deferred-update commit of a swap round for affected vertex u, from the
// flips of u itself and of its S neighbours (records w, c, d, K1, K2):
//   u == v: NN -w, NE -K2;  u == w: NN -v, NE -K1;
//   u == c: NN +d, NE +K2;  u == d: NN +c, NE +K1.
__device__ __forceinline__ void swap_commit_phase(Store S, const int* A, const int* nAp,
                                                  const int4* opA, const int* opK2,
                                                  const int* smark, int tag, DevStatus* st,
                                                  bool il = false) {
  const int first = first_entry(A, grank(il), S.vslots);
  const int n = *nAp;
  for (int i = grank(il); i < n; i += gsize()) {
    const int u = i < gsize() ? first : A[i];
    S.touch[u] = tag + 1;
    MeshCtx c = ctx_of(S, u);
    int lu = u - c.vb;
    int* nn = S.NN + (size_t)u * S.W;
    int* ne = S.NE + (size_t)u * S.W;
    if (swap_commit_short(S, u, c, lu, opA, opK2, smark, tag)) continue;
    int nnl = S.NNlen[u], nel = S.NElen[u];
    __align__(16) int nb[MAXW];  // read in chunks below
    int eb[MAXW];
    load_row(nn, nnl, nb);
    load_row(ne, nel, eb);
    int nn2 = nnl, ne2 = nel;
    bool ok = true;
    RowMask sel;
#pragma unroll 4
    for (int k = 0; k < nnl; ++k)
      if (smark[c.vb + nn[k]] == tag) sel.set(k);
    const bool self = smark[u] == tag;
    for (int k = -1; k < nnl; ++k) {
      if (k < 0 ? !self : !sel.test(k)) continue;
      int x = (k < 0) ? lu : nn[k];
      int xs = c.vb + x;
      int4 op = opA[xs];
      int K2 = opK2[xs];
      if (x == lu) {
        sorted_erase(nb, nn2, op.x);
        sorted_erase(eb, ne2, K2);
      }
      if (op.x == lu) {
        sorted_erase(nb, nn2, x);
        sorted_erase(eb, ne2, op.w);
      }
      if (op.y == lu) {
        ok &= sorted_insert(nb, nn2, MAXW, op.z);
        ok &= sorted_insert(eb, ne2, MAXW, K2);
      }
      if (op.z == lu) {
        ok &= sorted_insert(nb, nn2, MAXW, op.y);
        ok &= sorted_insert(eb, ne2, MAXW, op.w);
      }
    }
    if (!ok || nn2 > S.W || ne2 > S.W) {
      atomicExch(&st->overflow, 1);
      atomicMax(&st->maxdeg, max(nn2, ne2));
      continue;
    }
    for (int k = 0; k < nn2; ++k) nn[k] = nb[k];
    for (int k = 0; k < ne2; ++k) ne[k] = eb[k];
    S.NNlen[u] = nn2;
    S.NElen[u] = ne2;
    stamp_neighbours(S, nb, nn2, c.vb, tag + 1);
  }
}

__global__ void k_swap_commit(Store S, const int* A, const int* nAp, const int4* opA,
                              const int* opK2, const int* smark, int tag, DevStatus* st) {
  swap_commit_phase(S, A, nAp, opA, opK2, smark, tag, st);
}

// ---- smoothing (Sec. 2.4.4) -------------------------------------------------------

__device__ __forceinline__ double ball_min_quality(const Store& S, MeshCtx c, const int* ne,
                                                   int nel, double* qsum) {
  double qmin = 0.0, sum = 0.0;
#pragma unroll 4
  for (int k = 0; k < nel; ++k) {
    double q = S.qK[c.eb + ne[k]];
    if (k == 0 || dlt(q, qmin)) qmin = q;
    sum = sum + q;
  }
  if (qsum) *qsum = sum;
  return qmin;
}

// The w of a stored move (mvM): 0 no move; 1 its new ball qualities are stored too;
// 2 it certainly holds and they are evaluated after the move.  The last only in the
// rounds with a kernel per phase, whose filter leaves them open (`defer`): in a
// persistent round they would be one more phase and barrier, which lost 1% on
// meshes of up to 130k triangles; it evaluates again what it finds of them.
constexpr double kMoveEvaluated = 1.0, kMoveUnevaluated = 2.0;

// Smoothing evaluation in two passes.  Pass 1 (per pending vertex): reuse an
// unchanged earlier result, drop vertices whose ball is already good enough
// (cached qualities), list the rest for the full move evaluation.
__device__ __forceinline__ void smooth_scan_phase(Store S, const int* D, const int* nDp,
                                                  double4* mvM, int* C, int* nC, int* cmark,
                                                  int tag, int pass0, int* E, int* nE,
                                                  bool defer, bool il = false) {
  const int n = *nDp;
  for (int i0 = 0; i0 < n; i0 += gsize()) {
    int i = i0 + grank(il);
    int v = 0;
    bool reuse_cand = false, eval = false;
    if (i < n) {
      v = D[i];
      MeshCtx c = ctx_of(S, v);
      const double move = mvM[v].w;
      if (unchanged(S, v, c.vb, S.evm[v], pass0) && (defer || move != kMoveUnevaluated)) {
        reuse_cand = move != 0.0;
        if (reuse_cand) {
          cmark[v] = tag;
          S.tab.had[c.mi] = 1;
        }
      } else {
        S.evm[v] = tag;
        uint8_t f = S.vflag[v];
        if ((f & VF_ALIVE) && !(f & VF_BND)) {
          double qold = ball_min_quality(S, c, ne_row(S, v), S.NElen[v], nullptr);
          eval = dlt(qold, S.tab.q_thresh[c.mi]);
        }
        if (!eval) mvM[v].w = 0.0;
      }
    }
    warp_append(reuse_cand, v, C, nC);
    warp_append(eval, v, E, nE);
  }
}

__global__ void __launch_bounds__(256, 3)
k_smooth_scan(Store S, const int* D, const int* nDp, double4* mvM, int* C, int* nC, int* cmark,
              int tag, int pass0, int* E, int* nE) {
  smooth_scan_phase(S, D, nDp, mvM, C, nC, cmark, tag, pass0, E, nE, true);
}

// Minimum cached quality of v's ball (and, if asked, its sum in ascending
// element order).
__device__ double tile_ball_quality(const Tile& t, const Store& S, MeshCtx c, const int* ne,
                                    int nel, double* qsum) {
  double qmin = 1e300, sum = 0.0;
  for (int base = 0; base < nel; base += TW) {
    int k = base + t.tl;
    double q = (k < nel) ? S.qK[c.eb + ne[k]] : 1e300;
    qmin = dlt(q, qmin) ? q : qmin;
    if (qsum) {
      int cnt = min(TW, nel - base);
      for (int j = 0; j < cnt; ++j) sum = sum + tshfl(t, q, j);
    }
  }
  if (qsum) *qsum = sum;
  return tmin(t, qmin);
}

// Whether the closed element (a, b, d) contains X = px: the FP32 filters of the
// three sub-triangles first; a sign they leave open is taken exactly, unless
// another one is negative.
__device__ __forceinline__ bool contains(const Store& S, const VF& fx, double X, double Y, int sa,
                                         int sb, int sd) {
  const VF fa = load_vf(S, sa), fb = load_vf(S, sb), fd = load_vf(S, sd);
  const int f0 = f_orient(fx, fb, fd), f1 = f_orient(fa, fx, fd), f2 = f_orient(fa, fb, fx);
  if ((f0 | f1 | f2) < 0) return false;
  if (f0 > 0 && f1 > 0 && f2 > 0) return true;
  const VD px{X, Y, 0.0, 0.0, 0.0}, a = load_vd(S, sa), b = load_vd(S, sb), d = load_vd(S, sd);
  if (f0 == 0 && orient_sign(px, b, d) < 0) return false;
  if (f1 == 0 && orient_sign(a, px, d) < 0) return false;
  return f2 != 0 || orient_sign(a, b, px) >= 0;
}

// Barycentric interpolation of the metric at X in element e (canonical
// rotation).
__device__ __forceinline__ double4 interpolate_in(const Store& S, int vb, int4 e, double X,
                                                  double Y) {
  const VD px{X, Y, 0.0, 0.0, 0.0};
  int i0 = e.x, i1 = e.y, i2 = e.z;
  VD a = load_vd(S, vb + i0), b = load_vd(S, vb + i1), d = load_vd(S, vb + i2);
  canon(i0, i1, i2, a, b, d);
  const double o = orient3(a, b, d);
  const double l0 = orient3(px, b, d) / o, l1 = orient3(a, px, d) / o, l2 = orient3(a, b, px) / o;
  return make_double4((l0 * a.m00 + l1 * b.m00) + l2 * d.m00,
                      (l0 * a.m01 + l1 * b.m01) + l2 * d.m01,
                      (l0 * a.m11 + l1 * b.m11) + l2 * d.m11, 0.0);
}

// The same by the lanes of a tile, which all hold e: lanes 0 to 3 take one of the
// four areas each, lanes 0 to 2 one weight and one entry (about 24 FP64
// instructions of the warp instead of 73, the values by the same operations).
__device__ __forceinline__ double4 tile_interpolate_in(const Tile& t, const Store& S, int vb, int4 e,
                                                       double X, double Y) {
  const VD px{X, Y, 0.0, 0.0, 0.0};
  int i0 = e.x, i1 = e.y, i2 = e.z;
  VD a = load_vd(S, vb + i0), b = load_vd(S, vb + i1), d = load_vd(S, vb + i2);
  canon(i0, i1, i2, a, b, d);
  const double det = orient3(t.tl == 0 ? px : a, t.tl == 1 ? px : b, t.tl == 2 ? px : d);
  const double l = det / tshfl(t, det, 3);
  const double l0 = tshfl(t, l, 0), l1 = tshfl(t, l, 1), l2 = tshfl(t, l, 2);
  const double ma = t.tl == 0 ? a.m00 : (t.tl == 1 ? a.m01 : a.m11);
  const double mb = t.tl == 0 ? b.m00 : (t.tl == 1 ? b.m01 : b.m11);
  const double md = t.tl == 0 ? d.m00 : (t.tl == 1 ? d.m01 : d.m11);
  const double m = (l0 * ma + l1 * mb) + l2 * md;
  return make_double4(tshfl(t, m, 0), tshfl(t, m, 1), tshfl(t, m, 2), 0.0);
}

// Bounds of the quality of element e of v's ball with v at the record `fn`
// (relative error kx of its metric): the upper one is -1 when it is certainly not
// counter-clockwise, NaN when there is no useful bound; the lower one is -1 unless it
// is certainly counter-clockwise and the bound useful.
__device__ __forceinline__ FQual moved_quality(const Store& S, int vb, int lv, int4 e,
                                                  const VF& fn, float kx) {
  const VF a = e.x == lv ? fn : load_vf(S, vb + e.x), b = e.y == lv ? fn : load_vf(S, vb + e.y),
           c = e.z == lv ? fn : load_vf(S, vb + e.z);
  int sign;
  FQual q = f_quality(a, b, c, sign, kx);
  if (sign < 0) q.up = -1.0f;
  return q;
}

// The FP32 metric at X in element e into fn, its relative error bound.
__device__ __forceinline__ float metric_at(const Store& S, int vb, int4 e, const VF& fx, VF& fn) {
  fn = fx;
  return f_metric_at(fx, load_vf(S, vb + e.x), load_vf(S, vb + e.y), load_vf(S, vb + e.z), fn);
}

// Ball with v moved to (X, Y, Mv): every element counter-clockwise, and every
// quality above *floor (strict) or at least *floor (non-strict).  Writes each
// element's new quality to qout[k] and returns the ascending-order sum.
__device__ bool tile_ball_exact(const Tile& t, const Store& S, MeshCtx c, int lv,
                                const int* ne, int nel, double X, double Y, double4 Mv,
                                double floor, bool strict, double* qout, double* qsum) {
  VD nvd{X, Y, Mv.x, Mv.y, Mv.z};
  bool ok = true;
  double sum = 0.0;
  for (int base = 0; base < nel; base += TW) {
    int k = base + t.tl;
    double q = 0.0;
    if (k < nel) {
      int4 e = S.EN[c.eb + ne[k]];
      VD a = (e.x == lv) ? nvd : load_vd(S, c.vb + e.x);
      VD b = (e.y == lv) ? nvd : load_vd(S, c.vb + e.y);
      VD d = (e.z == lv) ? nvd : load_vd(S, c.vb + e.z);
      if (orient_sign(a, b, d) > 0) {
        q = quality_c(e.x, e.y, e.z, a, b, d);
        if (strict ? !dgt(q, floor) : dlt(q, floor)) ok = false;
        if (qout) qout[k] = q;
      } else {
        ok = false;
      }
    }
    if (qsum) {
      int cnt = min(TW, nel - base);
      for (int j = 0; j < cnt; ++j) sum = sum + tshfl(t, q, j);
    }
  }
  if (qsum) *qsum = sum;
  return tall(t, ok);
}

// A move of v to X, by v's tile: located in the first ball element (ascending
// id) that contains X with v at its current place, its metric interpolated there,
// and the ball checked.  Most moves fail, and the FP32 bounds mostly show it
// before the metric is interpolated in FP64: a quality certainly below `floor`,
// or (with qsum) a sum of the upper bounds below `sum_old`.
__device__ bool tile_try_move(const Tile& t, const Store& S, MeshCtx c, int lv, const int* ne,
                              int nel, double X, double Y, double floor, bool strict, double* qout,
                              double* qsum, double sum_old, double4& Mout, unsigned& ops) {
  const VF fx = make_vf_xy(X, Y);
  int4 eat = make_int4(0, 0, 0, 0);
  int src = -1;
  for (int base = 0; base < nel && src < 0; base += TW) {
    const int k = base + t.tl;
    bool inside = false;
    if (k < nel) {
      eat = S.EN[c.eb + ne[k]];
      inside = contains(S, fx, X, Y, c.vb + eat.x, c.vb + eat.y, c.vb + eat.z);
    }
    const unsigned bal = (__ballot_sync(t.mask, inside) >> t.shift) & 0xFFu;
    if (bal) src = __ffs(bal) - 1;
  }
  if (src < 0) return false;
  eat.x = __shfl_sync(t.mask, eat.x, src, TW);
  eat.y = __shfl_sync(t.mask, eat.y, src, TW);
  eat.z = __shfl_sync(t.mask, eat.z, src, TW);
  VF fn;
  const float kx = metric_at(S, c.vb, eat, fx, fn);
  const float ffloor = __double2float_rd(floor);
  bool fails = false;
  float up = 0.0f;
  for (int k = t.tl; k < nel; k += TW) {
    const float u = moved_quality(S, c.vb, lv, S.EN[c.eb + ne[k]], fn, kx).up;
    fails |= u < ffloor;
    up += u;
  }
  if (!tall(t, !fails)) return false;
  if (qsum) {
#pragma unroll
    for (int o = TW / 2; o > 0; o >>= 1) up += __shfl_xor_sync(t.mask, up, o, TW);
    // (the sum of at most 128 bounds is short by 128 u of itself at most)
    if (up * 1.00001f < __double2float_rd(sum_old)) return false;
  }
  Mout = tile_interpolate_in(t, S, c.vb, eat, X, Y);
  if (t.tl == 0) ops += 46 + 85 * nel;
  return tile_ball_exact(t, S, c, lv, ne, nel, X, Y, Mout, floor, strict, qout, qsum);
}

// Quality-constrained Laplacian move of v: metric-weighted neighbour mean,
// metric interpolated at the target, kept when the ball stays valid and its
// minimum quality strictly increases.
// `ops` receives the FP64 operations (+ - * / sqrt) of the path taken: 17 per
// neighbour (Laplacian), 11 (solve), 46 (barycentrics and metric) and 85 per
// element of the ball of an accepted move (orientation and quality).
__device__ bool tile_smooth_eval(const Tile& t, const Store& S, int v, MeshCtx c, double2& Xo,
                                 double4& Mo, double* qout, unsigned& ops) {
  uint8_t f = S.vflag[v];
  if (!(f & VF_ALIVE) || (f & VF_BND)) return false;
  const int* ne = ne_row(S, v);
  int nel = S.NElen[v];
  double qold = tile_ball_quality(t, S, c, ne, nel, nullptr);
  if (!dlt(qold, S.tab.q_thresh[c.mi])) return false;
  const int* nn = nn_row(S, v);
  int nnl = S.NNlen[v];
  double4 mv = S.M[v];
  // Five ordered sums over the neighbours, one on each of five lanes (through
  // shared memory: a sixth of the FP64 instructions of every lane adding all
  // five), then x on the even lanes and y on the odd ones.
  __shared__ double s_lap[kTileMax][TW][5];
  double (*lap)[5] = s_lap[(threadIdx.x / TW) % kTileMax];
  double acc = 0.0;
  for (int base = 0; base < nnl; base += TW) {
    const int k = base + t.tl;
    if (k < nnl) {
      const int js = c.vb + nn[k];
      const double2 pj = S.xy[js];
      const double4 mj = S.M[js];
      const double w00 = 0.5 * (mv.x + mj.x);
      const double w01 = 0.5 * (mv.y + mj.y);
      const double w11 = 0.5 * (mv.z + mj.z);
      lap[t.tl][0] = w00;
      lap[t.tl][1] = w01;
      lap[t.tl][2] = w11;
      lap[t.tl][3] = w00 * pj.x + w01 * pj.y;
      lap[t.tl][4] = w01 * pj.x + w11 * pj.y;
    }
    __syncwarp(t.mask);
    const int cnt = min(TW, nnl - base);
    if (t.tl < 5)
      for (int j = 0; j < cnt; ++j) acc = acc + lap[j][t.tl];
    __syncwarp(t.mask);
  }
  const double a00 = tshfl(t, acc, 0), a01 = tshfl(t, acc, 1), a11 = tshfl(t, acc, 2),
               b0 = tshfl(t, acc, 3), b1 = tshfl(t, acc, 4);
  if (t.tl == 0) ops += 17 * nnl + 3;
  const double det = a00 * a11 - a01 * a01;
  if (!dgt(det, 0.0)) return false;
  const bool odd = t.tl & 1;
  const double z = ((odd ? a00 : a11) * (odd ? b1 : b0) - a01 * (odd ? b0 : b1)) / det;
  const double x = tshfl(t, z, 0), y = tshfl(t, z, 1);
  if (t.tl == 0) ops += 8;
  Xo = make_double2(x, y);
  return tile_try_move(t, S, c, v - c.vb, ne, nel, x, y, qold, true, qout, nullptr, 0.0, Mo, ops);
}

// Pass 2 of the longer lists, one listed vertex per thread: the Laplacian sums,
// the 2x2 solve, the location and the interpolation run per thread (a tile of
// lanes per vertex repeats them in every lane: four vertices per warp instruction
// of FP64 instead of 32), and the FP32 bounds of the moved ball (its metric
// interpolated in FP32 first) drop the moves that certainly fail.  With `defer` those
// that certainly hold become candidates at once: their new qualities are evaluated
// when the move is made (half the candidates lose to a neighbour, and most of those
// are evaluated again after it has moved).  The others are listed for pass 3.
// The sums' and the solve's FP64 bounds it (pipe 76% active; the FP32 bounds run
// beside them).  Steps on 20M triangles, whole adaptation: a tile of lanes for all
// 171 ms, a thread per vertex and the filter 152, two passes 105, `defer` 87.9 -> 83.8.
__device__ __forceinline__ void smooth_filter_phase(Store S, const int* E, const int* nEp,
                                                    double2* mvxy, double4* mvM, int* R, int* nR,
                                                    int* C, int* nC, int* cmark, int tag,
                                                    bool defer, unsigned long long* work,
                                                    bool il = false) {
  const int first = first_entry(E, grank(il), S.vslots);
  const int n = *nEp;
  unsigned ops = 0;
  for (int j0 = 0; j0 < n; j0 += gsize()) {
    const int j = j0 + grank(il);
    int v = 0;
    bool may = false, sure = defer;
    if (j < n) {
      v = j0 == 0 ? first : E[j];
      const MeshCtx c = ctx_of(S, v);
      const int lv = v - c.vb;
      const int* ne = ne_row(S, v);
      const int nel = S.NElen[v];
      const int* nn = nn_row(S, v);
      const int nnl = S.NNlen[v];
      double qold = 1e300;
      for (int b = 0; b < nel; b += 8) {
        const Row8 r = row8(ne, b);
        double q[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) q[k] = b + k < nel ? S.qK[c.eb + r.a[k]] : 1e300;
#pragma unroll
        for (int k = 0; k < 8; ++k) qold = dlt(q[k], qold) ? q[k] : qold;
      }
      const double4 mv = S.M[v];
      double a00 = 0.0, a01 = 0.0, a11 = 0.0, b0 = 0.0, b1 = 0.0;
      for (int b = 0; b < nnl; b += 4) {
        const int4 r4 = *reinterpret_cast<const int4*>(nn + b);
        const int u4[4] = {r4.x, r4.y, r4.z, r4.w};
        double2 p[4];
        double4 mj[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int js = b + k < nnl ? c.vb + u4[k] : v;
          p[k] = S.xy[js];
          mj[k] = S.M[js];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (b + k >= nnl) continue;
          const double w00 = 0.5 * (mv.x + mj[k].x);
          const double w01 = 0.5 * (mv.y + mj[k].y);
          const double w11 = 0.5 * (mv.z + mj[k].z);
          a00 = a00 + w00;
          a01 = a01 + w01;
          a11 = a11 + w11;
          b0 = b0 + (w00 * p[k].x + w01 * p[k].y);
          b1 = b1 + (w01 * p[k].x + w11 * p[k].y);
        }
      }
      const double det = a00 * a11 - a01 * a01;
      ops += 17 * nnl + 3;
      if (dgt(det, 0.0)) {
        const double x = (a11 * b0 - a01 * b1) / det;
        const double y = (a00 * b1 - a01 * b0) / det;
        ops += 8;
        const VF fx = make_vf_xy(x, y);
        int4 e = make_int4(0, 0, 0, 0);
        for (int k = 0; k < nel && !may; ++k) {
          e = S.EN[c.eb + ne[k]];
          may = contains(S, fx, x, y, c.vb + e.x, c.vb + e.y, c.vb + e.z);
        }
        if (may) {
          VF fn;
          const float kx = metric_at(S, c.vb, e, fx, fn);
          const float ffloor = __double2float_rd(qold), fceil = __double2float_ru(qold);
#pragma unroll 2
          for (int k = 0; k < nel; ++k)
            if (may) {
              const FQual q = moved_quality(S, c.vb, lv, S.EN[c.eb + ne[k]], fn, kx);
              may = !(q.up < ffloor);
              sure = sure && q.lo > fceil;
            }
          if (may) {
            double4 Mn = interpolate_in(S, c.vb, e, x, y);
            ops += 46;
            Mn.w = sure ? kMoveUnevaluated : qold;  // (for pass 3)
            if (sure) {
              cmark[v] = tag;
              S.tab.had[c.mi] = 1;
            }
            mvxy[v] = make_double2(x, y);
            mvM[v] = Mn;
          }
        }
      }
      if (!may) mvM[v].w = 0.0;
    }
    const Room3 at = warp_reserve3(may && !sure ? 1 : 0, nR, may && sure ? 1 : 0, nC, 0, nullptr);
    if (may && !sure) R[at.a] = v;
    if (may && sure) C[at.b] = v;
  }
  add_work(work, ops);
}

// Pass 3 (one 8-lane tile per move that may succeed): the exact ball check.
// Every value of a move is computed by the same operations in the same order as
// in tile_smooth_eval.
__device__ __forceinline__ void smooth_exact_phase(Store S, const int* R, const int* nRp,
                                                   const double2* mvxy, double4* mvM,
                                                   double* qball, int* C, int* nC, int* cmark,
                                                   int tag, unsigned long long* work,
                                                   bool il = false) {
  const Tile t = tile_of();
  const int first = first_entry(R, trank(il), S.vslots);
  const int n = *nRp;
  unsigned ops = 0;
  for (int j0 = 0; j0 < n; j0 += tcount()) {
    const int j = j0 + trank(il);
    int v = 0;
    bool cand = false;
    if (j < n) {
      v = j0 == 0 ? first : R[j];
      const MeshCtx c = ctx_of(S, v);
      const int nel = S.NElen[v];
      const double2 X = mvxy[v];
      const double4 Mn = mvM[v];
      // the new ball qualities of an accepted move are kept for the apply
      cand = tile_ball_exact(t, S, c, v - c.vb, ne_row(S, v), nel, X.x, X.y, Mn, Mn.w, true,
                             qball + (size_t)v * S.W, nullptr);
      if (t.tl == 0) {
        ops += 85 * nel;
        mvM[v].w = cand ? kMoveEvaluated : 0.0;
        if (cand) {
          cmark[v] = tag;
          S.tab.had[c.mi] = 1;
        }
      }
    }
    warp_append(cand && t.tl == 0, v, C, nC);
  }
  add_work(work, ops);
}

// Passes 1 to 3 in one (persistent rounds whose list fits kFusePasses passes of the
// grid's tiles): an evaluation whose inputs carry no newer stamp stands, the
// others are made again.  The tile takes the stamp decision from lane 0, after every
// lane has read the stamp (the shuffle) and before lane 0 overwrites it.
__device__ __forceinline__ void smooth_scan_eval_phase(Store S, const int* D, const int* nDp,
                                                       double2* mvxy, double4* mvM, double* qball,
                                                       int* C, int* nC, int* cmark, int tag,
                                                       int pass0, unsigned long long* work) {
  const Tile t = tile_of();
  const int tile_rank = (threadIdx.x / TW) * gridDim.x + blockIdx.x;
  const int tiles = gridDim.x * (blockDim.x / TW);
  const int first = first_entry(D, tile_rank, S.vslots);
  const int n = *nDp;
  unsigned ops = 0;
  for (int j0 = 0; j0 < n; j0 += tiles) {
    int j = j0 + tile_rank;
    int v = 0;
    bool cand = false;
    if (j < n) {
      v = j0 == 0 ? first : D[j];
      MeshCtx c = ctx_of(S, v);
      const double move = mvM[v].w;
      bool keep = unchanged(S, v, c.vb, S.evm[v], pass0) && move != kMoveUnevaluated;
      keep = __shfl_sync(t.mask, keep, 0, TW);
      if (keep) {
        if (t.tl == 0) {
          cand = move != 0.0;
          if (cand) {
            cmark[v] = tag;
            S.tab.had[c.mi] = 1;
          }
        }
      } else {
        double2 X;
        double4 Mv;
        cand = tile_smooth_eval(t, S, v, c, X, Mv, qball + (size_t)v * S.W, ops);
        if (t.tl == 0) {
          S.evm[v] = tag;
          if (cand) {
            Mv.w = kMoveEvaluated;
            mvxy[v] = X;
            mvM[v] = Mv;
            cmark[v] = tag;
            S.tab.had[c.mi] = 1;
          } else {
            mvM[v].w = 0.0;
          }
        }
      }
    }
    warp_append(cand && t.tl == 0, v, C, nC);
  }
  add_work(work, ops);
}

// Pass 3 of the large rounds: the same with the ball elements of five or so moves
// side by side in a warp (a tile of 8 lanes per move leaves a quarter of them idle
// at six elements a ball, and the FP64 pipe is what bounds this pass).  Each warp
// walks a range of the list and takes as many moves at a time as fit 32 lanes; a
// ball of more than 32 elements takes the warp alone.  FP64 pipe 84% active; with the
// ordered sums of the tile form 94.8 -> 91.4 ms on 20M triangles.
__device__ __forceinline__ void smooth_exact_packed(Store S, const int* R, const int* nRp,
                                                    const double2* mvxy, double4* mvM,
                                                    double* qball, int* C, int* nC, int* cmark,
                                                    int tag, unsigned long long* work) {
  const int n = *nRp;
  const int lane = threadIdx.x & 31;
  const int warps = gridDim.x * (blockDim.x >> 5);
  const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int per = (n + warps - 1) / warps;
  const int end = min(n, (w + 1) * per);
  unsigned ops = 0;
  for (int pos = w * per; pos < end;) {
    // lanes 0..7: the next moves and their balls' places among the 32 lanes
    int v = 0, nel = 0;
    if (lane < 8 && pos + lane < end) {
      v = R[pos + lane];
      nel = S.NElen[v];
    }
    int incl = nel;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    const unsigned fit = __ballot_sync(0xffffffffu, lane < 8 && nel > 0 && incl <= 32);
    int cnt = __ffs(~fit) - 1;  // moves taken: the leading ones that fit
    if (cnt == 0) cnt = 1;
    // my move and element
    int own = -1, k = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int hi = __shfl_sync(0xffffffffu, incl, j), len = __shfl_sync(0xffffffffu, nel, j);
      if (j < cnt && lane >= hi - len && lane < hi) {
        own = j;
        k = lane - (hi - len);
      }
    }
    const int from = own >= 0 ? own : 0;
    const int mv_v = __shfl_sync(0xffffffffu, v, from);
    const int mv_n = __shfl_sync(0xffffffffu, nel, from);
    bool ok = true;
    if (own >= 0) {
      const MeshCtx c = ctx_of(S, mv_v);
      const int lv = mv_v - c.vb;
      const double2 X = mvxy[mv_v];
      const double4 M = mvM[mv_v];  // (its w holds the old minimum quality)
      const VD nvd{X.x, X.y, M.x, M.y, M.z};
      for (; k < mv_n; k += 32) {  // (one turn unless the ball takes the warp alone)
        const int4 e = S.EN[c.eb + ne_row(S, mv_v)[k]];
        const VD a = (e.x == lv) ? nvd : load_vd(S, c.vb + e.x);
        const VD b = (e.y == lv) ? nvd : load_vd(S, c.vb + e.y);
        const VD d = (e.z == lv) ? nvd : load_vd(S, c.vb + e.z);
        ops += kOpsOrient + kOpsQuality;
        if (orient_sign(a, b, d) > 0) {
          const double q = quality_c(e.x, e.y, e.z, a, b, d);
          ok &= dgt(q, M.w);
          // the new ball qualities of an accepted move are kept for the apply
          qball[(size_t)mv_v * S.W + k] = q;
        } else {
          ok = false;
        }
      }
    }
    const unsigned bad = __ballot_sync(0xffffffffu, !ok);
    // lane j < cnt: the answer of move j
    bool cand = false;
    if (lane < cnt) {
      const int lo = min(incl - nel, 32), hi = min(incl, 32);
      const unsigned mask = (hi >= 32 ? 0xffffffffu : (1u << hi) - 1u) &
                            ~(lo >= 32 ? 0xffffffffu : (1u << lo) - 1u);
      cand = (bad & mask) == 0u;
      mvM[v].w = cand ? kMoveEvaluated : 0.0;
      if (cand) {
        cmark[v] = tag;
        S.tab.had[ctx_of(S, v).mi] = 1;
      }
    }
    warp_append(cand, v, C, nC);
    pos += cnt;
  }
  add_work(work, ops);
}

__global__ void k_smooth_filter(Store S, const int* E, const int* nEp, double2* mvxy,
                                double4* mvM, int* R, int* nR, int* C, int* nC, int* cmark,
                                int tag, unsigned long long* work) {
  smooth_filter_phase(S, E, nEp, mvxy, mvM, R, nR, C, nC, cmark, tag, true, work);
}

__global__ void __launch_bounds__(256, 3)
k_smooth_eval(Store S, const int* R, const int* nRp, const double2* mvxy, double4* mvM,
              double* qball, int* C, int* nC, int* cmark, int tag, unsigned long long* work) {
  smooth_exact_packed(S, R, nRp, mvxy, mvM, qball, C, nC, cmark, tag, work);
}

// One round's independent set and its moves (see k_coarsen_select_apply); live
// interior neighbours of a moved vertex become pending for the next sweep (stamp
// pmark with the sweep tag).  What the move needs is loaded beside the
// independent set's gathers, and the round's lists share a reservation.  The elements
// of a move whose qualities were left open join list Q.  Gathers bound it
// (long-scoreboard stalls, DRAM 38%).
__device__ __forceinline__ void smooth_select_apply_phase(Store S, const int* C, const int* nCp,
                                                          const int* cmark, int* smark, int tag,
                                                          int* Dn, int* nDn, int* dmark,
                                                          const double2* mvxy, const double4* mvM,
                                                          const double* qball, int* P, int* nP,
                                                          int* pmark, int ptag, int stamp, int* Q,
                                                          int* nQ, bool il = false) {
  const int first = first_entry(C, grank(il), S.vslots);
  const int n = *nCp;
  for (int i0 = 0; i0 < n; i0 += gsize()) {
    int i = i0 + grank(il);
    bool win = false, lose = false;
    int v = 0, mi = 0, vb = 0, nnl = 0, eb = 0, nq = 0;
    const int* nn = nullptr;
    const int* ne = nullptr;
    RowMask take;
    if (i < n) {
      v = i0 == 0 ? first : C[i];
      const double2 p = mvxy[v];
      double4 mv = mvM[v];
      const MeshCtx c = ctx_of(S, v);
      ne = ne_row(S, v);
      Row8 er = row8(ne, 0);
      const int nel = S.NElen[v];
      win = local_max(S, v, cmark, tag);
      if (!win) lose = stamp_first(dmark, v, tag);
      if (win) {
        mi = c.mi;
        vb = c.vb;
        nn = nn_row(S, v);
        nnl = S.NNlen[v];
        for (int b = 0; b < nnl; b += 8) {
          const Row8 r = row8(nn, b);
          int op[8], f[8];
          // (a stamp on a vertex that is not taken is harmless: only interior
          // neighbours look at it)
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const bool in = b + k < nnl;
            const int s = vb + r.a[k];
            f[k] = in ? S.vflag[s] : VF_BND;
            op[k] = in ? atomicExch(pmark + s, ptag) : ptag;
            if (in) S.ntouch[s] = stamp;
          }
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (op[k] != ptag && (f[k] & VF_ALIVE) && !(f[k] & VF_BND)) take.set(b + k);
        }
        smark[v] = tag;
        if (mv.w == kMoveUnevaluated) nq = nel;
        eb = c.eb;
        mv.w = 0.0;
        S.xy[v] = p;
        S.M[v] = mv;
        store_vf(S, v, p, mv);
        S.touch[v] = stamp;
        for (int b = 0; nq == 0;) {
          double q[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) q[k] = b + k < nel ? qball[(size_t)v * S.W + b + k] : 0.0;
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (b + k < nel) S.qK[c.eb + er.a[k]] = q[k];
          b += 8;
          if (b >= nel) break;
          er = row8(ne, b);
        }
      }
    }
    count_op(S, win, mi);
    const Room3 at = warp_reserve3(take.count(), nP, lose ? 1 : 0, nDn, nq, nQ);
    write_row_bits(take, nn, vb, P, at.a);
    if (lose) Dn[at.b] = v;
    for (int k = 0; k < nq; ++k) Q[at.c + k] = eb + ne[k];
  }
}

__global__ void k_smooth_select_apply(Store S, const int* C, const int* nCp, const int* cmark,
                                      int* smark, int tag, int* Dn, int* nDn, int* dmark,
                                      const double2* mvxy, const double4* mvM, const double* qball,
                                      int* P, int* nP, int* pmark, int ptag, int stamp, int* Q,
                                      int* nQ, unsigned* done) {
  smooth_select_apply_phase(S, C, nCp, cmark, smark, tag, Dn, nDn, dmark, mvxy, mvM, qball, P, nP,
                            pmark, ptag, stamp, Q, nQ);
  round_done(S, done);
}

// d/dx and d/dy of the quality of element (i0, i1, i2) with respect to its
// vertex `own`: the operations of quality_grad_c that these two values need, in
// its order (the metric's derivatives, the other vertices' and those of the edge
// that does not touch the vertex are left out: about 200 FP64 instructions
// instead of 270).
__device__ __forceinline__ void quality_grad_xy(int i0, int i1, int i2, VD a, VD b, VD c, int own,
                                                double& gx, double& gy) {
  canon(i0, i1, i2, a, b, c);
  const int at = own == i0 ? 0 : (own == i1 ? 1 : 2);
  double k00 = div3((a.m00 + b.m00) + c.m00);
  double k01 = div3((a.m01 + b.m01) + c.m01);
  double k11 = div3((a.m11 + b.m11) + c.m11);
  double dx[3] = {b.x - a.x, c.x - b.x, a.x - c.x};
  double dy[3] = {b.y - a.y, c.y - b.y, a.y - c.y};
  double l[3];
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    double L2 = ((k00 * dx[e]) * dx[e] + ((2.0 * k01) * dx[e]) * dy[e]) + (k11 * dy[e]) * dy[e];
    l[e] = sqrt(L2);
  }
  double P = (l[0] + l[1]) + l[2];
  double area = 0.5 * orient3(a, b, c);
  double sd = sqrt(k00 * k11 - k01 * k01);
  double AM = sd * area;
  double xx = div3(P);
  bool left = (xx <= 1.0);
  double sv = left ? xx : 1.0 / xx;
  double f = sv * (2.0 - sv);
  double F = (f * f) * f;
  double PP = P * P;
  double t = (QC * AM) / PP;
  double gAM = (F * QC) / PP;
  double gP = -((2.0 * t) / P) * F;
  double gf = (3.0 * (f * f)) * t;
  double gs = (2.0 - 2.0 * sv) * gf;
  double gxx = left ? gs : -(gs / (xx * xx));
  gP = gP + div3(gxx);
  double go = 0.5 * (sd * gAM);
  // the edges before and after the vertex, and the opposite one's ends
  const double lb = at == 0 ? l[2] : (at == 1 ? l[0] : l[1]);
  const double la = at == 0 ? l[0] : (at == 1 ? l[1] : l[2]);
  const double bx = at == 0 ? dx[2] : (at == 1 ? dx[0] : dx[1]);
  const double by = at == 0 ? dy[2] : (at == 1 ? dy[0] : dy[1]);
  const double ax = at == 0 ? dx[0] : (at == 1 ? dx[1] : dx[2]);
  const double ay = at == 0 ? dy[0] : (at == 1 ? dy[1] : dy[2]);
  const double ya = at == 0 ? b.y : (at == 1 ? c.y : a.y), yb = at == 0 ? c.y : (at == 1 ? a.y : b.y);
  const double xa = at == 0 ? c.x : (at == 1 ? a.x : b.x), xb = at == 0 ? b.x : (at == 1 ? c.x : a.x);
  const double gLb = gP / (2.0 * lb), gLa = gP / (2.0 * la);
  const double bgx = ((2.0 * k00) * bx + (2.0 * k01) * by) * gLb;
  const double bgy = ((2.0 * k01) * bx + (2.0 * k11) * by) * gLb;
  const double agx = ((2.0 * k00) * ax + (2.0 * k01) * ay) * gLa;
  const double agy = ((2.0 * k01) * ax + (2.0 * k11) * ay) * gLa;
  // vertex 0 subtracts its own edge first, the others add the edge before first
  const double x0 = go * (ya - yb), y0 = go * (xa - xb);
  gx = at == 0 ? (x0 - agx) + bgx : (x0 + bgx) - agx;
  gy = at == 0 ? (y0 - agy) + bgy : (y0 + bgy) - agy;
}

// Optimisation-based smoothing of one member of S (gradient ascent of the
// ball's quality sum in v's coordinates, metric fixed; step 0.1 * shortest
// incident edge / |g|, halved up to five times; kept when every element stays
// counter-clockwise, the minimum quality does not drop and the sum rises),
// evaluated by an 8-lane tile.
__device__ bool tile_opt_eval(const Tile& t, const Store& S, int v, MeshCtx c, double2& Xo,
                              double4& Mo, double* qout) {
  uint8_t f = S.vflag[v];
  if (!(f & VF_ALIVE) || (f & VF_BND)) return false;
  int lv = v - c.vb;
  const int* ne = ne_row(S, v);
  int nel = S.NElen[v];
  double gx = 0.0, gy = 0.0;
  for (int base = 0; base < nel; base += TW) {
    int k = base + t.tl;
    double gxk = 0.0, gyk = 0.0;
    if (k < nel) {
      int4 e = S.EN[c.eb + ne[k]];
      quality_grad_xy(e.x, e.y, e.z, load_vd(S, c.vb + e.x), load_vd(S, c.vb + e.y),
                      load_vd(S, c.vb + e.z), lv, gxk, gyk);
    }
    int cnt = min(TW, nel - base);
    for (int j = 0; j < cnt; ++j) {
      gx = gx + tshfl(t, gxk, j);
      gy = gy + tshfl(t, gyk, j);
    }
  }
  double gn = sqrt(gx * gx + gy * gy);
  if (!(gn > 0.0)) return false;
  const int* nn = nn_row(S, v);
  int nnl = S.NNlen[v];
  double2 pv = S.xy[v];
  double lmin = 1e300;
  for (int k = t.tl; k < nnl; k += TW) {
    double2 pj = S.xy[c.vb + nn[k]];
    double dx = pj.x - pv.x;
    double dy = pj.y - pv.y;
    double l = sqrt(dx * dx + dy * dy);
    lmin = (l < lmin) ? l : lmin;
  }
  lmin = tmin(t, lmin);
  double qsum_old;
  double qmin_old = tile_ball_quality(t, S, c, ne, nel, &qsum_old);
  double alpha = (0.1 * lmin) / gn;
  unsigned ops = 0;
  for (int k = 0; k < 6; ++k) {
    double X = pv.x + alpha * gx;
    double Y = pv.y + alpha * gy;
    double4 Mn;
    double qsum;
    if (tile_try_move(t, S, c, lv, ne, nel, X, Y, qmin_old, false, qout, &qsum, qsum_old, Mn,
                      ops) &&
        qsum > qsum_old) {
      Xo = make_double2(X, Y);
      Mo = Mn;
      return true;
    }
    alpha = alpha * 0.5;
  }
  return false;
}

// Evaluate and apply in one pass (one tile per member of S): members are
// pairwise non-adjacent, so no member reads a vertex another member moves.
// FP64 bounds it (pipe 80% active).  20 rounds on 131k vertices: 11.9 ms with every
// trial step evaluated in full, 6.0 with the FP32 metric and quality bounds in front
// and the gradient of the moved vertex alone, 5.4 with the ordered sums spread over
// the tile's lanes.
__global__ void k_opt_apply(Store S, const int* Sl, const int* nSp, double* qball, int stamp) {
  advance_rounds(S);
  const int n = *nSp;
  const Tile t = tile_of();
  const int tiles_per_block = blockDim.x / TW;
  for (int j0 = blockIdx.x * tiles_per_block; j0 < n; j0 += gridDim.x * tiles_per_block) {
    int j = j0 + threadIdx.x / TW;
    bool moved = false;
    int mi = 0;
    if (j < n) {
      int v = Sl[j];
      MeshCtx c = ctx_of(S, v);
      mi = c.mi;
      double* qb = qball + (size_t)v * S.W;
      double2 X;
      double4 Mv;
      moved = tile_opt_eval(t, S, v, c, X, Mv, qb);
      __syncwarp(t.mask);
      if (moved && t.tl == 0) {
        S.xy[v] = X;
        S.M[v] = Mv;
        store_vf(S, v, X, Mv);
        S.touch[v] = stamp;
        const int* ne = ne_row(S, v);
        int nel = S.NElen[v];
        for (int k = 0; k < nel; ++k) S.qK[c.eb + ne[k]] = qb[k];
        stamp_neighbours(S, nn_row(S, v), S.NNlen[v], c.vb, stamp);
      }
    }
    count_op(S, moved && t.tl == 0, mi);
  }
}

// Every listed vertex is a candidate of this round.
__global__ void k_stamp_list(Store S, const int* L, const int* nLp, int* cmark, int tag) {
  const int n = *nLp;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int v = L[i];
    cmark[v] = tag;
    S.tab.had[mesh_of_vslot(S, v)] = 1;
  }
}

// ---- refinement (Sec. 2.4.2) -----------------------------------------------------

// Mark edges (a, b), a < b, longer than L_up: entry k of vmask[a] for NN entry k.
// A vertex unchanged since it was marked earlier in this pass keeps its mask;
// one unchanged since the end of an earlier complete pass has none.  The mask
// reads a's own row and the positions and metrics of a and its neighbours;
// inside one call vertices keep their positions and metrics until the
// operator loop ends (smoothing runs after it), so a's own stamp tells
// whether anything the mask read has changed: every change of a's row stamps a.
// A sweep over every slot that waits for its gathers: 48 registers, 40 warps an SM
// (9.7 -> 9.5 ms over the 29 launches of a 512-mesh batch; 80 registers 11.7).
__global__ void __launch_bounds__(256, 5)
k_refine_mark(Store S, int* cnt, RowMask* mask, int tag, int pass0, int lo, const int* before,
              const int* before2, const DevStatus* st) {
  if (!may_go(before, st)) return;
  tag += tags_of(before) + tags_of(before2);
  pass0 += tags_of(before) + tags_of(before2);
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < S.vused; s += gridDim.x * blockDim.x) {
    int mi = mesh_of_vslot(S, s);
    int vb = S.tab.vbase[mi];
    RowMask m;
    bool live = s - vb < S.tab.nv[mi] && S.tab.active[mi] && (S.vflag[s] & VF_ALIVE);
    const int et = live ? S.evr[s] : 0;
    const bool same = live && S.touch[s] <= et;
    if (same && et > pass0) {
      m = mask[s];  // kept as it is
    } else if (same && et > lo) {
      mask[s] = RowMask();
    } else if (live) {
      S.evr[s] = tag;
      int la = s - vb;
      const int* nn = nn_row(S, s);
      int nnl = S.NNlen[s];
      const VF fa = load_vf(S, s);
      unsigned ops = 0;
      // the row is sorted, so the neighbours above la form a suffix; four
      // lengths at a time so that their loads overlap
      int k0 = 0;
      // (a sweep over every slot hides the latency with resident warps: fewer
      // registers beat loads issued ahead, 150 against 187 us on 10M slots)
      while (k0 < nnl && nn[k0] <= la) ++k0;
#pragma unroll 4
      for (int k = k0; k < nnl; ++k)
        if (edge_longer(S, mi, fa, load_vf(S, vb + nn[k]), s, vb + nn[k], ops)) m.set(k);
      mask[s] = m;
    } else {
      mask[s] = RowMask();
    }
    cnt[s] = m.count();
  }
}

// Per-mesh number of new vertices (edges to split), after the counters, with
// the lists that the round's split fills cleared.
__global__ void k_refine_newcount(Store S, const int* vscan, int* counts, const int* before,
                                  const DevStatus* st) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  // (loaded together: the launch is a chain of latencies)
  const int go = before ? before[2] : 1, over = before ? st->overflow : 0;
  const int vb = i < S.nmesh ? S.tab.vbase[i] : 0, nv = i < S.nmesh ? S.tab.nv[i] : 0;
  if (go == 0 || over != 0) return;
  if (i == 0) counts[CN_EL] = counts[CN_CL] = 0;
  if (i < S.nmesh) counts[cn_newv(S.nmesh) + i] = vscan[vb + nv] - vscan[vb];
}

__device__ __forceinline__ int mid_id(const Store& S, int vb, int nv, const int* vscan,
                                      const RowMask* mask, int p, int q) {
  int a = p < q ? p : q, b = p < q ? q : p;
  const RowMask m = mask[vb + a];
  if (!m.any()) return -1;
  int k = row_find(nn_row(S, vb + a), S.NNlen[vb + a], b);
  if (k < 0 || !m.test(k)) return -1;
  int rank = m.below(k);
  return nv + (vscan[vb + a] - vscan[vb]) + rank;
}

__global__ void k_refine_newverts(Store S, const int* vscan, const RowMask* mask, int stamp,
                                  int4* owner) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < S.vused; s += gridDim.x * blockDim.x) {
    RowMask m = mask[s];
    if (!m.any()) continue;
    int mi = mesh_of_vslot(S, s);
    int vb = S.tab.vbase[mi], eb = S.tab.ebase[mi], nv = S.tab.nv[mi];
    const int* nn = nn_row(S, s);
    const int* ne = ne_row(S, s);
    int nel = S.NElen[s];
    int base = nv + (vscan[s] - vscan[vb]);
    int rank = 0;
    VD da = load_vd(S, s);
    while (m.any()) {
      int b = nn[m.pop()];
      VD db = load_vd(S, vb + b);
      int slot = vb + base + rank;
      ++rank;
      const double2 p = make_double2(0.5 * (da.x + db.x), 0.5 * (da.y + db.y));
      const double4 mid = make_double4(0.5 * (da.m00 + db.m00), 0.5 * (da.m01 + db.m01),
                                       0.5 * (da.m11 + db.m11), 0.0);
      S.xy[slot] = p;
      S.M[slot] = mid;
      store_vf(S, slot, p, mid);
      bool bedge = count_elems_with(S, ne, nel, eb, b) == 1;
      S.vflag[slot] = (uint8_t)(VF_ALIVE | (bedge ? VF_BND : 0));
      if (S.lid) S.lid[slot] = (slot - vb) - S.voff[mi];
      S.touch[slot] = stamp;
      S.evc[slot] = S.evs[slot] = S.evm[slot] = S.evr[slot] = 0;
      owner[slot] = make_int4(s - vb, b, 0, 0);  // the split edge (a, b)
    }
  }
}

// Extra children per live element (0..3); an element that splits gets the
// midpoint ids of its edges and joins the split list.
__global__ void k_refine_count(Store S, const int* vscan, const RowMask* mask, int* ecnt,
                               int4* emid, int* elist, int* nel) {
  for (int i0 = blockIdx.x * blockDim.x; i0 < S.eused; i0 += gridDim.x * blockDim.x) {
    int s = i0 + threadIdx.x;
    int extra = 0;
    if (s < S.eused) {
      int mi = mesh_of_eslot(S, s);
      int eb = S.tab.ebase[mi];
      if (s - eb < S.tab.ne[mi] && S.tab.active[mi]) {
        int4 e = S.EN[s];
        if (e.w) {
          int vb = S.tab.vbase[mi], nv = S.tab.nv[mi];
          int m0 = mid_id(S, vb, nv, vscan, mask, e.x, e.y);
          int m1 = mid_id(S, vb, nv, vscan, mask, e.y, e.z);
          int m2 = mid_id(S, vb, nv, vscan, mask, e.z, e.x);
          extra = (m0 >= 0) + (m1 >= 0) + (m2 >= 0);
          if (extra) emid[s] = make_int4(m0, m1, m2, extra);
        }
      }
      ecnt[s] = extra;
    }
    warp_append(extra > 0, s, elist, nel);
  }
}

// Templates: one split -> (a,m,o),(m,b,o); two splits -> (m0,u1,m1) plus the
// trapezoid (u0,m0,m1,u2) cut along its metric-shorter diagonal; three
// splits -> four children.  The first child keeps the parent's slot, the rest
// take ne + scan(extra children) in parent order.  Every child slot joins
// the list whose qualities k_refine_quality computes.
__global__ void k_refine_split(Store S, const int* escan, const int4* emid, const int* elist,
                               const int* nelp, int* clist, int* ncl, int stamp) {
  const int n = *nelp;
  for (int i0 = blockIdx.x * blockDim.x; i0 < n; i0 += gridDim.x * blockDim.x) {
    int i = i0 + threadIdx.x;
    int s = 0, nslot = 0, extra = 0;
    if (i < n) {
      s = elist[i];
      int mi = mesh_of_eslot(S, s);
      int eb = S.tab.ebase[mi];
      int4 e = S.EN[s];
      int4 md = emid[s];
      extra = md.w;
      int vb = S.tab.vbase[mi];
      nslot = eb + S.tab.ne[mi] + (escan[s] - escan[eb]);
      auto put = [&](int slot, int a, int b, int c) { S.EN[slot] = make_int4(a, b, c, 1); };
      int t[3] = {e.x, e.y, e.z};
      int mm[3] = {md.x, md.y, md.z};
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        S.touch[vb + t[k]] = stamp;
        if (mm[k] >= 0) S.touch[vb + mm[k]] = stamp;
      }
      if (md.w == 1) {
        int j = (mm[0] >= 0) ? 0 : (mm[1] >= 0) ? 1 : 2;
        int a = t[j], b = t[(j + 1) % 3], o = t[(j + 2) % 3], m = mm[j];
        put(s, a, m, o);
        put(nslot, m, b, o);
      } else if (md.w == 2) {
        int j = (mm[0] < 0) ? 0 : (mm[1] < 0) ? 1 : 2;
        int q = (j + 1) % 3;
        int u0 = t[q], u1 = t[(q + 1) % 3], u2 = t[(q + 2) % 3];
        int m0 = mm[q], m1 = mm[(q + 1) % 3];
        put(s, m0, u1, m1);
        double d1 = metric_len(load_vd(S, vb + u0), load_vd(S, vb + m1));
        double d2 = metric_len(load_vd(S, vb + m0), load_vd(S, vb + u2));
        if (!dgt(d1, d2)) {
          put(nslot, u0, m0, m1);
          put(nslot + 1, u0, m1, u2);
        } else {
          put(nslot, u0, m0, u2);
          put(nslot + 1, m0, m1, u2);
        }
      } else {
        put(s, t[0], mm[0], mm[2]);
        put(nslot, mm[0], t[1], mm[1]);
        put(nslot + 1, mm[2], mm[1], t[2]);
        put(nslot + 2, mm[0], mm[1], mm[2]);
      }
    }
    warp_append(i < n, s, clist, ncl);
    for (int j = 0; j < 3; ++j) warp_append(j < extra, nslot + j, clist, ncl);
  }
}

// Cached quality of every listed element slot (one element per thread): the
// children of a refinement round, the elements a collapse round changed.
__global__ void k_refine_quality(Store S, const int* clist, const int* nclp,
                                 unsigned long long* work) {
  elem_quality_phase(S, clist, nclp, work);
}

// Children of parent element K (local id) of this round: K itself and, when
// split, the extra slots ne + (escan[K] - escan[eb]) onwards.
__device__ __forceinline__ int refine_children(const Store& S, int mi, int eb, const int* escan,
                                               int K, int* out) {
  int s = eb + K;
  int e0 = escan[s], extra = escan[s + 1] - e0;
  out[0] = K;
  int first = S.tab.ne[mi] + (e0 - escan[eb]);
  for (int j = 0; j < extra; ++j) out[1 + j] = first + j;
  return 1 + extra;
}

// New rows of vertex slot s of a refinement round, from the old element row of
// `src`: NE = the children of those elements that contain the vertex, NN = the
// other vertices of those, both sorted.  Rows of up to 16 entries are made in
// registers; false, with nothing written, when one is longer.
// (They were built in a second buffer through local memory: a tenth of the adaptation
// of 20M triangles, 104.8 -> 99.6 ms, with the estimate of pm_mesh.cu in FP32.)
__device__ __forceinline__ bool refine_row_short(const Store& S, int s, int src, int mi, int vb,
                                                 int eb, const int* escan, int stamp) {
  const int lu = s - vb;
  const int nel = S.NElen[src];
  Row16 P;
  P.load(S.NE + (size_t)src * S.W, nel);
  if (nel > kRowReg) return false;
  const int base = S.tab.ne[mi] - escan[eb];
  Row16 N, E;
#pragma unroll
  for (int k = 0; k < kRowReg; ++k) N.a[k] = E.a[k] = kRowPad;
  bool ok = true;
  for (int k = 0; k < nel; ++k) {
    // (the row again, in cache: P is indexed by constants only)
    const int K = S.NE[(size_t)src * S.W + k];
    const int e0 = escan[eb + K], extra = escan[eb + K + 1] - e0;
    int4 e[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      e[j] = j <= extra ? S.EN[eb + (j == 0 ? K : base + e0 + j - 1)] : make_int4(-1, -1, -1, 0);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (e[j].x != lu && e[j].y != lu && e[j].z != lu) continue;
      ok &= E.insert(j == 0 ? K : base + e0 + j - 1);
      ok &= N.insert((e[j].x == lu) ? e[j].y : e[j].x);
      ok &= N.insert((e[j].z == lu) ? e[j].y : e[j].z);
    }
  }
  if (!ok) return false;
  const int nn2 = N.len(), ne2 = E.len();
  N.store(S.NN + (size_t)s * S.W, nn2);
  E.store(S.NE + (size_t)s * S.W, ne2);
  S.NNlen[s] = nn2;
  S.NElen[s] = ne2;
#pragma unroll
  for (int k = 0; k < kRowReg; ++k)
    if (k < nn2) S.ntouch[vb + N.a[k]] = stamp;
  return true;
}

// Rows of the vertices whose elements changed in this refinement round
// (stamped), in place, in two launches: the new vertices first (`fresh`), which
// read the old element row of their split edge's first end (the children that
// contain the new vertex are exactly those of the two parents on that edge), then
// the old ones, which read and write their own rows alone.  64 registers: 7.8 -> 6.5
// ms over the 28 launches of a 512-mesh batch (latency, not the 12 spilled bytes).
__global__ void __launch_bounds__(256, 4)
k_refine_rows(Store S, int vfirst, int vend, int fresh, const int* escan, const int4* owner,
              int stamp, DevStatus* st) {
  for (int s = vfirst + blockIdx.x * blockDim.x + threadIdx.x; s < vend;
       s += gridDim.x * blockDim.x) {
    if (S.touch[s] != stamp) continue;
    const int mi = mesh_of_vslot(S, s);
    const int vb = S.tab.vbase[mi], eb = S.tab.ebase[mi], nv = S.tab.nv[mi];
    const int lu = s - vb;
    if ((lu >= nv) != (fresh != 0)) continue;
    const int src = fresh ? vb + owner[s].x : s;
    if (refine_row_short(S, s, src, mi, vb, eb, escan, stamp)) continue;
    const int* ne = S.NE + (size_t)src * S.W;
    const int nel = S.NElen[src];
    __align__(16) int nb_[MAXW];  // read in chunks below
    int eb_[MAXW];
    int ne2 = 0, nn2 = 0;
    bool ok = true;
    for (int k = 0; k < nel; ++k) {
      int K = ne[k];
      int ch[4];
      int n = refine_children(S, mi, eb, escan, K, ch);
      for (int j = 0; j < n; ++j) {
        int4 e = S.EN[eb + ch[j]];
        if (e.x != lu && e.y != lu && e.z != lu) continue;
        ok &= sorted_insert(eb_, ne2, MAXW, ch[j]);
        int a = (e.x == lu) ? e.y : e.x;
        int b = (e.z == lu) ? e.y : e.z;
        ok &= sorted_insert(nb_, nn2, MAXW, a);
        ok &= sorted_insert(nb_, nn2, MAXW, b);
      }
    }
    if (!ok || ne2 > S.W || nn2 > S.W) {
      atomicExch(&st->overflow, 1);
      atomicMax(&st->maxdeg, max(ne2, nn2));
      // until the rows are rebuilt a new vertex has none (the marks queued behind
      // this round read them)
      if (fresh) S.NNlen[s] = S.NElen[s] = 0;
      continue;
    }
    int* wn = S.NN + (size_t)s * S.W;
    int* we = S.NE + (size_t)s * S.W;
    for (int k = 0; k < nn2; ++k) wn[k] = nb_[k];
    for (int k = 0; k < ne2; ++k) we[k] = eb_[k];
    S.NNlen[s] = nn2;
    S.NElen[s] = ne2;
    stamp_neighbours(S, nb_, nn2, vb, stamp);
  }
}

// The sizes after the round, in the table and after the counters; a mesh that
// splits edges counts the round and its splits.
__global__ void k_refine_sizes(Store S, const int* vscan, const int* escan, int* counts) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= S.nmesh) return;
  int vb = S.tab.vbase[i], eb = S.tab.ebase[i];
  int nv = S.tab.nv[i], ne = S.tab.ne[i];
  const int t = vscan[vb + nv] - vscan[vb];
  S.tab.nv[i] = counts[cn_sizes(S.nmesh) + i] = nv + t;
  S.tab.ne[i] = counts[cn_sizes(S.nmesh) + S.nmesh + i] = ne + (escan[eb + ne] - escan[eb]);
  if (t > 0) {
    S.tab.r[i] += 1;
    S.tab.ops[i] += (unsigned long long)t;
  }
}

// ---- persistent rounds ------------------------------------------------------------
//
// Once a pass's dirty list is small, a round does little work and its cost is
// launch and synchronisation latency.  Such rounds run back to back inside one
// cooperative launch (every block resident), with a grid-wide barrier between
// the phases and one read-back when the launch ends.  A collapse round
// evaluates in one phase (coarsen_eval_phase) and takes three barriers;
// smoothing scans and evaluates in one tile-parallel phase when the list fits
// kFusePasses passes of the grid's tiles (two barriers), else it keeps scan, filter and
// exact check apart (four); flips scan, evaluate and pick in one tile-parallel
// phase when the list fits as many passes (three barriers), else they keep their
// scan, item-parallel gains and pick (five).  The launch returns when a round finds no
// candidate (the pass is complete), when the next round's list outgrows `limit`, on a
// row overflow or an error, or after `max_rounds` rounds.
//
// Counters are reset where no block can still read or write them: the
// candidate count alternates between two slots (C of even rounds, C2 of odd
// ones); the other slot and the lists a round fills are cleared by block 0
// at least one barrier before their first use and after their last read.

constexpr unsigned long long kBarrierNs = 2000000000ull;  // a barrier wait gives up after 2 s

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ int ld_volatile(const int* p) { return *(volatile const int*)p; }

// Grid-wide barrier on a counter of arrivals that only grows (zeroed before
// the launch): the k-th barrier waits for k * gridDim.x arrivals.  Thread 0
// of each block arrives with a release after the block's __syncthreads (so
// every write of the block is published with it) and waits with acquire loads;
// nothing waits for the arrival's own round trip, and the error word travels
// with the waiting loads.  Returns false (the caller leaves the kernel) when the
// wait ran out (PM_ERR_TIMEOUT is recorded) or when an error had been recorded.
// An error recorded in the phase just left may be seen only at the next barrier
// (a block that leaves at once does not arrive there, and the others find the
// error while they wait), so a phase bounds its own reads by what the one before
// may have overrun.
__device__ bool grid_barrier(unsigned* bar, unsigned& target, DevStatus* st,
                             unsigned long long limit_ns = kBarrierNs) {
  __shared__ int s_ok;
  target += gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    unsigned long long t0 = 0;
    for (unsigned spin = 1;; ++spin) {
      int err;
      unsigned arrived;
      asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(err) : "l"(&st->err) : "memory");
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(arrived) : "l"(bar) : "memory");
      if (err != 0) {
        ok = 0;
        break;
      }
      if ((int)(arrived - target) >= 0) break;
      if ((spin & 255u) == 0) {
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 > limit_ns) {
          set_err(st, PM_ERR_TIMEOUT);
          ok = 0;
          break;
        }
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Test support: every block waits at a barrier whose target lies one arrival
// beyond the grid, so the wait can only end by its time limit.
__global__ void k_selftest_barrier(unsigned* bar, DevStatus* st, unsigned long long limit_ns) {
  unsigned target = 1;
  grid_barrier(bar, target, st, limit_ns);
}

// Flips and smoothing: lists of up to this many passes of the grid's tiles take
// the one-phase form (measured on a 201 x 201 mesh adapted to 670k triangles:
// flips 13.20 ms at one pass, 12.88 at two and three, 13.23 at eight; smoothing
// 12.80, 12.58, 13.01 at one, two, three).
constexpr int kFusePasses = 2;

struct RoundArgs {
  Store S;
  Work w;
  DevStatus* st;
  unsigned* bar;       // barrier arrivals (zeroed before the launch)
  int* res;            // out: rounds run, list index after, pass complete
  int cur;             // list index the first round reads
  int tag0;            // tag of the first round (then +2 per round)
  int pass0;
  int max_rounds;
  int limit;           // leave when the next list holds more entries
  int icap;            // flips: capacity of the item list
  int ptag;            // smoothing: stamp of the next sweep's list
  int sweeps;          // smoothing: sweeps left, the current one included
  int moved;           // smoothing: the current sweep has moved a vertex
  const int* before;   // flips: results of the rounds this launch is queued behind (may_go)
  int fuse;            // flips, smoothing: lists up to this size (and kFusePasses passes of
                       // tiles) take the one-phase evaluation
  unsigned long long* work;  // counted FP64 work (measurement) or null
};

__device__ __forceinline__ int* cand_count(int* cnt, int r) {
  return cnt + ((r & 1) ? CN_C2 : CN_C);
}

__device__ __forceinline__ void finish_rounds(const RoundArgs& a, int r, int cur, bool complete) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.res[0] = r;
    a.res[1] = cur;
    a.res[2] = complete ? 1 : 0;
  }
}

// Rounds of collapses: [evaluate] B1 [select + apply] B2 [commit] B3; rounds
// of flips whose list fits kFusePasses passes of the grid's tiles: [scan + gains +
// pick] B1 [select + apply] B2 [commit] B3; longer flip lists: [scan] B1
// [gains] [pick] [select + apply] [commit], five barriers.  Block 0 clears,
// before B1 of round r: A and the list round r
// fills (both last read before the last barrier of round r - 1); right after
// B1: the candidate slot of round r + 1 (last read before the last barrier of
// round r - 1); flips, after the pick: E and the item count (read by the pick
// and the gains).
template <bool FLIP>
__device__ __forceinline__ void topo_rounds(const RoundArgs& a) {
  const Work& w = a.w;
  int* cnt = w.counts;
  unsigned target = 0;
  int cur = a.cur, r = 0;
  bool complete = false;
  if (!may_go(a.before, a.st)) return;  // (the same answer in every block: all wait at B1 first)
  const int tag0 = a.tag0 + tags_of(a.before), pass0 = a.pass0 + tags_of(a.before);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *cand_count(cnt, 0) = 0;
    cnt[CN_E] = cnt[CN_I] = 0;
  }
  if (!grid_barrier(a.bar, target, a.st)) return;
  // a first list longer than the limit is left to the one-kernel-per-phase rounds
  const bool too_long = ld_volatile(cnt + cn_list(cur)) > a.limit;
  while (!too_long && r < a.max_rounds) {
    const int tag = tag0 + 2 * r, nxt = 1 - cur;
    int* nC = cand_count(cnt, r);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      cnt[CN_A] = 0;
      cnt[cn_list(nxt)] = 0;
      cnt[CN_CL] = 0;  // elements whose quality changes
    }
    if (FLIP && ld_volatile(cnt + cn_list(cur)) <= min(a.fuse, kFusePasses * tcount())) {
      // the list fits two passes of tiles: scan, gains and pick in one phase
      // (the list is complete since the last barrier: every block decides alike)
      swap_scan_eval_phase(a.S, w.D[cur], cnt + cn_list(cur), w.opA, w.opK2, w.C, nC, w.cmark,
                           tag, pass0, a.work);
      if (!grid_barrier(a.bar, target, a.st)) return;
      if (blockIdx.x == 0 && threadIdx.x == 0) *cand_count(cnt, r + 1) = 0;
    } else if (FLIP) {
      // a longer list keeps the three passes: item-parallel FP64 gains beat
      // two barriers saved
      swap_scan_phase(a.S, w.D[cur], cnt + cn_list(cur), w.opA, w.C, nC, w.cmark, tag, pass0,
                      w.E, cnt + CN_E, w.items, cnt + CN_I, a.icap, w.gains, a.st, true);
      if (!grid_barrier(a.bar, target, a.st)) return;
      if (blockIdx.x == 0 && threadIdx.x == 0) *cand_count(cnt, r + 1) = 0;
      swap_edge_phase(a.S, w.items, cnt + CN_I, a.icap, w.gains, tag, a.work, true);
      if (!grid_barrier(a.bar, target, a.st)) return;
      swap_pick_phase(a.S, w.E, cnt + CN_E, w.gains, w.opA, w.opK2, w.C, nC, w.cmark, tag, true);
      if (!grid_barrier(a.bar, target, a.st)) return;
      if (blockIdx.x == 0 && threadIdx.x == 0) cnt[CN_E] = cnt[CN_I] = 0;
    } else {
      coarsen_eval_phase(a.S, w.D[cur], cnt + cn_list(cur), w.target, w.cand, w.C, nC,
                         w.cmark, tag, pass0, a.work, true);
      if (!grid_barrier(a.bar, target, a.st)) return;
      if (blockIdx.x == 0 && threadIdx.x == 0) *cand_count(cnt, r + 1) = 0;
    }
    if (FLIP)
      swap_select_apply_phase(a.S, w.C, nC, w.cmark, w.smark, tag, w.opA, w.opK2, w.A,
                              cnt + CN_A, w.amark, w.D[nxt], cnt + cn_list(nxt), w.dmark, w.clist,
                              cnt + CN_CL, true);
    else
      coarsen_select_apply_phase(a.S, w.C, nC, w.cmark, w.smark, tag, w.target, w.A, cnt + CN_A,
                                 w.amark, w.D[nxt], cnt + cn_list(nxt), w.dmark, w.clist,
                                 cnt + CN_CL, true);
    if (!grid_barrier(a.bar, target, a.st)) return;
    const int nc = ld_volatile(nC), nd = ld_volatile(cnt + cn_list(nxt));
    advance_rounds(a.S);
    if (FLIP)
      swap_commit_phase(a.S, w.A, cnt + CN_A, w.opA, w.opK2, w.smark, tag, a.st, true);
    else
      coarsen_commit_phase(a.S, w.A, cnt + CN_A, w.target, w.smark, tag, a.st, true);
    elem_quality_phase(a.S, w.clist, cnt + CN_CL, a.work, true);
    if (!grid_barrier(a.bar, target, a.st)) return;
    ++r;
    if (nc == 0) {
      complete = true;
      break;
    }
    cur = nxt;
    if (ld_volatile(&a.st->overflow) != 0 || nd > a.limit) break;
  }
  // the host reads the candidates of the last round from the C slot
  if (blockIdx.x == 0 && threadIdx.x == 0 && r > 0)
    cnt[CN_C] = ld_volatile(cand_count(cnt, r - 1));
  finish_rounds(a, r, cur, complete);
}

__global__ void __launch_bounds__(256) k_coarsen_rounds(RoundArgs a) { topo_rounds<false>(a); }

__global__ void __launch_bounds__(256) k_swap_rounds(RoundArgs a) { topo_rounds<true>(a); }

// Colouring rounds of a list of at most `limit` vertices: [propose] B1 [resolve]
// B2, until no vertex is uncoloured.  (A colouring takes about 15 rounds, each of
// which was two launches and a wait.)  Block 0 clears the list a round fills
// before B1 (last read before the last round's B2).  A 129 x 129 mesh adapted by
// colour classes: 16.2 -> 13.3 ms, with the smoothing's longer lists in two passes.
__global__ void __launch_bounds__(256) k_colour_rounds(RoundArgs a) {
  const Work& w = a.w;
  int* cnt = w.counts;
  unsigned target = 0;
  int cur = a.cur, r = 0;
  int n = ld_volatile(cnt + cn_list(cur));
  while (n > 0 && n <= a.limit && r < a.max_rounds) {
    const int nxt = 1 - cur, rt = a.tag0 + 2 * r;
    if (blockIdx.x == 0 && threadIdx.x == 0) cnt[cn_list(nxt)] = 0;
    colour_propose_phase(a.S, w.D[cur], cnt + cn_list(cur), w.cprop, w.cstamp, rt, true);
    if (!grid_barrier(a.bar, target, a.st)) return;
    colour_resolve_phase(a.S, w.D[cur], cnt + cn_list(cur), w.cprop, w.cstamp, rt, w.D[nxt],
                         cnt + cn_list(nxt), true);
    if (!grid_barrier(a.bar, target, a.st)) return;
    n = ld_volatile(cnt + cn_list(nxt));
    cur = nxt;
    ++r;
  }
  finish_rounds(a, r, cur, n == 0);
}

// Sweeps of smoothing rounds.  A round whose list fits kFusePasses passes of the grid's
// tiles: [scan + evaluate] B1 [select + apply] B2; a longer one: [scan] B1
// [filter] B1' [exact] B1'' [select + apply] B2 (its threads then go to the
// vertices that need an evaluation, its tiles to the moves that may succeed).  A
// sweep ends with a round that finds no candidate;
// its pending list then becomes the current one and the next sweep starts in
// the same launch (ten sweeps used to be ten launches and read-backs, most of
// them for a handful of vertices: 1.86 -> 1.48 ms on a 41 x 41 mesh).  The three
// lists trade places by index, each with its own counter.  Block 0 clears, before B1 of
// round r: the list round r fills and, in a sweep's first round, its pending list (both
// last read by a scan and a decision before the last barrier); after B1: the candidate
// slot of round r + 1 (last read after B2 of round r - 1); after B1': E (read by the
// filter before B1'); after B1'': the filtered list.  The round counters advance after
// B2 from the flag set of the round's parity, so that round r + 1's evaluation can set
// the other set meanwhile.  The launch returns when the sweeps are over, after
// `max_rounds` rounds with candidates, or when the next list outgrows `limit`; the
// lists' counts are then put where the host expects them.
__global__ void __launch_bounds__(256) k_smooth_rounds(RoundArgs a) {
  const Work& w = a.w;
  int* cnt = w.counts;
  unsigned target = 0;
  int cur = 0, nxt = 1, pen = 2;
  auto list = [&](int b) { return b == 0 ? w.D[0] : (b == 1 ? w.D[1] : w.P); };
  auto count = [&](int b) { return cnt + (b == 2 ? CN_P : cn_list(b)); };
  int r = 0, rounds = 0, sweeps = 0, tag = a.tag0 - 2, ptag = a.ptag;
  bool moved = a.moved != 0, over = false, fresh = false;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *cand_count(cnt, 0) = 0;
    cnt[CN_E] = cnt[CN_S] = 0;
  }
  if (!grid_barrier(a.bar, target, a.st)) return;
  // a list longer than the limit is left to the one-kernel-per-phase rounds
  int n = ld_volatile(count(cur));
  const int tiles = gridDim.x * (blockDim.x / TW);
  while (!over && n <= a.limit && rounds < a.max_rounds) {
    tag += 2;
    int* nC = cand_count(cnt, r);
    Store S = a.S;
    S.tab.had = a.S.tab.had + (r & 1) * S.nmesh;
    // the list is complete since B2 of the last round: every block decides alike
    const bool fused = n <= min(a.fuse, kFusePasses * tiles);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      *count(nxt) = 0;
      if (fresh) *count(pen) = 0;
    }
    fresh = false;
    if (fused) {
      smooth_scan_eval_phase(S, list(cur), count(cur), w.mvxy, w.mvM, w.gains, w.C, nC, w.cmark,
                             tag, a.pass0, a.work);
      if (!grid_barrier(a.bar, target, a.st)) return;
      if (blockIdx.x == 0 && threadIdx.x == 0) *cand_count(cnt, r + 1) = 0;
    } else {
      smooth_scan_phase(S, list(cur), count(cur), w.mvM, w.C, nC, w.cmark, tag, a.pass0, w.E,
                        cnt + CN_E, false, true);
      if (!grid_barrier(a.bar, target, a.st)) return;
      if (blockIdx.x == 0 && threadIdx.x == 0) *cand_count(cnt, r + 1) = 0;
      smooth_filter_phase(S, w.E, cnt + CN_E, w.mvxy, w.mvM, w.Sl, cnt + CN_S, w.C, nC, w.cmark,
                          tag, false, a.work, true);
      if (!grid_barrier(a.bar, target, a.st)) return;
      if (blockIdx.x == 0 && threadIdx.x == 0) cnt[CN_E] = 0;
      smooth_exact_phase(S, w.Sl, cnt + CN_S, w.mvxy, w.mvM, w.gains, w.C, nC, w.cmark, tag,
                         a.work, true);
      if (!grid_barrier(a.bar, target, a.st)) return;
      if (blockIdx.x == 0 && threadIdx.x == 0) cnt[CN_S] = 0;
    }
    smooth_select_apply_phase(S, w.C, nC, w.cmark, w.smark, tag, list(nxt), count(nxt), w.dmark,
                              w.mvxy, w.mvM, w.gains, list(pen), count(pen), w.pmark, ptag, tag + 1,
                              nullptr, nullptr, true);
    if (!grid_barrier(a.bar, target, a.st)) return;
    const int nc = ld_volatile(nC), nd = ld_volatile(count(nxt)), np = ld_volatile(count(pen));
    advance_rounds(S);
    ++r;
    if (nc > 0) {
      ++rounds;
      moved = true;
      const int t = cur;
      cur = nxt;
      nxt = t;
      n = nd;
    } else {
      ++sweeps;
      over = !moved || sweeps == a.sweeps;
      if (!over) {
        const int t = cur;
        cur = pen;
        pen = t;
        n = np;
        tag += 2;
        ptag = tag;
        moved = false;
        fresh = true;
      }
    }
  }
  // every block has left the counters: the lists go to their places (D[0]
  // current, D[1] next, P pending)
  const int nn = ld_volatile(count(nxt)), np = fresh ? 0 : ld_volatile(count(pen));
  if (!grid_barrier(a.bar, target, a.st)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    cnt[CN_D0] = n;
    cnt[CN_D1] = nn;
    cnt[CN_P] = np;
    a.res[SR_ROUNDS] = rounds;
    a.res[SR_SWEEPS] = sweeps;
    a.res[SR_OVER] = over ? 1 : 0;
    a.res[SR_MOVED] = moved ? 1 : 0;
    a.res[SR_PERM] = cur | (nxt << 2) | (pen << 4);
    a.res[SR_TAGS] = (tag + 2 - a.tag0) / 2;
    a.res[SR_PTAG] = ptag;
  }
}

// ---- host helpers --------------------------------------------------------------

struct RoundIO {
  int nC;
  int overflow;
  int err;
};

RoundIO read_round(MeshSet& m) {
  RoundIO io;
  io.err = sync_counts(m, 0);
  io.nC = m.hcounts[CN_C];
  io.overflow = m.hst->overflow;
  return io;
}

void zero_counts(MeshSet& m, int first, int num) {
  cudaMemsetAsync(m.w.counts + first, 0, num * sizeof(int), m.stream);
}

// The counters of a new round (C, S, A, E, I) and of the list it fills
// (D[nxt]); the list it reads keeps its count.
void zero_round(MeshSet& m, int nxt) {
  static_assert(CN_D0 == 0 && CN_C == 1 && CN_I == 5 && CN_D1 == 7, "counter layout");
  zero_counts(m, nxt == 0 ? CN_D0 : CN_C, 7);
}

// A row overflow leaves some rows unwritten and the neighbour stamps of the
// rebuilt rows unset: rows are rebuilt from the elements and no evaluation
// made before is reused (every lo_* and the callers' pass start move to now).
int after_overflow(MeshSet& m) {
  int err = rebuild_adjacency(m, false, false);
  m.lo_coarsen = m.lo_swap = m.lo_refine = m.tag;
  return err;
}

int after_round(MeshSet& m, const RoundIO& io) {
  if (io.err) return io.err;
  if (io.overflow) return after_overflow(m);
  return PM_OK;
}

// Persistent rounds take over once a pass's list holds at most
// Tuning::rounds_limit vertices (and hand back when the next list outgrows
// it).  Defaults, measured on meshes of 8k to 20M triangles: 131072 for flips and
// smoothing (12.88 ms at 131072 against 13.2 at 32768 on the 201 x 201 mesh), 32768
// for collapses, whose longer lists run faster one vertex per thread on a full
// chip (8.08 against 8.80 ms on a 317 x 317 grid coarsened to 18k triangles).
// Colouring follows the smoothing's limit: its rounds are light too (gathers and a
// mask), and each costs two launches and a wait outside the persistent kernel.
constexpr int kRoundsThreads = 256;

// Blocks of a cooperative launch of the persistent round kernel `which`
// (0 collapse, 1 flip, 2 smoothing, 3 colouring) on this device: the tuning's blocks per
// SM (Tuning::rounds_blocks_per_sm, at most what its registers allow) on
// every SM, or 0 when the device cannot run it cooperatively (rounds stay one
// kernel per phase).
int rounds_grid(MeshSet& m, int which) {
  static std::mutex mu;
  static int occ[64][4];
  static bool known[64];
  const int dev = m.device;
  if (dev < 0 || dev >= 64 || which < 0 || which > 3) return 0;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!known[dev]) {
      int coop = 0;
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
      const void* ks[] = {(const void*)k_coarsen_rounds, (const void*)k_swap_rounds,
                          (const void*)k_smooth_rounds, (const void*)k_colour_rounds};
      for (int k = 0; k < 4; ++k) {
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, ks[k], kRoundsThreads, 0) !=
            cudaSuccess)
          b = 0;
        occ[dev][k] = coop ? b : 0;
      }
      cudaGetLastError();
      known[dev] = true;
    }
  }
  const int b = std::min(occ[dev][which], tuning().rounds_blocks_per_sm[which == 3 ? 0 : which]);
  return b >= 1 ? m.num_sms * b : 0;
}

RoundArgs round_args(MeshSet& m, int cur, int pass0, long long max_rounds) {
  RoundArgs a;
  a.S = m.S;
  a.w = m.w;
  a.st = m.st;
  a.bar = (unsigned*)(m.w.counts + CN_BAR);
  a.res = m.w.counts + CN_RES;
  a.cur = cur;
  a.tag0 = m.tag + 2;
  a.pass0 = pass0;
  a.max_rounds = (int)std::min<long long>(max_rounds, 1 << 30);
  a.limit = tuning().rounds_limit[0];
  a.icap = 0;
  a.ptag = 0;
  a.sweeps = 0;
  a.moved = 0;
  a.before = nullptr;
  a.fuse = 0;
  a.work = nullptr;
  return a;
}

struct RoundsOut {
  int rounds = 0;    // rounds run, the last one empty when the pass completed
  int cur = 0;       // list the next round reads
  int complete = 0;
  RoundIO io{0, 0, 0};
};

// One cooperative launch of persistent rounds.
int launch_rounds(MeshSet& m, int which, const void* kernel, const char* name, RoundArgs& a) {
  a.work = prof_work(name);
  void* args[] = {&a};
  __atomic_fetch_add(&g_launches, 1ull, __ATOMIC_RELAXED);
  int slot = g_prof_on ? prof_begin(name, m.stream) : -1;
  cudaError_t e = cudaLaunchCooperativeKernel(kernel, dim3(rounds_grid(m, which)),
                                              dim3(kRoundsThreads), args, 0, m.stream);
  if (slot >= 0) prof_end(slot, m.stream);
  if (e != cudaSuccess) {
    set_last_error(std::string("cooperative launch: ") + cudaGetErrorString(e));
    return PM_ERR_CUDA;
  }
  return PM_OK;
}

// The same, then the read-back of every counter and the status.  Advances the tag
// past the rounds that ran.
int run_rounds(MeshSet& m, int which, const void* kernel, const char* name, RoundArgs& a,
               RoundsOut& out, bool& bar_clear) {
  // (the first launch of an operator finds the counters cleared)
  if (!bar_clear) cudaMemsetAsync(a.bar, 0, sizeof(unsigned), m.stream);
  bar_clear = false;
  if (int err = launch_rounds(m, which, kernel, name, a)) return err;
  out.io = read_round(m);
  if (out.io.err) return out.io.err;
  if (which == 2) {
    m.tag += 2 * m.hcounts[CN_RES + SR_TAGS];
    return PM_OK;
  }
  out.rounds = m.hcounts[CN_RES];
  out.cur = m.hcounts[CN_RES + 1];
  out.complete = m.hcounts[CN_RES + 2];
  m.tag += 2 * out.rounds;
  return PM_OK;
}

// Colours every active mesh whose parameters ask for colour-class sets, at
// the start of a collapse, flip or smoothing pass: speculative rounds until
// no vertex is left uncoloured (each round keeps at least the proposal of
// the highest priority; the cap is far beyond any mesh's rounds).
int colour_set(MeshSet& m) {
  bool any = false;
  for (int x : m.select) any |= x == PM_SELECT_COLOUR;
  if (!any) return PM_OK;
  Work& w = m.w;
  const int g = grid_for(m, m.S.vused);
  const bool persist = rounds_grid(m, 3) > 0;
  const int limit = tuning().rounds_limit[2];
  bool bar_clear = true;
  zero_counts(m, 0, CN_NUM);
  PM_LAUNCH(k_colour_init, g, BLOCK, 0, m.stream, m.S, w.D[0], w.counts + CN_D0);
  int cur = 0, nlist = 0;  // entries of the list; unknown (0) at first
  for (int it = 0; it < (1 << 20); ++it) {
    if (persist && nlist <= limit) {
      RoundArgs a = round_args(m, cur, 0, 1 << 20);
      a.limit = limit;
      RoundsOut o;
      int err =
          run_rounds(m, 3, (const void*)k_colour_rounds, "k_colour_rounds", a, o, bar_clear);
      if (err) return err;
      if (o.complete) return PM_OK;
      cur = o.cur;
      nlist = m.hcounts[cn_list(cur)];
      if (nlist <= limit) continue;  // the round cap
    }
    const int nxt = 1 - cur;
    const int rt = (m.tag += 2);
    zero_counts(m, cn_list(nxt), 1);
    PM_LAUNCH(k_colour_propose, g, BLOCK, 0, m.stream, m.S, w.D[cur], w.counts + cn_list(cur),
              w.cprop, w.cstamp, rt);
    PM_LAUNCH(k_colour_resolve, g, BLOCK, 0, m.stream, m.S, w.D[cur], w.counts + cn_list(cur),
              w.cprop, w.cstamp, rt, w.D[nxt], w.counts + cn_list(nxt));
    RoundIO io = read_round(m);
    if (io.err) return io.err;
    cur = nxt;
    nlist = m.hcounts[cn_list(cur)];
    if (nlist == 0) return PM_OK;
  }
  set_last_error("colouring did not finish");
  return PM_ERR_INVALID_MESH;
}

}  // namespace

// ---------------------------------------------------------------------------
// Operator loops (host)
// ---------------------------------------------------------------------------

// An iteration's collapses, flips and first split marks waited on the host three
// times (10-20 us each on small meshes, the chip idle); queued one behind the other
// they wait once: 1140 against 1205 us on a 41 x 41 mesh, 11.80 against 11.92 ms at
// 201 x 201.  A launch that finds the pass before it incomplete (list too long, or a
// row that outgrew its width) does nothing, and the operators go on from there.
int ops_ahead(MeshSet& m, Ahead& h) {
  const Tuning tu = tuning();
  for (int x : m.select)
    if (x == PM_SELECT_COLOUR) return PM_OK;  // a colouring comes before each pass
  if (rounds_grid(m, 0) == 0 || rounds_grid(m, 1) == 0) return PM_OK;
  // the first lists of a call hold every vertex; the later ones are known only on the
  // device, where a pass whose list is too long hands back at once
  if (m.lo_coarsen == m.tag && m.S.vused > tu.rounds_limit[0]) return PM_OK;
  Work& w = m.w;
  const int n = m.nmesh;
  int* const second = w.counts + cn_second(n);
  const int* const none = nullptr;
  const int* const rounds_c = w.counts + CN_RES;
  const int* const rounds_s = second + CN_RES;
  const DevStatus* const st = m.st;
  zero_counts(m, 0, CN_NUM);
  cudaMemsetAsync(second, 0, CN_NUM * sizeof(int), m.stream);
  const int tag = m.tag;

  int bs = tu.block[TO_COARSEN];
  select_ops(m, OS_COARSEN);
  PM_LAUNCH(k_init_list, grid_tuned(m, m.S.vused, bs, tu.blocks_per_sm[TO_COARSEN]), bs, 0,
            m.stream, m.S, 0, w.D[0], w.counts + CN_D0, m.S.evc, m.lo_coarsen, none, st);
  RoundArgs a = round_args(m, 0, tag, 1 << 30);
  a.limit = tu.rounds_limit[0];
  if (int err = launch_rounds(m, 0, (const void*)k_coarsen_rounds, "k_coarsen_rounds", a))
    return err;

  bs = tu.block[TO_SWAP];
  select_ops(m, OS_SWAP);
  PM_LAUNCH(k_init_list, grid_tuned(m, m.S.vused, bs, tu.blocks_per_sm[TO_SWAP]), bs, 0, m.stream,
            m.S, 0, w.D[0], second + CN_D0, m.S.evs, m.lo_swap, rounds_c, st);
  a = round_args(m, 0, tag, 1 << 30);
  a.w.counts = second;
  a.bar = (unsigned*)(second + CN_BAR);
  a.res = second + CN_RES;
  a.icap = m.S.vslots * 6 + 64;
  a.limit = tu.rounds_limit[1];
  a.fuse = tu.fuse_limit[0];
  a.before = rounds_c;
  if (int err = launch_rounds(m, 1, (const void*)k_swap_rounds, "k_swap_rounds", a)) return err;

  bs = tu.block[TO_REFINE];
  select_ops(m, OS_REFINE);
  PM_LAUNCH(k_refine_mark, grid_tuned(m, m.S.vused, bs, tu.blocks_per_sm[TO_REFINE]), bs, 0,
            m.stream, m.S, w.vcnt, w.vmask, tag + 2, tag, m.lo_refine, rounds_s, rounds_c, st);
  // (without marks there are no counts either: the vertex slots are not read)
  scan_exclusive(w.vcnt, w.vscan, m.S.vused, m.scan, m.st, m.stream, rounds_s + 2);
  PM_LAUNCH(k_refine_newcount, (n + 127) / 128, 128, 0, m.stream, m.S, (const int*)w.vscan,
            w.counts, rounds_s, st);
  if (int err = sync_counts(m, kMeshWords * n + CN_NUM)) return err;

  const int* rc = m.hcounts + CN_RES;
  const int* rs = m.hcounts + cn_second(n) + CN_RES;
  m.tag = tag + 2 * rc[0];
  h.coarsen = rc[2] ? 1 : 2;
  h.pass0_c = tag;
  h.cur_c = rc[1];
  if (h.coarsen != 1) return PM_OK;
  h.swap = rs[2] ? 1 : 2;
  h.pass0_s = m.tag;
  h.cur_s = rs[1];
  m.tag += 2 * rs[0];
  if (h.swap == 1) {
    h.mark_tag = (m.tag += 2);
  } else {  // op_swap goes on with the first set of counters
    cudaMemcpyAsync(w.counts, second, CN_NUM * sizeof(int), cudaMemcpyDeviceToDevice, m.stream);
    std::copy(m.hcounts + cn_second(n), m.hcounts + cn_second(n) + CN_NUM, m.hcounts);
  }
  return PM_OK;
}

// Rounds of collapses until no dirty vertex has a valid collapse.  The first
// round's list leaves out vertices whose last collapse evaluation found
// nothing and whose inputs have not changed since.
int op_coarsen(MeshSet& m, int max_rounds, const Ahead& h) {
  if (h.coarsen == 1) return PM_OK;
  if (int err = colour_set(m)) return err;
  const Tuning tu = tuning();
  const int bs = tu.block[TO_COARSEN], bps = tu.blocks_per_sm[TO_COARSEN];
  const int rlimit = tu.rounds_limit[0];
  Work& w = m.w;
  const int gv = grid_tuned(m, m.S.vused, bs, bps);
  int pass0 = m.tag;
  const bool persist = rounds_grid(m, 0) > 0;
  bool bar_clear = h.coarsen == 0;
  if (h.coarsen == 0) {
    zero_counts(m, 0, CN_NUM);
    PM_LAUNCH(k_init_list, gv, bs, 0, m.stream, m.S, 0, w.D[0], w.counts + CN_D0, m.S.evc,
              m.lo_coarsen, (const int*)nullptr, (const DevStatus*)m.st);
  }
  // entries of the list the next round reads; unknown (0) at first: the
  // persistent launch itself hands a long first list back
  int nlist = 0;
  int cur = 0;
  bool complete = false;
  if (h.coarsen == 2) {  // behind the rounds of ops_ahead
    pass0 = h.pass0_c;
    cur = h.cur_c;
    if (m.hst->overflow)
      if (int err = after_overflow(m)) return err;
    nlist = m.hcounts[cn_list(cur)];
  }
  for (long long nr = 0; max_rounds == 0 || nr < max_rounds;) {
    if (m.lo_coarsen > pass0) pass0 = m.lo_coarsen;  // rows were rebuilt after an overflow
    if (persist && nlist >= 0 && nlist <= rlimit) {
      RoundArgs a = round_args(m, cur, pass0, max_rounds == 0 ? (1LL << 30) : max_rounds - nr);
      a.limit = rlimit;
      RoundsOut o;
      int err = run_rounds(m, 0, (const void*)k_coarsen_rounds, "k_coarsen_rounds", a, o, bar_clear);
      if (err) return err;
      nr += o.rounds - o.complete;
      cur = o.cur;
      if (o.complete) {
        complete = true;
        break;
      }
      if ((err = after_round(m, o.io))) return err;
      nlist = m.hcounts[cn_list(cur)];
      continue;
    }
    int tag = (m.tag += 2);
    int nxt = 1 - cur;
    zero_round(m, nxt);
    PM_LAUNCH(k_coarsen_scan, gv, bs, 0, m.stream, m.S, w.D[cur], w.counts + cn_list(cur),
              w.target, w.cand, w.C, w.counts + CN_C, w.cmark, tag, pass0, w.E,
              w.counts + CN_E);
    // one dense wave checking every vertex's first candidate, then the other
    // candidates of the vertices whose first one failed
    PM_LAUNCH(k_coarsen_check, gv, bs, 0, m.stream, m.S, w.E, w.counts + CN_E, w.Sl,
              w.counts + CN_S, w.target, w.cand, w.C, w.counts + CN_C, w.cmark, tag,
              prof_work("k_coarsen_check"));
    PM_LAUNCH(k_coarsen_rest, gv, bs, 0, m.stream, m.S, w.Sl, w.counts + CN_S, w.target, w.cand,
              w.C, w.counts + CN_C, w.cmark, tag, prof_work("k_coarsen_rest"));
    zero_counts(m, CN_CL, 1);
    PM_LAUNCH(k_coarsen_select_apply, gv, bs, 0, m.stream, m.S, w.C, w.counts + CN_C, w.cmark,
              w.smark, tag, w.target, w.A, w.counts + CN_A, w.amark, w.D[nxt],
              w.counts + cn_list(nxt), w.dmark, w.clist, w.counts + CN_CL,
              (unsigned*)(w.counts + CN_DONE));
    PM_LAUNCH(k_coarsen_commit, gv, bs, 0, m.stream, m.S, w.A, w.counts + CN_A, w.target,
              w.smark, tag, m.st);
    PM_LAUNCH(k_refine_quality, gv, bs, 0, m.stream, m.S, w.clist, w.counts + CN_CL, nullptr);
    RoundIO io = read_round(m);
    if (io.err) return io.err;
    if (io.nC == 0) {
      complete = true;
      break;
    }
    int err = after_round(m, io);
    if (err) return err;
    cur = nxt;
    ++nr;
    nlist = m.hcounts[cn_list(cur)];
  }
  if (!complete) m.lo_coarsen = m.tag;  // some vertex may still have a collapse
  return PM_OK;
}

// Rounds of flips until no dirty vertex has an improving flip.
int op_swap(MeshSet& m, int max_rounds, const Ahead& h) {
  if (h.swap == 1) return PM_OK;
  if (int err = colour_set(m)) return err;
  const Tuning tu = tuning();
  const int bs = tu.block[TO_SWAP], bps = tu.blocks_per_sm[TO_SWAP];
  const int rlimit = tu.rounds_limit[1];
  Work& w = m.w;
  const int gv = grid_tuned(m, m.S.vused, bs, bps);
  int pass0 = m.tag;
  const int icap = m.S.vslots * 6 + 64;
  const bool persist = rounds_grid(m, 1) > 0;
  bool bar_clear = h.swap == 0;
  if (h.swap == 0) {
    zero_counts(m, 0, CN_NUM);
    PM_LAUNCH(k_init_list, gv, bs, 0, m.stream, m.S, 0, w.D[0], w.counts + CN_D0, m.S.evs,
              m.lo_swap, (const int*)nullptr, (const DevStatus*)m.st);
  }
  int nlist = 0;  // unknown at first (see op_coarsen)
  int cur = 0;
  bool complete = false;
  if (h.swap == 2) {  // behind the rounds of ops_ahead
    pass0 = h.pass0_s;
    cur = h.cur_s;
    if (m.hst->overflow)
      if (int err = after_overflow(m)) return err;
    nlist = m.hcounts[cn_list(cur)];
  }
  for (long long nr = 0; max_rounds == 0 || nr < max_rounds;) {
    if (m.lo_swap > pass0) pass0 = m.lo_swap;  // rows were rebuilt after an overflow
    if (persist && nlist >= 0 && nlist <= rlimit) {
      RoundArgs a = round_args(m, cur, pass0, max_rounds == 0 ? (1LL << 30) : max_rounds - nr);
      a.icap = icap;
      a.limit = rlimit;
      a.fuse = tu.fuse_limit[0];
      RoundsOut o;
      int err = run_rounds(m, 1, (const void*)k_swap_rounds, "k_swap_rounds", a, o, bar_clear);
      if (err) return err;
      nr += o.rounds - o.complete;
      cur = o.cur;
      if (o.complete) {
        complete = true;
        break;
      }
      if ((err = after_round(m, o.io))) return err;
      nlist = m.hcounts[cn_list(cur)];
      continue;
    }
    int tag = (m.tag += 2);
    int nxt = 1 - cur;
    zero_round(m, nxt);
    PM_LAUNCH(k_swap_scan, gv, bs, 0, m.stream, m.S, w.D[cur], w.counts + cn_list(cur), w.opA,
              w.C, w.counts + CN_C, w.cmark, tag, pass0, w.E, w.counts + CN_E, w.items,
              w.counts + CN_I, icap, w.gains, m.st);
    PM_LAUNCH(k_swap_edge, grid_tuned(m, 6LL * m.S.vslots, bs, bps), bs, 0, m.stream, m.S, w.items,
              w.counts + CN_I, icap, w.gains, tag, prof_work("k_swap_edge"));
    PM_LAUNCH(k_swap_pick, gv, bs, 0, m.stream, m.S, w.E, w.counts + CN_E, w.gains, w.opA,
              w.opK2, w.C, w.counts + CN_C, w.cmark, tag);
    zero_counts(m, CN_CL, 1);
    PM_LAUNCH(k_swap_select_apply, gv, bs, 0, m.stream, m.S, w.C, w.counts + CN_C, w.cmark,
              w.smark, tag, w.opA, w.opK2, w.A, w.counts + CN_A, w.amark, w.D[nxt],
              w.counts + cn_list(nxt), w.dmark, w.clist, w.counts + CN_CL,
              (unsigned*)(w.counts + CN_DONE));
    PM_LAUNCH(k_swap_commit, gv, bs, 0, m.stream, m.S, w.A, w.counts + CN_A, w.opA, w.opK2,
              w.smark, tag, m.st);
    PM_LAUNCH(k_refine_quality, gv, bs, 0, m.stream, m.S, w.clist, w.counts + CN_CL, nullptr);
    RoundIO io = read_round(m);
    if (io.err) return io.err;
    if (io.nC == 0) {
      complete = true;
      break;
    }
    int err = after_round(m, io);
    if (err) return err;
    cur = nxt;
    ++nr;
    nlist = m.hcounts[cn_list(cur)];
  }
  if (!complete) m.lo_swap = m.tag;
  return PM_OK;
}

// Rounds of splits until no edge is longer than L_up.  Capacity is checked
// (and grown) before any new vertex or element is written.  A round's split is
// not waited for: the next round's marks are queued behind it, and one read-back
// brings the sizes after the split and the new marks' count (a row that outgrew W
// in the split voids those marks).  With `renumber_queued`, marks behind a split
// (which mostly find nothing) also take the renumbering's counts along.
int op_refine(MeshSet& m, int max_rounds, const Ahead& h, bool* renumber_queued) {
  const Tuning tu = tuning();
  const int bs = tu.block[TO_REFINE], bps = tu.blocks_per_sm[TO_REFINE];
  Work& w = m.w;
  const int n = m.nmesh;
  int pass0 = h.mark_tag ? h.mark_tag - 2 : m.tag;
  int marked = h.mark_tag;  // the first marks are there already, with their count
  bool complete = false;
  bool split = false;  // a split is queued whose sizes have not been read back
  std::vector<int> newv(n);
  // the sizes after a queued split; rows rebuilt wider when one outgrew W
  auto settle = [&](bool& again) -> int {
    for (int i = 0; i < n; ++i) {
      m.nv[i] = m.hcounts[cn_sizes(n) + i];
      m.ne[i] = m.hcounts[cn_sizes(n) + n + i];
    }
    set_used(m);
    split = false;
    again = m.hst->overflow != 0;
    return again ? after_overflow(m) : PM_OK;
  };
  for (long long nr = 0; max_rounds == 0 || nr < max_rounds;) {
    const int gv = grid_tuned(m, m.S.vused, bs, bps);
    const int tag = marked ? marked : (m.tag += 2);
    if (m.lo_refine > pass0) pass0 = m.lo_refine;  // storage was regrown
    const bool ahead = renumber_queued && split;
    if (!marked) {
      PM_LAUNCH(k_refine_mark, gv, bs, 0, m.stream, m.S, w.vcnt, w.vmask, tag, pass0, m.lo_refine,
                (const int*)nullptr, (const int*)nullptr, (const DevStatus*)m.st);
      scan_exclusive(w.vcnt, w.vscan, m.S.vused, m.scan, m.st, m.stream);
      PM_LAUNCH(k_refine_newcount, (n + 127) / 128, 128, 0, m.stream, m.S, (const int*)w.vscan,
                w.counts, (const int*)nullptr, (const DevStatus*)m.st);
      // (beside the marks' scan, which a split still needs; the counts are spent)
      if (ahead) renumber_queue(m, w.vcnt);
      if (int err = ahead ? sync_call(m) : sync_counts(m, kMeshWords * n)) return err;
    }
    marked = 0;
    std::copy(m.hcounts + cn_newv(n), m.hcounts + cn_newv(n) + n, newv.begin());
    if (split) {
      bool again = false;
      if (int err = settle(again)) return err;
      if (again) continue;
    }
    // A growth moves every mesh of the set, so when one mesh needs room, every
    // mesh that this round leaves with little gets half as much again as it
    // needs now, and some thousands at least (spare_slots; the next rounds of a
    // refinement pass usually split again).
    long long total = 0;
    bool need_grow = false;
    for (int i = 0; i < n; ++i) {
      total += newv[i];
      if ((long long)m.nv[i] + newv[i] > m.vcap[i] || (long long)m.ne[i] + 2LL * newv[i] > m.ecap[i])
        need_grow = true;
    }
    if (total == 0) {
      complete = true;
      if (ahead) {
        *renumber_queued = true;
        std::swap(w.vcnt, w.vscan);
      }
      break;
    }
    if (need_grow) {
      std::vector<int> vcap = m.vcap, ecap = m.ecap;
      for (int i = 0; i < n; ++i) {
        if (newv[i] == 0) continue;
        const long long vneed = (long long)m.nv[i] + newv[i] + 64;
        const long long eneed = (long long)m.ne[i] + 2LL * newv[i] + 64;
        if (vneed + vneed / 8 > m.vcap[i])
          vcap[i] = (int)std::min<long long>(
              vneed + std::max<long long>(vneed / 2, spare_slots(vneed, 8192, n)), 1LL << 30);
        if (eneed + eneed / 8 > m.ecap[i])
          ecap[i] = (int)std::min<long long>(
              eneed + std::max<long long>(eneed / 2, spare_slots(eneed, 16384, n)), 1LL << 30);
      }
      cudaError_t e = grow(m, vcap, ecap, m.S.W);
      if (e != cudaSuccess) {
        set_last_error(std::string("growing mesh storage: ") + cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? PM_ERR_OOM : PM_ERR_CUDA;
      }
      continue;  // redo this round on the new layout
    }
    const int ge = grid_tuned(m, m.S.eused, bs, bps);
    const int stamp = tag + 1;
    const int vend = m.vbase.back() + m.nv.back() + newv.back();  // above every new vertex
    PM_LAUNCH(k_refine_newverts, gv, bs, 0, m.stream, m.S, w.vscan, w.vmask, stamp, w.opA);
    PM_LAUNCH(k_refine_count, ge, bs, 0, m.stream, m.S, w.vscan, w.vmask, w.ecnt, w.emid,
              w.elist, w.counts + CN_EL);
    scan_exclusive(w.ecnt, w.escan, m.S.eused, m.scan, m.st, m.stream);
    PM_LAUNCH(k_refine_split, ge, bs, 0, m.stream, m.S, w.escan, w.emid, w.elist,
              w.counts + CN_EL, w.clist, w.counts + CN_CL, stamp);
    PM_LAUNCH(k_refine_quality, ge, bs, 0, m.stream, m.S, w.clist, w.counts + CN_CL, nullptr);
    // rows of the vertices whose elements changed: the new ones, then the old ones
    const int vnew = n == 1 ? m.nv[0] : 0;
    PM_LAUNCH(k_refine_rows, grid_tuned(m, vend - vnew, bs, bps), bs, 0, m.stream, m.S, vnew, vend, 1,
              (const int*)w.escan, (const int4*)w.opA, stamp, m.st);
    PM_LAUNCH(k_refine_rows, gv, bs, 0, m.stream, m.S, 0, m.S.vused, 0, (const int*)w.escan,
              (const int4*)w.opA, stamp, m.st);
    PM_LAUNCH(k_refine_sizes, (n + 127) / 128, 128, 0, m.stream, m.S, (const int*)w.vscan,
              (const int*)w.escan, w.counts);
    split = true;
    // every slot lies below these bounds (the exact element sizes follow with the
    // next read-back)
    m.S.vused = vend;
    m.S.eused = m.S.eused + 2 * newv.back();
    ++nr;
  }
  if (split) {
    if (int err = sync_counts(m, kMeshWords * n)) return err;
    bool again = false;
    if (int err = settle(again)) return err;
  }
  if (!complete) m.lo_refine = m.tag;
  return PM_OK;
}

// Laplacian sweeps, each a sequence of rounds over the sweep's pending set.
int op_smooth(MeshSet& m, int max_sweeps, int max_rounds) {
  // smoothing changes no topology: one colouring serves every sweep
  if (int err = colour_set(m)) return err;
  const Tuning tu = tuning();
  const int bs = tu.block[TO_SMOOTH], bps = tu.blocks_per_sm[TO_SMOOTH];
  const int rlimit = tu.rounds_limit[2];
  Work& w = m.w;
  const int gv = grid_tuned(m, m.S.vused, bs, bps);
  const int pass0 = m.tag;
  const bool persist = rounds_grid(m, 2) > 0;
  bool bar_clear = true;
  zero_counts(m, 0, CN_NUM);
  PM_LAUNCH(k_init_list, gv, bs, 0, m.stream, m.S, 1, w.D[0], w.counts + CN_D0, nullptr, 0,
            (const int*)nullptr, (const DevStatus*)m.st);
  int nlist = 0;  // unknown at first (see op_coarsen)
  long long nr = 0;
  int cur = 0, ptag = 0;
  bool moved = false, fresh = true;
  for (int sweep = 0; sweep < max_sweeps && (max_rounds == 0 || nr < max_rounds);) {
    if (fresh) {
      ptag = (m.tag += 2);  // stamp of the next sweep's pending list
      if (sweep > 0) zero_counts(m, CN_P, 1);
      moved = fresh = false;
    }
    if (persist && nlist >= 0 && nlist <= rlimit) {
      if (cur == 1) {  // the launch starts from D[0]
        std::swap(w.D[0], w.D[1]);
        cudaMemcpyAsync(w.counts + CN_D0, w.counts + CN_D1, sizeof(int), cudaMemcpyDeviceToDevice,
                        m.stream);
        cur = 0;
      }
      RoundArgs a = round_args(m, cur, pass0, max_rounds == 0 ? (1LL << 30) : max_rounds - nr);
      a.ptag = ptag;
      a.sweeps = max_sweeps - sweep;
      a.moved = moved ? 1 : 0;
      a.limit = rlimit;
      a.fuse = tu.fuse_limit[1];
      RoundsOut o;
      int err = run_rounds(m, 2, (const void*)k_smooth_rounds, "k_smooth_rounds", a, o, bar_clear);
      if (err) return err;
      const int* res = m.hcounts + CN_RES;
      nr += res[SR_ROUNDS];
      sweep += res[SR_SWEEPS];
      moved = res[SR_MOVED] != 0;
      ptag = res[SR_PTAG];
      int* const buf[3] = {w.D[0], w.D[1], w.P};
      w.D[0] = buf[res[SR_PERM] & 3];
      w.D[1] = buf[(res[SR_PERM] >> 2) & 3];
      w.P = buf[(res[SR_PERM] >> 4) & 3];
      nlist = m.hcounts[CN_D0];
      if (res[SR_OVER]) break;
      continue;
    }
    int tag = (m.tag += 2);
    int nxt = 1 - cur;
    zero_round(m, nxt);
    PM_LAUNCH(k_smooth_scan, gv, bs, 0, m.stream, m.S, w.D[cur], w.counts + cn_list(cur),
              w.mvM, w.C, w.counts + CN_C, w.cmark, tag, pass0, w.E, w.counts + CN_E);
    PM_LAUNCH(k_smooth_filter, gv, bs, 0, m.stream, m.S, w.E, w.counts + CN_E, w.mvxy, w.mvM,
              w.Sl, w.counts + CN_S, w.C, w.counts + CN_C, w.cmark, tag,
              prof_work("k_smooth_filter"));
    PM_LAUNCH(k_smooth_eval, grid_tuned(m, (long long)m.S.vused * TW, bs, bps), bs, 0, m.stream,
              m.S, w.Sl, w.counts + CN_S, w.mvxy, w.mvM, w.gains, w.C, w.counts + CN_C, w.cmark,
              tag, prof_work("k_smooth_eval"));
    zero_counts(m, CN_CL, 1);
    PM_LAUNCH(k_smooth_select_apply, gv, bs, 0, m.stream, m.S, w.C, w.counts + CN_C,
              w.cmark, w.smark, tag, w.D[nxt], w.counts + cn_list(nxt), w.dmark, w.mvxy, w.mvM,
              w.gains, w.P, w.counts + CN_P, w.pmark, ptag, tag + 1, w.clist, w.counts + CN_CL,
              (unsigned*)(w.counts + CN_DONE));
    PM_LAUNCH(k_refine_quality, gv, bs, 0, m.stream, m.S, w.clist, w.counts + CN_CL, nullptr);
    RoundIO io = read_round(m);
    if (io.err) return io.err;
    if (io.nC > 0) {
      ++nr;
      moved = true;
      cur = nxt;
      nlist = m.hcounts[cn_list(cur)];
      continue;
    }
    ++sweep;
    if (!moved) break;
    // the next sweep's pending list becomes the current list
    std::swap(w.D[0], w.P);
    cudaMemcpyAsync(w.counts + CN_D0, w.counts + CN_P, sizeof(int), cudaMemcpyDeviceToDevice,
                    m.stream);
    cur = 0;
    nlist = m.hcounts[CN_P];
    fresh = true;
  }
  return PM_OK;
}

// Rounds of optimisation-based smoothing over all interior vertices.
int op_opt_smooth(MeshSet& m, int nrounds, int max_rounds) {
  const Tuning tu = tuning();
  const int bs = tu.block[TO_SMOOTH], bps = tu.blocks_per_sm[TO_SMOOTH];
  Work& w = m.w;
  const int gv = grid_tuned(m, m.S.vused, bs, bps);
  zero_counts(m, 0, CN_NUM);
  PM_LAUNCH(k_init_list, gv, bs, 0, m.stream, m.S, 1, w.C, w.counts + CN_C, nullptr, 0,
            (const int*)nullptr, (const DevStatus*)m.st);
  for (int it = 0; it < nrounds && (max_rounds == 0 || it < max_rounds); ++it) {
    int tag = (m.tag += 2);
    zero_counts(m, CN_S, 1);
    PM_LAUNCH(k_stamp_list, gv, bs, 0, m.stream, m.S, w.C, w.counts + CN_C, w.cmark, tag);
    PM_LAUNCH(k_select, gv, bs, 0, m.stream, m.S, w.C, w.counts + CN_C, w.cmark, w.smark, tag,
              w.Sl, w.counts + CN_S, nullptr, nullptr, nullptr);
    PM_LAUNCH(k_opt_apply, grid_tuned(m, (long long)m.S.vused * TW, bs, bps), bs, 0, m.stream, m.S, w.Sl,
              w.counts + CN_S, w.gains, tag + 1);
  }
  return PM_OK;  // the caller's read-back waits
}

}  // namespace pm

// Test support (see pm.h): a grid barrier that nothing completes gives up
// after limit_ms and reports PM_ERR_TIMEOUT through the status word.
extern "C" pm_status pm_selftest_wait_timeout(double limit_ms, int32_t* device_status,
                                              double* elapsed_ms) {
  using namespace pm;
  if (!device_status || !elapsed_ms || !(limit_ms > 0.0) || !(limit_ms <= 2000.0))
    return PM_ERR_INVALID_ARG;
  int dev = 0, sms = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess)
    return PM_ERR_CUDA;
  if (!coop || sms < 1) return PM_ERR_CUDA;
  unsigned* bar = nullptr;
  DevStatus* st = nullptr;
  if (cudaMalloc(&bar, sizeof(unsigned)) != cudaSuccess) return PM_ERR_OOM;
  if (cudaMalloc(&st, sizeof(DevStatus)) != cudaSuccess) {
    cudaFree(bar);
    return PM_ERR_OOM;
  }
  cudaMemset(bar, 0, sizeof(unsigned));
  cudaMemset(st, 0, sizeof(DevStatus));
  unsigned long long limit_ns = (unsigned long long)(limit_ms * 1e6);
  void* args[] = {&bar, &st, &limit_ns};
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  cudaEventRecord(e0);
  cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_selftest_barrier, dim3(sms),
                                              dim3(256), args, 0, 0);
  cudaEventRecord(e1);
  if (e == cudaSuccess) e = cudaEventSynchronize(e1);
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  DevStatus h{};
  if (e == cudaSuccess) e = cudaMemcpy(&h, st, sizeof(DevStatus), cudaMemcpyDeviceToHost);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(bar);
  cudaFree(st);
  if (e != cudaSuccess) return PM_ERR_CUDA;
  *device_status = h.err;
  *elapsed_ms = ms;
  return PM_OK;
}
