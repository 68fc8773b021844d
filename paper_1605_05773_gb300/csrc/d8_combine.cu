// d8_combine.cu -- the combine of the unit-count pipeline (Algorithms 5-6),
// layered as the paper's conclusion suggests.
//
// Level 0 units are the tiles; each has a perimeter summary (per perimeter
// slot: the exit of the slot's in-tile path, and the in-tile count at exits).
// A level-l unit ("group") is a G x G block of level-(l-1) units.  The exits
// of the children form a forest inside the group: a child exit's parent is
// the child exit that its successor's path reaches next.  k_group_up solves
// that forest in shared memory with the same last-arriver walks as the tiles
// (Algorithm 2 on the exit forest) and writes the group's own perimeter
// summary in the same format -- so the next level runs the same kernel.
// Above the last shared-memory level, k_top_* solve the remaining exit forest
// in global memory: the master's queue method (Algorithms 5-6) with global
// atomics, a short walk because few units remain.  k_group_down then runs
// each level back down: the resolved inflow across a group's border seeds
// its child exits and the same walks give every child exit its final area;
// at level 0 the final areas of the tile exits give the tiles' receivers their
// inflow, which the finalising pass reads.
//
// Unit counts travel as uint32, weighted areas as float-float values (fp32
// arithmetic throughout, with compensated atomic adds).
#include <cstring>
#include <type_traits>

#include "d8_device.cuh"

namespace d8 {

namespace cmb {

// threads per group: 8 or 16 child slots each (with 16 at 4096 slots too the combine
// of weighted areas took 136 us at 1001 x 777, where a group's latency counts,
// for 112 at the time; 416 and 418 us at 8192 x 8192)
template <int S, int G>
constexpr int NTG = G * G * 4 * S >= 8192 ? 1024 : G * G * 4 * S / 8;
constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr uint16_t N_ROOT = 0xFFFFu;  // path ends inside the group
constexpr uint16_t N_OUT = 0xFFFEu;   // parent lies outside the group (a group exit)
constexpr uint16_t N_NONE = 0xFFFDu;  // not an exit slot

template <int S, int G, class V>
struct GroupLayout {
  static constexpr int NS = G * G * 4 * S;  // child slots of a group
  static constexpr size_t off_spx = 0;                                       // u16 child exit codes
  static constexpr size_t off_val = ((size_t)NS * 2 + 15) / 16 * 16;         // value
  static constexpr size_t off_pd = off_val + (size_t)NS * sizeof(V);         // u32 parent << 16 | children left
  static constexpr size_t off_src = off_pd + (size_t)NS * 4;                 // u16 source lists
  // (parents, counts and sources together also hold the receivers' inflow)
  static constexpr size_t off_misc = off_pd + (size_t)NS * (sizeof(V) > 6 ? sizeof(V) : 6);
  static constexpr size_t bytes = off_misc + 64;
};

__device__ __forceinline__ DemDesc dem_by_index(const DemTable& t, int k) { return t.ndem == 1 ? t.one : t.table[k]; }

// Value arithmetic: uint32 counts, or float-float areas.  A float-float
// atomic add (fp32 atomics exist in shared and global memory; fp64 arithmetic
// is slow on this GPU) adds the high part with an atomic that returns the old
// value, takes that add's exact rounding error by TwoSum and adds it with the
// low part into the low word: only the rounding of the low word's own sums is
// lost.  The parts are not renormalised between adds, which float-float
// addition tolerates.
__device__ __forceinline__ uint32_t vadd(uint32_t a, uint32_t b) { return a + b; }
__device__ __forceinline__ ff vadd(ff a, ff b) { return ff_add(a, b); }
__device__ __forceinline__ void vatomic_add(uint32_t* p, uint32_t x) { atomicAdd(p, x); }
__device__ __forceinline__ void vatomic_add(ff* p, ff x) {
  const float old = atomicAdd(&p->hi, x.hi);
  const float s = __fadd_rn(old, x.hi);
  const float bv = __fsub_rn(s, old);
  const float err = __fadd_rn(__fsub_rn(old, __fsub_rn(s, bv)), __fsub_rn(x.hi, bv));
  atomicAdd(&p->lo, __fadd_rn(err, x.lo));
}
__device__ __forceinline__ uint32_t vload_volatile(const uint32_t* p) { return *(volatile const uint32_t*)p; }
__device__ __forceinline__ ff vload_volatile(const ff* p) {
  return ff{*(volatile const float*)&p->hi, *(volatile const float*)&p->lo};
}

struct UnitGeo {
  int64_t i0, j0;
  int h, w;
};

__device__ __forceinline__ UnitGeo unit_geo(const DemDesc& d, int64_t uy, int64_t ux, int S) {
  UnitGeo u;
  u.i0 = uy * S;
  u.j0 = ux * S;
  u.h = (int)min64(S, d.H - u.i0);
  u.w = (int)min64(S, d.W - u.j0);
  return u;
}

// Load the children of group (gy, gx) and compute every child exit's parent
// inside the group and the children count of every node.
// Returns the number of child exits this thread loaded.
// pd[n]: node n's parent (bits 16..31, or N_ROOT / N_OUT / N_NONE) and its
// number of unfinished children (bits 0..14: a node's children drain into its
// child unit's perimeter of 4 S cells, each with at most five cells outside),
// one 32-bit word so that both live in native 32-bit atomics.  SINGLE: the node
// has one child in all (marked in groups of long chains, group_walk).
__device__ __forceinline__ uint32_t pd_par(uint32_t w) { return w >> 16; }
constexpr uint32_t SINGLE = 0x8000u;
__device__ __forceinline__ uint32_t pd_deg(uint32_t w) { return w & (SINGLE - 1u); }

// A group's extent in cells (ragged at the right and bottom), and that of its
// child (a, b): everything inside a group is 32-bit arithmetic.
struct GroupGeo {
  int h, w;
};
template <int S, int G>
__device__ __forceinline__ GroupGeo group_geo(const DemDesc& d, int64_t gy, int64_t gx) {
  return GroupGeo{(int)min64(G * S, d.H - gy * (G * S)), (int)min64(G * S, d.W - gx * (G * S))};
}
template <int S>
__device__ __forceinline__ int child_h(const GroupGeo& g, int a) { return min(S, g.h - a * S); }
template <int S>
__device__ __forceinline__ int child_w(const GroupGeo& g, int b) { return min(S, g.w - b * S); }

// node of the group's cell (i, j), which lies on its child's perimeter
template <int S, int G>
__device__ __forceinline__ int node_of(const GroupGeo& g, int i, int j) {
  const int a = (int)((unsigned)i / S), b = (int)((unsigned)j / S);
  return (a * G + b) * (4 * S) + slot_of(i - a * S, j - b * S, child_h<S>(g, a), child_w<S>(g, b), S);
}

// the cell of node n, relative to the group
template <int S, int G>
__device__ __forceinline__ void cell_of(const GroupGeo& g, int n, int& i, int& j) {
  const int lt = (int)((unsigned)n / (4 * S)), a = (int)((unsigned)lt / G), b = (int)((unsigned)lt % G);
  slot_cell(n - lt * (4 * S), child_h<S>(g, a), child_w<S>(g, b), S, i, j);
  i += a * S;
  j += b * S;
}

// The node that child exit n (exit code pe) drains into, or -1 if its cell
// lies in another group.
template <int S, int G>
__device__ __forceinline__ int target_node(const GroupGeo& g, int n, uint16_t pe) {
  int i, j;
  cell_of<S, G>(g, n, i, j);
  i += code_di(pe & 7);
  j += code_dj(pe & 7);
  if ((unsigned)i >= (unsigned)(G * S) || (unsigned)j >= (unsigned)(G * S)) return -1;
  return node_of<S, G>(g, i, j);
}

// spx[] of a child exit once it is loaded: the node it drains into, or XN_OUT and
// its code when that lies in another group.  (Finding the node takes some fifty
// instructions, and the receivers' inflow asks for it again: with that, the
// border's codes requested at once and 16-byte stores of the inflow the combine
// went from 1.70 to 1.62 ms at 32768 x 32768, and a 512 x 512 grid's whole
// accumulation from 66 to 62 us.)
constexpr uint16_t XN_OUT = 0x4000u;

template <int S, int G, int NT, class V, class CV>
__device__ int group_load(const DemDesc& cd, const GroupGeo& gg, int64_t gy, int64_t gx, const uint16_t* cpex,
                          const CV* cpval, uint16_t* spx, V* val, uint32_t* pd) {
  constexpr int NS = G * G * 4 * S;
  constexpr int SPT = 4 * S;  // slots per child, a multiple of 8
  constexpr int NQ = NS / 8 / NT > 0 ? NS / 8 / NT : 1;
  static_assert(SPT % 8 == 0 && NS % (8 * NT) == 0, "eight slots per load, whole rounds per thread");
  static_assert(NS <= XN_OUT, "a node fits below the exit codes' flags");
  int exits = 0;
  // eight consecutive slots of one child per 16-byte load of codes, with
  // their values loaded unconditionally beside them: every load of this
  // thread is issued before any is used (one round trip to memory)
  uint4 pe8[NQ];
  CV v8[NQ][8];
#pragma unroll
  for (int r = 0; r < NQ; r++) {
    const int n = (threadIdx.x + r * NT) * 8;
    const int lt = n / SPT, s = n - lt * SPT;
    const int64_t cy = gy * G + lt / G, cx = gx * G + lt % G;
    pe8[r] = make_uint4(PEX_TERM | (PEX_TERM << 16), PEX_TERM | (PEX_TERM << 16), PEX_TERM | (PEX_TERM << 16),
                        PEX_TERM | (PEX_TERM << 16));
    if (cy < cd.nty && cx < cd.ntx) {
      const int64_t g0 = (cd.tile_base + cy * cd.ntx + cx) * SPT + s;
      pe8[r] = *reinterpret_cast<const uint4*>(cpex + g0);
      const uint4* vp = reinterpret_cast<const uint4*>(cpval + g0);
      uint4 raw[8 * sizeof(CV) / 16];
#pragma unroll
      for (int k = 0; k < (int)(8 * sizeof(CV) / 16); k++) raw[k] = vp[k];
      memcpy(v8[r], raw, sizeof(raw));
    }
  }
#pragma unroll
  for (int r = 0; r < NQ; r++) {
    const int n = (threadIdx.x + r * NT) * 8;
    const uint16_t* pe = reinterpret_cast<const uint16_t*>(&pe8[r]);
    V vo[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const bool ex = (pe[k] & PEX_EXIT) != 0;
      exits += ex;
      vo[k] = ex ? V(v8[r][k]) : V{};
    }
    *reinterpret_cast<uint4*>(spx + n) = pe8[r];
#pragma unroll
    for (int k = 0; k < 8; k++) val[n + k] = vo[k];
    *reinterpret_cast<uint4*>(pd + n) = make_uint4(0, 0, 0, 0);
    *reinterpret_cast<uint4*>(pd + n + 4) = make_uint4(0, 0, 0, 0);
  }
  __syncthreads();
  for (int n = threadIdx.x; n < NS; n += NT) {
    const uint16_t pe = spx[n];
    uint16_t pr = N_NONE;
    if (pe & PEX_EXIT) {
      const int n2 = target_node<S, G>(gg, n, pe);
      spx[n] = (uint16_t)(PEX_EXIT | (n2 >= 0 ? n2 : XN_OUT | (pe & 7)));  // (others look at PEX_EXIT alone)
      if (n2 >= 0) {
        const uint16_t pe2 = spx[n2];
        if (pe2 & PEX_EXIT)
          pr = (uint16_t)n2;
        else if (pe2 == PEX_TERM)
          pr = N_ROOT;
        else
          pr = (uint16_t)(n2 / (4 * S) * (4 * S) + pe2);
        if (pr < N_NONE) atomicAdd(&pd[pr], 1u);
      } else {
        pr = N_OUT;
      }
    }
    if (pr != 0) atomicAdd(&pd[n], (uint32_t)pr << 16);
  }
  __syncthreads();
  return exits;
}

// The walks of a warp's n sources.  CHAINS: a walk past LONG_RUN steps takes up to
// CHAIN_STEPS nodes marked SINGLE at a time.  Nobody else adds to those, so a
// step is a load of the node's word and three operations, where the atomics'
// replies take 240 cycles.
constexpr int LONG_RUN = 16, CHAIN_STEPS = 64;
template <bool CHAINS, class V>
__device__ __forceinline__ int walk_sources(const uint16_t* my, int n, V* val, uint32_t* pd) {
  const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
  int done = 0, head = 0, cur = -1, run = 0;
  V v{};
  for (;;) {
    if (head < n) {
      const unsigned need = __ballot_sync(FULL, cur < 0);
      const int idx = head + __popc(need & lt);
      if (cur < 0 && idx < n) {
        cur = my[idx];
        v = val[cur];
        done++;
        run = 0;
      }
      head += __popc(need);
    } else if (!__any_sync(FULL, cur >= 0)) {
      break;
    }
    if (cur >= 0) {
      uint32_t p = pd_par(pd[cur]);
      if (CHAINS && ++run > LONG_RUN) {
        for (int k = 0; k < CHAIN_STEPS && p < N_NONE; k++) {
          const uint32_t w = pd[p];
          if (!(w & SINGLE)) break;
          v = vadd(val[p], v);
          val[p] = v;
          cur = (int)p;
          p = pd_par(w);
          done++;
        }
      }
      if (p >= N_NONE) {
        cur = -1;
        continue;
      }
      vatomic_add(&val[p], v);
      // the addition above is released by the count's atomic; the last child
      // reads the parent's value after it (acquire)
      const uint32_t old = atomic_add_acq_rel_cta(&pd[p], 0u - 1u);
      if (pd_deg(old) == 1u) {
        cur = p;
        v = vload_volatile(&val[p]);
        done++;
      } else {
        cur = -1;
      }
    }
  }
  return done;
}

// Algorithm 2 on the exit forest of a group: last-arriver walks from the
// nodes without unfinished children.  A finished node adds its value to its
// parent, then (after a block fence) decrements the parent's children count;
// the last child continues at the parent (its acquire-release count atomic
// orders it after every child's addition).  Returns the number of nodes this thread finished.
//
// Unit counts: in a group whose channels wind, few exits are sources (4 to 12 %
// on boustrophedons and spirals, 80 to 86 % on fractals and planes), and the walks
// are chains.  There the nodes with one child are marked first, so that the walks
// need no atomics on them.  A block decides as a whole, by its warps' sources (a
// count that the barrier takes along: a sum of sources and exits cost fractals
// 1 to 2 % of the combine, marks and chains in every group 1 to 3 % of the call).
// Whole accumulation of a 512 x 512 boustrophedon and spiral: 217 and 230 us (553
// and 615 without; 326 and 621 with groups of 4 x 4 tiles and of 2 x 2, whose
// chains are shorter), 300 x 257 spiral in 32 x 32 tiles 220 (443, 243), 600 x 700
// spiral 346 (567, 473).
template <int S, int G, int NT, class V>
__device__ int group_walk(uint16_t* spx, V* val, uint32_t* pd, uint16_t* srcl) {
  constexpr int NS = G * G * 4 * S;
  constexpr int NW = NT / 32;
  static_assert(5 * 4 * S < (int)SINGLE, "a children count fits below the mark");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint16_t* my = srcl + warp * (NS / NW);
  int n = 0;
  for (int r = 0; r < NS / NT; r++) {
    const int c = threadIdx.x + r * NT;
    const bool s = (spx[c] & PEX_EXIT) && pd_deg(pd[c]) == 0u;
    const unsigned m = __ballot_sync(FULL, s);
    if (s) my[n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)c;
    n += __popc(m);
  }
  if constexpr (std::is_same<V, uint32_t>::value && NS >= 8192) {
    // the group winds if hardly a warp found sources in more than an eighth of its slots
    if (__syncthreads_count(n > NS / NW / 8) <= NT / 8) {
      for (int c = threadIdx.x; c < NS; c += NT)
        if (pd_deg(pd[c]) == 1u) pd[c] |= SINGLE;
      __syncthreads();
      return walk_sources<true, V>(my, n, val, pd);
    }
  } else {
    __syncthreads();
  }
  return walk_sources<false, V>(my, n, val, pd);
}

template <int S, int G, class V, class CV>
__global__ void __launch_bounds__(NTG<S, G>) k_group_up(DemTable cdt, DemTable gdt, const uint16_t* cpex, const CV* cpval,
                                                    uint16_t* gpex, V* gpval, unsigned long long* node,
                                                    int64_t ngroups, uint32_t* queue, uint32_t* status) {
  using L = GroupLayout<S, G, V>;
  extern __shared__ __align__(16) unsigned char sm[];
  uint16_t* spx = reinterpret_cast<uint16_t*>(sm + L::off_spx);
  V* val = reinterpret_cast<V*>(sm + L::off_val);
  uint32_t* pd = reinterpret_cast<uint32_t*>(sm + L::off_pd);
  uint16_t* srcl = reinterpret_cast<uint16_t*>(sm + L::off_src);
  int* misc = reinterpret_cast<int*>(sm + L::off_misc);
  constexpr int NS = L::NS, NT = NTG<S, G>;
  constexpr int GS = G * S;
  TileQueue tq(queue, ngroups);
  for (int64_t gu = tq.first(); gu < ngroups; gu = tq.next()) {
    const DemDesc gd = dem_of(gdt, gu);
    const int dem = gdt.ndem == 1 ? 0 : gdt.tile_dem[gu];
    const DemDesc cd = dem_by_index(cdt, dem);
    const int64_t lg = gu - gd.tile_base;
    const int64_t gy = lg / gd.ntx, gx = lg % gd.ntx;
    if (threadIdx.x == 0) {
      misc[0] = 0;
      misc[1] = 0;
    }
    const GroupGeo gg = group_geo<S, G>(gd, gy, gx);
    const int exits = group_load<S, G, NT, V, CV>(cd, gg, gy, gx, cpex, cpval, spx, val, pd);
    const int done = group_walk<S, G, NT, V>(spx, val, pd, srcl);
    atomicAdd(&misc[0], done);
    atomicAdd(&misc[1], exits);
    __syncthreads();
    // every exit node must have been finished, else the exit graph has a cycle
    if (threadIdx.x == 0 && misc[0] != misc[1]) set_status(status, D8_ERR_CYCLE);
    // the group's own perimeter summary
    for (int gs = threadIdx.x; gs < 4 * GS; gs += NT) {
      int ci, cj;
      uint16_t gpe = PEX_TERM;
      V gv{};
      if (slot_cell(gs, gg.h, gg.w, GS, ci, cj)) {
        const int n0 = node_of<S, G>(gg, ci, cj);
        const uint16_t pe = spx[n0];
        int x = -1;
        if (pe & PEX_EXIT) {
          if (pd_par(pd[n0]) == N_OUT) {
            gpe = (uint16_t)(PEX_EXIT | (pe & 7));
            gv = val[n0];
          } else {
            x = n0;
          }
        } else if (pe != PEX_TERM) {
          x = n0 / (4 * S) * (4 * S) + pe;
        }
        if (x >= 0) {
          for (int it = 0; it < NS && pd_par(pd[x]) < N_NONE; it++) x = (int)pd_par(pd[x]);
          if (pd_par(pd[x]) == N_OUT) {
            int xi, xj;
            cell_of<S, G>(gg, x, xi, xj);
            gpe = (uint16_t)slot_of(xi, xj, gg.h, gg.w, GS);
          }
        }
      }
      gpex[gu * (4 * GS) + gs] = gpe;
      gpval[gu * (4 * GS) + gs] = gv;
      if (node) node[gu * (4 * GS) + gs] = 0ull;  // below the top level: its words start at zero
    }
    // (the queue's barrier protects shared memory before the next group)
  }
}

// infl[n] = the sum of the final areas of the group's child exits that drain
// into node n's cell
template <int NS, int NT, class V>
__device__ __forceinline__ void receivers_inflow(const uint16_t* spx, const V* val, V* infl) {
  constexpr int Q = 16 / sizeof(V);
  for (int q = threadIdx.x; q < NS / Q; q += NT) reinterpret_cast<uint4*>(infl)[q] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  for (int n = threadIdx.x; n < NS; n += NT) {
    const uint16_t pe = spx[n];
    if ((pe & (PEX_EXIT | XN_OUT)) == PEX_EXIT) vatomic_add(&infl[pe & (XN_OUT - 1)], val[n]);
  }
}

// ... and to the children's slots, a 16-byte word at a time
template <int S, int G, int NT, class V>
__device__ __forceinline__ void store_inflow(const DemDesc& cd, int64_t gy, int64_t gx, const V* infl, V* cfin) {
  constexpr int NS = G * G * 4 * S, Q = 16 / sizeof(V);
  for (int q = threadIdx.x; q < NS / Q; q += NT) {
    const int n = q * Q, lt = n / (4 * S), s = n - lt * (4 * S);
    const int64_t cy = gy * G + lt / G, cx = gx * G + lt % G;
    if (cy < cd.nty && cx < cd.ntx)
      *reinterpret_cast<uint4*>(cfin + (cd.tile_base + cy * cd.ntx + cx) * (4 * S) + s) =
          reinterpret_cast<const uint4*>(infl)[q];
  }
}

// The group's border inflow and its children's final values.  RECV (the
// children are tiles): cfin gets per slot not the exits' final
// areas but the receivers' inflow, the sum of the final areas of the exits of
// other tiles that drain into the slot's cell, which is what the finalising
// pass needs (it then reads one contiguous row per tile; gathering the areas
// there took the codes around every tile and scattered loads).
template <int S, int G, class V, class CV, bool RECV>
__global__ void __launch_bounds__(NTG<S, G>) k_group_down(DemTable cdt, DemTable gdt, const uint16_t* cpex, const CV* cpval,
                                                      V* cfin, const V* gfin, int64_t ngroups, uint32_t* queue,
                                                      const uint32_t* counters, uint32_t* status) {
  using L = GroupLayout<S, G, V>;
  extern __shared__ __align__(16) unsigned char sm[];
  uint16_t* spx = reinterpret_cast<uint16_t*>(sm + L::off_spx);
  V* val = reinterpret_cast<V*>(sm + L::off_val);
  uint32_t* pd = reinterpret_cast<uint32_t*>(sm + L::off_pd);
  uint16_t* srcl = reinterpret_cast<uint16_t*>(sm + L::off_src);
  constexpr int NS = L::NS, NT = NTG<S, G>;
  constexpr int GS = G * S;
  // below the top level: an exit its walks never finished lies on a cycle
  if (counters && blockIdx.x == 0 && threadIdx.x == 0 && counters[1] != counters[2]) set_status(status, D8_ERR_CYCLE);
  TileQueue tq(queue, ngroups);
  for (int64_t gu = tq.first(); gu < ngroups; gu = tq.next()) {
    const DemDesc gd = dem_of(gdt, gu);
    const int dem = gdt.ndem == 1 ? 0 : gdt.tile_dem[gu];
    const DemDesc cd = dem_by_index(cdt, dem);
    const int64_t lg = gu - gd.tile_base;
    const int64_t gy = lg / gd.ntx, gx = lg % gd.ntx;
    const GroupGeo gg = group_geo<S, G>(gd, gy, gx);
    group_load<S, G, NT, V, CV>(cd, gg, gy, gx, cpex, cpval, spx, val, pd);
    // inflow across the group border: each border cell r receives the final
    // areas of the outside cells draining into it; the inflow then follows
    // r's path inside its child unit to that child's exit
    constexpr int NB = 4 * GS / NT;  // border slots per thread
    static_assert(4 * GS % NT == 0, "whole rounds over the border");
    V bin[RECV ? NB : 1];  // inflow across the border and the child slot it enters
    int bslot[RECV ? NB : 1];
#pragma unroll 1
    for (int r = 0; r < NB; r++) {
      const int gs = threadIdx.x + r * NT;
      if (RECV) bslot[RECV ? r : 0] = -1;
      int ci, cj;
      if (!slot_cell(gs, gg.h, gg.w, GS, ci, cj)) continue;
      const int64_t gi = gy * GS + ci, gj = gx * GS + cj;
      // the codes outside are all requested before the first is looked at
      uint32_t code[8];
#pragma unroll
      for (int k = 0; k < 8; k++) {
        const int li = ci + code_di(k), lj = cj + code_dj(k);
        const int64_t ni = gi + code_di(k), nj = gj + code_dj(k);
        const bool outside = (unsigned)li >= (unsigned)gg.h || (unsigned)lj >= (unsigned)gg.w;
        code[k] = 9;
        if (outside && ni >= 0 && nj >= 0 && ni < gd.H && nj < gd.W) code[k] = __ldg(gd.dir + ni * gd.lddir + nj);
      }
      uint32_t from = 0;
#pragma unroll
      for (int k = 0; k < 8; k++) from |= (code[k] == (uint32_t)opposite(k) ? 1u : 0u) << k;
      if (!from) continue;
      V in{};
      for (uint32_t m = from; m; m &= m - 1) {
        const int k = __ffs(m) - 1;
        in = vadd(in, gfin[global_slot(gd, gi + code_di(k), gj + code_dj(k), GS)]);
      }
      const int n0 = node_of<S, G>(gg, ci, cj);
      const uint16_t pe = spx[n0];
      if (pe & PEX_EXIT)
        vatomic_add(&val[n0], in);
      else if (pe != PEX_TERM)
        vatomic_add(&val[n0 / (4 * S) * (4 * S) + pe], in);
      if (RECV) {
        bin[RECV ? r : 0] = in;
        bslot[RECV ? r : 0] = n0;
      }
    }
    __syncthreads();
    group_walk<S, G, NT, V>(spx, val, pd, srcl);
    __syncthreads();
    if constexpr (RECV) {
      V* infl = reinterpret_cast<V*>(pd);  // the walk is done with it
      receivers_inflow<NS, NT, V>(spx, val, infl);
#pragma unroll 1
      for (int r = 0; r < NB; r++)
        if (bslot[r] >= 0) vatomic_add(&infl[bslot[r]], bin[r]);
      __syncthreads();
      store_inflow<S, G, NT, V>(cd, gy, gx, infl, cfin);
    } else {
      for (int n = threadIdx.x; n < NS; n += NT) {
        if (!(spx[n] & PEX_EXIT)) continue;
        const int lt = n / (4 * S), s = n - lt * (4 * S);
        const int64_t cy = gy * G + lt / G, cx = gx * G + lt % G;
        cfin[(cd.tile_base + cy * cd.ntx + cx) * (4 * S) + s] = val[n];
      }
    }
  }
}

// The whole combine of a grid that one group covers (unit counts): load, walk,
// receivers' inflow, one block of NTS threads per DEM.  One launch instead of
// two up and two down; a 512 x 512 grid's 64 tiles are one group of 8 x 8.
constexpr int NTS = 1024;
template <int S, int G>
__global__ void __launch_bounds__(NTS) k_group_solve(DemTable dt, const uint16_t* pex, const uint32_t* pval,
                                                       uint32_t* inflow, uint32_t* status) {
  using L = GroupLayout<S, G, uint32_t>;
  extern __shared__ __align__(16) unsigned char sm[];
  uint16_t* spx = reinterpret_cast<uint16_t*>(sm + L::off_spx);
  uint32_t* val = reinterpret_cast<uint32_t*>(sm + L::off_val);
  uint32_t* pd = reinterpret_cast<uint32_t*>(sm + L::off_pd);
  uint16_t* srcl = reinterpret_cast<uint16_t*>(sm + L::off_src);
  int* misc = reinterpret_cast<int*>(sm + L::off_misc);
  const DemDesc d = dem_by_index(dt, blockIdx.x);
  const GroupGeo gg = group_geo<S, G>(d, 0, 0);
  if (threadIdx.x < 2) misc[threadIdx.x] = 0;
  const int exits = group_load<S, G, NTS, uint32_t, uint32_t>(d, gg, 0, 0, pex, pval, spx, val, pd);
  const int done = group_walk<S, G, NTS, uint32_t>(spx, val, pd, srcl);
  atomicAdd(&misc[0], done);
  atomicAdd(&misc[1], exits);
  __syncthreads();
  if (threadIdx.x == 0 && misc[0] != misc[1]) set_status(status, D8_ERR_CYCLE);
  receivers_inflow<L::NS, NTS, uint32_t>(spx, val, pd);
  __syncthreads();
  store_inflow<S, G, NTS, uint32_t>(d, 0, 0, pd, inflow);
}

template <int S, int G>
static cudaError_t launch_solve(const HLevel& t, uint32_t* status, cudaStream_t s) {
  constexpr size_t bytes = GroupLayout<S, G, uint32_t>::bytes;
  auto k = k_group_solve<S, G>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  k<<<(unsigned)t.dt.ndem, NTS, bytes, s>>>(t.dt, t.pex, static_cast<const uint32_t*>(t.pval),
                                            static_cast<uint32_t*>(t.fin), status);
  return cudaGetLastError();
}

// ---- top level: Algorithms 5-6 over the remaining units, in global memory

// A node's word: children left (bits 32..47), children in all (bits 48..63)
// and, unit counts, the value (low half).  The count of all children tells the
// sources (exits without any) from nodes whose children have arrived.  (A unit
// of side 512 has 2048 slots and at most nine units drain into one: 16 bits.)
constexpr unsigned long long CHILD = (1ull << 32) | (1ull << 48), LEFT = 1ull << 32;
__device__ __forceinline__ uint32_t left_of(unsigned long long w) { return (uint32_t)(w >> 32) & 0xFFFFu; }
__device__ __forceinline__ uint32_t children(const unsigned long long* node, uint32_t p) {
  return (uint32_t)(*(volatile const unsigned long long*)&node[p] >> 48);
}
constexpr uint32_t LONG_WALK = 64;  // steps

// parents, children counts and values (the words were zeroed by the level below)
template <int S, class V, class CV>
__global__ void k_top_init(DemTable dt, const uint16_t* pex, const CV* pval, V* fin, uint32_t* par,
                           unsigned long long* node, int64_t nslots) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < nslots; g += stride) {
    const uint16_t pe = pex[g];
    if (!(pe & PEX_EXIT)) continue;
    const int64_t t = g / (4 * S);
    const int s = (int)(g - t * (4 * S));
    const DemDesc d = dem_of(dt, t);
    const int64_t lt = t - d.tile_base;
    const UnitGeo u = unit_geo(d, lt / d.ntx, lt % d.ntx, S);
    int i, j;
    slot_cell(s, u.h, u.w, S, i, j);
    const int k = pe & 7;
    const int64_t y = global_slot(d, u.i0 + i + code_di(k), u.j0 + j + code_dj(k), S);
    const uint16_t pey = pex[y];
    uint32_t pr = ROOT;
    if (pey & PEX_EXIT)
      pr = (uint32_t)y;
    else if (pey != PEX_TERM)
      pr = (uint32_t)((y / (4 * S)) * (4 * S) + pey);
    if (pr != ROOT) atomicAdd(&node[pr], CHILD);
    if constexpr (std::is_same<V, uint32_t>::value)
      atomicAdd(&node[g], (unsigned long long)pval[g]);
    else
      fin[g] = pval[g];
    par[g] = pr;
  }
}

// Algorithm 6 with global atomics: last-arriver walks up the exit forest from
// the sources, each started by the thread that comes across it (the slots'
// walks are short; a list of the sources, to give every thread one, took two
// passes of its own: 8192 x 8192 11 us and 27 for the walks, 32768 x 32768 37
// and 188).  Unit counts: one 64-bit atomic per step delivers the value and
// tells the last child (no fences); each finished node stores its value for
// the down sweep.  Float-float: value add, then children count, released and
// acquired by its atomic.  The next parent is loaded beside the atomic, so a
// step waits for one reply, not two.  A walk that has gone far is on a chain,
// where most nodes have one child: nobody else adds to those, so plain loads do.
// (Looking from the first step on costs short walks more than it saves: 32768 x
// 32768 combine 1.56 and 1.62 ms.)  An 8192 x 8192 boustrophedon, 122,895 steps:
// 32.6 ms (50.4 before, 42.8 without the plain loads), weighted 56 (155).
// counters: [1] exits, [2] finished.
template <class V>
__global__ void __launch_bounds__(256) k_top_walk(const uint16_t* pex, const uint32_t* par, V* fin,
                                                  unsigned long long* node, uint32_t* counters, int64_t nslots) {
  uint32_t done = 0, exits = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < nslots; g += stride) {
    if (!(pex[g] & PEX_EXIT)) continue;
    exits++;
    const unsigned long long w = *(volatile const unsigned long long*)&node[g];
    if (w >> 48) continue;  // has children: their walks come here
    uint32_t x = (uint32_t)g, run = 0;
    if constexpr (std::is_same<V, uint32_t>::value) {
      uint32_t v = (uint32_t)w, p = par[x];
      for (;;) {
        fin[x] = v;
        done++;
        if (p == ROOT) break;
        const uint32_t next = par[p];  // in flight beside the atomic: a step waits for one reply, not two
        if (++run > LONG_WALK && children(node, p) == 1u) {
          v += (uint32_t)node[p];
          x = p;
          p = next;
          continue;
        }
        const unsigned long long old = atomicAdd(&node[p], (unsigned long long)v - LEFT);
        if (left_of(old) != 1u) break;
        v += (uint32_t)old;
        x = p;
        p = next;
      }
    } else {
      V v = fin[x];
      uint32_t p = par[x];
      done++;
      for (;;) {
        if (p == ROOT) break;
        const uint32_t next = par[p];
        if (++run > LONG_WALK && children(node, p) == 1u) {
          v = vadd(fin[p], v);
          fin[p] = v;
          p = next;
          done++;
          continue;
        }
        vatomic_add(&fin[p], v);
        // the high half of the word: releases the addition; acquires the others'
        const uint32_t old = atomic_add_acq_rel_gpu(reinterpret_cast<uint32_t*>(&node[p]) + 1, 0u - 1u);
        if ((old & 0xFFFFu) != 1u) break;
        v = vload_volatile(&fin[p]);
        p = next;
        done++;
      }
    }
  }
  __shared__ uint32_t sum[2];
  if (threadIdx.x < 2) sum[threadIdx.x] = 0u;
  __syncthreads();
  if (exits) atomicAdd(&sum[0], exits);
  if (done) atomicAdd(&sum[1], done);
  __syncthreads();
  if (threadIdx.x < 2 && sum[threadIdx.x]) atomicAdd(&counters[1 + threadIdx.x], sum[threadIdx.x]);
}

// ---- top level by pointer jumping (strategy 2).  The queue walk above costs
// one dependent global atomic per node of the longest chain, which a channel
// crossing the top-level units 10^5 times makes tens of milliseconds.  Here
// every exit y keeps P(y) = its 2^r-th ancestor (ROOT past the root); a round
// adds each exit's partial sum to P(y) and jumps (P(y) = P(P(y))), and after
// ceil(log2(depth)) rounds every exit holds its subtree sum (Algorithm 6's
// result).  Rounds after the last active one return at once (a per-round flag).
//
// The partial sum of y is its own value plus all that was added to it so far.
// Even rounds add to add[], odd ones to add2[], so the buffer of the round
// before stands still while its additions are read, and nothing has to be
// applied or set to zero between rounds: in round r
//   sum(y) = fin(y) + (r - 1's buffer)(y),  fin(y) <- own value + (r - 1's buffer)(y),
// where fin holds the own value plus r's buffer as it was before this round.
// (On an 8192 x 8192 boustrophedon the whole combine takes 361 us; 490 with a
// pass after each round that applied the additions and cleared one buffer.)

// parents, values (fin = pval at exits), additions zeroed, first round flag
template <int S, class V, class CV>
__global__ void k_topj_init(DemTable dt, const uint16_t* pex, const CV* pval, V* fin, uint32_t* par, V* add, V* add2,
                            uint32_t* flags, int64_t nslots) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  bool any = false;
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < nslots; g += stride) {
    const uint16_t pe = pex[g];
    uint32_t pr = ROOT;
    if (pe & PEX_EXIT) {
      const int64_t t = g / (4 * S);
      const int s = (int)(g - t * (4 * S));
      const DemDesc d = dem_of(dt, t);
      const int64_t lt = t - d.tile_base;
      const UnitGeo u = unit_geo(d, lt / d.ntx, lt % d.ntx, S);
      int i, j;
      slot_cell(s, u.h, u.w, S, i, j);
      const int k = pe & 7;
      const int64_t y = global_slot(d, u.i0 + i + code_di(k), u.j0 + j + code_dj(k), S);
      const uint16_t pey = pex[y];
      if (pey & PEX_EXIT)
        pr = (uint32_t)y;
      else if (pey != PEX_TERM)
        pr = (uint32_t)((y / (4 * S)) * (4 * S) + pey);
      fin[g] = V(pval[g]);
      add[g] = add2[g] = V{};
      any |= pr != ROOT;
    }
    par[g] = pr;
  }
  if (__syncthreads_or(any) && threadIdx.x == 0) raise_flag(&flags[0]);
}

// one round over the listed exits: scatter to the 2^r-th ancestor, then jump
// (every block writing the round flag took 48 us a round at 8192 x 8192, of
// which 40 were the writes; raised once it takes 9 to 20).  last: the other
// buffer, which holds the additions of the round before.
template <class V, class CV>
__global__ void k_topj_round(const uint32_t* list, const uint32_t* counters, const uint32_t* pc, uint32_t* pn,
                             const CV* pval, V* fin, V* add, const V* last, uint32_t* flags, int r) {
  if (*(volatile const uint32_t*)&flags[r] == 0u) return;
  const uint32_t n = counters[0];
  bool active = false;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t y = list[i];
    const uint32_t a = pc[y];
    if (a == ROOT) {
      pn[y] = ROOT;
      continue;
    }
    const V in = last[y];
    vatomic_add(&add[a], vadd(fin[y], in));
    fin[y] = vadd(V(pval[y]), in);
    const uint32_t aa = pc[a];
    pn[y] = aa;
    active |= aa != ROOT;
  }
  if (__syncthreads_or(active) && threadIdx.x == 0) raise_flag(&flags[r + 1]);
}

// every listed exit's subtree sum
template <class V, class CV>
__global__ void k_topj_apply(const uint32_t* list, const uint32_t* counters, const CV* pval, V* fin, const V* add,
                             const V* add2) {
  const uint32_t n = counters[0];
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t y = list[i];
    fin[y] = vadd(V(pval[y]), vadd(add[y], add2[y]));
  }
}

// exits still jumping after the last round: the exit forest has a cycle
__global__ void k_topj_check(const uint32_t* flags, int R, uint32_t* status) {
  if (threadIdx.x == 0 && blockIdx.x == 0 && flags[R] != 0u) set_status(status, D8_ERR_CYCLE);
}

// every exit listed, with one atomic per block on the list's length: a first
// pass counts this thread's exits, a block scan (Hillis-Steele) gives each
// thread its offset inside the block's range, a second pass writes them
__global__ void __launch_bounds__(256) k_topj_list(const uint16_t* pex, uint32_t* list, uint32_t* counters,
                                                   int64_t nslots) {
  __shared__ uint32_t sh[256];
  __shared__ uint32_t sh_base;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t g0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t nex = 0;
  for (int64_t g = g0; g < nslots; g += stride) nex += (pex[g] & PEX_EXIT) != 0;
  sh[threadIdx.x] = nex;
  __syncthreads();
  for (int off = 1; off < 256; off <<= 1) {
    const uint32_t a = threadIdx.x >= off ? sh[threadIdx.x - off] : 0u;
    __syncthreads();
    sh[threadIdx.x] += a;
    __syncthreads();
  }
  if (threadIdx.x == 255) sh_base = sh[255] ? atomicAdd(&counters[0], sh[255]) : 0u;
  __syncthreads();
  uint32_t pos = sh_base + sh[threadIdx.x] - nex;
  if (nex)
    for (int64_t g = g0; g < nslots; g += stride)
      if (pex[g] & PEX_EXIT) list[pos++] = (uint32_t)g;
}

template <int S, int G, class V, class CV>
static cudaError_t launch_level_up(const DemTable& cdt, const DemTable& gdt, const uint16_t* cpex, const void* cpval,
                                   uint16_t* gpex, void* gpval, unsigned long long* node, int64_t ngroups,
                                   uint32_t* queue, uint32_t* status, cudaStream_t s) {
  using L = GroupLayout<S, G, V>;
  auto k = k_group_up<S, G, V, CV>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes);
  if (e != cudaSuccess) return e;
  int per_sm = 1, dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, NTG<S, G>, L::bytes);
  int64_t grid = (int64_t)(per_sm < 1 ? 1 : per_sm) * sms;
  if (grid > ngroups) grid = ngroups;
  k<<<(unsigned)grid, NTG<S, G>, L::bytes, s>>>(cdt, gdt, cpex, static_cast<const CV*>(cpval), gpex,
                                                static_cast<V*>(gpval), node, ngroups, queue, status);
  return cudaGetLastError();
}

template <int S, int G, class V, class CV, bool RECV>
static cudaError_t launch_level_down(const DemTable& cdt, const DemTable& gdt, const uint16_t* cpex, const void* cpval,
                                     void* cfin, const void* gfin, int64_t ngroups, uint32_t* queue,
                                     const uint32_t* counters, uint32_t* status, cudaStream_t s) {
  using L = GroupLayout<S, G, V>;
  auto k = k_group_down<S, G, V, CV, RECV>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes);
  if (e != cudaSuccess) return e;
  int per_sm = 1, dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, NTG<S, G>, L::bytes);
  int64_t grid = (int64_t)(per_sm < 1 ? 1 : per_sm) * sms;
  if (grid > ngroups) grid = ngroups;
  k<<<(unsigned)grid, NTG<S, G>, L::bytes, s>>>(cdt, gdt, cpex, static_cast<const CV*>(cpval), static_cast<V*>(cfin),
                                                static_cast<const V*>(gfin), ngroups, queue, counters, status);
  return cudaGetLastError();
}

template <int S, class V, class CV>
static cudaError_t launch_top_jump(const DemTable& dt, const HLevel& lv, const HTop& top, cudaStream_t s, int* nl) {
  const int64_t ns = lv.nunits * 4 * S;
  cudaError_t e = cudaMemsetAsync(top.flags, 0, sizeof(uint32_t) * (MAX_ROUNDS + 2), s);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int64_t b = (ns + 255) / 256;
  if (b > (int64_t)sms * 16) b = (int64_t)sms * 16;
  if (b < 1) b = 1;
  V* fin = static_cast<V*>(lv.fin);
  V* add = reinterpret_cast<V*>(top.node);
  V* add2 = add + ns;
  const CV* pval = static_cast<const CV*>(lv.pval);
  k_topj_init<S, V, CV><<<(unsigned)b, 256, 0, s>>>(dt, lv.pex, pval, fin, top.par, add, add2, top.flags, ns);
  k_topj_list<<<(unsigned)b, 256, 0, s>>>(lv.pex, top.list, top.counters, ns);
  // rounds: enough for a chain through every slot
  int R = 1;
  while (R < MAX_ROUNDS && ((int64_t)1 << R) < ns) R++;
  for (int r = 0; r < R; r++) {
    uint32_t* pc = (r & 1) ? top.par2 : top.par;
    uint32_t* pn = (r & 1) ? top.par : top.par2;
    k_topj_round<V, CV><<<(unsigned)b, 256, 0, s>>>(top.list, top.counters, pc, pn, pval, fin, (r & 1) ? add2 : add,
                                                    (r & 1) ? add : add2, top.flags, r);
  }
  k_topj_apply<V, CV><<<(unsigned)b, 256, 0, s>>>(top.list, top.counters, pval, fin, add, add2);
  k_topj_check<<<1, 32, 0, s>>>(top.flags, R, top.status);
  *nl += 4 + R;
  return cudaGetLastError();
}

template <int S, class V, class CV>
static cudaError_t launch_top(const DemTable& dt, const HLevel& lv, const HTop& top, cudaStream_t s, int* nl) {
  if (top.jump) return launch_top_jump<S, V, CV>(dt, lv, top, s, nl);
  const int64_t ns = lv.nunits * 4 * S;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const unsigned b = (unsigned)min64((ns + 255) / 256, (int64_t)sms * 16);
  k_top_init<S, V, CV><<<b, 256, 0, s>>>(dt, lv.pex, static_cast<const CV*>(lv.pval), static_cast<V*>(lv.fin), top.par,
                                         top.node, ns);
  k_top_walk<V><<<(unsigned)min64(b, (int64_t)sms * 8), 256, 0, s>>>(lv.pex, top.par, static_cast<V*>(lv.fin), top.node,
                                                                     top.counters, ns);
  *nl += 2;
  return cudaGetLastError();
}

}  // namespace cmb

// Level schedule: groups of 8 x 8 tiles (wide; 32 or 64 a side), or of 4 x 4,
// then of 2 x 2 children, up to a group side of 512 cells; the global queue
// solve takes the rest.  (A 1024-cell level cost more than the longer
// top-level chains it saves: measured at 8192^2 and 32768^2.)  One level of 8 x
// 8 in blocks of 1024 threads instead of 4 x 4 and 2 x 2 in smaller ones: the
// whole combine takes 144 us at 8192^2 (181), 1.60 ms at 32768^2 (2.01), 80 us
// at 3001 x 5003 (89).  Not for float-float values (8 x 8 children do not fit
// shared memory), nor under strategy "jump", whose long chains are walked
// inside a group: two levels halve them.
int hier_levels(int T, int64_t max_side, bool wide, int* S, int* G, int max_levels) {
  int n = 0;
  int s = T;
  while (n < max_levels && s < max_side && s < 512) {
    const int g = (s <= 64) ? (wide ? 8 : 4) : 2;
    S[n] = s;
    G[n] = g;
    s *= g;
    n++;
  }
  return n;
}

namespace cmb {

// V: accumulation type above the tiles; CV0: the tiles' stored pval type
template <class V, class CV0>
static cudaError_t combine_hier_t(const HPlan& hp, cudaStream_t s, int* nlaunch) {
  cudaError_t e = cudaSuccess;
  // up: level l-1 -> l
  for (int l = 1; l <= hp.nlev && e == cudaSuccess; l++) {
    const HLevel& c = hp.lev[l - 1];
    const HLevel& g = hp.lev[l];
    const int S = c.S, G = g.S / c.S;
#define D8_UP(SS, GG)                                                                                             \
  if (S == SS && G == GG) {                                                                                      \
    unsigned long long* node = l == hp.nlev && hp.need_top && !hp.top.jump ? hp.top.node : nullptr;               \
    e = l == 1 ? launch_level_up<SS, GG, V, CV0>(c.dt, g.dt, c.pex, c.pval, g.pex, g.pval, node, g.nunits,         \
                                                 hp.queue + l, hp.status, s)                                      \
               : launch_level_up<SS, GG, V, V>(c.dt, g.dt, c.pex, c.pval, g.pex, g.pval, node, g.nunits,           \
                                               hp.queue + l, hp.status, s);                                       \
    ++*nlaunch;                                                                                                  \
    continue;                                                                                                    \
  }
    if constexpr (std::is_same<V, uint32_t>::value) {
      D8_UP(32, 8) D8_UP(64, 8)
    }
    D8_UP(32, 4) D8_UP(64, 4) D8_UP(128, 2) D8_UP(256, 2)
#undef D8_UP
    return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  // top
  const HLevel& t = hp.lev[hp.nlev];
  if (hp.need_top) {
    // (a grid of more than one unit has levels up to 512)
    if (t.S != 512) return cudaErrorInvalidValue;
    e = launch_top<512, V, V>(t.dt, t, hp.top, s, nlaunch);
    if (e != cudaSuccess) return e;
  }
  // down: level l -> l-1 (at the tiles: the receivers' inflow)
  for (int l = hp.nlev; l >= 1 && e == cudaSuccess; l--) {
    const HLevel& c = hp.lev[l - 1];
    const HLevel& g = hp.lev[l];
    const int S = c.S, G = g.S / c.S;
#define D8_DN(SS, GG)                                                                                               \
  if (S == SS && G == GG) {                                                                                        \
    const uint32_t* cnt = l == hp.nlev && hp.need_top && !hp.top.jump ? hp.top.counters : nullptr;                \
    e = l == 1 ? launch_level_down<SS, GG, V, CV0, true>(c.dt, g.dt, c.pex, c.pval, c.fin, g.fin, g.nunits,         \
                                                         hp.queue + 16 + l, cnt, hp.status, s)                    \
               : launch_level_down<SS, GG, V, V, false>(c.dt, g.dt, c.pex, c.pval, c.fin, g.fin, g.nunits,          \
                                                        hp.queue + 16 + l, cnt, hp.status, s);                    \
    ++*nlaunch;                                                                                                    \
    continue;                                                                                                      \
  }
    if constexpr (std::is_same<V, uint32_t>::value) {
      D8_DN(32, 8) D8_DN(64, 8)
    }
    D8_DN(32, 4) D8_DN(64, 4) D8_DN(128, 2) D8_DN(256, 2)
#undef D8_DN
    return cudaErrorInvalidValue;
  }
  return e;
}

}  // namespace cmb

int solve_side(int T) { return T == 128 ? 512 : 8 * T; }

cudaError_t launch_combine_hier(const HPlan& hp, cudaStream_t s, int* nlaunch) {
  if (hp.solve) {
    ++*nlaunch;
    switch (hp.lev[0].S) {
      case 32: return cmb::launch_solve<32, 8>(hp.lev[0], hp.status, s);
      case 64: return cmb::launch_solve<64, 8>(hp.lev[0], hp.status, s);
      case 128: return cmb::launch_solve<128, 4>(hp.lev[0], hp.status, s);
    }
    return cudaErrorInvalidValue;
  }
  if (!hp.weighted) return cmb::combine_hier_t<uint32_t, uint32_t>(hp, s, nlaunch);
  return cmb::combine_hier_t<ff, ff>(hp, s, nlaunch);
}

}  // namespace d8
