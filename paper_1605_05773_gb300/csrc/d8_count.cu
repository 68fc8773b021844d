// d8_count.cu -- the unit-count tile pass (the headline path) for tiles of side
// 32 and 64: per tile, codes from the direction field, the in-tile input counts
// (Algorithm 1), the in-tile up-slope counts with inflow from other tiles
// unknown = 0 (Algorithms 2-4), written to A, and the perimeter summary.
//
// Layout choices for GB300:
//  * one packed 32-bit word per cell in shared memory holds all there is to a
//    cell (Cell): its in-tile count, its number of unfinished in-tile inputs,
//    class bits and a link, the byte offset of its down-slope cell's word.  One
//    shared atomicAdd both delivers a finished cell's count to its down-slope
//    cell and tells the sender whether it was the last input; only then does
//    the sender continue (Algorithm 2's tail recursion);
//  * words are stored in an order (Place) in which a warp's four-cell groups
//    hit 32 banks, and the down-slope offset is read from an 8-byte table per
//    column of the group, so a code costs few instructions and no conflicts;
//  * sources are delivered in one sweep, and the walks start at the cells the
//    sweep completed.  A walk advances STEPS cells in a batch of 32, then goes
//    back to its warp's stack, so that batches stay full; a step has no
//    branches (lanes with nothing to deliver add to a spare word);
//  * once a warp has fewer than 32 walks left it hands them to a pool, and the
//    last warp to do so finishes the pool alone: the long chains (about 90
//    cells on a 64 x 64 fractal tile, with 25 walks left after 15 steps) then
//    occupy one warp instead of four, and need no atomics but at junctions;
//  * these last walks point the link of each cell they leave at the cell they
//    started from, and that cell's link at the place where they stopped, so
//    following links from any cell reaches the end of its in-tile path in a
//    short chase: the exits of the perimeter cells.
//  * the next tile's codes are requested before this one's walks.
//
// Measured, T = 64: 32768 x 32768 fractal 3.77 ms, 8192 x 8192 261 us (before:
// 6.53 ms and 435 us, 128 threads, a 16-bit segment record per cell beside the
// word, 8 tiles per SM, one ring of starts per warp); 3001 x 5003, rows at odd
// addresses: 85 us (110 with byte loads and strided stores).  11264 warp
// instructions per tile (21000).  Where the 261 us go: words 40, sweep 43,
// batches 60, the last walks 57, counts to A 12, summary 32, the rest 17.
#include "d8_device.cuh"

namespace d8 {
namespace count {

// NT, the threads of a tile's block, is 64 with 12 tiles per SM: 262 us at 8192
// x 8192; 128 threads, 8 tiles: 320 (two more warps wait out the last walks).
// Few tiles: see launch_t.
constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int STEPS = 4;   // cells a walk advances per batch (3: 274 us, 6: 276, 4: 271 at the time)
constexpr int SWEEP = 4;   // rows of the block's cells swept at once (1: 309 us, 2: 297, 4: 293 at the time)
// walks on a warp's stack: 31 and a sweep's, or what all warps leave over
constexpr int cap(int warps) { return 32 * (1 + SWEEP > warps ? 1 + SWEEP : warps); }

// Where cell (i, j) of a tile is stored: within its row by (column mod 4,
// column / 4), rows rotated among the bank groups, so that the cells k of 32
// consecutive four-cell groups lie in 32 banks.
template <int T>
struct Place {
  static constexpr int Q = T / 4;            // four-cell groups per row
  static constexpr int RM = 32 / Q - 1;      // rows per warp-wide set of groups, less one
  __host__ __device__ static constexpr int col(int i, int j) { return ((j & 3) * Q + (j >> 2)) ^ ((i & RM) * Q); }
  __device__ static __forceinline__ int of(int i, int j) { return i * T + col(i, j); }
  __device__ static __forceinline__ int row(int p) { return p / T; }
  __device__ static __forceinline__ int column(int p) {
    const int x = (p & (T - 1)) ^ ((row(p) & RM) * Q);
    return (x & (Q - 1)) * 4 + x / Q;
  }
};

// The packed word: bits 0, 1 IN (target inside the tile) and EXIT (target in
// another tile); then the link, a byte offset into word[] (a multiple of 4) of
// IN cells (others: the code << 2); the count from bit CB; inputs still to
// arrive in bits 28..31, so one unsigned compare of the value an atomic
// returns tells the last arriver (left was 1 iff old < 2 << 28).
constexpr uint32_t IN = 1u, EXIT = 2u, LEFT1 = 1u << 28;
template <int T>
struct Cell {
  static constexpr int CB = 14;
  static constexpr uint32_t ONE = 1u << CB;
  static constexpr uint32_t CNT = (LEFT1 - 1u) & ~(ONE - 1u);
  static constexpr uint32_t LINK = (uint32_t)(T * T - 1) << 2;
  static_assert((uint32_t)(T * T) <= (CNT >> CB) && LINK < ONE, "the largest count fits, above the link");
  __device__ static __forceinline__ bool last(uint32_t old) { return old < 2 * LEFT1; }
  __device__ static __forceinline__ int code(uint32_t w) { return (int)((w >> 2) & 0xFu); }  // cells that are not IN
};

template <int T, int NT>
struct Layout {
  static constexpr int NW = NT / 32, CAP = cap(NW);
  static constexpr size_t TT = (size_t)T * T;
  static constexpr size_t off_word = 0;                         // uint32 per cell
  static constexpr size_t off_spare = TT * 4;                   // uint32 [32], right after word: see spare()
  static constexpr size_t off_tab = off_spare + 128;            // int8: see Table
  static constexpr size_t off_misc = off_tab + 3 * 3 * (Place<T>::RM + 1) * 4 * 8;
  static constexpr size_t off_stack = off_misc + 16;            // uint16 [NW + 1][CAP]: walks (byte offsets); the pool last
  static constexpr size_t bytes = (off_stack + (size_t)(NW + 1) * CAP * 2 + 15) / 16 * 16;
};

__device__ __forceinline__ uint32_t& at(uint32_t* word, uint32_t o) {
  return *reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(word) + o);
}
// Byte offset of a word for this lane that nobody reads: lanes with nothing to
// deliver add to it, so that a step has no branches (which cost more
// instructions than the step).
template <int T>
__device__ __forceinline__ uint32_t spare() {
  return (uint32_t)(T * T * 4 + 4 * (threadIdx.x & 31));
}

// One cell of a ragged tile: its own word and one more input for its target.  A
// code 0..7 whose target is outside the tile is an exit when the target is on the
// grid, otherwise the path ends there.
template <int T>
__device__ __forceinline__ void add_cell(uint32_t* word, int i, int j, int code, const TileGeo& g, const DemDesc& d,
                                         uint32_t* status) {
  using P = Place<T>;
  using C = Cell<T>;
  uint32_t own = C::ONE;
  if (code < 8) {
    const int ti = i + code_di(code), tj = j + code_dj(code);
    if ((unsigned)ti < (unsigned)g.th && (unsigned)tj < (unsigned)g.tw) {
      const uint32_t t = 4u * (uint32_t)P::of(ti, tj);
      atomicAdd(&at(word, t), LEFT1);
      own |= IN | t;
    } else {
      const int64_t gi = g.i0 + ti, gj = g.j0 + tj;
      if (gi >= 0 && gj >= 0 && gi < d.H && gj < d.W) own |= EXIT;
      own |= (uint32_t)code << 2;
    }
  } else {
    if (code > 9) {
      set_status(status, D8_ERR_ARG);
      code = 10;
    }
    own |= (uint32_t)code << 2;
  }
  atomicAdd(&word[P::of(i, j)], own);
}

// The offsets table of Layout::off_tab: for row class rc and column k of a
// four-cell group, the distance in places from a cell to its neighbour in
// direction code (a signed byte), OUTSIDE where that lies outside the tile: in
// the first or last row (rk 0, 2; else 1) or in the first or last group (ck).
constexpr int OUTSIDE = -128;  // no distance is: the largest is 64 + 49
template <int T>
struct Table {
  static constexpr int CLASSES = Place<T>::RM + 1;
  static constexpr int BYTES = 3 * 3 * CLASSES * 4 * 8;
  // entry of column 0 of a group, in units of 8 bytes (columns follow)
  __device__ static __forceinline__ int of(int rk, int ck, int rc) { return ((rk * 3 + ck) * CLASSES + rc) * 4; }
};
template <int T, int NT>
__device__ __forceinline__ void fill_table(int8_t* tab) {
  using P = Place<T>;
  for (int e = threadIdx.x; e < Table<T>::BYTES; e += NT) {
    const int code = e & 7, k = (e / 8) & 3, rc = (e / 32) & P::RM, ck = e / (32 * (P::RM + 1)) % 3,
              rk = e / (32 * (P::RM + 1)) / 3;
    const int i = rc + P::RM + 1, j = 4 + k;  // any cell of that class away from the tile's edge
    const int di = code_di(code), dj = code_dj(code);
    const bool out = (rk == 0 && di < 0) || (rk == 2 && di > 0) || (ck == 0 && k == 0 && dj < 0) ||
                     (ck == 2 && k == 3 && dj > 0);
    tab[e] = (int8_t)(out ? OUTSIDE : di * T + P::col(i + di, j + dj) - P::col(i, j));
  }
}

// byte k of v, sign-extended (k below 8: prmt's selectors k + 8 copy its sign)
__device__ __forceinline__ int signed_byte(uint2 v, uint32_t k) {
  int r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(v.x), "r"(v.y), "r"(k * 0x1111u + 0x8880u));
  return r;
}

// The codes of a whole tile, loaded ahead: four consecutive cells of a row per
// 32-bit word, rows i0, i0 + RS, ... of group q per thread.  Every load is
// issued before any is used, one word per group.  Rows that start at an odd
// address are read as the aligned words that cover them and shifted into place
// when they are used; the word after a row's last group is held by the lane of
// that row's number among the thread's.  (Ragged tiles read theirs later.)
template <int T, int NT>
struct Codes {
  static constexpr int Q = Place<T>::Q;
  static constexpr int NQ = T * T / 4 / NT;  // four-cell groups per thread
  static constexpr int RS = NT / Q;          // rows from one group of a thread to its next
  static_assert(NQ <= Q, "a lane per row for the words after the rows");
  uint32_t word[NQ], after;
  __device__ static __forceinline__ int row0() { return threadIdx.x / Q; }
  __device__ static __forceinline__ int group() { return threadIdx.x & (Q - 1); }
  // address of the codes of this thread's group in row0() + r * RS
  __device__ static __forceinline__ const uint8_t* first(const DemDesc& d, const TileGeo& g, int r) {
    return d.dir + (g.i0 + row0() + r * RS) * d.lddir + (g.j0 + 4 * group());
  }
  __device__ static __forceinline__ bool aligned(const DemDesc& d) {
    return ((reinterpret_cast<uintptr_t>(d.dir) | (uintptr_t)d.lddir) & 3u) == 0;
  }

  __device__ __forceinline__ void load(const DemDesc& d, const TileGeo& g) {
    if (g.tw != T || g.th != T) return;
    if (aligned(d)) {
#pragma unroll
      for (int r = 0; r < NQ; r++) word[r] = __ldg(reinterpret_cast<const unsigned int*>(first(d, g, r)));
    } else {
#pragma unroll
      for (int r = 0; r < NQ; r++)
        word[r] = __ldg(reinterpret_cast<const unsigned int*>(reinterpret_cast<uintptr_t>(first(d, g, r)) & ~(uintptr_t)3));
      // lane q: the word that ends row row0() + q * RS, where its bytes are needed
      after = 0;
      if (group() < NQ) {
        const uintptr_t end = reinterpret_cast<uintptr_t>(d.dir + (g.i0 + row0() + group() * RS) * d.lddir + g.j0 + T);
        if (end & 3u) after = __ldg(reinterpret_cast<const unsigned int*>(end & ~(uintptr_t)3));
      }
    }
  }
  // once loaded: word[r] becomes the codes of group r
  __device__ __forceinline__ void shift(const DemDesc& d, const TileGeo& g) {
    if (g.tw != T || g.th != T || aligned(d)) return;
#pragma unroll
    for (int r = 0; r < NQ; r++)
      word[r] = unaligned_four<Q>(word[r], __shfl_sync(FULL, after, r, Q), first(d, g, r));
  }
};

// The words of tile g (zeroed before) from its codes: Algorithm 1.
template <int T, int NT, bool NARROW>
__device__ __forceinline__ void set_words(const Codes<T, NT>& codes, const DemDesc& d, const TileGeo& g, uint32_t* word,
                                          const uint2* tab, uint32_t* status) {
  using P = Place<T>;
  using C = Cell<T>;
  constexpr int NQ = Codes<T, NT>::NQ, RS = Codes<T, NT>::RS;
  const int i0 = Codes<T, NT>::row0(), q = Codes<T, NT>::group();
  if (g.th == T && g.tw == T) {
    // whole tiles: the tables give the places of the targets inside the tile
    const int ck = q == 0 ? 0 : (q == P::Q - 1 ? 2 : 1), rc = i0 & P::RM;
    uint32_t own_at[4];  // byte offset of the word of cell k of the first group
#pragma unroll
    for (int k = 0; k < 4; k++) own_at[k] = 4u * (uint32_t)(i0 * T + ((k * P::Q + q) ^ (rc * P::Q)));
    uint2 inner[4];  // the entries of the rows between the first and the last
#pragma unroll
    for (int k = 0; k < 4; k++) inner[k] = tab[Table<T>::of(1, ck, rc) + k];
    uint32_t wrong = 0;
#pragma unroll
    for (int r = 0; r < NQ; r++) {
      const uint32_t four = codes.word[r];
      wrong |= ((four & 0x7F7F7F7Fu) + 0x76767676u) | four;  // bit 7 of a byte: above 9
      uint2 dist_of[4];
#pragma unroll
      for (int k = 0; k < 4; k++) {
        dist_of[k] = inner[k];
        if (r == 0 && i0 == 0) dist_of[k] = tab[Table<T>::of(0, ck, rc) + k];
        if (r == NQ - 1 && i0 == RS - 1) dist_of[k] = tab[Table<T>::of(2, ck, rc) + k];
      }
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const uint32_t code = (four >> (8 * k)) & 0xFFu;
        const int dist = signed_byte(dist_of[k], code);
        const bool flows = code < 8u, in = flows && dist != OUTSIDE;
        const uint32_t o_at = own_at[k] + r * RS * T * 4, t = o_at + 4 * dist;
        atomicAdd(&at(word, in ? t : spare<T>()), LEFT1);
        atomicAdd(&at(word, o_at), in ? t + (C::ONE | IN) : code * 4u + (flows ? C::ONE + EXIT : C::ONE));
      }
    }
    if (wrong & 0x80808080u) set_status(status, D8_ERR_ARG);  // (such a cell's path ends there)
    return;
  }
  constexpr int U = 16;  // codes read at once
  const int sh = NARROW ? width_shift(g) : T == 64 ? 6 : 5, end = NARROW ? g.th << sh : T * T;
  static_assert(T == 64 || T == 32, "the shift of whole rows");
#pragma unroll 1
  for (int c0 = threadIdx.x; c0 < end; c0 += U * NT) {
    uint8_t code[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int c = c0 + u * NT, i = c >> sh, j = c & ((1 << sh) - 1);
      code[u] = i < g.th && j < g.tw ? __ldg(d.dir + (g.i0 + i) * d.lddir + (g.j0 + j)) : (uint8_t)0;
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int c = c0 + u * NT, i = c >> sh, j = c & ((1 << sh) - 1);
      if (i < g.th && j < g.tw) add_cell<T>(word, i, j, code[u], g, d, status);
    }
  }
}

// At the grid's edge a target off the grid is a path end, not an exit (whole
// tiles; set_words took every target outside the tile for an exit).
template <int T, int NT>
__device__ __forceinline__ void end_at_grid_edge(const DemDesc& d, const TileGeo& g, uint32_t* word) {
  using C = Cell<T>;
  if (g.th != T || g.tw != T || (g.i0 > 0 && g.j0 > 0 && g.i0 + T < d.H && g.j0 + T < d.W)) return;
  for (int s = threadIdx.x; s < 4 * T; s += NT) {
    int i, j;
    if (!slot_cell(s, T, T, T, i, j)) continue;
    uint32_t* w = &word[Place<T>::of(i, j)];
    const uint32_t v = *(volatile uint32_t*)w;
    if ((v & (IN | EXIT)) != EXIT) continue;
    const int64_t gi = g.i0 + i + code_di(C::code(v)), gj = g.j0 + j + code_dj(C::code(v));
    if (gi < 0 || gj < 0 || gi >= d.H || gj >= d.W) atomicAdd(w, 0u - EXIT);
  }
}

// A[tile] = the in-tile counts: four consecutive cells per thread in one 16-byte
// store when the layout allows, else one.  Returns whether one of this thread's
// cells still waits for an input: it lies on or below a cycle.
template <int T, int NT, bool NARROW>
__device__ __forceinline__ bool store_counts(const DemDesc& d, const TileGeo& g, const uint32_t* word) {
  using P = Place<T>;
  using C = Cell<T>;
  uint32_t left = 0;
  const bool vec = g.tw == T && g.th == T && ((reinterpret_cast<uintptr_t>(d.A) & 15u) == 0) && (d.ldA & 3) == 0;
  if (vec) {
    constexpr int RS = NT / P::Q;  // rows from one group of a thread to its next
    const int i0 = threadIdx.x / P::Q, j = 4 * (threadIdx.x & (P::Q - 1));
    uint32_t* dst = static_cast<uint32_t*>(d.A) + (g.i0 + i0) * d.ldA + (g.j0 + j);
    const uint32_t* w0[4];
#pragma unroll
    for (int k = 0; k < 4; k++) w0[k] = word + P::of(i0, j + k);
#pragma unroll
    for (int r = 0; r < T / RS; r++) {
      uint32_t w[4];
#pragma unroll
      for (int k = 0; k < 4; k++) w[k] = w0[k][r * RS * T];
      left |= (w[0] | w[1]) | (w[2] | w[3]);
      // (a cell that still waits has no count yet; the call reports it)
      *reinterpret_cast<uint4*>(dst) = make_uint4(w[0] >> C::CB, w[1] >> C::CB, w[2] >> C::CB, w[3] >> C::CB);
      dst += RS * d.ldA;
    }
  } else {
    // consecutive lanes store consecutive columns
    const int sh = NARROW ? width_shift(g) : T == 64 ? 6 : 5;
    const int RS = NT >> sh;  // rows at once
    const int i0 = threadIdx.x >> sh, j = threadIdx.x & ((1 << sh) - 1);
    uint32_t* dst = static_cast<uint32_t*>(d.A) + (g.i0 + i0) * d.ldA + (g.j0 + j);
    if (j < g.tw) {
#pragma unroll 8
      for (int i = i0; i < g.th; i += RS) {
        const uint32_t w = word[P::of(i, j)];
        left |= w;
        *dst = w >> C::CB;
        dst += RS * d.ldA;
      }
    }
  }
  return left >= LEFT1;
}

// Perimeter summary of a finished tile: for each perimeter slot, the exit of
// the cell's in-tile path (Algorithms 3-4 seen from the exit side) found by
// following links, and the in-tile count at the slot.
template <int T, int NT>
__device__ __forceinline__ void perimeter_summary(const TileGeo& g, int64_t t, uint32_t* word, bool cyc,
                                                  const Pipe& p) {
  using P = Place<T>;
  using C = Cell<T>;
  constexpr int N = 4 * T / NT;  // slots per thread, followed side by side
  uint16_t* pex = p.pex + t * (4 * T);
  uint32_t* pval = static_cast<uint32_t*>(p.pval) + t * (4 * T);
  uint32_t w[N], o[N], v[N];
#pragma unroll
  for (int r = 0; r < N; r++) {
    int i, j;
    w[r] = 0u;
    o[r] = 0u;
    if (slot_cell(threadIdx.x + r * NT, g.th, g.tw, T, i, j)) {
      o[r] = 4u * (uint32_t)P::of(i, j);
      w[r] = at(word, o[r]);
    }
    v[r] = cyc ? 0u : w[r];
    pval[threadIdx.x + r * NT] = w[r] >> C::CB;
  }
  for (int guard = 0; guard < 2 * T * T; guard++) {
    uint32_t any = 0;
#pragma unroll
    for (int r = 0; r < N; r++) {
      if (v[r] & IN) {
        o[r] = v[r] & C::LINK;
        v[r] = at(word, o[r]);
        any |= v[r];
      }
    }
    if (!(any & IN)) break;
  }
#pragma unroll
  for (int r = 0; r < N; r++) {
    uint16_t pe = PEX_TERM;
    if ((w[r] & (IN | EXIT)) == EXIT)
      pe = (uint16_t)(PEX_EXIT | C::code(w[r]));
    else if ((w[r] & IN) && (v[r] & (IN | EXIT)) == EXIT)
      pe = (uint16_t)slot_of(P::row(o[r] >> 2), P::column(o[r] >> 2), g.th, g.tw, T);
    pex[threadIdx.x + r * NT] = pe;
  }
}

// Algorithm 2 for one walk per lane, up to STEPS cells.  A walk is the cell it
// finished last: o, the byte offset of its word, and w, the word with the
// cell's complete count.  Each step delivers that count to the cell's target;
// if it was the target's last input the walk finishes it and goes on there.
// Returns whether the walk is still under way.  The cell it starts from gets a
// link to where it came (the last finished cell, or the junction that waits
// for others): a shorter way for those who follow links later.
template <int T>
__device__ __forceinline__ bool advance(uint32_t& o, uint32_t* word) {
  using C = Cell<T>;
  const uint32_t start = o, w0 = at(word, o);
  uint32_t w = w0;
  bool go = true;
#pragma unroll
  for (int u = 0; u < STEPS; u++) {
    const bool in = go && (w & IN) != 0u;
    const uint32_t t = in ? w & C::LINK : spare<T>(), add = (w & C::CNT) - LEFT1;
    const uint32_t old = atomicAdd(&at(word, t), add);
    go = in && C::last(old);
    w = old + add;
    o = in ? t : o;
  }
  if (w0 & IN) at(word, start) = (w0 & ~C::LINK) | o;
  return go;
}

// The last walks of a tile, one per lane, to their ends.  No other warp moves
// any more, so a target that waits for one input waits for this lane's walk
// and is finished by a plain load and store: the chain per cell is one load
// and two operations, not an atomic's reply.  Only junctions that wait for
// more take the atomic.
template <int T>
__device__ __forceinline__ void finish(uint32_t o, bool on, uint32_t* word) {
  using C = Cell<T>;
  const uint32_t start = o;
  uint32_t w = at(word, o);
  bool go = on;
  while (__any_sync(FULL, go)) {
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const bool in = go && (w & IN) != 0u;
      const uint32_t t = in ? w & C::LINK : spare<T>(), add = (w & C::CNT) - LEFT1;
      uint32_t old = *(volatile uint32_t*)&at(word, t);
      go = in && C::last(old);
      const bool meets = in && !go, alone = go;
      if (__any_sync(FULL, meets)) {
        if (meets) old = atomicAdd(&at(word, t), add);
        go = in && C::last(old);
      }
      if (go && o != start) at(word, o) = (w & ~C::LINK) | start;
      w = go ? old + add : w;
      if (alone) *(volatile uint32_t*)&at(word, t) = w;
      o = go ? t : o;
    }
  }
  if (on && o != start) at(word, start) = (at(word, start) & ~C::LINK) | o;
}

// NARROW (narrow_grid): the loops over a tile's cells
// end with its rows, and its rows are counted by their own width.
template <int T, int NT, bool NARROW>
__global__ void __launch_bounds__(NT, NT <= 64 ? 12 : 4) k_up_count(DemTable dt, Pipe p) {
  using L = Layout<T, NT>;
  using C = Cell<T>;
  constexpr int TT = T * T, ROWS = TT / NT, NW = L::NW, CAP = L::CAP;
  extern __shared__ __align__(16) unsigned char sm[];
  uint32_t* word = reinterpret_cast<uint32_t*>(sm + L::off_word);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint16_t* stacks = reinterpret_cast<uint16_t*>(sm + L::off_stack);
  uint16_t* pool = stacks + NW * CAP;
  const uint2* tab = reinterpret_cast<const uint2*>(sm + L::off_tab);
  uint32_t* misc = reinterpret_cast<uint32_t*>(sm + L::off_misc);  // pooled walks, warps done, next tile
  const unsigned lt = (1u << lane) - 1u;

  fill_table<T, NT>(reinterpret_cast<int8_t*>(sm + L::off_tab));
  // Block b starts with tile b, later ones come from the queue, one ahead:
  // the next tile's codes are requested before this one's walks.
  Codes<T, NT> codes;
  int64_t t = blockIdx.x;
  if (t < p.ntiles) {
    const DemDesc d = dem_of(dt, t);
    codes.load(d, tile_geo(d, t - d.tile_base, T));
  }
  for (int64_t next; t < p.ntiles; t = next) {
    const DemDesc d = dem_of(dt, t);
    const TileGeo g = tile_geo(d, t - d.tile_base, T);
    __syncthreads();  // everyone is done with the tile before
    uint4* w4 = reinterpret_cast<uint4*>(word);
    for (int c = threadIdx.x; c < TT / 4; c += NT) w4[c] = make_uint4(0, 0, 0, 0);
    if (threadIdx.x == 0) {
      misc[0] = misc[1] = 0;
      misc[2] = gridDim.x + atomicAdd(p.queue, 1u);
    }
    __syncthreads();
    codes.shift(d, g);
    set_words<T, NT, NARROW>(codes, d, g, word, tab, p.status);
    __syncthreads();
    end_at_grid_edge<T, NT>(d, g, word);  // (only the summary reads what it changes)
    next = misc[2];
    if (next < p.ntiles) {
      const DemDesc dn = dem_of(dt, next);
      codes.load(dn, tile_geo(dn, next - dn.tile_base, T));
    }
    // Algorithm 2.  Sources (count 1, no input) are swept, a row of the block's
    // cells at a time: each delivers its 1 to its target (its link already
    // says so), and the source that delivers a target's last input queues a
    // walk from there.  (A cell that is no source never looks like one: its
    // count is above 1 once its last input has arrived.)
    uint16_t* stack = stacks + warp * CAP;
    int n = 0;           // walks on the stack
    bool alone = false;  // this warp came last and finishes the tile's walks
    const int rows = NARROW ? (g.th * T + NT * SWEEP - 1) / (NT * SWEEP) * SWEEP : ROWS;
    for (int r = 0;;) {
      while (r < rows && n < 32) {
        uint32_t s[SWEEP];
        bool ready[SWEEP];
#pragma unroll
        for (int u = 0; u < SWEEP; u++) {
          const uint32_t w = word[threadIdx.x + (r + u) * NT];
          const bool src = (w & (~(C::ONE - 1u) | IN)) == (C::ONE | IN);  // with a target in the tile
          s[u] = src ? w & C::LINK : spare<T>();
          const uint32_t old = atomicAdd(&at(word, s[u]), C::ONE - LEFT1);
          ready[u] = src && C::last(old);
        }
#pragma unroll
        for (int u = 0; u < SWEEP; u++) {
          const unsigned m = __ballot_sync(FULL, ready[u]);
          if (ready[u]) stack[n + __popc(m & lt)] = (uint16_t)s[u];
          n += __popc(m);
        }
        r += SWEEP;
      }
      __syncwarp();
      if (n < 32) {  // swept, and no full batch left
        if (alone) break;
        // the walks left go to the pool; the last warp to come goes on with it
        uint32_t base = 0, come = 0;
        if (lane == 0) base = atomicAdd(&misc[0], (uint32_t)n);
        base = __shfl_sync(FULL, base, 0);
        if (lane < n) pool[base + lane] = stack[lane];
        __syncwarp();
        __threadfence_block();  // the pooled walks, and the cells they finished, before the arrival
        if (lane == 0) come = atomicAdd(&misc[1], 1u);
        come = __shfl_sync(FULL, come, 0);
        if (come != NW - 1) break;
        __threadfence_block();
        alone = true;
        stack = pool;
        n = (int)*(volatile uint32_t*)&misc[0];
        if (n < 32) break;
      }
      n -= 32;
      uint32_t o = *(volatile uint16_t*)&stack[n + lane];
      const bool on = advance<T>(o, word);
      const unsigned m = __ballot_sync(FULL, on);  // (the batch has been read before its places are written again)
      if (on) stack[n + __popc(m & lt)] = (uint16_t)o;
      n += __popc(m);
      __syncwarp();
    }
    if (alone) finish<T>(lane < n ? *(volatile uint16_t*)&stack[lane] : spare<T>(), lane < n, word);
    __syncthreads();
    const bool cyc = __syncthreads_or(store_counts<T, NT, NARROW>(d, g, word));
    if (threadIdx.x == 0 && cyc) set_status(p.status, D8_ERR_CYCLE);
    perimeter_summary<T, NT>(g, t, word, cyc, p);
  }
}

// Blocks of kernel k that run at once on the device.
template <class K>
static int64_t resident(K k, int threads, size_t bytes) {
  int dev = 0, sms = 1, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, bytes) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  return (int64_t)per_sm * sms;
}

// Wide blocks where all tiles are under way at once: a tile's own latency is
// what the pass takes then.  512 x 512 (64 tiles): 17 us, 27 in blocks of 64
// threads; 576 tiles: 25 and 29; 676, more than the 608 wide blocks that fit at
// once: 33 and 30.  32 x 32 tiles, 256 of them: 12.8 and 15.8.
template <int T, int NT, bool NARROW>
static cudaError_t launch_nt(const DemTable& dt, const Pipe& p, bool resident_only, bool* done, cudaStream_t s) {
  auto k = k_up_count<T, NT, NARROW>;
  constexpr size_t bytes = Layout<T, NT>::bytes;
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  const int64_t at_once = resident(k, NT, bytes);
  *done = !resident_only || p.ntiles <= at_once;
  if (!*done) return cudaSuccess;
  const int64_t grid = min64(at_once, p.ntiles);
  k<<<(unsigned)(grid < 1 ? 1 : grid), NT, bytes, s>>>(dt, p);
  return cudaGetLastError();
}

template <int T>
static cudaError_t launch_t(const DemTable& dt, const Pipe& p, cudaStream_t s) {
  constexpr int WIDE = 4 * T, NT = 64;
  bool done = false;
  const cudaError_t e = launch_nt<T, WIDE, false>(dt, p, true, &done, s);
  if (e != cudaSuccess || done) return e;
  return narrow_grid(dt, T) ? launch_nt<T, NT, true>(dt, p, false, &done, s)
                            : launch_nt<T, NT, false>(dt, p, false, &done, s);
}

}  // namespace count

cudaError_t launch_up_count(const DemTable& dt, const Pipe& p, cudaStream_t s) {
  switch (p.T) {
    case 32: return count::launch_t<32>(dt, p, s);
    case 64: return count::launch_t<64>(dt, p, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace d8
