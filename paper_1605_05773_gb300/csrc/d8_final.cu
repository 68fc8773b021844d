// d8_final.cu -- the finalise (Algorithms 7-8) after the layered combine,
// restricted to where it changes anything: unit counts, and weighted areas.
//
// The final count is A(c) + F(c), where A holds the in-tile counts and F(c) is
// the inflow from other tiles routed through c.  Inflow enters a tile only at
// its receivers (perimeter cells with an up-slope neighbour in another tile);
// the combine leaves it per perimeter slot.  It follows the unique down-slope
// path from there, so each receiver walks its path once adding its inflow to
// every cell on it: additions commute, so the walks need no ordering between
// them and no reply from the shared atomics, and only the cells down-slope of
// a receiver (about a sixth of a 64 x 64 tile on fractal terrain) are touched.
// Then the 16-byte quads of A with inflow are read, added to and written.
//
// The walks are chains of a code's load and six operations per cell, so what
// counts is few instructions per step and many tiles per SM: the codes of
// perimeter cells that leave the tile are replaced by a path end beforehand
// (no bounds in the walk), offsets come from a table in two registers, and the
// next tile's inflow and codes are requested before this one's walks.
//
// Measured, T = 64: 32768 x 32768 fractal 2.03 ms, 8192 x 8192 140 us (before,
// with the receivers found and their inflow gathered here: 3.06 ms, 203 us; with
// rows of 64 cells, whose vertical neighbours share a bank: 2.38 ms, 160 us, and
// 312 instead of 151 us on an 8192 x 8192 boustrophedon); 3001 x 5003, rows at
// odd addresses: 47 us (73 when their codes and counts were read one by one).
// The receivers' paths overlap (65 receivers, 2800 additions to 540 cells of a
// tile), so the shared-memory pipe is what bounds it.
#include "d8_device.cuh"

namespace d8 {
namespace fin {

constexpr int NTN = 128;  // threads per tile block
constexpr unsigned FULL = 0xFFFFFFFFu;

// Cells are numbered with a row stride of T + 4: vertical neighbours lie in
// different banks, and a row of codes that starts at an odd address fits with
// the bytes around it (Ahead).
template <int T>
struct Layout {
  static constexpr int S = T + 4;
  static constexpr size_t TS = (size_t)T * S;
  static constexpr size_t off_f = 0;                         // uint32 per cell: inflow routed through it
  static constexpr size_t off_code = TS * 4;                 // uint8 [2][TS]: codes of this tile and the next
  static constexpr size_t off_rin = off_code + 2 * TS;       // uint32 per receiver: its inflow
  static constexpr size_t off_rcell = off_rin + (size_t)4 * T * 4;  // uint16 per receiver: its cell
  static constexpr size_t off_misc = off_rcell + (size_t)4 * T * 2;
  static constexpr size_t bytes = off_misc + 16;
};

// distance in cells to the neighbour in direction code
template <int T>
__device__ __forceinline__ int step_of(uint32_t code) {
  constexpr int S = T + 4;
  if (T <= 64) {  // signed bytes N, NE, E, SE / S, SW, W, NW (prmt's selectors k + 8 copy byte k's sign)
    constexpr uint32_t lo = (uint32_t)(-S & 0xFF) | (uint32_t)((1 - S) & 0xFF) << 8 | 1u << 16 | (uint32_t)(S + 1) << 24;
    constexpr uint32_t hi = (uint32_t)S | (uint32_t)(S - 1) << 8 | 0xFFu << 16 | (uint32_t)((-S - 1) & 0xFF) << 24;
    int r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(lo), "r"(hi), "r"(code * 0x1111u + 0x8880u));
    return r;
  }
  return code_di((int)code) * S + code_dj((int)code);
}

// What a tile needs, requested ahead: the inflow of this thread's slots, and
// the codes by asynchronous copies into code[].  Rows of whole tiles are copied
// as the aligned words that cover them, one more word than the row has when it
// starts at an odd address, and shifted into place in finish().
template <int T, int NT, class V, bool NARROW = false>
struct Ahead {
  static constexpr int S = T + 4;
  static constexpr int NS = (4 * T + NT - 1) / NT;           // slots per thread
  static constexpr int Q = T / 4;                            // words per row
  static constexpr int RS = NT / Q, NQ = T * Q / NT;       // rows at once, words per thread
  V in[NS];

  __device__ static __forceinline__ bool whole(const TileGeo& g) { return g.tw == T && g.th == T; }
  __device__ static __forceinline__ bool aligned(const DemDesc& d) {
    return ((reinterpret_cast<uintptr_t>(d.dir) | (uintptr_t)d.lddir) & 3u) == 0;
  }

  __device__ __forceinline__ void load(const Pipe& p, const DemDesc& d, const TileGeo& g, int64_t t, uint8_t* code) {
    const V* inflow = static_cast<const V*>(p.S);
#pragma unroll
    for (int r = 0; r < NS; r++) {
      const int s = threadIdx.x + r * NT;
      in[r] = inflow && s < 4 * T ? inflow[t * (4 * T) + s] : V{};
    }
    const int i0 = threadIdx.x / Q, q = threadIdx.x % Q;
    if (whole(g)) {
      const uint8_t* src = d.dir + (g.i0 + i0) * d.lddir + (g.j0 + 4 * q);
      uint8_t* dst = code + i0 * S + 4 * q;
#pragma unroll 4
      for (int r = 0; r < NQ; r++) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(src) & ~(uintptr_t)3;
        cp_async4(dst, reinterpret_cast<const void*>(a), 4);
        if (q == Q - 1 && a != reinterpret_cast<uintptr_t>(src)) cp_async4(dst + 4, reinterpret_cast<const void*>(a + 4), 4);
        src += RS * d.lddir;
        dst += RS * S;
      }
    } else {
      const int sh = width_shift(g), end = NARROW ? g.th << sh : T * T;
#pragma unroll 8
      for (int c = threadIdx.x; c < end; c += NT) {
        const int i = NARROW ? c >> sh : c / T, j = NARROW ? c & ((1 << sh) - 1) : c % T;
        if (i < g.th && j < g.tw) code[i * S + j] = __ldg(d.dir + (g.i0 + i) * d.lddir + (g.j0 + j));
      }
    }
    cp_async_commit();
  }
  // waits for this thread's copies and puts its part of the codes in place
  __device__ __forceinline__ void finish(const DemDesc& d, const TileGeo& g, uint8_t* code) const {
    cp_async_wait<0>();
    if (!whole(g) || aligned(d)) return;
    const int i0 = threadIdx.x / Q, q = threadIdx.x % Q;
    const uintptr_t src = reinterpret_cast<uintptr_t>(d.dir + (g.i0 + i0) * d.lddir + g.j0);
    uint32_t* w = reinterpret_cast<uint32_t*>(code + i0 * S) + q;
    __syncwarp();  // a row's words were copied by lanes of this warp
    uint32_t f[NQ];
#pragma unroll
    for (int r = 0; r < NQ; r++)
      f[r] = __funnelshift_r(w[r * RS * (S / 4)], w[r * RS * (S / 4) + 1],
                             8u * (uint32_t)((src + r * RS * (uintptr_t)d.lddir) & 3u));
    __syncwarp();  // and read before one is written
#pragma unroll
    for (int r = 0; r < NQ; r++) w[r * RS * (S / 4)] = f[r];
  }
};

// NARROW (narrow_grid): the loops over a tile's cells end with its rows, and its
// rows are counted by their own width.
template <int T, bool NARROW>
__global__ void __launch_bounds__(NTN, 8) k_fin_count(DemTable dt, Pipe p) {
  using L = Layout<T>;
  using AH = Ahead<T, NTN, uint32_t, NARROW>;
  constexpr int TT = T * T, S = L::S, TS = (int)L::TS, NS = AH::NS;
  extern __shared__ __align__(16) unsigned char sm[];
  uint32_t* F = reinterpret_cast<uint32_t*>(sm + L::off_f);
  uint32_t* rin = reinterpret_cast<uint32_t*>(sm + L::off_rin);
  uint16_t* rcell = reinterpret_cast<uint16_t*>(sm + L::off_rcell);
  uint32_t* misc = reinterpret_cast<uint32_t*>(sm + L::off_misc);  // receivers (by tile parity), next tile
  const int lane = threadIdx.x & 31;

  // F starts at zero; every tile leaves the words it touched at zero again
  for (int q = threadIdx.x; q < TS / 4; q += NTN) reinterpret_cast<uint4*>(F)[q] = make_uint4(0, 0, 0, 0);
  if (threadIdx.x < 2) misc[threadIdx.x] = 0u;
  AH ahead;
  int64_t t = blockIdx.x;
  if (t < p.ntiles) {
    const DemDesc d = dem_of(dt, t);
    ahead.load(p, d, tile_geo(d, t - d.tile_base, T), t, sm + L::off_code);
  }
  int buf = 0;
  for (int64_t next; t < p.ntiles; t = next, buf ^= 1) {
    const DemDesc d = dem_of(dt, t);
    const TileGeo g = tile_geo(d, t - d.tile_base, T);
    uint8_t* code = sm + L::off_code + buf * TS;
    if (threadIdx.x == 0) misc[2] = gridDim.x + atomicAdd(p.queue + 1, 1u);
    ahead.finish(d, g, code);
    __syncthreads();  // codes landed; everyone is done with the tile before
    // Algorithm 7: the receivers listed; codes that leave the tile end the walk
#pragma unroll
    for (int r = 0; r < NS; r++) {
      int i, j;
      uint32_t in = ahead.in[r];
      const bool cell = slot_cell(threadIdx.x + r * NTN, g.th, g.tw, T, i, j);
      if (cell) {
        const uint32_t k = code[i * S + j];
        const int ti = i + code_di(k & 7), tj = j + code_dj(k & 7);
        if (k < 8u && ((unsigned)ti >= (unsigned)g.th || (unsigned)tj >= (unsigned)g.tw)) code[i * S + j] = 8;
        // flow entering across the grid's first or last row (a strip)
        if (p.top_in && g.i0 + i == 0) in += p.top_in[g.j0 + j];
        if (p.bot_in && g.i0 + i == d.H - 1) in += p.bot_in[g.j0 + j];
      }
      const unsigned m = __ballot_sync(FULL, cell && in != 0u);
      uint32_t base = 0;
      if (lane == 0 && m) base = atomicAdd(&misc[buf], (uint32_t)__popc(m));
      base = __shfl_sync(FULL, base, 0);
      if (cell && in != 0u) {
        const int at = (int)base + __popc(m & ((1u << lane) - 1u));
        rcell[at] = (uint16_t)(i * S + j);
        rin[at] = in;
      }
    }
    __syncthreads();
    const int nrec = (int)misc[buf];
    if (threadIdx.x == 0) misc[buf ^ 1] = 0u;
    next = misc[2];
    if (next < p.ntiles) {
      const DemDesc dn = dem_of(dt, next);
      ahead.load(p, dn, tile_geo(dn, next - dn.tile_base, T), next, sm + L::off_code + (buf ^ 1) * TS);
    }
    // Algorithm 8 on the receivers' paths (a path inside one tile has at most
    // T^2 cells; the bound only matters for a field with a cycle, which the
    // tile pass reports)
    for (int r = threadIdx.x; r < nrec; r += NTN) {
      const uint32_t in = rin[r];
      int c = rcell[r];
      for (int n = 0; n < TT; n++) {
        atomicAdd(&F[c], in);
        const uint32_t k = code[c];
        if (k >= 8u) break;
        c += step_of<T>(k);
      }
    }
    __syncthreads();
    // A += F where F is not zero; those words go back to zero.  16-byte quads
    // when the layout allows, else single cells, in consecutive lanes; the
    // reads of U of them are issued before any is used.
    uint32_t* const A0 = static_cast<uint32_t*>(d.A) + g.i0 * d.ldA + g.j0;
    if constexpr (NARROW) {
      const int sh = width_shift(g), jm = (1 << sh) - 1;
#pragma unroll 1
      for (int q = threadIdx.x; q < g.th << sh; q += NTN) {
        const int i = q >> sh, j = q & jm;  // (columns off the tile have no inflow)
        const uint32_t f = F[i * S + j];
        if (f) {
          F[i * S + j] = 0u;
          A0[i * d.ldA + j] += f;
        }
      }
    } else if (g.tw == T && ((reinterpret_cast<uintptr_t>(d.A) & 15u) == 0) && (d.ldA & 3) == 0) {
      constexpr int NQ = TT / 4 / NTN, U = NQ < 4 ? NQ : 4;
#pragma unroll 1
      for (int r0 = 0; r0 < NQ; r0 += U) {
        uint4 f[U], a[U];
        bool on[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int q = threadIdx.x + (r0 + u) * NTN;
          uint4* fq = reinterpret_cast<uint4*>(F) + q / (T / 4) * (S / 4) + q % (T / 4);
          f[u] = *fq;
          on[u] = (f[u].x | f[u].y | f[u].z | f[u].w) != 0u;
          if (on[u]) {
            *fq = make_uint4(0, 0, 0, 0);
            a[u] = *reinterpret_cast<const uint4*>(A0 + q / (T / 4) * d.ldA + q % (T / 4) * 4);
          }
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int q = threadIdx.x + (r0 + u) * NTN;
          if (on[u])
            *reinterpret_cast<uint4*>(A0 + q / (T / 4) * d.ldA + q % (T / 4) * 4) =
                make_uint4(a[u].x + f[u].x, a[u].y + f[u].y, a[u].z + f[u].z, a[u].w + f[u].w);
        }
      }
    } else {
      constexpr int NQ = TT / NTN, U = 8;
#pragma unroll 1
      for (int r0 = 0; r0 < NQ; r0 += U) {
        uint32_t f[U], a[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int q = threadIdx.x + (r0 + u) * NTN;  // (cells off a ragged tile have no inflow)
          uint32_t* fq = F + q / T * S + q % T;
          f[u] = *fq;
          if (f[u]) {
            *fq = 0u;
            a[u] = A0[q / T * d.ldA + q % T];
          }
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int q = threadIdx.x + (r0 + u) * NTN;
          if (f[u]) A0[q / T * d.ldA + q % T] = a[u] + f[u];
        }
      }
    }
  }
  cp_async_wait<0>();
}

// ---- weighted areas
constexpr int NTW = 256;  // threads per tile block

// 96-bit two's-complement fixed point, three 32-bit words (w0 lowest).
struct fx96 {
  uint32_t w0, w1, w2;
};

// round(f * 2^q) (ties away from zero) for a finite f with |f| 2^q < 2^94
__device__ __forceinline__ fx96 fx96_of(float f, int q) {
  const uint32_t bits = __float_as_uint(f);
  const int E = (int)((bits >> 23) & 0xFFu);
  const uint32_t mant = (bits & 0x7FFFFFu) | (E ? 0x800000u : 0u);
  const int s = (E ? E : 1) - 150 + q;  // f * 2^q = mant * 2^s
  uint64_t lo = 0;
  uint32_t hi = 0;
  if (mant != 0u) {
    if (s >= 64) {
      hi = mant << (s - 64);
    } else if (s >= 0) {
      lo = (uint64_t)mant << s;
      hi = s > 40 ? (uint32_t)(mant >> (64 - s)) : 0u;
    } else if (s > -26) {
      lo = ((uint64_t)mant + (1ull << (-s - 1))) >> (-s);
    }
  }
  if (bits >> 31) {  // negate the 96-bit value
    lo = ~lo + 1ull;
    hi = ~hi + (lo == 0ull ? 1u : 0u);
  }
  return fx96{(uint32_t)lo, (uint32_t)(lo >> 32), hi};
}

__device__ __forceinline__ fx96 fx96_add(fx96 a, fx96 b) {
  const uint64_t al = a.w0 | ((uint64_t)a.w1 << 32), bl = b.w0 | ((uint64_t)b.w1 << 32);
  const uint64_t l = al + bl;
  return fx96{(uint32_t)l, (uint32_t)(l >> 32), a.w2 + b.w2 + (l < al ? 1u : 0u)};
}

// The finalise's per-cell fixed-point accumulator: word 0 is the low 32 bits,
// summed modulo 2^32 with the carry of each addition taken from the atomic's
// reply; words 1 and 2 are limbs of LB bits (unsigned, then signed) summed
// without carries, their spare bits absorbing up to 4T additions (one per
// receiver).  A value x with |x| < 2^(32 + 2 LB) enters as x0 = x mod 2^32,
// x1 = (x >> 32) mod 2^LB, x2 = x >> (32 + LB); the three words then hold the
// exact sum as w0 + w1 2^32 + w2 2^(32 + LB), whatever the order.
template <int T>
struct FxLimbs {
  static constexpr int LB = T >= 128 ? 22 : (T >= 64 ? 23 : 24);  // 4T (LB-bit limb + carry) sums < 2^31
  static constexpr int VB = 32 + 2 * LB;                          // value bits, sign included
};

template <int T>
__device__ __forceinline__ void fx_split(fx96 v, uint32_t& x0, uint32_t& x1, uint32_t& x2) {
  constexpr int LB = FxLimbs<T>::LB;
  const long long rest = (long long)(v.w1 | ((unsigned long long)v.w2 << 32));  // v >> 32, |rest| < 2^(2 LB)
  x0 = v.w0;
  x1 = (uint32_t)rest & ((1u << LB) - 1u);
  x2 = (uint32_t)(int)(rest >> LB);
}

// the three words of a cell back to a 96-bit two's-complement value
template <int T>
__device__ __forceinline__ fx96 fx_join(uint32_t w0, uint32_t w1, uint32_t w2) {
  constexpr int LB = FxLimbs<T>::LB;
  const uint64_t lo = (uint64_t)w0 + ((uint64_t)w1 << 32);  // w1 < 2^31
  const long long t = (long long)(int)w2;                  // signed sum of the top limbs
  const uint64_t tl = (uint64_t)t << (32 + LB);
  const fx96 a{(uint32_t)lo, (uint32_t)(lo >> 32), 0u};
  const fx96 b{(uint32_t)tl, (uint32_t)(tl >> 32), (uint32_t)(t >> (32 - LB))};
  return fx96_add(a, b);
}

// 2^k as fp32 for -126 <= k <= 127 (built from its exponent field: exact)
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((127 + k) << 23); }

// The fixed-point value (w0, w1, w2) * 2^-q as float-float: the top 62 bits
// of the magnitude rounded to fp32, plus their exact remainder rounded to
// fp32 (a relative error of at most 2^-48 from the remainder's rounding and
// 2^-61 from the bits below the top 62).  2^-q is passed as two powers of two
// p1 * p2 of the normal range; each product below is exact until the last,
// which rounds once.
__device__ __forceinline__ ff fx96_to_ff(uint32_t w0, uint32_t w1, uint32_t w2, float p1, float p2) {
  uint64_t lo = w0 | ((uint64_t)w1 << 32);
  uint32_t hi = w2;
  const bool neg = (hi >> 31) != 0u;
  if (neg) {
    lo = ~lo + 1ull;
    hi = ~hi + (lo == 0ull ? 1u : 0u);
  }
  const int p = hi ? 95 - __clz(hi) : (lo ? 63 - __clzll(lo) : 0);  // leading bit
  int sh = 0;
  uint64_t U = lo;
  if (p > 61) {
    sh = p - 61;
    U = (lo >> sh) | (hi ? ((uint64_t)hi << (64 - sh)) : 0ull);
  }
  const float fh = __ull2float_rn(U);  // U < 2^62 rounded to 24 bits: an integer
  const float fl = __ll2float_rn((long long)(U - __float2ull_rn(fh)));
  const float sc = pow2f(sh);  // sh <= 34
  const ff r{__fmul_rn(__fmul_rn(__fmul_rn(fh, sc), p1), p2), __fmul_rn(__fmul_rn(__fmul_rn(fl, sc), p1), p2)};
  return neg ? ff{-r.hi, -r.lo} : r;
}

// The same value with |lo| at most half an ulp of hi (TwoSum: exact whatever the
// parts' sizes; the combine's sums are not normalised, and where they cancel
// the low part can be all there is).
__device__ __forceinline__ ff normalised(ff a) {
  const float s = __fadd_rn(a.hi, a.lo);
  const float b = __fsub_rn(s, a.hi);
  return ff{s, __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, b)), __fsub_rn(a.lo, b))};
}

// The tile's codes lie with the padded row stride of Ahead; the fixed-point
// words of cell (i, j) at i * T + (j ^ 4 (i mod 8)), which puts vertical
// neighbours in different banks without the padding's memory (four tiles per
// SM need it).
template <int T>
struct LayoutW {
  static constexpr int S = T + 4;
  static constexpr size_t TT = (size_t)T * T;
  static constexpr size_t off_w = 0;                     // uint32 [3][TT]
  static constexpr size_t off_code = TT * 12;            // uint8 code per cell
  static constexpr size_t off_rin = (off_code + (size_t)T * S + 15) / 16 * 16;  // ff per receiver
  static constexpr size_t off_rcell = off_rin + (size_t)4 * T * sizeof(ff);     // uint16 per receiver: i * S + j
  static constexpr size_t off_misc = off_rcell + (size_t)4 * T * 2;
  static constexpr size_t bytes = off_misc + 32;
};
template <int T>
__device__ __forceinline__ int word_at(int i, int j) {
  return i * T + (j ^ ((i & 7) * 4));
}

// Algorithms 7-8 for weighted areas, with the same walks as the unit counts.
// The inflow is added in fixed point so that the additions stay exact and
// commute: F(c) is an integer in units of 2^-q.  The scale is set per tile from
// the receivers' inflows: with |in_r| < 2^e_r, S = sum over receivers of 2^e_r
// (an exact integer sum of powers of two, so the same in every run) bounds the
// sum of their magnitudes.
//
// q makes S * 2^q <= 2^(VB - 2), so that no partial sum of the three words
// (FxLimbs: VB = 78 value bits for 64 x 64 tiles) reaches 2^(VB - 1) in
// magnitude.  Each receiver's float-float inflow is rounded once to a multiple
// of 2^-q, an error below 2^-q <= 2^-(VB - 4) * sum |in_r| (2^-74 for 64 x 64
// tiles), far below fp32 resolution even when the tile's inflows span twenty
// orders of magnitude.
//
// After the rounding the sums are exact, so this pass does not depend on the
// schedule.  Finally A = fp32(A + F), F converted to float-float.  A non-finite
// inflow (non-finite weights) cannot be scaled: the tile keeps its in-tile
// areas and D8_ERR_NONFINITE is raised.
//
// Measured, T = 64, 8192 x 8192 fractal: 581 us; 690 us when this pass gathered
// its receivers' inflow itself, tested bounds at each step and had vertical
// neighbours in one bank (the combine, which now leaves the inflow, went from
// 400 to 434 us).  A second accumulator of 64 bits for tiles whose inflows lie
// close together took 527 us, at less precision: not used.

// Each receiver's walk, adding its inflow to every cell on its path.
template <int T>
__device__ __forceinline__ void add_inflow(const uint8_t* code, uint32_t* F0, const uint16_t* rcell, const ff* rin,
                                           int nrec, int q) {
  constexpr int TT = T * T, S = T + 4;
  for (int r = threadIdx.x; r < nrec; r += NTW) {
    const ff in = rin[r];
    const fx96 v = fx96_add(fx96_of(in.hi, q), fx96_of(in.lo, q));
    uint32_t x0, x1, x2;
    fx_split<T>(v, x0, x1, x2);
    int c = rcell[r], i = c / S, w = i * T + (c - i * S);  // w: i * T + j
    for (int step = 0; step < TT; step++) {
      uint32_t* f = F0 + (w ^ ((w / T & 7) * 4));
      const uint32_t o0 = atomicAdd(f, x0);
      const uint32_t k = code[c];  // the walk goes on while the reply is in flight
      const uint32_t up = x1 + ((o0 + x0 < o0) ? 1u : 0u);
      if (up) atomicAdd(f + TT, up);
      if (x2) atomicAdd(f + 2 * TT, x2);
      if (k >= 8u) break;
      const int d = step_of<T>(k);
      c += d;
      w += d - 4 * code_di((int)k);
    }
  }
}

// A = fp32(A + F) where F is not zero; those words go back to zero.
template <int T>
__device__ __forceinline__ void add_to_areas(const DemDesc& d, const TileGeo& g, uint32_t* F0, float p1, float p2) {
  constexpr int TT = T * T;
  const bool vec = g.tw == T && ((reinterpret_cast<uintptr_t>(d.A) & 15u) == 0) && (d.ldA & 3) == 0;
  float* const A0 = static_cast<float*>(d.A) + g.i0 * d.ldA + g.j0;
  constexpr int NQ = TT / 4 / NTW > 0 ? TT / 4 / NTW : 1, U = NQ < 2 ? NQ : 2;  // quads per thread, read at once
#pragma unroll 1
  for (int r0 = 0; r0 < NQ; r0 += U) {
    uint4 f[U][3];
    float4 a[U];
    bool on[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int qd = threadIdx.x + (r0 + u) * NTW, i = qd / (T / 4), j = qd % (T / 4) * 4;
      uint4* f0 = reinterpret_cast<uint4*>(F0 + word_at<T>(i, j));
      f[u][0] = f0[0];
      f[u][1] = f0[TT / 4];
      f[u][2] = f0[2 * TT / 4];
      uint32_t any = 0;
#pragma unroll
      for (int l = 0; l < 3; l++) any |= f[u][l].x | f[u][l].y | f[u][l].z | f[u][l].w;
      on[u] = any != 0u && i < g.th;
      if (any) {
        f0[0] = f0[TT / 4] = f0[2 * TT / 4] = make_uint4(0, 0, 0, 0);
      }
      if (on[u] && vec) a[u] = *reinterpret_cast<const float4*>(A0 + i * d.ldA + j);
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      if (!on[u]) continue;
      const int qd = threadIdx.x + (r0 + u) * NTW, i = qd / (T / 4), j = qd % (T / 4) * 4;
      float* dst = A0 + i * d.ldA + j;
      const uint32_t w0[4] = {f[u][0].x, f[u][0].y, f[u][0].z, f[u][0].w};
      const uint32_t w1[4] = {f[u][1].x, f[u][1].y, f[u][1].z, f[u][1].w};
      const uint32_t w2[4] = {f[u][2].x, f[u][2].y, f[u][2].z, f[u][2].w};
      float av[4] = {a[u].x, a[u].y, a[u].z, a[u].w};
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const fx96 v = fx_join<T>(w0[k], w1[k], w2[k]);
        const bool any = (v.w0 | v.w1 | v.w2) != 0u;
        if (any && (vec || j + k < g.tw)) {
          const float was = vec ? av[k] : dst[k];
          const ff r = ff_add(ff{was, 0.0f}, fx96_to_ff(v.w0, v.w1, v.w2, p1, p2));
          av[k] = __fadd_rn(r.hi, r.lo);
          if (!vec) dst[k] = av[k];
        }
      }
      if (vec) *reinterpret_cast<float4*>(dst) = make_float4(av[0], av[1], av[2], av[3]);
    }
  }
}

template <int T>
__global__ void __launch_bounds__(NTW, T >= 128 ? 1 : (T >= 64 ? 4 : 8)) k_fin_area(DemTable dt, Pipe p) {
  using L = LayoutW<T>;
  using AH = Ahead<T, NTW, ff>;
  constexpr int TT = T * T, S = L::S, NS = AH::NS;
  extern __shared__ __align__(16) unsigned char sm[];
  uint32_t* F0 = reinterpret_cast<uint32_t*>(sm + L::off_w);  // words 0, 1, 2 at F0, F0 + TT, F0 + 2 TT
  uint8_t* code = sm + L::off_code;
  uint16_t* rcell = reinterpret_cast<uint16_t*>(sm + L::off_rcell);
  ff* rin = reinterpret_cast<ff*>(sm + L::off_rin);
  // receivers, largest exponent bound + 1024, non-finite seen, next tile; the sum of bounds
  uint32_t* misc = reinterpret_cast<uint32_t*>(sm + L::off_misc);
  unsigned long long* sum = reinterpret_cast<unsigned long long*>(misc + 4);

  for (int q = threadIdx.x; q < 3 * TT / 4; q += NTW) reinterpret_cast<uint4*>(F0)[q] = make_uint4(0, 0, 0, 0);
  // |x| < 2^ebound(x) for finite x (subnormals and zero: 2^-126)
  auto ebound = [](float x) -> int {
    const int eb = (int)((__float_as_uint(x) >> 23) & 0xFFu);
    return eb == 0 ? -126 : eb - 126;
  };
  AH ahead;
  int64_t t = blockIdx.x;
  for (int64_t next; t < p.ntiles; t = next) {
    const DemDesc d = dem_of(dt, t);
    const TileGeo g = tile_geo(d, t - d.tile_base, T);
    __syncthreads();  // everyone is done with the tile before
    ahead.load(p, d, g, t, code);
    if (threadIdx.x == 0) {
      misc[0] = misc[1] = misc[2] = 0u;
      *sum = 0ull;
      misc[3] = gridDim.x + atomicAdd(p.queue + 1, 1u);
    }
    ahead.finish(d, g, code);
    __syncthreads();
    next = misc[3];
    // Algorithm 7: the receivers listed; codes that leave the tile end the walk
#pragma unroll
    for (int r = 0; r < NS; r++) {
      int i, j;
      const int s = threadIdx.x + r * NTW;
      if (s >= 4 * T || !slot_cell(s, g.th, g.tw, T, i, j)) continue;
      const uint32_t k = code[i * S + j];
      const int ti = i + code_di(k & 7), tj = j + code_dj(k & 7);
      if (k < 8u && ((unsigned)ti >= (unsigned)g.th || (unsigned)tj >= (unsigned)g.tw)) code[i * S + j] = 8;
      const ff in = normalised(ahead.in[r]);
      if (in.hi == 0.0f && in.lo == 0.0f) continue;
      const uint32_t at = atomicAdd(&misc[0], 1u);
      rcell[at] = (uint16_t)(i * S + j);
      rin[at] = in;
      if (isfinite(in.hi)) {
        atomicMax(&misc[1], (uint32_t)(1024 + ebound(in.hi)));
      } else {
        misc[2] = 1u;
      }
    }
    __syncthreads();
    const int nrec = (int)misc[0];
    if (misc[2]) {  // an infinite or NaN inflow
      if (threadIdx.x == 0) set_status(p.status, D8_ERR_NONFINITE);
      continue;
    }
    if (nrec == 0) continue;  // no inflow: A is final
    // S = sum of 2^(e_r - emax + 40), each term rounded up to at least 1
    const int emax = (int)misc[1] - 1024;
    for (int r = threadIdx.x; r < nrec; r += NTW) {
      const int sh = ebound(rin[r].hi) - emax + 40;
      atomicAdd(sum, sh <= 0 ? 1ull : 1ull << sh);
    }
    __syncthreads();
    // sum |in_r| < S * 2^(emax - 40) <= 2^(ceil(log2 S) + emax - 40)
    const int q = FxLimbs<T>::VB - 2 - (64 - __clzll(*sum - 1ull)) - (emax - 40);
    // 2^-q as two powers of two of the normal range (|q| <= 250: -126 <= emax <= 128)
    const float p1 = pow2f(-q / 2), p2 = pow2f(-q - (-q / 2));
    // Algorithm 8 on the receivers' paths, in fixed point
    add_inflow<T>(code, F0, rcell, rin, nrec, q);
    __syncthreads();
    add_to_areas<T>(d, g, F0, p1, p2);
  }
}

template <class K>
static cudaError_t launch_k(K k, int threads, size_t bytes, const DemTable& dt, const Pipe& p, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 1, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, bytes) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  const int64_t grid = min64((int64_t)per_sm * sms, p.ntiles);
  k<<<(unsigned)(grid < 1 ? 1 : grid), threads, bytes, s>>>(dt, p);
  return cudaGetLastError();
}

template <int T>
static cudaError_t launch_t(const DemTable& dt, const Pipe& p, bool weighted, cudaStream_t s) {
  if (weighted) return launch_k(k_fin_area<T>, NTW, LayoutW<T>::bytes, dt, p, s);
  return narrow_grid(dt, T) ? launch_k(k_fin_count<T, true>, NTN, Layout<T>::bytes, dt, p, s)
                            : launch_k(k_fin_count<T, false>, NTN, Layout<T>::bytes, dt, p, s);
}

}  // namespace fin

cudaError_t launch_down_recv(const DemTable& dt, const Pipe& p, bool weighted, cudaStream_t s) {
  switch (p.T) {
    case 32: return fin::launch_t<32>(dt, p, weighted, s);
    case 64: return fin::launch_t<64>(dt, p, weighted, s);
    case 128: return fin::launch_t<128>(dt, p, weighted, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace d8
