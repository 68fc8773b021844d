// d8_final.cu -- the finalise of unit counts (Algorithms 7-8) after the layered
// combine, restricted to where it changes anything.
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
  constexpr int S = Layout<T>::S;
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
template <int T>
struct Ahead {
  static constexpr int S = Layout<T>::S;
  static constexpr int NS = 4 * T / NTN;                     // slots per thread
  static constexpr int Q = T / 4;                            // words per row
  static constexpr int RS = NTN / Q, NQ = T * Q / NTN;       // rows at once, words per thread
  uint32_t in[NS];

  __device__ static __forceinline__ bool whole(const TileGeo& g) { return g.tw == T && g.th == T; }
  __device__ static __forceinline__ bool aligned(const DemDesc& d) {
    return ((reinterpret_cast<uintptr_t>(d.dir) | (uintptr_t)d.lddir) & 3u) == 0;
  }

  __device__ __forceinline__ void load(const Pipe& p, const DemDesc& d, const TileGeo& g, int64_t t, uint8_t* code) {
    const uint32_t* inflow = static_cast<const uint32_t*>(p.S);
#pragma unroll
    for (int r = 0; r < NS; r++) in[r] = inflow ? __ldg(inflow + t * (4 * T) + threadIdx.x + r * NTN) : 0u;
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
#pragma unroll 8
      for (int c = threadIdx.x; c < T * T; c += NTN) {
        const int i = c / T, j = c % T;
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

template <int T>
__global__ void __launch_bounds__(NTN, 8) k_fin_count(DemTable dt, Pipe p) {
  using L = Layout<T>;
  constexpr int TT = T * T, S = L::S, TS = (int)L::TS, NS = Ahead<T>::NS;
  extern __shared__ __align__(16) unsigned char sm[];
  uint32_t* F = reinterpret_cast<uint32_t*>(sm + L::off_f);
  uint32_t* rin = reinterpret_cast<uint32_t*>(sm + L::off_rin);
  uint16_t* rcell = reinterpret_cast<uint16_t*>(sm + L::off_rcell);
  uint32_t* misc = reinterpret_cast<uint32_t*>(sm + L::off_misc);  // receivers (by tile parity), next tile
  const int lane = threadIdx.x & 31;

  // F starts at zero; every tile leaves the words it touched at zero again
  for (int q = threadIdx.x; q < TS / 4; q += NTN) reinterpret_cast<uint4*>(F)[q] = make_uint4(0, 0, 0, 0);
  if (threadIdx.x < 2) misc[threadIdx.x] = 0u;
  Ahead<T> ahead;
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
    if (g.tw == T && ((reinterpret_cast<uintptr_t>(d.A) & 15u) == 0) && (d.ldA & 3) == 0) {
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

template <int T>
static cudaError_t launch_t(const DemTable& dt, const Pipe& p, cudaStream_t s) {
  constexpr size_t bytes = Layout<T>::bytes;
  auto k = k_fin_count<T>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 1, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, NTN, bytes) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  const int64_t grid = min64((int64_t)per_sm * sms, p.ntiles);
  k<<<(unsigned)(grid < 1 ? 1 : grid), NTN, bytes, s>>>(dt, p);
  return cudaGetLastError();
}

}  // namespace fin

cudaError_t launch_down_count(const DemTable& dt, const Pipe& p, cudaStream_t s) {
  switch (p.T) {
    case 32: return fin::launch_t<32>(dt, p, s);
    case 64: return fin::launch_t<64>(dt, p, s);
    case 128: return fin::launch_t<128>(dt, p, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace d8
