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
// Measured, T = 64: 32768 x 32768 fractal 2.39 ms, 8192 x 8192 160 us (before,
// with the receivers found and their inflow gathered here: 3.06 ms, 203 us);
// 4240 warp instructions per tile (8200), the shared-memory pipe 82 % busy:
// the receivers' paths overlap (65 receivers, 2800 additions to 540 cells).
#include "d8_device.cuh"

namespace d8 {
namespace fin {

constexpr int NTN = 128;  // threads per tile block
constexpr unsigned FULL = 0xFFFFFFFFu;

template <int T>
struct Layout {
  static constexpr size_t TT = (size_t)T * T;
  static constexpr size_t off_f = 0;                         // uint32 per cell: inflow routed through it
  static constexpr size_t off_code = TT * 4;                 // uint8 [2][TT]: codes of this tile and the next
  static constexpr size_t off_rin = off_code + 2 * TT;       // uint32 per receiver: its inflow
  static constexpr size_t off_rcell = off_rin + (size_t)4 * T * 4;  // uint16 per receiver: its cell
  static constexpr size_t off_misc = off_rcell + (size_t)4 * T * 2;
  static constexpr size_t bytes = off_misc + 16;
};

// distance in cells to the neighbour in direction code
template <int T>
__device__ __forceinline__ int step_of(uint32_t code) {
  if (T <= 64) {  // signed bytes N, NE, E, SE / S, SW, W, NW (prmt's selectors k + 8 copy byte k's sign)
    constexpr uint32_t lo = (uint32_t)(-T & 0xFF) | (uint32_t)((1 - T) & 0xFF) << 8 | 1u << 16 | (uint32_t)(T + 1) << 24;
    constexpr uint32_t hi = (uint32_t)T | (uint32_t)(T - 1) << 8 | 0xFFu << 16 | (uint32_t)((-T - 1) & 0xFF) << 24;
    int r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(lo), "r"(hi), "r"(code * 0x1111u + 0x8880u));
    return r;
  }
  return code_di((int)code) * T + code_dj((int)code);
}

// What a tile needs, requested ahead: the inflow of this thread's slots, and
// the codes by asynchronous copies into code[] (waited for by the caller).
template <int T>
struct Ahead {
  static constexpr int NS = 4 * T / NTN;  // slots per thread
  uint32_t in[NS];

  __device__ __forceinline__ void load(const Pipe& p, const DemDesc& d, const TileGeo& g, int64_t t, uint8_t* code) {
    const uint32_t* inflow = static_cast<const uint32_t*>(p.S);
#pragma unroll
    for (int r = 0; r < NS; r++) in[r] = inflow ? __ldg(inflow + t * (4 * T) + threadIdx.x + r * NTN) : 0u;
    const bool vec = g.tw == T && ((reinterpret_cast<uintptr_t>(d.dir) & 15u) == 0) && (d.lddir % 16 == 0);
    for (int q = threadIdx.x; q < T * T / 16; q += NTN) {  // 16 codes at a time
      const int i = q / (T / 16), j = q % (T / 16) * 16;
      if (i >= g.th) break;
      const uint8_t* src = d.dir + (g.i0 + i) * d.lddir + (g.j0 + j);
      uint8_t* dst = code + i * T + j;
      if (vec) {
        cp_async16(dst, src, 16);
      } else {
        uint32_t w[4] = {0x08080808u, 0x08080808u, 0x08080808u, 0x08080808u};
#pragma unroll
        for (int k = 0; k < 16; k++)
          if (j + k < g.tw) w[k / 4] = (w[k / 4] & ~(0xFFu << (8 * (k & 3)))) | (uint32_t)__ldg(src + k) << (8 * (k & 3));
        *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    cp_async_commit();
  }
};

template <int T>
__global__ void __launch_bounds__(NTN) k_fin_count(DemTable dt, Pipe p) {
  using L = Layout<T>;
  constexpr int TT = T * T, NS = Ahead<T>::NS;
  extern __shared__ __align__(16) unsigned char sm[];
  uint32_t* F = reinterpret_cast<uint32_t*>(sm + L::off_f);
  uint32_t* rin = reinterpret_cast<uint32_t*>(sm + L::off_rin);
  uint16_t* rcell = reinterpret_cast<uint16_t*>(sm + L::off_rcell);
  uint32_t* misc = reinterpret_cast<uint32_t*>(sm + L::off_misc);  // receivers (by tile parity), next tile
  const int lane = threadIdx.x & 31;

  // F starts at zero; every tile leaves the words it touched at zero again
  for (int q = threadIdx.x; q < TT / 4; q += NTN) reinterpret_cast<uint4*>(F)[q] = make_uint4(0, 0, 0, 0);
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
    uint8_t* code = sm + L::off_code + buf * TT;
    if (threadIdx.x == 0) misc[2] = gridDim.x + atomicAdd(p.queue + 1, 1u);
    cp_async_wait<0>();
    __syncthreads();  // codes landed; everyone is done with the tile before
    // Algorithm 7: the receivers listed; codes that leave the tile end the walk
#pragma unroll
    for (int r = 0; r < NS; r++) {
      int i, j;
      uint32_t in = ahead.in[r];
      const bool cell = slot_cell(threadIdx.x + r * NTN, g.th, g.tw, T, i, j);
      if (cell) {
        const uint32_t k = code[i * T + j];
        const int ti = i + code_di(k & 7), tj = j + code_dj(k & 7);
        if (k < 8u && ((unsigned)ti >= (unsigned)g.th || (unsigned)tj >= (unsigned)g.tw)) code[i * T + j] = 8;
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
        rcell[at] = (uint16_t)(i * T + j);
        rin[at] = in;
      }
    }
    __syncthreads();
    const int nrec = (int)misc[buf];
    if (threadIdx.x == 0) misc[buf ^ 1] = 0u;
    next = misc[2];
    if (next < p.ntiles) {
      const DemDesc dn = dem_of(dt, next);
      ahead.load(p, dn, tile_geo(dn, next - dn.tile_base, T), next, sm + L::off_code + (buf ^ 1) * TT);
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
    // A += F where F is not zero; those words go back to zero
    constexpr int NQ = TT / 4 / NTN, U = NQ < 4 ? NQ : 4;  // quads per thread, quads read at once
    const bool vec = g.tw == T && ((reinterpret_cast<uintptr_t>(d.A) & 15u) == 0) && (d.ldA & 3) == 0;
    uint32_t* const A0 = static_cast<uint32_t*>(d.A) + g.i0 * d.ldA + g.j0;
#pragma unroll 1
    for (int r0 = 0; r0 < NQ; r0 += U) {
      uint4 f[U], a[U];
      bool on[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        const int q = threadIdx.x + (r0 + u) * NTN, i = q / (T / 4), j = q % (T / 4) * 4;
        f[u] = reinterpret_cast<const uint4*>(F)[q];
        on[u] = (f[u].x | f[u].y | f[u].z | f[u].w) != 0u;
        if (on[u]) {
          reinterpret_cast<uint4*>(F)[q] = make_uint4(0, 0, 0, 0);
          if (vec) a[u] = *reinterpret_cast<const uint4*>(A0 + i * d.ldA + j);
        }
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        if (!on[u]) continue;
        const int q = threadIdx.x + (r0 + u) * NTN, i = q / (T / 4), j = q % (T / 4) * 4;
        uint32_t* dst = A0 + i * d.ldA + j;
        if (vec) {
          *reinterpret_cast<uint4*>(dst) = make_uint4(a[u].x + f[u].x, a[u].y + f[u].y, a[u].z + f[u].z, a[u].w + f[u].w);
        } else {
          if (f[u].x) dst[0] += f[u].x;  // (cells off a ragged tile have none)
          if (f[u].y) dst[1] += f[u].y;
          if (f[u].z) dst[2] += f[u].z;
          if (f[u].w) dst[3] += f[u].w;
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
