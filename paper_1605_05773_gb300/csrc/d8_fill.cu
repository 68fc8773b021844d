// d8_fill.cu -- pit and flat removal by epsilon filling on the GPU (the
// method's precondition, "The Algorithm", first paragraph: pits raised and
// flats resolved so that every interior cell drains).
//
// The filled surface F is the unique array with F = z on the grid's edge and,
// for every interior cell c with m = the lowest of its 8 neighbouring F,
//     F(c) = z(c) if z(c) > m,   else   F(c) = up(m) = max(fl32(m + eps), next fp32 above m).
// The update G(F)(c) = (z(c) > m ? z(c) : up(m)) is monotone in F and every
// fixed point is the same array, so iterating it from any start above F
// converges to F exactly, whatever the order in which cells are updated:
// starting from +inf inside, every value only ever decreases, and reading a
// neighbour's older (higher) value can only delay, never spoil, the result.
//
// GPU layout: 64 x 64 tiles.  A round visits the tiles listed for it: a block
// of 64 threads loads the tile's z and the current F of the tile, each with a
// one-cell halo, into shared memory and relaxes the tile to a fixed point of
// that halo in directional passes (thread r walks row r left to right, then
// right to left, then column r down and up; a pass carries a change across
// the whole tile).  Every pass evaluates every cell, so the first pass that
// changes nothing ends the visit.  Then the tile is written back, and a
// neighbouring tile is listed for the next round if one of its cells beside
// this tile would drop under this tile's new border.  A round that lists
// nothing ends the fill: every tile is then at a fixed point of its final
// halo, so F is the global fixed point.
//
// Measured: 8192 x 8192 raw fractal 6.7 ms, 700 x 933 0.47 ms (before: 105 and
// 4.7 ms, 256 threads per tile with two waves over dirty cells, then sweeps of
// four passes each until a whole sweep changed nothing; its lanes down a row
// shared banks, and every change of a tile's border listed all eight
// neighbours).
#include <cmath>
#include <cstdio>

#include "d8_device.cuh"

namespace d8 {
namespace fill {

constexpr int T = 64;
constexpr int NTF = T;                  // one thread per row, or column, of the tile
constexpr int HW = T + 2;               // rows and columns of a tile with its halo
constexpr int RS = T + 3;               // row stride of those arrays: odd, so lanes down a column hit distinct banks
constexpr int MAX_PASSES = 16 * T;      // passes before a visit gives up and lists its own tile again
constexpr unsigned FULL = 0xFFFFFFFFu;

struct Layout {
  static constexpr size_t off_f = 0;                                          // float [HW][RS]: F with halo
  static constexpr size_t off_z = ((size_t)HW * RS * 4 + 15) / 16 * 16;       // float [HW][RS]: z with halo
  static constexpr size_t off_misc = off_z + ((size_t)HW * RS * 4 + 15) / 16 * 16;
  static constexpr size_t bytes = off_misc + 16;
};

// max(fl32(m + eps), next fp32 above m) for finite m, with eps at least the
// smallest positive fp32.  |m| (2^-24 + 2^-44) is more than half and less than
// one and a half of the distance to the next value, so one fused add of it
// rounds to that value; where it is too small (|m| below 2^-125) eps reaches
// the next value.  (Checked against nextafterf for every finite m.)
__device__ __forceinline__ float up(float m, float eps) {
  return fmaxf(__fadd_rn(m, eps), __fmaf_rn(fabsf(m), 0x1.00001p-24f, m));
}

__device__ __forceinline__ float relaxed(float zc, float m, float eps) { return zc > m ? zc : up(m, eps); }

__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// F = z on the grid's edge, +inf inside; non-finite z reported; the tiles on
// the grid's border listed for the first round (no cell of another tile can
// drop before one of them has: those start at +inf with +inf around)
__global__ void k_fill_init(const float* z, int64_t H, int64_t W, int64_t ldz, float* F, int64_t ldF, int64_t ntx,
                            int64_t nty, uint32_t* list, uint32_t* count, uint32_t* status) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x, t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool bad = false;
  for (int64_t c = t0; c < H * W; c += stride) {
    const int64_t i = c / W, j = c - i * W;
    const float zc = z[i * ldz + j];
    bad |= !isfinite(zc);
    const bool edge = i == 0 || j == 0 || i == H - 1 || j == W - 1;
    F[i * ldF + j] = edge ? zc : INFINITY;
  }
  for (int64_t t = t0; t < ntx * nty; t += stride) {
    const int64_t ty = t / ntx, tx = t - ty * ntx;
    if (ty == 0 || tx == 0 || ty == nty - 1 || tx == ntx - 1) list[atomicAdd(count, 1u)] = (uint32_t)t;
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) set_status(status, D8_ERR_NONFINITE);
}

// One directional pass: this thread relaxes the T cells at f, f + DS, ...,
// its neighbours in the block the lines at f - DL and f + DL, all in step.
// Cell q's three neighbours behind (q - 1) carry this pass's values: the own
// line's from a register, the adjacent lines' by shuffles.  At a warp's first
// and last lane a shuffle returns the own line's value, so the values read of
// the adjacent lines two steps earlier enter the minimum for every lane: they
// are older, so never lower, than the shuffled ones, and the pass that
// changes nothing has no older values.  The loads of step q + 1's column are
// issued before step q's store.  The chain per step is shuffle, minimum,
// raise, select, minimum: about 50 cycles; the strides are compile-time
// constants so that a step is about 20 instructions.
template <int DS, int DL>
__device__ __forceinline__ bool relax_pass(float* f, const float* zc, float eps) {
  float su = f[-DS - DL], l = f[-DS], sd = f[-DS + DL];
  float cu = f[-DL], c = f[0], cd = f[DL];
  float ru = f[DS - DL], r = f[DS], rd = f[DS + DL];
  float zq = zc[0];
  float behind = fminf(su, sd);  // the adjacent lines' q - 1, as read
  bool changed = false;
#pragma unroll 8
  for (int q = 0; q < T; q++) {
    float nu = 0.0f, n = 0.0f, nd = 0.0f, zn = 0.0f;
    if (q < T - 1) {
      nu = f[2 * DS - DL];
      n = f[2 * DS];
      nd = f[2 * DS + DL];
      zn = zc[DS];
    }
    const float beside = fminf(cu, cd);
    const float known = fminf(l, min3(min3(ru, r, rd), beside, behind));
    const float v = relaxed(zq, min3(su, sd, known), eps);
    changed |= v < c;
    c = fminf(v, c);
    f[0] = c;
    su = __shfl_up_sync(FULL, c, 1);
    sd = __shfl_down_sync(FULL, c, 1);
    l = c;
    behind = beside;
    cu = ru;
    c = r;
    cd = rd;
    ru = nu;
    r = n;
    rd = nd;
    zq = zn;
    f += DS;
    zc += DS;
  }
  return changed;
}

// pass k: line tid left to right, right to left, then down, up
__device__ __forceinline__ bool relax_dir(int k, float* Fh, const float* zh, float eps) {
  const int p = threadIdx.x + 1, row = p * RS, a = row + 1, b = row + T, c = RS + p, d = T * RS + p;
  switch (k & 3) {
    case 0: return relax_pass<1, RS>(Fh + a, zh + a, eps);
    case 1: return relax_pass<-1, RS>(Fh + b, zh + b, eps);
    case 2: return relax_pass<RS, 1>(Fh + c, zh + c, eps);
    default: return relax_pass<-RS, 1>(Fh + d, zh + d, eps);
  }
}

// One round over the listed tiles.  list / count: this round's tiles;
// next / next_count: the tiles listed for the next round, each once
// (mark[t] = stamp once t is listed).
__global__ void __launch_bounds__(NTF) k_fill_round(const float* z, int64_t H, int64_t W, int64_t ldz, float* F,
                                                    int64_t ldF, float eps, int64_t ntx, int64_t nty,
                                                    const uint32_t* list, const uint32_t* count, uint32_t* next,
                                                    uint32_t* next_count, uint32_t* queue, uint32_t* mark,
                                                    uint32_t stamp) {
  extern __shared__ __align__(16) unsigned char sm[];
  float* Fh = reinterpret_cast<float*>(sm + Layout::off_f);
  float* zh = reinterpret_cast<float*>(sm + Layout::off_z);
  uint32_t* dirs = reinterpret_cast<uint32_t*>(sm + Layout::off_misc);  // neighbours to list, one bit each
  const int tid = threadIdx.x;
  const int64_t n = *count;
  TileQueue tq(queue, n);
  for (int64_t at = tq.first(); at < n; at = tq.next()) {
    const int64_t t = list[at];
    const int64_t ty = t / ntx, tx = t - ty * ntx, i0 = ty * T, j0 = tx * T;
    const int th = (int)min64(T, H - i0), tw = (int)min64(T, W - j0);
    if (tid == 0) *dirs = 0u;
    // F and z with the halo; F is +inf off the grid.  z is +inf for every
    // cell that never changes (off the grid, or on its edge, where F = z
    // already), so that no relaxation lowers it.
    auto load = [&](int hi, int hj) {
      const int64_t gi = i0 + hi - 1, gj = j0 + hj - 1;
      float *fd = Fh + hi * RS + hj, *zd = zh + hi * RS + hj;
      if (gi >= 0 && gj >= 0 && gi < H && gj < W)
        cp_async4(fd, F + gi * ldF + gj, 4);
      else
        *fd = INFINITY;
      if (gi > 0 && gj > 0 && gi < H - 1 && gj < W - 1)
        cp_async4(zd, z + gi * ldz + gj, 4);
      else
        *zd = INFINITY;
    };
    for (int hi = 0; hi < HW; hi++) load(hi, tid + 1);
    for (int q = tid; q < 2 * HW; q += NTF) load(q >> 1, (q & 1) * (HW - 1));
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    bool any = false, settled = false;
    for (int k = 0; k < MAX_PASSES; k++) {
      if (!__syncthreads_or(relax_dir(k, Fh, zh, eps))) {
        settled = true;
        break;
      }
      any = true;
    }
    if (any) {
      if (tid < tw)
#pragma unroll 8
        for (int i = 0; i < th; i++) F[(i0 + i) * ldF + (j0 + tid)] = Fh[(i + 1) * RS + tid + 1];
      // halo cells that would drop under the new border: their tiles go on
      // the next round's list (their F here may be older, so higher, than
      // their tile's own: then the tile may be listed for nothing)
      for (int q = tid; q < 4 * (HW - 1); q += NTF) {
        const int side = q / (HW - 1), p = q % (HW - 1);
        const int hi = side == 0 ? 0 : side == 1 ? HW - 1 : side == 2 ? p + 1 : p;
        const int hj = side == 0 ? p : side == 1 ? p + 1 : side == 2 ? 0 : HW - 1;
        float m = INFINITY;
#pragma unroll
        for (int k = 0; k < 8; k++) {
          const int a = hi + code_di(k), b = hj + code_dj(k);
          if (a >= 1 && b >= 1 && a <= T && b <= T) m = fminf(m, Fh[a * RS + b]);
        }
        if (relaxed(zh[hi * RS + hj], m, eps) < Fh[hi * RS + hj]) {
          const int di = hi == 0 ? 0 : hi == HW - 1 ? 2 : 1, dj = hj == 0 ? 0 : hj == HW - 1 ? 2 : 1;
          atomicOr(dirs, 1u << (3 * di + dj));
        }
      }
      __syncthreads();
    }
    if (tid < 9 && (tid == 4 ? !settled : (any && ((*dirs >> tid) & 1u)))) {
      const int64_t nt = (ty + tid / 3 - 1) * ntx + (tx + tid % 3 - 1);
      if (atomicExch(&mark[nt], stamp) != stamp) next[atomicAdd(next_count, 1u)] = (uint32_t)nt;
    }
  }
}

}  // namespace fill

constexpr int CHUNK = 16;  // rounds between host checks

// workspace: counts of listed tiles (CHUNK + 1) and work queues (CHUNK), one
// mark and two list entries per tile
size_t fill_ws_bytes(int64_t H, int64_t W) {
  const int64_t ntiles = ((H + fill::T - 1) / fill::T) * ((W + fill::T - 1) / fill::T);
  return 256 + sizeof(uint32_t) * 3 * (size_t)ntiles;
}

// The fill: init, then rounds until one lists nothing.  The host reads the
// rounds' list counts every CHUNK rounds (synchronising the stream) and stops
// after max_rounds with D8_ERR_TIMEOUT.
cudaError_t run_fill(const float* z, int64_t H, int64_t W, int64_t ldz, float eps, float* F, int64_t ldF, void* ws,
                     uint32_t* status, cudaStream_t s, int64_t max_rounds, int64_t* rounds_out, bool* timed_out,
                     int* nlaunch) {
  using namespace fill;
  const int64_t ntx = (W + T - 1) / T, nty = (H + T - 1) / T, ntiles = ntx * nty;
  static_assert(sizeof(uint32_t) * (2 * CHUNK + 1) <= 256, "counts and queues fit the workspace's head");
  uint32_t* counts = static_cast<uint32_t*>(ws);  // counts[k]: tiles listed for round k of the chunk
  uint32_t* queues = counts + CHUNK + 1;
  uint32_t* mark = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + 256);
  uint32_t* list[2] = {mark + ntiles, mark + 2 * ntiles};
  *timed_out = false;
  eps = fmaxf(eps, 0x1p-149f);  // see up()
  int dev = 0, sms = 1, per_sm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e = cudaFuncSetAttribute(k_fill_round, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Layout::bytes);
  if (e != cudaSuccess) return e;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fill_round, NTF, Layout::bytes) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  int64_t grid = (int64_t)per_sm * sms;
  if (grid > ntiles) grid = ntiles;
  e = cudaMemsetAsync(ws, 0, 256 + sizeof(uint32_t) * (size_t)ntiles, s);
  if (e != cudaSuccess) return e;
  int64_t nb = (H * W + 255) / 256;
  if (nb > (int64_t)sms * 16) nb = (int64_t)sms * 16;
  k_fill_init<<<(unsigned)(nb < 1 ? 1 : nb), 256, 0, s>>>(z, H, W, ldz, F, ldF, ntx, nty, list[0], counts, status);
  ++*nlaunch;
  int64_t r = 0;
  for (;;) {
    for (int k = 0; k < CHUNK; k++, r++) {
      k_fill_round<<<(unsigned)grid, NTF, Layout::bytes, s>>>(z, H, W, ldz, F, ldF, eps, ntx, nty, list[r & 1],
                                                              counts + k, list[(r + 1) & 1], counts + k + 1,
                                                              queues + k, mark, (uint32_t)(r + 1));
      ++*nlaunch;
    }
    uint32_t h[CHUNK + 1];
    e = cudaMemcpyAsync(h, counts, sizeof(h), cudaMemcpyDeviceToHost, s);
    // the last count is the next chunk's first
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(counts, counts + CHUNK, sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(counts + 1, 0, sizeof(uint32_t) * 2 * CHUNK, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    for (int k = 1; k <= CHUNK; k++) {
      if (h[k] == 0) {  // the first round that listed nothing
        *rounds_out = r - CHUNK + k;
        return cudaGetLastError();
      }
    }
    if (r >= max_rounds) {
      *rounds_out = r;
      *timed_out = true;
      return cudaGetLastError();
    }
  }
}

}  // namespace d8
