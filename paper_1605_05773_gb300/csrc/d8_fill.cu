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
// loads the tile's z and the current F of the tile, each with a
// one-cell halo, into shared memory and relaxes the tile to a fixed point of
// that halo in directional passes (thread r walks row r left to right, then
// right to left, then column r down and up; a pass carries a change across
// the whole tile).  Every pass evaluates every cell, so a pass that changes
// nothing ends the visit; so does the fourth, and the tile is then listed for
// the next round itself.  (A change has crossed the tile by then: going on to
// the fixed point, 10 to 12 passes, makes the neighbours wait for work that
// their own changes undo again.)  Then the tile is written back, and a
// neighbouring tile is listed for the next round if one of its cells beside
// this tile would drop under this tile's new border.  A round that lists
// nothing ends the fill: every tile is then at a fixed point of its final
// halo, so F is the global fixed point.
// A visit is a chain of latencies, 64 steps a pass; the other threads of its
// block only share in loading, storing and looking at the border, whose loops
// would add half of the passes' time (64 threads: 8192 x 8192 5.14 ms, 700 x
// 933 358 us; 128: 4.71 and 314; 256: 4.58 and 293).
//
// Start from above: the fixed point is reached from any start that is nowhere
// below it, and the nearer the start, the fewer visits.  So the fill is first
// bounded on coarser grids, side ratio 4 (k_fill_pool, then the same rounds).
// A coarse cell is a block B of n x n cells with Z(B) its highest z, and its
// value bounds F over the block: the block's cells can be reached from any
// cell of an adjacent block in at most n steps inside B, each raising by one
// up() and to no more than Z(B), so with X = max(Z(B), lowest adjacent value)
//     max of F over B <= up^n(X) <= X + |X| b + a        (BlockBound below),
// and blocks holding cells of the grid's edge keep the bound with X = Z(B).
// Every state of that iteration from +inf bounds F, settled or not, so the
// coarse grids get one round each and no host check; each level starts from
// the bounds of the level above it.
//
// Measured, 8192 x 8192 raw fractals, 8192 x 8192 noisy plane, 700 x 933 fractals:
// 3.1 to 5.2 (by the field), 0.90 and 0.19 to 0.30 ms.  One set of fields, 4.4,
// 0.93 and 0.25 ms, took with more rounds on the coarse grids 4.6, 1.02 and
// 0.29; in blocks of 64 threads too 5.1, 1.09 and 0.36 (at most 3 passes a visit
// 5.5 ms and 0.45 for the fractals, 5 passes 5.5 and 0.37); visits to the fixed
// point 5.9, 1.12 and 0.40; without the coarse grids 6.5, 3.2 and 0.45 (the
// fractal's lakes, thousands of cells wide, still fill one tile a round);
// before (two waves over dirty cells, then sweeps of four passes until a whole
// sweep changed nothing; lanes down a row shared banks, and every change of a
// tile's border listed all eight neighbours) the fractals took 105 and 4.7 ms.
// One channel that winds through every tile, behind a dam, 1024 x 1024: 157 ms (3.8
// s), 7900 rounds.
#include <cmath>
#include <type_traits>

#include "d8_device.cuh"

namespace d8 {
namespace fill {

constexpr int T = 64;
constexpr int RATIO = 4;                // side ratio of a level to the next finer one
constexpr int NTF = 256;                // threads per tile; the first T take a row, or a column, each
constexpr int LINES = NTF / T;          // rows moved at once
constexpr int HW = T + 2;               // rows and columns of a tile with its halo
constexpr int RS = T + 3;               // row stride of those arrays: odd, so lanes down a column hit distinct banks
constexpr int MAX_PASSES = 4;           // passes before a visit ends and lists its own tile again
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

// The value a cell of elevation zc takes above its lowest neighbour m: on the
// grid itself, and on a grid of blocks of n x n cells (a bound, see above).
struct CellRaise {
  float eps;
  __device__ __forceinline__ float operator()(float zc, float m) const { return zc > m ? zc : up(m, eps); }
};

// up^n(x) <= x + n eps + n ulp(V), V the largest magnitude on the way, at most
// (|x| + n eps)(1 + n 2^-22); ulp(V) <= 2^-23 V + 2^-149.  The factors leave
// twice that and 8 2^-22 (|x| + n eps) more for this evaluation's roundings.
struct BlockBound {
  float a, b;
  BlockBound(float n, float eps) : a(n * eps * 1.001f + (n + 8.0f) * 0x1p-22f * n * eps + 1e-38f), b((n + 8.0f) * 0x1p-22f) {}
  __device__ __forceinline__ float of(float x) const { return __fadd_rn(__fmaf_rn(fabsf(x), b, x), a); }
  __device__ __forceinline__ float operator()(float zc, float m) const { return of(fmaxf(zc, m)); }
};

__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// A level's start: its edge at z (blocks: at their bound), the inside at the
// bounds of the next coarser level, or +inf without one; its tiles listed for
// the first round, only those on its border when the inside is at +inf (no
// other cell can drop before one of them has).  check: report non-finite z.
template <class Raise>
__global__ void k_fill_init(const float* z, int64_t H, int64_t W, int64_t ldz, float* F, int64_t ldF, Raise raise,
                            const float* coarse, int64_t cW, int64_t ntx, int64_t nty, uint32_t* list,
                            uint32_t* count, bool check, uint32_t* status) {
  const int64_t stride = (int64_t)gridDim.x * gridDim.y * blockDim.x;
  const int64_t t0 = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x;
  bool bad = false;
  // RATIO cells of a row per thread: they share one coarser cell
  const int64_t j0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * RATIO;
  const bool vec = (reinterpret_cast<uintptr_t>(F) & 15u) == 0 && ldF % RATIO == 0 && j0 + RATIO <= W;
  for (int64_t i = blockIdx.y; i < H && j0 < W; i += gridDim.y) {
    const float inside = coarse ? __ldg(&coarse[(i / RATIO) * cW + j0 / RATIO]) : INFINITY;
    const bool row_edge = i == 0 || i == H - 1;
    float v[RATIO];
#pragma unroll
    for (int k = 0; k < RATIO; k++) {
      const int64_t j = j0 + k;
      const bool edge = row_edge || j == 0 || j == W - 1;
      v[k] = inside;
      if (j < W && (edge || check)) {
        const float zc = z[i * ldz + j];
        bad |= check && !isfinite(zc);
        if (edge) v[k] = zc;
        if constexpr (std::is_same<Raise, BlockBound>::value)
          if (edge) v[k] = raise.of(zc);
      }
    }
    float* dst = F + i * ldF + j0;
    if (vec) {
      *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int k = 0; k < RATIO; k++)
        if (j0 + k < W) dst[k] = v[k];
    }
  }
  for (int64_t t = t0; t < ntx * nty; t += stride) {
    const int64_t ty = t / ntx, tx = t - ty * ntx;
    if (coarse)
      list[t] = (uint32_t)t;
    else if (ty == 0 || tx == 0 || ty == nty - 1 || tx == ntx - 1)
      list[atomicAdd(count, 1u)] = (uint32_t)t;
  }
  if (coarse && t0 == 0) *count = (uint32_t)(ntx * nty);
  if (__syncthreads_or(bad) && threadIdx.x == 0) set_status(status, D8_ERR_NONFINITE);
}

// highest z of each RATIO x RATIO block (vec: rows of z are 16-byte aligned);
// check: report non-finite z
__global__ void k_fill_pool(const float* z, int64_t H, int64_t W, int64_t ldz, float* zc, int64_t cH, int64_t cW,
                            bool vec, bool check, uint32_t* status) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  bool bad = false;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < cH * cW; c += stride) {
    const int64_t bi = c / cW, bj = c - bi * cW;
    const int h = (int)min64(RATIO, H - bi * RATIO), w = (int)min64(RATIO, W - bj * RATIO);
    const float* p = z + bi * RATIO * ldz + bj * RATIO;
    float m = -INFINITY;
    bool fin = true;
#pragma unroll
    for (int i = 0; i < RATIO; i++) {
      if (i >= h) break;
      if (vec && w == RATIO) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p + i * ldz));
        m = fmaxf(m, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
        fin &= isfinite(v.x) && isfinite(v.y) && isfinite(v.z) && isfinite(v.w);
      } else {
        for (int j = 0; j < w; j++) {
          const float v = __ldg(p + i * ldz + j);
          m = fmaxf(m, v);
          fin &= isfinite(v);
        }
      }
    }
    zc[c] = m;
    bad |= check && !fin;
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
template <int DS, int DL, class Raise>
__device__ __forceinline__ bool relax_pass(float* f, const float* zc, Raise raise) {
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
    const float v = raise(zq, min3(su, sd, known));
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
template <class Raise>
__device__ __forceinline__ bool relax_dir(int k, float* Fh, const float* zh, Raise raise) {
  const int p = threadIdx.x + 1, row = p * RS, a = row + 1, b = row + T, c = RS + p, d = T * RS + p;
  switch (k & 3) {
    case 0: return relax_pass<1, RS>(Fh + a, zh + a, raise);
    case 1: return relax_pass<-1, RS>(Fh + b, zh + b, raise);
    case 2: return relax_pass<RS, 1>(Fh + c, zh + c, raise);
    default: return relax_pass<-RS, 1>(Fh + d, zh + d, raise);
  }
}

// One round over the listed tiles.  list / count: this round's tiles;
// next / next_count: the tiles listed for the next round, each once
// (mark[t] = stamp once t is listed).
template <class Raise>
__global__ void __launch_bounds__(NTF) k_fill_round(const float* z, int64_t H, int64_t W, int64_t ldz, float* F,
                                                    int64_t ldF, Raise raise, int64_t ntx, int64_t nty,
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
    for (int hi = tid / T; hi < HW; hi += LINES) load(hi, tid % T + 1);
    for (int q = tid; q < 2 * HW; q += NTF) load(q >> 1, (q & 1) * (HW - 1));
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    bool any = false, settled = false;
    for (int k = 0; k < MAX_PASSES; k++) {
      if (!__syncthreads_or(tid < T && relax_dir(k, Fh, zh, raise))) {
        settled = true;
        break;
      }
      any = true;
    }
    if (any) {
      if (tid % T < tw)
#pragma unroll 8
        for (int i = tid / T; i < th; i += LINES) F[(i0 + i) * ldF + (j0 + tid % T)] = Fh[(i + 1) * RS + tid % T + 1];
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
        if (raise(zh[hi * RS + hj], m) < Fh[hi * RS + hj]) {
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

namespace fill {

constexpr int CHUNK = 8;      // rounds between host checks
constexpr int MAX_LEVELS = 8;
constexpr size_t HEAD = 256;  // bytes of a level's counts (CHUNK + 1) and work queues (CHUNK)
static_assert(RATIO == 4, "k_fill_init and k_fill_pool move blocks' rows as float4");
static_assert(sizeof(uint32_t) * (2 * CHUNK + 1) <= HEAD, "counts and queues fit the head");

// A level's grid and its part of the workspace.  Level 0 is the grid itself.
struct Level {
  int64_t H, W, ntx, nty, ntiles;
  const float* z;
  int64_t ldz;
  float* F;
  int64_t ldF;
  uint32_t* counts;  // counts[k]: tiles listed for round k of the chunk
  uint32_t* queues;
  uint32_t* mark;
  uint32_t* list[2];
};

static size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

// Levels are added while the last one has more than one tile, for grids of
// more than 8 tiles a side: smaller ones settle in about as many rounds as the
// coarse grids would take (two fractals each, with and without levels: 500 x 500
// 174 and 186 us, 151 and 219; 600 x 600 188 and 192, 227 and 249; 700 x 933 204 and
// 192, 269 and 263; 3000 x 3000 629 and 1410, 925 and 1345; 8192 x 8192 3.06 and 5.19
// ms, 3.92 and 4.90).  Returns their number; bytes: the workspace.
// What must be zero at the start comes first, `zeroed` bytes of it.
static int levels(int64_t H, int64_t W, bool coarse, void* ws, Level* lv, size_t* zeroed, size_t* bytes) {
  int n = 0;
  size_t at = 0;
  char* base = static_cast<char*>(ws);
  for (;;) {
    Level& L = lv[n++];
    L = Level{};
    L.H = H;
    L.W = W;
    L.ntx = (W + T - 1) / T;
    L.nty = (H + T - 1) / T;
    L.ntiles = L.ntx * L.nty;
    L.counts = reinterpret_cast<uint32_t*>(base + at);
    L.queues = L.counts + CHUNK + 1;
    L.mark = reinterpret_cast<uint32_t*>(base + at + HEAD);
    at += HEAD + a256(sizeof(uint32_t) * (size_t)L.ntiles);
    if (!coarse || n == MAX_LEVELS || L.ntiles == 1 || (n == 1 && min64(L.ntx, L.nty) <= 8)) break;
    H = (H + RATIO - 1) / RATIO;
    W = (W + RATIO - 1) / RATIO;
  }
  *zeroed = at;
  for (int l = 0; l < n; l++) {
    Level& L = lv[l];
    for (auto& q : L.list) {
      q = reinterpret_cast<uint32_t*>(base + at);
      at += a256(sizeof(uint32_t) * (size_t)L.ntiles);
    }
    if (l == 0) continue;
    const size_t cells = a256(sizeof(float) * (size_t)L.H * (size_t)L.W);
    L.z = reinterpret_cast<const float*>(base + at);
    L.F = reinterpret_cast<float*>(base + at + cells);
    L.ldz = L.ldF = L.W;
    at += 2 * cells;
  }
  *bytes = at;
  return n;
}

static unsigned blocks_for(int64_t n, int sms) {
  int64_t b = (n + 255) / 256;
  if (b > (int64_t)sms * 16) b = (int64_t)sms * 16;
  return (unsigned)(b < 1 ? 1 : b);
}

template <class Raise>
static cudaError_t start_level(const Level& L, const Level* coarser, Raise raise, bool check, uint32_t* status, int sms,
                               cudaStream_t s, int* nlaunch) {
  const int64_t gx = (L.W + 256 * RATIO - 1) / (256 * RATIO);  // 256 threads, RATIO cells each, along a row
  int64_t gy = (int64_t)sms * 16 / gx;
  if (gy > L.H) gy = L.H;
  if (gy > 65535) gy = 65535;
  if (gy < 1) gy = 1;
  k_fill_init<Raise><<<dim3((unsigned)gx, (unsigned)gy), 256, 0, s>>>(
      L.z, L.H, L.W, L.ldz, L.F, L.ldF, raise, coarser ? coarser->F : nullptr, coarser ? coarser->W : 0, L.ntx, L.nty,
      L.list[0], L.counts, check, status);
  ++*nlaunch;
  return cudaGetLastError();
}

// rounds first .. first + n - 1 of a level (n <= CHUNK), counts and queues at 0
template <class Raise>
static cudaError_t rounds(const Level& L, Raise raise, int64_t first, int n, int sms, cudaStream_t s, int* nlaunch) {
  int per_sm = 1;
  auto kern = k_fill_round<Raise>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Layout::bytes);
  if (e != cudaSuccess) return e;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NTF, Layout::bytes) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  const int64_t grid = min64((int64_t)per_sm * sms, L.ntiles);
  for (int k = 0; k < n; k++) {
    const int64_t r = first + k;
    kern<<<(unsigned)grid, NTF, Layout::bytes, s>>>(L.z, L.H, L.W, L.ldz, L.F, L.ldF, raise, L.ntx, L.nty,
                                                    L.list[r & 1], L.counts + k, L.list[(r + 1) & 1],
                                                    L.counts + k + 1, L.queues + k, L.mark, (uint32_t)(r + 1));
    ++*nlaunch;
  }
  return cudaGetLastError();
}

}  // namespace fill

size_t fill_ws_bytes(int64_t H, int64_t W, bool coarse) {
  fill::Level lv[fill::MAX_LEVELS];
  size_t zeroed, bytes;
  fill::levels(H, W, coarse, nullptr, lv, &zeroed, &bytes);
  return bytes;
}

// The fill: the coarser levels from the coarsest, then the grid itself in
// rounds until one lists nothing.  The host reads the rounds' list counts
// every CHUNK rounds (synchronising the stream) and stops after max_rounds
// with D8_ERR_TIMEOUT.
cudaError_t run_fill(const float* z, int64_t H, int64_t W, int64_t ldz, float eps, float* F, int64_t ldF, void* ws,
                     bool coarse, uint32_t* status, cudaStream_t s, int64_t max_rounds, int64_t* rounds_out, bool* timed_out,
                     int* nlaunch) {
  using namespace fill;
  Level lv[MAX_LEVELS];
  size_t zeroed, bytes;
  const int n = levels(H, W, coarse, ws, lv, &zeroed, &bytes);
  Level& G = lv[0];
  G.z = z;
  G.ldz = ldz;
  G.F = F;
  G.ldF = ldF;
  eps = fmaxf(eps, 0x1p-149f);  // see up()
  *timed_out = false;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e = cudaMemsetAsync(ws, 0, zeroed, s);
  for (int l = 1; l < n && e == cudaSuccess; l++) {
    const Level &f = lv[l - 1], &c = lv[l];
    const bool vec = (reinterpret_cast<uintptr_t>(f.z) & 15u) == 0 && f.ldz % 4 == 0;
    k_fill_pool<<<blocks_for(c.H * c.W, sms), 256, 0, s>>>(f.z, f.H, f.W, f.ldz, const_cast<float*>(c.z), c.H, c.W, vec,
                                                           l == 1, status);
    ++*nlaunch;
    e = cudaGetLastError();
  }
  for (int l = n - 1; l >= 1 && e == cudaSuccess; l--) {
    const BlockBound bound((float)(1 << (2 * l)), eps);
    e = start_level(lv[l], l + 1 < n ? &lv[l + 1] : nullptr, bound, false, status, sms, s, nlaunch);
    // bounds left higher than they could be only cost the finer level visits,
    // and not as many as more rounds here take (k of them, up to 8, for a
    // level of 2 (k - 3) tiles a side: 8192 x 8192 fractal 4.58 ms, 4.36 with
    // one; noisy plane 1.03 and 0.93; 700 x 933 fractal 308 us and 247; 4096 x
    // 4096 noisy bowl 3.31 ms and 3.15)
    if (e == cudaSuccess) e = rounds(lv[l], bound, 0, 1, sms, s, nlaunch);
  }
  if (e == cudaSuccess) e = start_level(G, n > 1 ? &lv[1] : nullptr, CellRaise{eps}, n == 1, status, sms, s, nlaunch);
  if (e != cudaSuccess) return e;
  int64_t r = 0;
  for (;;) {
    constexpr int m = CHUNK;
    e = rounds(G, CellRaise{eps}, r, m, sms, s, nlaunch);
    r += m;
    uint32_t h[m + 1];
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, G.counts, sizeof(uint32_t) * (m + 1), cudaMemcpyDeviceToHost, s);
    // the last count is the next chunk's first
    if (e == cudaSuccess) e = cudaMemcpyAsync(G.counts, G.counts + m, sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(G.counts + 1, 0, sizeof(uint32_t) * 2 * CHUNK, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    for (int k = 1; k <= m; k++) {
      if (h[k] == 0) {  // the first round that listed nothing
        *rounds_out = r - m + k;
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
