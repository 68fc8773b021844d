// d8_flowdir.cu -- the D8 direction stencil ("The Algorithm": steepest slope
// over the eight neighbours, slope = drop / distance between cell centres;
// "Introduction": lowest neighbour) as a streaming kernel.
//
// Reads 4 bytes of z and writes 1 byte of code per cell.  The comparisons and
// selections run at half the rate of the additions, so they, not HBM, bound
// it; the layout below is chosen to need few of them:
//  * a lane owns 4 adjacent columns and walks down its rows; T / 4 lanes make
//    a tile of the pipeline's tiling, so a warp takes 4, 2 or 1 tiles (T = 32,
//    64, 128) and a batch of DEMs maps onto warps through the tile table;
//  * rows go through a ring of PD rows per tile in shared memory by
//    asynchronous copies (16 bytes per lane), PD - 1 rows ahead; loads into
//    registers waited for one another instead (a warp has six scoreboards);
//    a lane reads its four columns and the two beside them;
//  * steepest: the slope towards a neighbour is the exact negation of the
//    neighbour's slope back, so each difference is formed once and serves two
//    cells (E / W, S / N, SE / NW, SW / NE: 7.25 operations per cell, not 12);
//  * the lowest of the eight values comes from four three-input minima, and
//    the code from five comparisons and predicated additions;
//  * whole items inside the grid run a loop without any of the edges' tests
//    (walk_inside); an item at the grid's edge, or one in which a non-finite
//    elevation turned up that the rule does not mask, runs the general one
//    (walk_any).
// Rows that are not 16-byte aligned take 4-byte copies.  Grids
// with few tiles are cut into shorter row segments, so that a small call
// still fills the GPU (launch_t).
//
// Measured (steepest): 32768 x 32768 1.31 ms, 4.1 TB/s (before: 2.90 ms, one
// warp per tile, 2 columns per lane, eight ordered compare-and-selects per
// cell); 8192 x 8192 97 us (195), 3001 x 5003 with masks and a hundredth of it NaN
// 41 us (85), 512 x 512 9 us (27).  41 warp instructions per 32 cells, 79 % issue active,
// half-rate pipe 65 % busy, DRAM 42 %.
#include "d8_device.cuh"

namespace d8 {
namespace fdir {

constexpr int NTF = 128;  // threads per block
constexpr int CPL = 4;    // columns per lane
constexpr int PD = 8;     // rows of the ring
constexpr unsigned FULL = 0xFFFFFFFFu;

__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// x = v where a == b, on the addition pipe: v + nz with nz = -0 is v
__device__ __forceinline__ void set_if_eq(float a, float b, float& x, float v, float nz) {
  asm("{.reg .pred p; setp.eq.f32 p, %1, %2; @p add.f32 %0, %3, %4;}" : "+f"(x) : "f"(a), "f"(b), "f"(v), "f"(nz));
}
__device__ __forceinline__ void set3_if_eq(float a, float b, float& x, float xv, float& y, float yv, float& c, float cv,
                                           float nz) {
  asm("{.reg .pred p; setp.eq.f32 p, %3, %4; @p add.f32 %0, %5, %8; @p add.f32 %1, %6, %8; @p add.f32 %2, %7, %8;}"
      : "+f"(x), "+f"(y), "+f"(c)
      : "f"(a), "f"(b), "f"(xv), "f"(yv), "f"(cv), "f"(nz));
}

// Code (plus `add`, as a float) of the lowest of the eight values, in the
// order N, NE, E, SE, S, SW, W, NW: the first of equal ones, if it is below
// `than`, else SINK.  NaN values are never the lowest and never equal to it.
// The values are grouped 3 + 3 + 2: the first group that holds the minimum,
// then the place in it, is four minima, five comparisons and eight predicated
// additions (nz = -0, unknown to the compiler, which would make them
// selections): comparisons, minima and selections run at half the rate of
// additions and are what bounds the kernel.
__device__ __forceinline__ float lowest_code(float v0, float v1, float v2, float v3, float v4, float v5, float v6,
                                             float v7, float than, float add, float nz) {
  const float g0 = min3(v0, v1, v2), g1 = min3(v3, v4, v5);
  const float m = min3(g0, g1, fminf(v6, v7));
  // first and second value of the group (copies, also as additions); code of its third
  float x = __fadd_rn(v6, nz), y = __fadd_rn(v7, nz), third = add + 8.0f;
  set3_if_eq(g1, m, x, v3, y, v4, third, add + 5.0f, nz);
  set3_if_eq(g0, m, x, v0, y, v1, third, add + 2.0f, nz);
  float code = third;
  set_if_eq(y, m, code, third, -1.0f);
  set_if_eq(x, m, code, third, -2.0f);
  asm("{.reg .pred p; setp.geu.f32 p, %1, %2; @p add.f32 %0, %3, %4;}" : "+f"(code) : "f"(m), "f"(than), "f"(add + 9.0f), "f"(nz));
  return code;
}

// four codes, those of the even columns with 2^23 added, as bytes
__device__ __forceinline__ uint32_t pack_codes(float c0, float c1, float c2, float c3) {
  const float lo = __fmaf_rn(c1, 256.0f, c0), hi = __fmaf_rn(c3, 256.0f, c2);  // exact: below 2^24
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x5410);
}
constexpr float EVEN = 0x1p23f;

// One row as a lane sees it: columns jb - 1 .. jb + 4.
struct Row {
  float v[CPL + 2];
};

// The slopes between a row b and the row c below it, as drops towards the
// lower row are negative: S of each own column; SE of columns -1 .. 3 and SW
// of columns 0 .. 4, each one rounded difference and one rounded product with
// R = fp32(1/sqrt 2).  Negated they are c's N, NW and NE slopes.
struct Slopes {
  float s[CPL], se[CPL + 1], sw[CPL + 1];
};

__device__ __forceinline__ Slopes slopes_between(const Row& b, const Row& c) {
  Slopes o;
#pragma unroll
  for (int k = 0; k < CPL; k++) o.s[k] = __fsub_rn(c.v[k + 1], b.v[k + 1]);
#pragma unroll
  for (int k = 0; k <= CPL; k++) {
    o.se[k] = __fmul_rn(__fsub_rn(c.v[k + 1], b.v[k]), inv_sqrt2_f32());
    o.sw[k] = __fmul_rn(__fsub_rn(c.v[k], b.v[k + 1]), inv_sqrt2_f32());
  }
  return o;
}

// The codes of a lane's four cells in row b, as bytes; a and c the rows above
// and below it, up and dn the slopes between them (a is unused by the
// steepest rule, up and dn by the lowest).
template <bool LOWEST>
__device__ __forceinline__ uint32_t row_codes(const Row& a, const Row& b, const Row& c, const Slopes& up,
                                              const Slopes& dn, float nz) {
  float code[CPL], e[CPL + 1];  // e: E slope of columns -1 .. 3; negated, the W slope of columns 0 .. 4
#pragma unroll
  for (int k = 0; k <= CPL; k++) e[k] = LOWEST ? 0.0f : __fsub_rn(b.v[k + 1], b.v[k]);
#pragma unroll
  for (int k = 0; k < CPL; k++) {
    const float add = k & 1 ? 0.0f : EVEN;
    code[k] = LOWEST ? lowest_code(a.v[k + 1], a.v[k + 2], b.v[k + 2], c.v[k + 2], c.v[k + 1], c.v[k], b.v[k], a.v[k],
                                   b.v[k + 1], add, nz)
                     : lowest_code(-up.s[k], -up.sw[k + 1], e[k + 1], dn.se[k + 1], dn.s[k], dn.sw[k], -e[k],
                                   -up.se[k], 0.0f, add, nz);
  }
  return pack_codes(code[0], code[1], code[2], code[3]);
}

// A lane's part of a work item: rows 0 .. n - 1 of four columns of a tile.
struct Item {
  const float* z;     // row -1, first own column (only formed, not read, when off the grid)
  const float* h;     // row -1, the column beside the tile for its first and last lane, else z
  int64_t ldz, lddir;
  uint8_t* dir;       // row 0, first own column
  int n, ncols;       // rows; own columns present
  bool first, last;   // the tile's first, last lane
  bool hval;          // h's column is on the grid
  bool right;         // the column right of the tile is on the grid
  int qlo, qhi;       // rows q - 1, q in [qlo, qhi), are on the grid (or in the halo of a strip)
  int top, bottom;    // the row that is the grid's first, last; negative if none is
  uint32_t colmask;   // bytes of the columns on the grid's edge
};

__device__ __forceinline__ Row row_of(const Item& it, const float (&x)[CPL], float h) {
  Row r;
#pragma unroll
  for (int k = 0; k < CPL; k++) r.v[k + 1] = x[k];
  const float l = __shfl_up_sync(FULL, x[CPL - 1], 1), e = __shfl_down_sync(FULL, x[0], 1);
  r.v[0] = it.first ? h : l;
  r.v[CPL + 1] = it.last ? h : e;
  return r;
}

// NaN when a value of the row is not finite (the own columns; NODATA: also the
// ones beside), else acc
template <bool NODATA>
__device__ __forceinline__ float nonfinite(const Row& r, float acc) {
#pragma unroll
  for (int k = NODATA ? 0 : 1; k < CPL + (NODATA ? 2 : 1); k++) acc = __fmaf_rn(r.v[k], 0.0f, acc);
  return acc;
}

// asynchronous copies under a predicate (no branch around them)
__device__ __forceinline__ void copy16_if(bool on, float* dst, const float* src) {
  asm volatile("{.reg .pred p; setp.ne.s32 p, %2, 0; @p cp.async.cg.shared.global [%0], [%1], 16;}"
               :: "r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"((int)on) : "memory");
}
__device__ __forceinline__ void copy4_if(bool on, float* dst, const float* src) {
  asm volatile("{.reg .pred p; setp.ne.s32 p, %2, 0; @p cp.async.ca.shared.global [%0], [%1], 4;}"
               :: "r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"((int)on) : "memory");
}

// Under NODATA: OUTLET for the cells of row b that are not finite or lie next to
// a cell that is not.
__device__ __forceinline__ uint32_t mask_nodata(const Row& a, const Row& b, const Row& c, uint32_t packed) {
  float col[CPL + 2];  // NaN for a column with such a cell in the three rows
#pragma unroll
  for (int k = 0; k < CPL + 2; k++) col[k] = __fmaf_rn(a.v[k], 0.0f, __fmaf_rn(b.v[k], 0.0f, __fmul_rn(c.v[k], 0.0f)));
#pragma unroll
  for (int k = 0; k < CPL; k++) {
    const float near = __fadd_rn(__fadd_rn(col[k], col[k + 1]), col[k + 2]);
    if (near != near) packed = (packed & ~(0xFFu << (8 * k))) | (8u << (8 * k));
  }
  return packed;
}

// Items whose rows -1 .. n and own columns all lie on the grid and whose n is
// a multiple of 4.  ring: PD rows of RW floats, columns j0 - 4 .. j0 + T + 3
// of the tile; row k sits at place (k + 7) % 8.  Returns whether the warp met
// a non-finite elevation under a rule without masks (an error: the codes are
// then redone by walk_any).  With masks such rows are masked in place: a raster
// with a border or holes of NaN has whole tiles of them.
template <int T, bool LOWEST, bool NODATA, bool VEC>
__device__ __forceinline__ bool walk_inside(Item it, float* ring, float nz) {
  constexpr int LPT = T / CPL, RW = T + 8;
  static_assert(PD == 8, "places of rows in the ring");
  const int li = (threadIdx.x & 31) & (LPT - 1);
  // this lane's part of a row's copy: its own columns and, for the first and
  // last lane, the one beside the tile; or the columns li, li + LPT, ... of
  // those from j0 - 1 on
  const float* src = VEC ? it.z : it.z - li * CPL - 1 + li;
  const int own = VEC ? CPL + li * CPL : CPL - 1 + li;
  const int beside = it.first ? CPL - 1 : CPL + T;
  const bool lo = li > 0 || it.hval, hi = li == 1 && it.right;  // !VEC: the first and the last column are on the grid
  auto fetch = [&](float* row, bool on) {
    if (VEC) {
      copy16_if(on, row + own, src);
      copy4_if(on && it.hval, row + beside, it.h);
    } else {
      copy4_if(on && lo, row + own, src);
#pragma unroll
      for (int k = 1; k < CPL; k++) copy4_if(on, row + own + k * LPT, src + k * LPT);
      copy4_if(on && (li == 0 || hi), row + own + CPL * LPT, src + CPL * LPT);
    }
    cp_async_commit();
    src += it.ldz;
    it.h += it.ldz;
  };
  const int mine = li * CPL;
  auto take = [&](const float* row) {
    cp_async_wait<PD - 2>();
    __syncwarp();  // every lane's part has landed, and every lane is done with the row before this one
    Row r;
    const float4 v = *reinterpret_cast<const float4*>(row + CPL + mine);
    r.v[0] = row[CPL - 1 + mine];
    r.v[1] = v.x;
    r.v[2] = v.y;
    r.v[3] = v.z;
    r.v[4] = v.w;
    r.v[5] = row[2 * CPL + mine];
    return r;
  };
#pragma unroll
  for (int k = -1; k < PD - 2; k++) fetch(ring + ((k + PD - 1) % PD) * RW, true);
  Row a = take(ring + 6 * RW);
  fetch(ring + 5 * RW, true);  // row 6
  Row b = take(ring + 7 * RW);
  fetch(ring + 6 * RW, true);  // row 7
  Slopes up, dn;
  if (!LOWEST) up = slopes_between(a, b);
  float acc = nonfinite<NODATA>(b, 0.0f);  // NODATA: of row b alone, else of all rows so far
  float above = NODATA ? nonfinite<NODATA>(a, 0.0f) : 0.0f;  // of row a
  for (int i = 0; i < it.n; i += 4) {
    float *cur = ring + (i & 4) * RW, *other = ring + ((i & 4) ^ 4) * RW;
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const Row c = take(cur + u * RW);
      fetch(u ? cur + (u - 1) * RW : other + 3 * RW, i + u + PD <= it.n);  // row i + u + 8
      const float next = nonfinite<NODATA>(c, NODATA ? 0.0f : acc);
      if (!LOWEST) dn = slopes_between(b, c);
      uint32_t packed = row_codes<LOWEST>(a, b, c, up, dn, nz);
      if (NODATA) {
        const float any = __fadd_rn(__fadd_rn(above, acc), next);
        if (any != any) packed = mask_nodata(a, b, c, packed);
        above = acc;
      }
      acc = next;
      packed = (packed & ~it.colmask) | (0x08080808u & it.colmask);
      if (VEC) {
        *reinterpret_cast<uint32_t*>(it.dir) = packed;
      } else {
#pragma unroll
        for (int k = 0; k < CPL; k++) it.dir[k] = (uint8_t)(packed >> (8 * k));
      }
      it.dir += it.lddir;
      a = b;
      b = c;
      up = dn;
    }
  }
  cp_async_wait<0>();  // nothing may land in the ring after the item is done
  __syncwarp();
  return !NODATA && __any_sync(FULL, acc != acc);
}

// Any item.  Off the grid rows and columns read as zero: they only neighbour
// edge cells, whose code is OUTLET.  Returns whether an own cell of a rule
// without masks is not finite.
template <bool LOWEST, bool NODATA>
__device__ __forceinline__ bool walk_any(Item it, float nz) {
  auto load = [&](int q) {
    float x[CPL] = {0.0f, 0.0f, 0.0f, 0.0f}, h = 0.0f;
    if (q >= it.qlo && q < it.qhi) {
#pragma unroll
      for (int k = 0; k < CPL; k++)
        if (k < it.ncols) x[k] = __ldg(it.z + k);
      if (it.hval) h = __ldg(it.h);
    }
    it.z += it.ldz;
    it.h += it.ldz;
    return row_of(it, x, h);
  };
  const int nmax = __reduce_max_sync(FULL, it.n);
  Row a = load(0), b = load(1), c = load(2);
  Slopes up, dn;
  if (!LOWEST) up = slopes_between(a, b);
  bool report = false;
  for (int i = 0; i < nmax; i++) {
    const Row ahead = load(i + 3);
    if (!LOWEST) dn = slopes_between(b, c);
    uint32_t packed = row_codes<LOWEST>(a, b, c, up, dn, nz);
    float bad = nonfinite<NODATA>(b, 0.0f);
    if (NODATA) bad = nonfinite<NODATA>(a, nonfinite<NODATA>(c, bad));
    if (bad != bad && i < it.n) {
      if (NODATA) {
        packed = mask_nodata(a, b, c, packed);
      } else {
#pragma unroll
        for (int k = 0; k < CPL; k++)
          if (!isfinite(b.v[k + 1])) packed = (packed & ~(0xFFu << (8 * k))) | (9u << (8 * k));
        report = true;
      }
    }
    const uint32_t m = (i == it.top || i == it.bottom) ? 0xFFFFFFFFu : it.colmask;
    packed = (packed & ~m) | (0x08080808u & m);
    if (i < it.n) {
#pragma unroll
      for (int k = 0; k < CPL; k++)
        if (k < it.ncols) it.dir[k] = (uint8_t)(packed >> (8 * k));
    }
    it.dir += it.lddir;
    a = b;
    b = c;
    c = ahead;
    up = dn;
  }
  return report;
}

// NODATA masks (the rule's NODATA bit): a cell with a non-finite elevation is
// outside the study area and gets OUTLET, and so does every cell next to one
// (the area's edge drains off it, as the grid's edge does); nothing is
// reported as an error.  nseg: work items per tile, of seg_rows rows (a divisor of T).
// nz: -0 (lowest_code).
template <int T, bool LOWEST, bool NODATA>
__global__ void __launch_bounds__(NTF, 5) k_flowdir_rows(DemTable dt, int64_t ntiles, int nseg, int seg_rows, float nz,
                                                         uint32_t* status) {
  constexpr int LPT = T / CPL;   // lanes per tile
  constexpr int IPW = 32 / LPT;  // items per warp
  const int lane = threadIdx.x & 31, li = lane & (LPT - 1);
  __shared__ __align__(16) float rings[NTF / LPT][PD * (T + 8)];
  float* ring = rings[threadIdx.x / LPT];
  const int64_t nitems = ntiles * nseg;
  const int64_t step = (int64_t)gridDim.x * (NTF / 32) * IPW;
  const int64_t first = ((int64_t)blockIdx.x * (NTF / 32) + (threadIdx.x >> 5)) * IPW;
  for (int64_t base = first; base < nitems; base += step) {
    // the warp's items are consecutive; one past the end has no rows
    const bool present = base + lane / LPT < nitems;
    const int64_t item = present ? base + lane / LPT : nitems - 1;
    const int64_t t = item / nseg;
    const DemDesc d = dem_of(dt, t);
    const TileGeo g = tile_geo(d, t - d.tile_base, T);
    const int r0 = (int)(item - t * nseg) * seg_rows;
    const int64_t i0 = g.i0 + r0, gj = g.j0 + li * CPL;  // first row, first own column
    Item it;
    it.n = present ? max(0, min(seg_rows, g.th - r0)) : 0;
    it.ncols = max(0, min(CPL, g.tw - li * CPL));
    it.ldz = d.ldz;
    it.lddir = d.lddir;
    it.z = d.z + (i0 - 1) * d.ldz + gj;
    it.dir = d.dir + i0 * d.lddir + gj;
    it.first = li == 0;
    it.last = li == LPT - 1;
    it.right = g.j0 + T < d.W;
    it.hval = it.first ? g.j0 > 0 : (it.last && it.right);
    it.h = it.hval ? it.z + (it.first ? -1 : CPL) : it.z;
    const bool above = i0 > 0 || (d.halo & 1), below = i0 + it.n < d.H || (d.halo & 2);
    it.qlo = above ? 0 : 1;
    it.qhi = it.n == 0 ? it.qlo : it.n + (below ? 2 : 1);
    it.top = above ? -1 : 0;
    it.bottom = below ? -1 : it.n - 1;
    it.colmask = gj == 0 ? 0xFFu : 0u;
#pragma unroll
    for (int k = 0; k < CPL; k++)
      if (gj + k == d.W - 1) it.colmask |= 0xFFu << (8 * k);
    const bool inside = it.n == seg_rows && it.ncols == CPL && above && below;
    const bool vec = ((reinterpret_cast<uintptr_t>(it.z) & 15u) == 0) && (d.ldz & 3) == 0 &&
                     ((reinterpret_cast<uintptr_t>(it.dir) & 3u) == 0) && (d.lddir & 3) == 0;
    bool redo = true;
    if (__all_sync(FULL, inside)) {
      redo = __all_sync(FULL, vec) ? walk_inside<T, LOWEST, NODATA, true>(it, ring, nz)
                                    : walk_inside<T, LOWEST, NODATA, false>(it, ring, nz);
    }
    if (redo && walk_any<LOWEST, NODATA>(it, nz)) set_status(status, D8_ERR_NONFINITE);
  }
}

// Rows per item: whole tiles for grids that fill the GPU with them (two rows
// in T are then read twice); below MIN_WARPS_PER_SM warps the tiles are cut
// into segments of T / 2, T / 4, ... down to 8 rows.  (About 20 warps fit an
// SM; with 35 here 8192 x 8192 runs 2.7 rounds of them and takes 121 us, with
// 70 it halves its tiles and takes 97, with 140 it quarters them: 104.  With 35,
// 70 and 140: 1024 x 1024 10.7, 9.7, 9.5 us; 3001 x 5003 33, 37, 37; 6000 x 6000
// 76, 67, 69; 10000 x 7000 125, 109, 114; 12000 x 12000 217, 217, 200; 2048 x 2048,
// 16384 x 16384 and 32768 x 32768 the same.)  A grid
// lower than a tile is cut into segments of its own rows: 8 x 400000 takes 14 us,
// 25 to 33 when two thirds of the segments lay below the grid.
constexpr int64_t MIN_WARPS_PER_SM = 70;

template <int T, bool LOWEST, bool NODATA>
static cudaError_t launch_t(const DemTable& dt, int64_t ntiles, uint32_t* status, cudaStream_t s) {
  int dev = 0, sms = 1, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  auto k = k_flowdir_rows<T, LOWEST, NODATA>;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, NTF, 0) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  constexpr int IPW = 32 / (T / CPL), IPB = IPW * (NTF / 32);
  const int span = (int)(dt.ndem == 1 ? min64(T, dt.one.H) : T);  // rows of the highest tile
  int rows = T;
  auto segments = [&]() { return (span + rows - 1) / rows; };
  while (rows > 8 && ntiles * segments() < MIN_WARPS_PER_SM * IPW * sms) rows /= 2;
  const int nseg = segments();
  int64_t grid = (ntiles * nseg + IPB - 1) / IPB;
  const int64_t cap = (int64_t)sms * per_sm;
  if (grid > cap) grid = cap;
  k<<<(unsigned)(grid < 1 ? 1 : grid), NTF, 0, s>>>(dt, ntiles, nseg, rows, -0.0f, status);
  return cudaGetLastError();
}

template <int T>
static cudaError_t launch_rule(const DemTable& dt, int64_t ntiles, int rule, uint32_t* status, cudaStream_t s) {
  switch (rule) {
    case 0: return launch_t<T, false, false>(dt, ntiles, status, s);
    case 1: return launch_t<T, true, false>(dt, ntiles, status, s);
    case 2: return launch_t<T, false, true>(dt, ntiles, status, s);
    case 3: return launch_t<T, true, true>(dt, ntiles, status, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace fdir

cudaError_t launch_flowdir(const DemTable& dt, int64_t ntiles, int T, int rule, uint32_t* status, cudaStream_t s,
                           int* nlaunch) {
  ++*nlaunch;
  switch (T) {
    case 32: return fdir::launch_rule<32>(dt, ntiles, rule, status, s);
    case 64: return fdir::launch_rule<64>(dt, ntiles, rule, status, s);
    case 128: return fdir::launch_rule<128>(dt, ntiles, rule, status, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace d8
