// Float64 local operators in block fixed point (fx.hpp): the operators A_II^-1
// and K_GG of every subdomain as lower triangles of tiles (fx_pack.hpp), times a
// block of right-hand sides (sm_103a).
//
// What bounds it: as float64 the pass is bound by the 2 FMAs per SM and clock
// of GB300's float64 pipe, far below HBM. In fixed point a stored entry costs
// 6 integer multiply-adds (3 for its row's and 3 for its column's product, 32
// lanes per SM and clock), about half of the time its 8 bytes take from HBM, so
// storing the triangle pays; at one column DRAM is 68 to 74 % busy and the integer
// pipe 46 to 51 %, the rest the end of a unit, where every warp waits. From two columns
// on the integer multiply-adds are the larger part (3 per full entry and column
// against one float64 FMA at a sixteenth of their rate).
//
// Split. One block of up to 12 warps owns one unit, an operator and up to NC
// columns, at a time; the tiles are dealt to the warps, and every warp streams its
// own ones through a private ring of bulk copies that runs on into the next unit,
// so no warp waits for another one but at a unit's end. A tile is read twice from
// shared memory, so that neither use needs a reduction across the warp: once with a
// row per lane (its row's products with x_J), once with two columns per lane (the
// products with x_I of the mirrored tile). The sums go to shared memory with 32-bit
// integer atomics that nothing waits for: exact, so the result depends on no order.
//
// Rows whose certificate does not hold (fx.hpp) are listed at the unit's end and
// summed in float64, a warp each, from the float64 form of the tiles: a few in 10^5
// for dense operands, 0.1 to 0.6 % in the iterations of a solve with lognormal
// conductivities (up to a tenth of one operator: that solve takes 26.9 ms on 96^3
// elements, 25.9 without a certificate and 49.1 in float64), a third or so for an
// operand with one entry.
//
// Measured on 1728 operators of 343 rows at one column: 165 us, 5.6 TB/s of stored
// entries (the float64 kernel: 401 us); on 512 of them at 8 columns 322 us, half
// of the integer multiply-add rate (the float64 kernel: 1085 us). (Row-major
// triangles with whole rows per warp took 270 to 430 us: rows of many lengths cost
// more instructions in control and reductions than in products.)
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "async.cuh"
#include "fx_pack.hpp"
#include "kernels.cuh"

namespace bddc {

namespace {
constexpr int kFxWarps = 12;                // of a block at most; kFxFewWarps where more rings don't fit
constexpr int kFxFewWarps = 8;
constexpr int kFxTileBytes = kFxTileElems * 8;
constexpr int kFxMaxSlots = 2;              // tiles in flight per warp
constexpr size_t kFxSmemCap = kSmemMost;
constexpr int kFxSmemSm = 228 * 1024;       // of an SM; every block takes 1 KB beside its own and the static arrays
constexpr int kFarList = 256;

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ int4 lds16(uint32_t addr) {
  int4 v;
  asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
// (h, m) += the product of the entries {al, ah} and {xl, xh}. (In C++: written
// as inline mad.wide the kernel ran 1.2 times the instructions, five times
// the 32-bit adds among them.)
__device__ __forceinline__ void fx_mac(int64_t& h, int64_t& m, int al, int ah, int xl, int xh) {
  h += (int64_t)ah * xh;
  m += (int64_t)ah * xl;
  m += (int64_t)al * xh;
}

// (hi + frac 2^-kFxFrac) 2^k, rounded
__device__ __forceinline__ double fx_value(int64_t hi, int64_t frac, int k) {
  const double v = fma((double)frac, 1.0 / (double)(1 << kFxFrac), (double)hi);
  // (|v| is 0 or between 2^-24 and 2^63)
  if (k > -990 && k < 960) return v * __longlong_as_double((long long)(k + 1023) << 52);
  return scalbn(v, k);
}

// Row i of an n x n operator times the column at x, in float64: every lane a 32nd
// of the row, the loads of kRowTiles tiles in flight together (a row is a chain of
// loads otherwise), then a tree over the lanes.
constexpr int kRowTiles = 12;
__device__ __noinline__ double fx_row64(const double* __restrict__ values, const double* __restrict__ x, int nrhs, int n,
                                        int i, int lane) {
  const int I = i / kFxTile, r = i % kFxTile;
  double s = 0.0;
  for (int J0 = 0; J0 * kFxTile < n; J0 += kRowTiles) {
    double a[kRowTiles], v[kRowTiles];
#pragma unroll
    for (int q = 0; q < kRowTiles; ++q) {
      const int J = J0 + q, j = J * kFxTile + lane;
      const double* tile = values + (int64_t)fx_tile_at(I, J) * kFxTileElems;
      a[q] = j < n ? __ldg(tile + (J <= I ? r * kFxTile + lane : lane * kFxTile + r)) : 0.0;
      v[q] = j < n ? x[(int64_t)j * nrhs] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < kRowTiles; ++q) s = fma(a[q], v[q], s);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

__device__ __forceinline__ int64_t shfl_xor64(int64_t v, int o) {
  int lo = (int)v, hi = (int)(v >> 32);
  lo = __shfl_xor_sync(0xffffffffu, lo, o);
  hi = __shfl_xor_sync(0xffffffffu, hi, o);
  return (int64_t)((uint32_t)lo) | ((int64_t)hi << 32);
}

// The fixed-point tiles of all operators from the float64 ones, an operator per
// block at a time.
__global__ void __launch_bounds__(256) k_fx_quantize(const WorkItem* __restrict__ items, int n_items,
                                                     const double* __restrict__ values, const int32_t* __restrict__ rexp,
                                                     const int8_t* __restrict__ shift, int2* __restrict__ halves) {
  for (int u = blockIdx.x; u < n_items; u += gridDim.x) {
    const WorkItem w = items[u];
    const int n = w.ncols;
    int64_t at = w.moff;
    for (int I = 0; I * kFxTile < n; ++I)
      for (int J = 0; J <= I; ++J, at += kFxTileElems) {
        const int s = shift[at / kFxTileElems];
        for (int e = threadIdx.x; e < kFxTileElems; e += blockDim.x) {
          const int r = e / kFxTile, k = e % kFxTile, i = I * kFxTile + r, j = J * kFxTile + k;
          int2 q;
          fx_entry((uint64_t)__double_as_longlong(values[at + e]), i < n ? rexp[w.yoff + i] : 0,
                   j < n ? rexp[w.yoff + j] : 0, s, q.x, q.y);
          halves[at + fx_place(r, k)] = q;
        }
      }
  }
}

// Shared memory of one block, in this order; T = tile rows of the largest
// operator, npad its rows padded to whole tiles.
struct FxSmem {
  int T, npad, nc;
  __host__ __device__ FxSmem(int max_n, int nc_) : T((max_n + kFxTile - 1) / kFxTile), npad(T * kFxTile), nc(nc_) {}
  __host__ __device__ int shift_bytes() const { return (T * (T + 1) / 2 + 3 + 15) / 16 * 16; }
  __host__ __device__ size_t total(int nw, int nst) const {
    // rings and barriers; per row: operand halves, next operand, totals and
    // magnitudes of every column, the operator's row exponent; per tile row and
    // column: operand exponent, two buffers of unit and certificate; the tiles'
    // shifts, two buffers
    return (size_t)nw * nst * (kFxTileBytes + 8) + (size_t)npad * ((8 + 8 + 16) * nc + 4) + (size_t)T * nc * (4 + 2 * 12) +
           2 * shift_bytes();
  }
};

// Units: (operator, slice, columns [NC b, NC b + NC)), ncb column blocks. With
// one slice (S = 1) a unit's tasks are the operator's tiles, each for its rows
// and its columns. With S > 1 slices, slice s owns the tile rows s, s + S, ..
// of the result, and a task is one half: tile (I, J) for rows I where J <= I, or
// tile (J, I) for its columns I; a tile is then read by two blocks.
struct FxUnits {
  int n_items, ncb, S;
  __device__ int count() const { return n_items * S * ncb; }
  __device__ int item(int u) const { return u / (S * ncb); }
  __device__ int slice(int u) const { return u % (S * ncb) / ncb; }
  __device__ int col(int u) const { return u % ncb; }
  // tasks of a slice of an operator of T tile rows
  __device__ int tasks(int s, int T) const { return S == 1 ? T * (T + 1) / 2 : s < T ? ((T - 1 - s) / S + 1) * T : 0; }
};
// Cursor over the tasks of one warp: tasks warp, warp + (warps of a block), .. of unit
// u, then those of the block's next unit.
struct FxCursor {
  int u, t, nt;          // unit, task, tasks of the unit
  int T, s;              // tile rows of its operator, its slice
  const int2* base;      // the operator's tiles
};

// Y = Op X.
template <int NC>
__global__ void __launch_bounds__(kFxWarps * 32, 1)
    k_fx_gemm(const WorkItem* __restrict__ items, FxUnits U, FxForm A, const double* __restrict__ X,
              double* __restrict__ Y, const int32_t* __restrict__ yscatter, int nrhs, int nst, int max_n,
              int32_t* __restrict__ err) {
  constexpr int NG = NC < 4 ? NC : 4;   // columns whose sums are held at once
  extern __shared__ __align__(128) unsigned char smem[];
  const FxSmem L(max_n, NC);
  const int npad = L.npad, ldT = L.T, n_units = U.count();
  const int2* arena = reinterpret_cast<const int2*>(A.halves);
  int2* xq = reinterpret_cast<int2*>(smem + (size_t)(blockDim.x >> 5) * nst * kFxTileBytes);   // operand [NC][npad]
  double* xraw = reinterpret_cast<double*>(xq + NC * npad);                                    // next operand
  uint64_t* bars = reinterpret_cast<uint64_t*>(xraw + NC * npad);
  uint32_t* sums = reinterpret_cast<uint32_t*>(bars + (blockDim.x >> 5) * nst);   // totals, magnitudes [4][NC][npad]
  int32_t* xexp = reinterpret_cast<int32_t*>(sums + 4 * NC * npad);      // row exponents of the next operand
  int32_t* xe = xexp + npad;                                             // exponents of the operand's blocks [NC][T]
  int32_t* top_of = xe + NC * ldT;                                       // of this unit and the next: unit of a tile
  const int top_buf = 3 * NC * ldT;                                      // row's totals [NC][T], certificate [2][NC][T]
  int8_t* shift = reinterpret_cast<int8_t*>(top_of + 2 * top_buf);       // of this operator's and the next one's tiles
  const int shift_buf = L.shift_bytes();
  __shared__ uint16_t far_list[kFarList];   // rows and columns left for float64, while there is room
  __shared__ int far_count[2];         // of this unit and the next
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  uint64_t* full = bars + warp * nst;
  unsigned char* ring = smem + (size_t)warp * nst * kFxTileBytes;

  if (tid == 0) {
    far_count[0] = far_count[1] = 0;
    for (int s = 0; s < nw * nst; ++s) mbar_init(&bars[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const int lim = NC * npad;
  for (int i = tid; i < 4 * lim; i += blockDim.x) sums[i] = 0;
  auto add = [&](int at, int64_t h0, int64_t m0, int64_t h1, int64_t m1, int d) {
    int64_t hi;
    uint32_t f;
    fx_scaled_sum(h0, m0, h1, m1, d, hi, f);
    atomicAdd(&sums[at], f);
    atomicAdd(&sums[lim + at], fx_limb0(hi));
    atomicAdd(&sums[2 * lim + at], (uint32_t)fx_limb1(hi));
    atomicAdd(&sums[3 * lim + at], fx_magnitude(h0, h1, d));
  };

  auto enter = [&](FxCursor& c) {   // the first unit from c.u on that has a task for this warp
    for (; c.u < n_units; c.u += gridDim.x) {
      const WorkItem w = items[U.item(c.u)];
      c.T = (w.ncols + kFxTile - 1) / kFxTile;
      c.s = U.slice(c.u);
      c.nt = U.tasks(c.s, c.T);
      c.base = arena + w.moff;
      if (c.t < c.nt) return;
    }
  };
  // lane 0 keeps nst tiles of the warp in flight
  FxCursor in{(int)blockIdx.x, warp, 0, 0, 0, nullptr};
  enter(in);
  int in_slot = 0, flying = 0;
  auto issue = [&]() {
    if (in.u >= n_units) return;
    int tile = in.t;
    if (U.S > 1) {
      const int I = in.s + U.S * (in.t / in.T), J = in.t % in.T, a = max(I, J), b = min(I, J);
      tile = a * (a + 1) / 2 + b;
    }
    if (lane == 0) {
      mbar_expect_tx(&full[in_slot], kFxTileBytes);
      bulk_load(ring + (size_t)in_slot * kFxTileBytes, in.base + (int64_t)tile * (kFxTile * kFxTile), kFxTileBytes,
                &full[in_slot]);
    }
    ++flying;
    if (++in_slot == nst) in_slot = 0;
    if ((in.t += nw) >= in.nt) {
      in.u += gridDim.x;
      in.t = warp;
      enter(in);
    }
  };
  // shifts of an operator's tiles: copied from the word that holds the first one
  auto tile0 = [](const WorkItem& w) { return (int)(w.moff / kFxTileElems); };
  auto prefetch_operand = [&](int uu, int p) {
    const WorkItem wn = items[U.item(uu)];
    const int k0 = U.col(uu) * NC, nk = min(NC, nrhs - k0);
    for (int j = tid; j < NC * npad; j += blockDim.x) {
      const int i = j / NC, k = j - i * NC;
      if (i < wn.ncols && k < nk)
        cp_async8(xraw + k * npad + i, X + (int64_t)(wn.xoff + i) * nrhs + k0 + k);
      else
        xraw[k * npad + i] = 0.0;
    }
    for (int i = tid; i < npad; i += blockDim.x) {
      if (i < wn.ncols)
        cp_async4(xexp + i, A.rexp + wn.yoff + i);
      else
        xexp[i] = 0;
    }
    const int t0 = tile0(wn), words = ((t0 & 3) + fx_tiles(wn.ncols) + 3) / 4;
    for (int i = tid; i < words; i += blockDim.x) cp_async4(shift + p * shift_buf + 4 * i, A.shift + (t0 & ~3) + 4 * i);
    cp_async_commit();
  };
  // Three block barriers per unit: (A) all sums added and the next operand
  // landed, (B) the next operand converted, a block per warp at a time, (C) the
  // unit's results stored and the sums cleared, the next one's tile rows' units and
  // certificates known.
  auto convert_operand = [&]() {
    for (int b = warp; b < NC * ldT; b += nw) {
      const int k = NC == 1 ? 0 : b / ldT, i = (b - k * ldT) * kFxTile + lane, at = k * npad + i;
      const uint64_t v = (uint64_t)__double_as_longlong(xraw[at]);
      const int ei = xexp[i];
      int E = __reduce_max_sync(0xffffffffu, fx_scaled_exponent(v, ei));
      int2 h = make_int2(0, 0);
      if (E != kFxZero && E != kFxNonFinite) {
        auto round = [&]() {
          const int64_t q = ei != kFxZero ? fx_quantize(v, kFxBits - E + ei) : 0;
          h = make_int2(fx_lo(q), fx_hi(q));
        };
        round();
        const uint32_t part = fx_part(h.y), all = __reduce_add_sync(0xffffffffu, part);
        if (fx_half_exceeds(all)) {   // the lower and upper, the even and odd half
          const uint32_t low = __reduce_add_sync(0xffffffffu, lane < 16 ? part : 0);
          const uint32_t even = __reduce_add_sync(0xffffffffu, lane & 1 ? 0 : part);
          if (fx_half_exceeds(max(max(low, all - low), max(even, all - even)))) {
            ++E;
            round();
          }
        }
      }
      xq[at] = h;
      if (lane == 0) xe[b] = E;
    }
  };
  auto row_scales = [&](int uu, int p) {
    const WorkItem wn = items[U.item(uu)];
    const int T = (wn.ncols + kFxTile - 1) / kFxTile;
    const int8_t* sh = shift + p * shift_buf + (tile0(wn) & 3);
    int32_t* top = top_of + p * top_buf;
    for (int b = warp; b < NC * T; b += nw) {   // a tile row and column per warp, a block per lane
      const int k = NC == 1 ? 0 : b / T, I = b - k * T;
      const int32_t* e = xe + k * ldT;
      auto scale = [&](int J) { return J < T ? fx_block_scale(e[J], sh[fx_tile_at(I, J)]) : kFxZero; };
      int hi = kFxZero;
      for (int J = lane; J < T; J += 32) hi = max(hi, scale(J));
      hi = __reduce_max_sync(0xffffffffu, hi);
      uint32_t s1 = 0, s2 = 0;
      if (hi >= kFxNonFinite) {
        s2 = lane == 0;
      } else if (hi != kFxZero) {
        for (int J = lane; J < T; J += 32) {
          const int d = hi - scale(J);
          s1 += fx_s1(d);
          s2 += fx_s2(d);
        }
        s1 = __reduce_add_sync(0xffffffffu, s1);
        s2 = __reduce_add_sync(0xffffffffu, s2);
      }
      if (lane == 0) {
        top[k * ldT + I] = hi >= kFxNonFinite ? 0 : hi;
        top[(NC + k) * ldT + I] = (int32_t)s1;
        top[(2 * NC + k) * ldT + I] = (int32_t)s2;
      }
    }
  };

  int par = 0;
  __syncthreads();   // barriers initialised, sums cleared
  for (int s = 0; s < nst; ++s) issue();
  if (blockIdx.x < n_units) {
    prefetch_operand(blockIdx.x, par);
    cp_async_wait_all();
    __syncthreads();                          // operand landed
    convert_operand();
    __syncthreads();                          // xq and xe complete; xraw free
    row_scales(blockIdx.x, par);
    __syncthreads();                          // top and cert complete
    if (blockIdx.x + (int)gridDim.x < n_units) prefetch_operand(blockIdx.x + gridDim.x, par ^ 1);
  }
  int slot = 0;
  uint32_t phase = 0;
  bool aborted = false;
  // shared addresses: row view (row lane, vector v at v ^ (lane & 7)), column
  // view (vector lane & 15 of rows t + 16 (lane >> 4))
  const uint32_t xq_addr = smem_addr(xq), ring_addr = smem_addr(ring), xcol = (uint32_t)npad * 8u;
  const uint32_t sw = (uint32_t)(lane & 7) << 4;
  const uint32_t rowv = (uint32_t)lane * 256u, colv = (uint32_t)(lane >> 4) * 16u * 256u;
  const uint32_t vec = (uint32_t)(lane & 15) << 4;
  for (int u = blockIdx.x; u < n_units; u += gridDim.x) {
    const WorkItem w = items[U.item(u)];
    const int n = w.ncols, T = (n + kFxTile - 1) / kFxTile, sl = U.slice(u), nt = U.tasks(sl, T);
    const int k0 = U.col(u) * NC, nk = min(NC, nrhs - k0);
    const bool has_next = u + (int)gridDim.x < n_units;
    const int8_t* sh = shift + par * shift_buf + (tile0(w) & 3);
    const int32_t* top = top_of + par * top_buf;
    int I = 0, first = 0;   // S = 1: tile row of t, and its first tile
    for (int t = warp; t < nt; t += nw) {
      int J;
      bool rows = true, cols;   // the halves of this task: rows I times x_J, columns J times x_I
      if (U.S == 1) {
        while (t > first + I) first += ++I;
        J = t - first;
        cols = I != J;
      } else {
        const int i = sl + U.S * (t / T), j = t % T;
        I = max(i, j);
        J = min(i, j);
        rows = i >= j;
        cols = !rows;
      }
      if (!aborted && !mbar_wait(&full[slot], phase)) {
        if (lane == 0) atomicExch(err, BDDC_ERR_TIMEOUT);
        aborted = true;
      }
      aborted = __any_sync(0xffffffffu, aborted);
      if (aborted) break;
      --flying;
      const uint32_t tile = ring_addr + (uint32_t)slot * kFxTileBytes;
      const int ts = sh[fx_tile_at(I, J)];
#pragma unroll 1
      for (int g = 0; g < (NC > NG ? nk : 1); g += NG) {
        if (rows) {
          // rows: lane's row times x_J
          const uint32_t ad = tile + rowv, xa = xq_addr + (uint32_t)J * (kFxTile * 8) + g * xcol;
          int64_t h[NG][2], m[NG][2];
#pragma unroll
          for (int k = 0; k < NG; ++k) h[k][0] = h[k][1] = m[k][0] = m[k][1] = 0;
#pragma unroll
          for (int v = 0; v < kFxTile / 2; ++v) {
            const int4 a = lds16(ad + (((uint32_t)v << 4) ^ sw));
#pragma unroll
            for (int k = 0; k < NG; ++k) {
              const int4 x = lds16(xa + k * xcol + 16u * v);
              fx_mac(h[k][0], m[k][0], a.x, a.y, x.x, x.y);
              fx_mac(h[k][1], m[k][1], a.z, a.w, x.z, x.w);
            }
          }
#pragma unroll
          for (int k = 0; k < NG; ++k) {
            const int c = (g + k) * ldT, d = max(0, top[c + I] - xe[c + J] + ts);
            add((g + k) * npad + I * kFxTile + lane, h[k][0], m[k][0], h[k][1], m[k][1], d);
          }
        }
        if (cols) {
          // columns: two per lane, rows r and r + 16 on the half warps, times x_I
          const uint32_t ad = tile + colv;
          const uint32_t xa = xq_addr + (uint32_t)I * (kFxTile * 8) + (uint32_t)(lane >> 4) * 128u + g * xcol;
          int64_t h[NG][2], m[NG][2];
#pragma unroll
          for (int k = 0; k < NG; ++k) h[k][0] = h[k][1] = m[k][0] = m[k][1] = 0;
#pragma unroll
          for (int r = 0; r < kFxTile / 2; r += 2) {
            const int4 a = lds16(ad + 256u * r + (vec ^ ((uint32_t)(r & 7) << 4)));
            const int4 b = lds16(ad + 256u * (r + 1) + (vec ^ ((uint32_t)((r + 1) & 7) << 4)));
#pragma unroll
            for (int k = 0; k < NG; ++k) {
              const int4 x = lds16(xa + k * xcol + 8u * r);   // the operand at rows r and r + 1
              fx_mac(h[k][0], m[k][0], a.x, a.y, x.x, x.y);
              fx_mac(h[k][1], m[k][1], a.z, a.w, x.x, x.y);
              fx_mac(h[k][0], m[k][0], b.x, b.y, x.z, x.w);
              fx_mac(h[k][1], m[k][1], b.z, b.w, x.z, x.w);
            }
          }
          // the half warps' sums: the lower half keeps the first column
          const bool up = lane >= 16;
#pragma unroll
          for (int k = 0; k < NG; ++k) {
            const int64_t ho = shfl_xor64(up ? h[k][0] : h[k][1], 16), mo = shfl_xor64(up ? m[k][0] : m[k][1], 16);
            const int c = (g + k) * ldT, d = max(0, top[c + J] - xe[c + I] + ts);
            add((g + k) * npad + J * kFxTile + 2 * (lane & 15) + up, up ? h[k][1] : h[k][0], up ? m[k][1] : m[k][0], ho,
                mo, d);
          }
        }
      }
      __syncwarp();   // the tile is read: its slot may be refilled
      issue();
      if (++slot == nst) { slot = 0; phase ^= 1u; }
    }
    cp_async_wait_all();                      // this thread's copies of the next operand landed
    __syncthreads();                          // A: sums added; xq and xe no longer read
    if (has_next) convert_operand();
    __syncthreads();                          // B: xq and xe complete; xraw free
    auto store = [&](int j, double y) {
      const int64_t jy = (int64_t)w.yoff + j / NC;
      Y[(yscatter ? (int64_t)yscatter[jy] : jy) * nrhs + k0 + j % NC] = y;
    };
    auto row64 = [&](int j) {
      const double y = fx_row64(A.values + w.moff, X + (int64_t)w.xoff * nrhs + k0 + j % NC, nrhs, n, j / NC, lane);
      if (lane == 0) store(j, y);
    };
    for (int j0 = warp * 32; j0 < NC * n; j0 += blockDim.x) {
      const int j = j0 + lane, c = j / NC, k = j - c * NC, at = k * npad + c, I = c / kFxTile;
      bool far = false;   // not accurate in fixed point
      if (j < NC * n && (U.S == 1 || I % U.S == sl) && k < nk) {
        const int E = top[k * ldT + I], ec = A.rexp[w.yoff + c];
        const uint32_t s1 = top[(NC + k) * ldT + I], s2 = top[(2 * NC + k) * ldT + I];
        far = !fx_holds(sums[3 * lim + at], s1, s2) && (ec != kFxZero || s1 == 0);   // (a row of zeros is exact)
        double y = 0.0;
        if (E != kFxZero && ec != kFxZero)
          y = fx_value(fx_total(sums[lim + at], (int32_t)sums[2 * lim + at]), sums[at], fx_unit(ec, E));
        if (!far) store(j, y);
      }
      if (j < NC * n) sums[at] = sums[lim + at] = sums[2 * lim + at] = sums[3 * lim + at] = 0;
      const uint32_t left = __ballot_sync(0xffffffffu, far);
      if (left) {
        int at0 = 0;
        if (lane == 0) at0 = atomicAdd(&far_count[par], __popc(left));
        const int pos = __shfl_sync(0xffffffffu, at0, 0) + __popc(left & ((1u << lane) - 1));
        if (far && pos < kFarList) far_list[pos] = (uint16_t)j;
        for (uint32_t rest = __ballot_sync(0xffffffffu, far && pos >= kFarList); rest; rest &= rest - 1)
          row64(j0 + __ffs(rest) - 1);
      }
    }
    if (has_next) row_scales(u + gridDim.x, par ^ 1);
    __syncthreads();                          // C: sums clear; the next top, far_list and far_count complete
    // (from the last warp on: the tiles are dealt from the first one on)
    for (int q = nw - 1 - warp; q < min(far_count[par], kFarList); q += nw) row64(far_list[q]);
    par ^= 1;
    if (tid == 0) far_count[par] = 0;         // (added to after the next B)
    if (u + 2 * (int)gridDim.x < n_units) prefetch_operand(u + 2 * gridDim.x, par ^ 1);
  }
  cp_async_wait_all();
  // after a timeout: this warp's copies in flight land before the block exits
  for (; aborted && flying > 0; --flying) {
    if (!mbar_wait(&full[slot], phase)) break;
    if (++slot == nst) { slot = 0; phase ^= 1u; }
  }
}

template <int NC>
cudaError_t run_fx(const WorkItem* items, int n_items, int max_n, int S, const FxForm& A, const double* X, double* Y,
                   const int32_t* yscatter, int nrhs, int32_t* err, cudaStream_t st) {
  const FxSmem L(max_n, NC);
  const FxUnits U{n_items, (nrhs + NC - 1) / NC, S};
  const int64_t units = (int64_t)n_items * U.ncb * S;
  auto fits = [&](int nw, int nst) { return L.total(nw, nst) <= kFxSmemCap; };
  auto blocks = [&](int nw) { return std::min(kFxWarps / nw, (int)(kFxSmemSm / (L.total(nw, kFxMaxSlots) + 2048))); };
  // Warps of a block: as many as the largest operator has tiles, up to 12, in one
  // block per SM; narrower blocks, several to an SM, where there are more units than
  // SMs: the waits at a unit's end and its chain of loads then overlap with other
  // units. Three (two) blocks of 4 warps for operators of up to 6 tile rows, two of
  // 6 warps for larger ones at one or two columns, as far as both fit (1728
  // operators, one column: 64 rows 24 us against 59 with 12 warps, 125 rows 40
  // against 67, 343 rows 165 against 171; 4 columns of 125 rows 110 against 128;
  // 8 columns of 196 rows, where one block of 4 warps fits, 613 against 397).
  int nw = std::max(4, std::min(kFxWarps, fx_tiles(max_n)));
  if (units > num_sms()) {
    if (L.T <= 6 && blocks(4) >= 2) nw = 4;
    else if (NC <= 2 && nw > 6 && blocks(6) >= 2) nw = 6;
  }
  const int nst = fits(nw, kFxMaxSlots) ? kFxMaxSlots : 1;
  if (!fits(nw, nst)) nw = kFxFewWarps;
  const size_t smem = L.total(nw, nst);
  cudaError_t e = allow_smem(k_fx_gemm<NC>, smem);
  if (e != cudaSuccess) return e;
  const int per_sm = nst == kFxMaxSlots ? std::max(1, blocks(nw)) : 1;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(units, (int64_t)per_sm * num_sms()));
  k_fx_gemm<NC><<<grid, nw * 32, smem, st>>>(items, U, A, X, Y, yscatter, nrhs, nst, max_n, err);
  return cudaGetLastError();
}

}  // namespace

bool fx_gemm_supported(int max_n) {
  return max_n <= kFxMaxBlocks * kFxTile && FxSmem(max_n, 1).total(kFxFewWarps, 1) <= kFxSmemCap;
}

cudaError_t launch_fx_quantize(const WorkItem* items, int n_items, const FxForm& A, int32_t* halves, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  k_fx_quantize<<<std::min(n_items, 8 * num_sms()), 256, 0, st>>>(items, n_items, A.values, A.rexp, A.shift,
                                                                  reinterpret_cast<int2*>(halves));
  return cudaGetLastError();
}

cudaError_t launch_fx_gemm(const WorkItem* items, int n_items, int max_n, double share, const FxForm& A, const double* X,
                           double* Y, const int32_t* yscatter, int nrhs, int32_t* err, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  if (!fx_gemm_supported(max_n)) return cudaErrorInvalidValue;
  // columns per unit: the most that nrhs fills and shared memory holds
  int nc = nrhs > 4 ? 8 : nrhs > 2 ? 4 : nrhs;
  while (nc > 1 && FxSmem(max_n, nc).total(kFxWarps, 1) > kFxSmemCap) nc /= 2;
  // slices: so that the largest unit is at most an SM's share of the work, or
  // half of it at several columns, where the second reading of the tiles costs
  // nothing (216 operators of 343 rows on 152 SMs: 35 us with 1 slice and 43
  // with 2 at one column, 146 with 2, 156 with 1 and 162 with 3 at 8)
  const int ncb = (nrhs + nc - 1) / nc;
  const int S = (int)std::min<double>((max_n + kFxTile - 1) / kFxTile,
                                      std::max(1.0, std::ceil((nrhs > 1 ? 2.0 : 1.0) * share * num_sms() / ncb - 0.01)));
  switch (nc) {
    case 8: return run_fx<8>(items, n_items, max_n, S, A, X, Y, yscatter, nrhs, err, st);
    case 4: return run_fx<4>(items, n_items, max_n, S, A, X, Y, yscatter, nrhs, err, st);
    case 2: return run_fx<2>(items, n_items, max_n, S, A, X, Y, yscatter, nrhs, err, st);
    default: return run_fx<1>(items, n_items, max_n, S, A, X, Y, yscatter, nrhs, err, st);
  }
}

}  // namespace bddc
