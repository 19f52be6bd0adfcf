// Float64 local operators in block fixed point (fx.hpp): the operators A_II^-1
// and K_GG of every subdomain as lower triangles of tiles, times a block of
// right-hand sides (sm_103a).
//
// What bounds it: as float64 the pass is bound by the 2 FMAs per SM and clock
// of GB300's float64 pipe, far below HBM. In fixed point a stored entry costs
// 6 integer multiply-adds (3 for its row's and 3 for its column's product, 32
// lanes per SM and clock), about half of the time its 8 bytes take from HBM, so
// storing the triangle pays and HBM is the bound again at one column. From two
// columns on the integer multiply-adds are (3 per full entry and column against
// one float64 FMA at a sixteenth of their rate).
//
// Scales. Operator entry (i, j) is held relative to 2^(e_i + e_j), e_i the
// exponent of row i (about that of sqrt(a_ii): both operators are symmetric
// and, in exact arithmetic, positive semidefinite, so |a_ij| <= sqrt(a_ii
// a_jj)); the operand is scaled by 2^e_j entry by entry and rounded to
// 58 bits of its largest scaled entry when it is staged, and a result is
// scaled by 2^e_i when it is converted back.
//
// Layout. Entries are {low, high} halves, 8 bytes, in tiles of 32 x 32 (8 KB):
// tile (I, J), J <= I, at position I (I + 1) / 2 + J, the diagonal ones whole,
// rows and columns beyond n zero. Within a tile, vector v (two entries) of row
// r stands at v ^ (r & 7), which makes reading a row across lanes and one
// vector of 8 rows across lanes both free of bank conflicts.
//
// Split. One block of 12 warps owns one unit, an operator and up to NC columns,
// at a time; the tiles are dealt
// to the warps, and every warp streams its own ones through a private ring of
// bulk copies that runs on into the next unit, so no warp waits for another
// one but at a unit's end. A tile is read twice from shared
// memory, so that neither use needs a reduction across the warp: once with a
// row per lane (its row's products with x_J), once with two columns per lane
// (the products with x_I of the mirrored tile). The sums go to shared
// memory with 32-bit integer atomics that nothing waits for: exact, so the
// result depends on no order.
// Measured on 1728 operators of 343 rows at one column: 171 us, 5.45 TB/s of
// stored entries (the float64 kernel: 401 us); with 8 warps of 3 tiles 10 %
// longer, with 6 of 4 30 %. At 8 columns 844 us, 65 % of the integer multiply-add
// rate (the float64 kernel: 3650 us). (Row-major triangles with whole rows per
// warp, in four forms, took 270 to 430 us at one column, against 133 us for
// streaming them alone: rows of many lengths cost more instructions in control
// and reductions than in products.)
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <memory>
#include <thread>
#include <vector>

#include "async.cuh"
#include "fx.hpp"
#include "kernels.cuh"

namespace bddc {

namespace {
constexpr int kFxWarps = 12;
constexpr int kFxThreads = kFxWarps * 32;
constexpr int kFxTile = 32;
constexpr int kFxTileBytes = kFxTile * kFxTile * 8;
constexpr int kFxMaxSlots = 2;              // tiles in flight per warp
constexpr int kFxSmemCap = 222 * 1024;
#ifndef BAL
#define BAL 1.0
#define BAL8 2.0
#define FXW 12
#endif
static_assert(kFxTile == kFxBlock, "sums run over the rows and columns of a tile");

__host__ __device__ __forceinline__ int fx_tiles(int n) {
  const int t = (n + kFxTile - 1) / kFxTile;
  return t * (t + 1) / 2;
}
// Entry (g, c) of an operator, in entries; c / 32 <= g / 32.
__host__ __device__ __forceinline__ int64_t fx_entry(int g, int c) {
  const int I = g / kFxTile, J = c / kFxTile, r = g % kFxTile, k = c % kFxTile;
  return (int64_t)(I * (I + 1) / 2 + J) * (kFxTile * kFxTile) + r * kFxTile + (((k / 2) ^ (r & 7)) * 2 + k % 2);
}

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

__device__ __forceinline__ int64_t shfl_xor64(int64_t v, int o) {
  int lo = (int)v, hi = (int)(v >> 32);
  lo = __shfl_xor_sync(0xffffffffu, lo, o);
  hi = __shfl_xor_sync(0xffffffffu, hi, o);
  return (int64_t)((uint32_t)lo) | ((int64_t)hi << 32);
}

// Shared memory of one block after the rings, in this order; npad = the
// largest operator padded to whole tiles.
struct FxSmem {
  int npad, nc;
  __host__ __device__ FxSmem(int max_n, int nc_) : npad((max_n + kFxTile - 1) / kFxTile * kFxTile), nc(nc_) {}
  __host__ __device__ size_t total(int nst) const {
    // per column: operand halves, totals (12 bytes), next operand; the
    // operator's row exponents, barriers
    return (size_t)kFxWarps * nst * (kFxTileBytes + 8) + (size_t)npad * ((8 + 12 + 8) * nc + 4);
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
// Cursor over the tasks of one warp: tasks warp, warp + kFxWarps, .. of unit
// u, then those of the block's next unit.
struct FxCursor {
  int u, t, nt;          // unit, task, tasks of the unit
  int T, s;              // tile rows of its operator, its slice
  const int2* base;      // the operator's tiles
};

// Y = Op X.
template <int NC>
__global__ void __launch_bounds__(kFxThreads, 1)
    k_fx_gemm(const WorkItem* __restrict__ items, FxUnits U, const int2* __restrict__ arena,
              const int32_t* __restrict__ rexp, const double* __restrict__ X, double* __restrict__ Y,
              const int32_t* __restrict__ yscatter, int nrhs, int nst, int max_n, int32_t* __restrict__ err) {
  constexpr int NG = NC < 4 ? NC : 4;   // columns whose sums are held at once
  extern __shared__ __align__(128) unsigned char smem[];
  const FxSmem L(max_n, NC);
  const int npad = L.npad, n_units = U.count();
  int2* xq = reinterpret_cast<int2*>(smem + (size_t)kFxWarps * nst * kFxTileBytes);   // operand halves [NC][npad]
  double* xraw = reinterpret_cast<double*>(xq + NC * npad);                           // next operand
  uint64_t* bars = reinterpret_cast<uint64_t*>(xraw + NC * npad);
  uint32_t* sums = reinterpret_cast<uint32_t*>(bars + kFxWarps * nst);                // totals [3][NC][npad]
  int32_t* xexp = reinterpret_cast<int32_t*>(sums + 3 * NC * npad);                   // row exponents of the next operand
  __shared__ int xe[2][NC];   // exponents of the columns of this operand and the next
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint64_t* full = bars + warp * nst;
  unsigned char* ring = smem + (size_t)warp * nst * kFxTileBytes;

  if (tid == 0) {
    for (int s = 0; s < kFxWarps * nst; ++s) mbar_init(&bars[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const int lim = NC * npad;
  for (int i = tid; i < 3 * lim; i += kFxThreads) sums[i] = 0;
  auto add = [&](int at, int64_t hi, uint32_t f) {
    atomicAdd(&sums[at], f);
    atomicAdd(&sums[lim + at], fx_limb0(hi));
    atomicAdd(&sums[2 * lim + at], (uint32_t)fx_limb1(hi));
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
    if ((in.t += kFxWarps) >= in.nt) {
      in.u += gridDim.x;
      in.t = warp;
      enter(in);
    }
  };
  auto prefetch_operand = [&](int uu) {
    const WorkItem wn = items[U.item(uu)];
    const int k0 = U.col(uu) * NC, nk = min(NC, nrhs - k0);
    for (int j = tid; j < NC * npad; j += kFxThreads) {
      const int i = j / NC, k = j - i * NC;
      if (i < wn.ncols && k < nk)
        cp_async8(xraw + k * npad + i, X + (int64_t)(wn.xoff + i) * nrhs + k0 + k);
      else
        xraw[k * npad + i] = 0.0;
    }
    for (int i = tid; i < npad; i += kFxThreads) {
      if (i < wn.ncols)
        cp_async4(xexp + i, rexp + wn.yoff + i);
      else
        xexp[i] = 0;
    }
    cp_async_commit();
  };
  // Two block barriers per unit at one column: (A) all sums added and the
  // next operand landed, (B) the next operand converted, the sums cleared and
  // xraw free. The exponents of the columns come between them: at one column
  // every warp takes the maximum over the whole operand by itself, at several
  // the warps share them out and a third barrier follows.
  int par = 0;
  auto convert_operand = [&](int p) {
    for (int k = NC == 1 ? 0 : warp; k < NC; k += NC == 1 ? 1 : kFxWarps) {
      int E = kFxZero;
      for (int i = lane; i < npad; i += 32) {
        const int e = fx_exponent((uint64_t)__double_as_longlong(xraw[k * npad + i]));
        E = max(E, e == kFxNonFinite || e == kFxZero ? e : e + xexp[i]);
      }
      E = __reduce_max_sync(0xffffffffu, E);
      if (lane == 0) xe[p][k] = E;
    }
    if (NC > 1) __syncthreads();
    else __syncwarp();
    for (int j = tid; j < NC * npad; j += kFxThreads) {
      const int k = NC == 1 ? 0 : j / npad, i = NC == 1 ? j : j - k * npad, E = xe[p][k];
      int64_t q = 0;
      if (E != kFxZero && E != kFxNonFinite)
        q = fx_quantize((uint64_t)__double_as_longlong(xraw[j]), kFxBits - E + xexp[i]);
      xq[j] = make_int2(fx_lo(q), fx_hi(q));
    }
  };

  __syncthreads();   // barriers initialised, sums cleared
  for (int s = 0; s < nst; ++s) issue();
  if (blockIdx.x < n_units) {
    prefetch_operand(blockIdx.x);
    cp_async_wait_all();
    __syncthreads();                          // operand landed
    convert_operand(par);
    __syncthreads();                          // xq complete; xraw free
    if (blockIdx.x + (int)gridDim.x < n_units) prefetch_operand(blockIdx.x + gridDim.x);
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
    int I = 0, first = 0;   // S = 1: tile row of t, and its first tile
    for (int t = warp; t < nt; t += kFxWarps) {
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
            int64_t hi;
            uint32_t f;
            fx_block_sum(h[k][0], m[k][0], h[k][1], m[k][1], hi, f);
            add((g + k) * npad + I * kFxTile + lane, hi, f);
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
            int64_t hi;
            uint32_t f;
            fx_block_sum(up ? h[k][1] : h[k][0], up ? m[k][1] : m[k][0], ho, mo, hi, f);
            add((g + k) * npad + J * kFxTile + 2 * (lane & 15) + up, hi, f);
          }
        }
      }
      __syncwarp();   // the tile is read: its slot may be refilled
      issue();
      if (++slot == nst) { slot = 0; phase ^= 1u; }
    }
    cp_async_wait_all();                      // this thread's copies of the next operand landed
    __syncthreads();                          // A: sums added; xq no longer read
    for (int j = tid; j < NC * n; j += kFxThreads) {
      const int c = j / NC, k = j - c * NC, at = k * npad + c, E = xe[par][k];
      if (U.S > 1 && c / kFxTile % U.S != sl) continue;
      const int64_t jy = (int64_t)w.yoff + c;
      const int ec = rexp[jy];
      double y = 0.0;
      if (E == kFxNonFinite) {
        // an operand with an infinity or NaN: the float64 products themselves
        for (int i = 0; i < n && k < nk; ++i) {
          const int2 a = arena[w.moff + fx_entry(max(c, i), min(c, i))];
          const double q = (double)(((int64_t)a.y << kFxLow) + a.x);
          y = fma(scalbn(q, ec + rexp[w.yoff + i] - kFxBits), X[(int64_t)(w.xoff + i) * nrhs + k0 + k], y);
        }
      } else if (E != kFxZero) {
        y = fx_value(fx_total(sums[lim + at], (int32_t)sums[2 * lim + at]), sums[at], fx_unit(ec, E));
      }
      sums[at] = sums[lim + at] = sums[2 * lim + at] = 0;
      if (k < nk) Y[(yscatter ? (int64_t)yscatter[jy] : jy) * nrhs + k0 + k] = y;
    }
    par ^= 1;
    if (has_next) convert_operand(par);
    __syncthreads();                          // B: xq complete; sums and xraw free
    if (u + 2 * (int)gridDim.x < n_units) prefetch_operand(u + 2 * gridDim.x);
  }
  cp_async_wait_all();
  // after a timeout: this warp's copies in flight land before the block exits
  for (; aborted && flying > 0; --flying) {
    if (!mbar_wait(&full[slot], phase)) break;
    if (++slot == nst) { slot = 0; phase ^= 1u; }
  }
}

template <int NC>
cudaError_t run_fx(const WorkItem* items, int n_items, int max_n, int S, const int2* arena, const int32_t* rexp,
                   const double* X, double* Y, const int32_t* yscatter, int nrhs, int32_t* err, cudaStream_t st) {
  const FxSmem L(max_n, NC);
  const int nst = L.total(kFxMaxSlots) <= (size_t)kFxSmemCap ? kFxMaxSlots : 1;
  const size_t smem = L.total(nst);
  cudaError_t e = cudaFuncSetAttribute(k_fx_gemm<NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const FxUnits U{n_items, (nrhs + NC - 1) / NC, S};
  // one block per SM: the rings take its shared memory
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)n_items * U.ncb * S, num_sms()));
  k_fx_gemm<NC><<<grid, kFxThreads, smem, st>>>(items, U, arena, rexp, X, Y, yscatter, nrhs, nst, max_n, err);
  return cudaGetLastError();
}

}  // namespace

int64_t fx_packed_elems(int n) { return (int64_t)fx_tiles(n) * (kFxTile * kFxTile); }

bool fx_gemm_supported(int max_n) {
  return max_n <= kFxMaxBlocks * kFxTile && FxSmem(max_n, 1).total(1) <= (size_t)kFxSmemCap;
}

// S = (A + A^T) / 2 by tiles (the transposed reads stay in cache), row-major.
static void fx_symmetric_part(const double* A, int n, double* S) {
  for (int i0 = 0; i0 < n; i0 += kFxTile)
    for (int j0 = 0; j0 <= i0; j0 += kFxTile)
      for (int i = i0; i < std::min(n, i0 + kFxTile); ++i)
        for (int j = j0; j < std::min(n, j0 + kFxTile); ++j) {
          const double v = 0.5 * (A[(size_t)i * n + j] + A[(size_t)j * n + i]);
          S[(size_t)i * n + j] = v;
          S[(size_t)j * n + i] = v;
        }
}

// Row exponents of the symmetric S.
static void fx_row_scales(const double* S, int n, int32_t* e) {
  // |s_ij| < 2^(e_i + e_j): from the diagonal, raised where rounding (or a
  // row that vanishes in exact arithmetic) breaks the bound of the semidefinite case
  auto exponent = [](double v) {
    uint64_t b;
    std::memcpy(&b, &v, 8);
    return fx_exponent(b);
  };
  for (int i = 0; i < n; ++i) {
    const double d = S[(size_t)i * n + i];
    e[i] = d != 0.0 ? (exponent(d) + 2049) / 2 - 1024 : -400;
  }
  std::vector<double> inv(n), size(n);
  for (int i = 0; i < n; ++i) size[i] = std::ldexp(1.0, e[i]);
  for (int i = 0; i < n; ++i) {
    const double* row = S + (size_t)i * n;
    for (int j = 0; j < i; ++j) {
      if (std::fabs(row[j]) < size[i] * size[j]) continue;   // the common case
      const int need = exponent(row[j]) - e[i] - e[j];
      if (need <= 0) continue;
      const int up = e[i] < e[j] ? i : j;
      e[up] += need;
      size[up] = std::ldexp(1.0, e[up]);
    }
  }
  // the largest absolute sums of a row, over one block and in all, in units
  // of the scales
  for (int i = 0; i < n; ++i) inv[i] = std::ldexp(1.0, -e[i]);
  double block = 0.0, most = 0.0;
  for (int i = 0; i < n; ++i) {
    const double* row = S + (size_t)i * n;
    double all = 0.0;
    for (int j0 = 0; j0 < n; j0 += kFxBlock) {
      double s = 0.0;
      for (int j = j0; j < std::min(n, j0 + kFxBlock); ++j) s += std::fabs(row[j]) * inv[j];
      block = std::max(block, s * inv[i]);
      all += s;
    }
    most = std::max(most, all * inv[i]);
  }
  int up = 0;
  while (up < 16 && (block > (double)kFxBlockSum * (1 << (2 * up)) || most > (double)kFxRowSum * (1 << (2 * up)))) ++up;
  for (int i = 0; i < n; ++i) e[i] += up;
}

void fx_pack_lower(const std::vector<std::vector<double>>& ops, const std::vector<int>& dims,
                   const std::vector<int32_t>& voff, int threads, std::vector<int64_t>& off,
                   std::unique_ptr<int2[]>& arena, int64_t& elems, std::vector<int32_t>& rexp) {
  off.assign(ops.size(), 0);
  int64_t cur = 0, rows = 0;
  for (size_t s = 0; s < ops.size(); ++s) {
    off[s] = cur;   // (whole tiles: 8 KB blocks)
    cur += fx_packed_elems(dims[s]);
    rows = std::max<int64_t>(rows, (int64_t)voff[s] + dims[s]);
  }
  elems = std::max<int64_t>(cur, 1);
  arena.reset(new int2[elems]);   // (every entry is written below, by the threads)
  rexp.assign((size_t)std::max<int64_t>(rows, 1), 0);
  auto work = [&](int t, int nt) {
    std::vector<double> S;
    for (size_t s = t; s < ops.size(); s += nt) {
      const int n = dims[s];
      int32_t* e = &rexp[voff[s]];
      if (n == 0) continue;
      S.resize((size_t)n * n);
      fx_symmetric_part(ops[s].data(), n, S.data());
      fx_row_scales(S.data(), n, e);
      int2* out = arena.get() + off[s];
      for (int I = 0; I * kFxTile < n; ++I)
        for (int J = 0; J <= I; ++J)
          for (int r = 0; r < kFxTile; ++r, out += kFxTile) {
            const int g = I * kFxTile + r, c0 = J * kFxTile;
            for (int k = 0; k < kFxTile; ++k) {
              int64_t q = 0;
              if (g < n && c0 + k < n) {
                uint64_t b;
                std::memcpy(&b, &S[(size_t)g * n + c0 + k], 8);
                if (b << 1) q = fx_quantize(b, kFxBits - e[g] - e[c0 + k]);
              }
              out[((k / 2) ^ (r & 7)) * 2 + k % 2] = make_int2(fx_lo(q), fx_hi(q));   // as fx_entry
            }
          }
    }
  };
  // a thread per 65536 entries, not more than asked for
  const int nt = (int)std::max<int64_t>(1, std::min<int64_t>(threads, cur >> 16));
  std::vector<std::thread> pool;
  for (int t = 1; t < nt; ++t) pool.emplace_back(work, t, nt);
  work(0, nt);
  for (auto& t : pool) t.join();
}

cudaError_t launch_fx_gemm(const WorkItem* items, int n_items, int max_n, double share, const void* arena,
                           const int32_t* rexp, const double* X, double* Y, const int32_t* yscatter, int nrhs,
                           int32_t* err, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  if (!fx_gemm_supported(max_n)) return cudaErrorInvalidValue;
  const int2* A = static_cast<const int2*>(arena);
  // columns per unit: the most that nrhs fills and shared memory holds
  int nc = nrhs > 4 ? 8 : nrhs > 2 ? 4 : nrhs;
  while (nc > 1 && FxSmem(max_n, nc).total(1) > (size_t)kFxSmemCap) nc /= 2;
  // slices: so that the largest unit is at most an SM's share of the work, or
  // half of it at several columns, where the second reading of the tiles costs
  // nothing (216 operators of 343 rows on 152 SMs: 35 us with 1 slice and 43
  // with 2 at one column, 146 with 2, 156 with 1 and 162 with 3 at 8)
  const int ncb = (nrhs + nc - 1) / nc;
  const int S = (int)std::min<double>((max_n + kFxTile - 1) / kFxTile,
                                      std::max(1.0, std::ceil((nrhs > 1 ? 2.0 : 1.0) * share * num_sms() / ncb - 0.01)));
  switch (nc) {
    case 8: return run_fx<8>(items, n_items, max_n, S, A, rexp, X, Y, yscatter, nrhs, err, st);
    case 4: return run_fx<4>(items, n_items, max_n, S, A, rexp, X, Y, yscatter, nrhs, err, st);
    case 2: return run_fx<2>(items, n_items, max_n, S, A, rexp, X, Y, yscatter, nrhs, err, st);
    default: return run_fx<1>(items, n_items, max_n, S, A, rexp, X, Y, yscatter, nrhs, err, st);
  }
}

}  // namespace bddc
