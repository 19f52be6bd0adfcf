// Float32 local operators times blocks of right-hand sides on the CUDA cores
// (sm_103a): Y = Op X for the operators of all subdomains, row-major, rows padded
// to 16 bytes.
//
// What bounds it: the float32 pipe (32 columns: 8 FMAs per operator byte). The
// streamed GEMV (bddc_bgemv_tma.cu) keeps the whole operand of an operator in
// shared memory, so operators of 1000 rows and more run with 4 columns per pass
// and one block per SM, at 3 % of that pipe's rate. Here the operand is cut along
// the operator's columns like the operator itself: a unit is RT rows of one
// operator times 8 CB columns, and a ring stage holds kFgK of the operator's
// columns for both, fetched by 16-byte asynchronous copies of all threads two
// stages ahead, on into the next unit. (Bulk copies of one 512-byte row piece
// each ran at 1.2 TB/s.)
//
// Summation order, kept from the streamed GEMV so that the results are the same
// values: a sum over an operator row is 16 partial sums, lane g of a half warp
// taking the 16-byte vectors g, g + 16, .. in ascending order, then a binary tree
// over the lanes (8, 4, 2, 1 apart). A lane holds 8 rows x 8 columns of partial
// sums: 256 FMAs for 16 shared-memory loads.
//
// The operand is converted to float32 once per launch (k_fg_pack) into blocks
// of 4 rows x 8 columns padded to 144 bytes, which spreads the 16 lanes' reads
// over the banks.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "async.cuh"
#include "kernels.cuh"

namespace bddc {

namespace {

constexpr int kFgK = 128;              // operator columns per stage
constexpr int kFgCols = 8;             // right-hand sides per column block
constexpr int kFgBlk = 36;             // floats of an operand block: 4 rows x 8 columns, and 4 of padding
constexpr int kFgStages = 3;
constexpr int kFgRows = 8;             // rows per lane
constexpr int kFgLanes = 16;           // lanes per row

// Shape of a unit: NW warps, CB column blocks; a warp takes 16 rows of one of them.
template <int NW, int CB> struct FgShape {
  static constexpr int RT = 16 * NW / CB;
  static constexpr int a_bytes = RT * kFgK * 4;
  static constexpr int x_bytes = CB * (kFgK / 4) * kFgBlk * 4;
  static constexpr int stage = a_bytes + x_bytes;
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Operand of operator s: n rows from xoff, packed from block xblk on, for every
// column block (cstride floats apart); rows beyond n and columns beyond nrhs are 0.
__global__ void __launch_bounds__(256) k_fg_pack(const FgOperand* __restrict__ ops, int n_ops, int nrhs, int ncb,
                                                 int64_t cstride, const double* __restrict__ X, float* __restrict__ P) {
  for (int s = blockIdx.x; s < n_ops; s += gridDim.x) {
    const FgOperand w = ops[s];
    const int rows = (w.n + 3) / 4 * 4, wc = ncb * kFgCols;
    for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < rows * wc; i += gridDim.y * blockDim.x) {
      const int c = i / wc, k = i - c * wc;
      const float v = c < w.n && k < nrhs ? (float)X[(int64_t)(w.xoff + c) * nrhs + k] : 0.0f;
      P[(k / kFgCols) * cstride + (int64_t)(w.xblk + c / 4) * kFgBlk + (c % 4) * kFgCols + k % kFgCols] = v;
    }
  }
}

template <int NW, int CB>
__global__ void __launch_bounds__(NW * 32, 16 / NW)
    k_fgemm(const FgItem* __restrict__ items, int n_items, int ncg, const float* __restrict__ arena,
            const float* __restrict__ P, int64_t cstride, double* __restrict__ Y,
            const int32_t* __restrict__ yscatter, int nrhs) {
  using Sh = FgShape<NW, CB>;
  constexpr int kFgWarps = NW, kFgThreads = NW * 32;
  extern __shared__ __align__(128) unsigned char smem[];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int ncb = (nrhs + kFgCols - 1) / kFgCols;   // column blocks in all
  const int total = n_items * ncg;
  const uint32_t base = smem_addr(smem);

  // the stage to be fetched next: unit fu, operator column fc
  int fu = blockIdx.x, fc = 0, fslot = 0;
  FgItem fw{};
  if (fu < total) fw = items[fu / ncg];
  auto fetch = [&]() {
    if (fu < total) {
      const uint32_t st = base + (uint32_t)fslot * Sh::stage;
      const int kv = min(kFgK, fw.lda - fc) / 4;   // vectors of a row in this stage
      const float* A = arena + fw.moff + (int64_t)fw.row0 * fw.lda + fc;
      if (lane < kv)
#pragma unroll
        for (int r = 0; r < Sh::RT / kFgWarps; ++r) {   // a warp per row: 32 vectors
          const int row = r * kFgWarps + warp;
          if (row < fw.nrows) cp_async16(st + (uint32_t)(row * kFgK + lane * 4) * 4u, A + (int64_t)row * fw.lda + lane * 4);
        }
      const int cb0 = (fu % ncg) * CB, ncu = min(CB, ncb - cb0);
      const int xv = kv * (kFgBlk / 4);                 // vectors of a column block's operand
      for (int q = 0; q < ncu; ++q) {
        const float* X = P + (cb0 + q) * cstride + (int64_t)(fw.xblk + fc / 4) * kFgBlk;
        for (int i = t; i < xv; i += kFgThreads)
          cp_async16(st + Sh::a_bytes + (uint32_t)(q * (kFgK / 4) * kFgBlk + i * 4) * 4u, X + i * 4);
      }
      fc += kFgK;
      if (fc >= fw.lda) {
        fc = 0;
        fu += gridDim.x;
        if (fu < total) fw = items[fu / ncg];
      }
    }
    cp_async_commit();   // (an empty group where nothing is left, so that groups count stages)
    if (++fslot == kFgStages) fslot = 0;
  };
  for (int s = 0; s < kFgStages - 1; ++s) fetch();

  const int cb = warp % CB, rg = warp / CB;                    // column block, group of 16 rows
  const int gl = lane % kFgLanes, half = lane / kFgLanes;      // vector class, 8 of the 16 rows
  const int r0 = rg * 16 + half * kFgRows;
  int slot = 0;
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const FgItem w = items[u / ncg];
    const int k0 = ((u % ncg) * CB + cb) * kFgCols;            // first right-hand side of this warp
    const bool idle = k0 >= nrhs || rg * 16 >= w.nrows;
    float acc[kFgRows * kFgCols];
#pragma unroll
    for (int e = 0; e < kFgRows * kFgCols; ++e) acc[e] = 0.0f;
    for (int c0 = 0; c0 < w.lda; c0 += kFgK) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kFgStages - 2) : "memory");
      __syncthreads();   // the stage has landed for all; the one before it is read by all
      fetch();           // (into that one's slot)
      if (!idle) {
        const unsigned char* st = smem + slot * Sh::stage;
        const float* A = reinterpret_cast<const float*>(st) + r0 * kFgK + gl * 4;
        const float* Xb = reinterpret_cast<const float*>(st + Sh::a_bytes) + (cb * (kFgK / 4) + gl) * kFgBlk;
        const int kc = min(kFgK, w.lda - c0);
#pragma unroll
        for (int h = 0; h < kFgK / 64; ++h)
          if (h * 64 + gl * 4 < kc) {   // (all lanes, but in an operator's last stage)
            float4 a[kFgRows];
#pragma unroll
            for (int r = 0; r < kFgRows; ++r) a[r] = *reinterpret_cast<const float4*>(A + h * 64 + r * kFgK);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              float x[kFgCols];
#pragma unroll
              for (int q = 0; q < kFgCols; q += 4) {
                const float4 y = *reinterpret_cast<const float4*>(Xb + h * 16 * kFgBlk + v * kFgCols + q);
                x[q] = y.x; x[q + 1] = y.y; x[q + 2] = y.z; x[q + 3] = y.w;
              }
#pragma unroll
              for (int r = 0; r < kFgRows; ++r) {
                const float av = v == 0 ? a[r].x : v == 1 ? a[r].y : v == 2 ? a[r].z : a[r].w;
#pragma unroll
                for (int k = 0; k < kFgCols; ++k) acc[r * kFgCols + k] = fmaf(av, x[k], acc[r * kFgCols + k]);
              }
            }
          }
      }
      if (++slot == kFgStages) slot = 0;
    }
    if (idle) continue;
    // the tree over the 16 lanes; lane gl keeps entries 4 gl .. 4 gl + 3 (row
    // gl / 2 of its 8, columns 4 (gl & 1) ..)
#pragma unroll
    for (int o = kFgLanes / 2, n = kFgRows * kFgCols; o >= 1; o >>= 1, n >>= 1) {
      const bool upper = (gl & o) != 0;
#pragma unroll
      for (int i = 0; i < n / 2; ++i) {
        const float send = upper ? acc[i] : acc[i + n / 2];
        const float keep = upper ? acc[i + n / 2] : acc[i];
        acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    const int row = r0 + gl / 2;
    if (row < w.nrows) {
      const int64_t jy = (int64_t)w.yoff + w.row0 + row;
      double* out = Y + (yscatter ? (int64_t)yscatter[jy] : jy) * nrhs;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = k0 + 4 * (gl & 1) + i;
        if (k < nrhs) out[k] = (double)acc[i];
      }
    }
  }
  cp_async_wait_all();
}

template <int NW, int CB>
cudaError_t run_fgemm(const FgOperators& F, const float* P, int64_t cstride, double* Y, const int32_t* yscatter,
                      int nrhs, cudaStream_t st) {
  using Sh = FgShape<NW, CB>;
  constexpr int cls = Sh::RT == 32 ? 0 : Sh::RT == 64 ? 1 : 2;
  static_assert(Sh::RT == 32 << cls, "row tiles of the item lists");
  constexpr int smem = kFgStages * Sh::stage;
  auto kern = k_fgemm<NW, CB>;
  cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  const int ncg = (nrhs + kFgCols * CB - 1) / (kFgCols * CB);
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NW * 32, smem);
  if (e != cudaSuccess) return e;
  const int grid = std::max(1, std::min(F.n_items[cls] * ncg, std::max(per_sm, 1) * num_sms()));
  kern<<<grid, NW * 32, smem, st>>>(F.items[cls], F.n_items[cls], ncg, F.arena, P, cstride, Y, yscatter, nrhs);
  return cudaGetLastError();
}

}  // namespace

size_t fgemm_operand_floats(int64_t blocks, int nrhs_max) {
  return (size_t)blocks * kFgBlk * ((nrhs_max + kFgCols - 1) / kFgCols);
}

cudaError_t launch_fgemm(const FgOperators& F, float* P, const double* X, double* Y, const int32_t* yscatter, int nrhs,
                         cudaStream_t st) {
  if (F.n_ops == 0) return cudaSuccess;
  const int ncb = (nrhs + kFgCols - 1) / kFgCols;
  const int64_t cstride = F.blocks * kFgBlk;
  const int per = std::max(1, std::min(8, 4 * num_sms() / F.n_ops));
  k_fg_pack<<<dim3(std::min(F.n_ops, 4 * num_sms()), per), 256, 0, st>>>(F.ops, F.n_ops, nrhs, ncb, cstride, X, P);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // long row tiles share the operand, short ones give more units: blocks of two
  // warps per column block where the long ones would leave SMs idle
  const int room = 2 * num_sms();
  if (ncb == 1)
    return F.n_items[2] >= room ? run_fgemm<8, 1>(F, P, cstride, Y, yscatter, nrhs, st)
                                : run_fgemm<2, 1>(F, P, cstride, Y, yscatter, nrhs, st);
  if (ncb == 2)
    return F.n_items[1] >= room ? run_fgemm<8, 2>(F, P, cstride, Y, yscatter, nrhs, st)
                                : run_fgemm<4, 2>(F, P, cstride, Y, yscatter, nrhs, st);
  return run_fgemm<8, 4>(F, P, cstride, Y, yscatter, nrhs, st);
}

}  // namespace bddc
