// Circuit unitary in FP32 on the CUDA cores (sm_103a): column j of U = S_m ...
// S_1 is the circuit applied to |j>, so a block of columns is a batch of
// copies of one fused program, each from its own basis state, which the fused
// kernel runs with the state in shared memory.  In the chain U <- S_k U
// (Algorithm 1) all but 2 or 4 terms of an entry's sum come from zero entries
// of S_k per factor; here only the others are formed.  The columns are written
// one after the other (rows of U^T) and then transposed into U.
//
// Against the chain as dense FP32 products (64 x 64 tiles, four real products):
// n = 10, 40 steps (20 layers of U3 and CNOTs): 8.95 ms before, 198 us now, n = 12
// 412 ms before, 3.0 ms now (bound by the fused kernel's instruction issue);
// error against FP64 3.5e-6 before, 4.9e-7 now (one rounding per rotation
// instead of a sum over 2^n terms per step).
#include <algorithm>

#include "checked.h"
#include "tqs_internal.h"

namespace tqs {
namespace {

// circs[i]: the program of *base from the basis state |col0 + i> (leading X
// gates are folded into the program's start index, which they flip).
__global__ void column_circs_kernel(const FusedCirc* __restrict__ base, FusedCirc* __restrict__ circs,
                                    int32_t* __restrict__ order, int col0, int ncols) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ncols) return;
  FusedCirc c = *base;
  c.gen_index ^= col0 + i;
  c.out_off = static_cast<int64_t>(i) << c.n;
  circs[TQS_IX(i, ncols)] = c;
  order[TQS_IX(i, ncols)] = i;
}

// U[r * ldu + j] = V[j][r] for j < M, r < N: 32 x 32 tiles through shared
// memory, so both sides move 256-byte runs.
__global__ void __launch_bounds__(256)
    transpose_kernel(const float2* __restrict__ V, float2* __restrict__ U, int N, int M, int64_t ldu) {
  __shared__ float2 t[32][33];
  const int r0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
  for (int k = threadIdx.y; k < 32; k += 8)
    if (j0 + k < M && r0 + static_cast<int>(threadIdx.x) < N)
      t[k][threadIdx.x] = V[TQS_IX(static_cast<size_t>(j0 + k) * N + r0 + threadIdx.x, static_cast<size_t>(M) * N)];
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += 8)
    if (r0 + k < N && j0 + static_cast<int>(threadIdx.x) < M)
      U[TQS_IX(static_cast<size_t>(r0 + k) * static_cast<size_t>(ldu) + j0 + threadIdx.x,
               static_cast<size_t>(N - 1) * static_cast<size_t>(ldu) + M)] = t[threadIdx.x][k];
}

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

}  // namespace

TQS_DEFINE_VIOLATIONS(violations_columns)

size_t columns_scratch_bytes(int n, int ncols) {
  return align256(size_t(ncols) * sizeof(FusedCirc)) + align256(size_t(ncols) * sizeof(int32_t)) + 256 +
         (size_t(ncols) << n) * sizeof(float2);
}

// Columns [col0, col0 + ncols) of the unitary of the program that L's arrays
// hold (its FusedCirc at L.circs), nint internal qubits, into d_U[r * ldu + j].
cudaError_t launch_columns(FusedLaunch L, int n, int nint, int col0, int ncols, float2* d_U, int64_t ldu,
                           void* scratch, int sms, cudaStream_t s) {
  char* p = static_cast<char*>(scratch);
  FusedCirc* circs = reinterpret_cast<FusedCirc*>(p);
  p += align256(size_t(ncols) * sizeof(FusedCirc));
  int32_t* order = reinterpret_cast<int32_t*>(p);
  p += align256(size_t(ncols) * sizeof(int32_t));
  L.counter = reinterpret_cast<int32_t*>(p);
  L.out = reinterpret_cast<float2*>(p + 256);
  cudaError_t e = cudaMemsetAsync(L.counter, 0, sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  column_circs_kernel<<<(ncols + 127) / 128, 128, 0, s>>>(L.circs, circs, order, col0, ncols);
  count_launches(1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  L.circs = circs;
  L.order = order;
  L.n_jobs = ncols;
  // a CTA per column, a thread per group of 16 amplitudes (from 2^14 on two
  // groups): a column's passes then take one round, and 512 threads' worth of
  // CTAs fill an SM's registers at every n
  L.team = TEAM_CTA;
  L.slice_q = nint;
  L.warps_per_cta = std::min(kCtaThreads, std::max(32, 1 << (nint - 4))) / 32;
  const int per_sm = std::max(1, fused_max_ctas_per_sm(TEAM_CTA, L.warps_per_cta, L.slice_q));
  L.grid = std::min(ncols, per_sm * sms);
  if ((e = launch_fused(L, s)) != cudaSuccess) return e;
  const int N = 1 << n;
  transpose_kernel<<<dim3((N + 31) / 32, (ncols + 31) / 32), dim3(32, 8), 0, s>>>(L.out, d_U, N, ncols, ldu);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace tqs
