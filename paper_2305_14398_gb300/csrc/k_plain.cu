// Plain materialised form (sm_103a): stage 4 (Algorithm 2, the step unitary
// written out as a dense matrix) and stage 6 applied per step (eq. 11, dense
// matrix-vector product).  This is the baseline the fused kernel is measured
// against; both kernels stream the 2^n x 2^n complex64 matrix through HBM.
#include "checked.h"
#include "step_entry.h"
#include "tqs_internal.h"

namespace tqs {
namespace {

// S[r][c] = prod_f M_f[bits_f(r)][bits_f(c)] when r and c agree on every idle
// qubit (identity factors), else 0 (step_entry.h).  Factors are staged in
// shared memory.
constexpr int kMatThreads = 256;
constexpr int kMaxFactors = 16;

// Small matrices and few factors (expansion_pays): one product over the factors per entry.
__global__ void __launch_bounds__(kMatThreads)
    materialize_small_kernel(const StepFactor* __restrict__ factors, int nf, uint32_t idle, int n,
                       float2* __restrict__ S) {
  __shared__ StepFactor fs[kMaxFactors];
  for (int i = threadIdx.x; i < nf * static_cast<int>(sizeof(StepFactor) / 8); i += blockDim.x)
    reinterpret_cast<float2*>(fs)[TQS_IX(i, int(sizeof(fs) / 8))] =
        reinterpret_cast<const float2*>(factors)[i];
  __syncthreads();
  const int64_t N = int64_t(1) << n;
  const int64_t pairs = (N * N) >> 1;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < pairs; e += stride) {
    const int64_t flat = e << 1;
    const uint32_t r = static_cast<uint32_t>(flat >> n);
    const uint32_t c = static_cast<uint32_t>(flat & (N - 1));
    const float2 v0 = step_entry(fs, nf, idle, r, c);
    const float2 v1 = step_entry(fs, nf, idle, r, c + 1);
    __stcs(reinterpret_cast<float4*>(S) + TQS_IX(e, pairs), make_float4(v0.x, v0.y, v1.x, v1.y));
  }
}

// Larger matrices.  Per entry the product costs a complex multiply and an
// entry lookup per factor (n = 12, a layer of 12 single-qubit gates: 196 us,
// 0.68 TB/s written, bound by instruction issue), but entries of a row share
// their partial products: a row is expanded qubit by qubit, x(c | b << q) =
// x(c) f_q(r, c | b << q), where f_q is the entry of the factor whose highest
// qubit is q (1 where q is a lower qubit of its factor, the delta where it
// is idle).  The last expansion costs two multiplies per entry (one for each
// parent), all before it half as much again.  A block of 256 threads works 2^14
// entries (kRows rows, as many as fill it): every thread forms one product
// over the lowest n - 6 qubits, expands it by 3 qubits into shared memory, and
// then expands 8 of those by the top 3 qubits into the matrix, two neighbours
// at once, so that a warp's store covers 512 contiguous bytes.  Same matrix:
// 29 us, and n = 14 at 6.9 TB/s, the measured copy rate (n = 12, 13: 4.7, 6.3 TB/s).
// Where expansion is the faster: its time hardly depends on the factors (n = 10
// 9..11 us, n = 11 11..13 us, n = 12 25..29 us), the small kernel's grows with their
// number (n = 10, 2 to 6 factors 8.2..8.6 us, 8 9.9, 10 16.6; n = 11, 2 and 3 9.5 us, 4 12.0, 6
// 18.7; n = 12, 3 25.9 us, 6 60); n = 9 9 us against 12.
inline bool expansion_pays(int n, int factors) { return n >= 12 || (n == 11 && factors > 4) || (n == 10 && factors > 8); }
constexpr int kMatMid = 2048;  // entries of the 2^(n-3)-entry row parts of a block

// How the expansion by qubit q multiplies: the index of the factor whose
// highest qubit q is, or one of these.
constexpr int kLevelIdle = -1, kLevelCopy = -2;

__device__ __noinline__ float2 custom_entry(const StepFactor& f, uint32_t r, uint32_t c) {
  return factor_entry(f, r, c);
}

// x: the row's value with the qubits from q on left out (at column bits c);
// out[i]: with the 3 qubits q, q + 1, q + 2 at the bits of i.
__device__ __forceinline__ void expand3(const StepFactor* fs, const int* level, int q, uint32_t r, uint32_t c,
                                        float2 x, float2 (&out)[8]) {
  out[0] = x;
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    const int k = level[TQS_IX(q + l, 16)];
    const uint32_t bit = 1u << (q + l);
    if (k < 0) {
      const bool one = k == kLevelCopy || (r & bit) != 0, zero = k == kLevelCopy || (r & bit) == 0;
#pragma unroll
      for (int i = 0; i < (1 << l); ++i) {
        out[i | (1 << l)] = one ? out[i] : make_float2(0.f, 0.f);
        out[i] = zero ? out[i] : make_float2(0.f, 0.f);
      }
    } else if (fs[k].custom) {
#pragma unroll
      for (int i = 0; i < (1 << l); ++i) {
        const uint32_t ci = c | (static_cast<uint32_t>(i) << q);
        out[i | (1 << l)] = step_cmul(out[i], custom_entry(fs[k], r, ci | bit));
        out[i] = step_cmul(out[i], custom_entry(fs[k], r, ci));
      }
    } else if (fs[k].nq == 1) {
      const float2* m = fs[k].m + ((r & bit) ? 2 : 0);
      const float2 f0 = m[0], f1 = m[1];
#pragma unroll
      for (int i = 0; i < (1 << l); ++i) {
        out[i | (1 << l)] = step_cmul(out[i], f1);
        out[i] = step_cmul(out[i], f0);
      }
    } else {
      // the row's entries at this qubit's bit, for both bits of the partner
      const int q0 = fs[k].q0, q1 = fs[k].q1, part = q0 == q + l ? q1 : q0;
      const float2* m = fs[k].m + 4 * ((((r >> q0) & 1) << 1) | ((r >> q1) & 1));
      const int sb = q0 == q + l ? 2 : 1, sp = 3 - sb;
      const float2 f00 = m[0], f01 = m[sb], f10 = m[sp], f11 = m[3];
#pragma unroll
      for (int i = 0; i < (1 << l); ++i) {
        const bool p = ((c | (static_cast<uint32_t>(i) << q)) >> part) & 1;
        const float2 f0 = make_float2(p ? f10.x : f00.x, p ? f10.y : f00.y);
        const float2 f1 = make_float2(p ? f11.x : f01.x, p ? f11.y : f01.y);
        out[i | (1 << l)] = step_cmul(out[i], f1);
        out[i] = step_cmul(out[i], f0);
      }
    }
  }
}

__global__ void __launch_bounds__(kMatThreads)
    materialize_kernel(const StepFactor* __restrict__ factors, int nf, uint32_t idle, int n,
                       float2* __restrict__ S) {
  __shared__ StepFactor fs[kMaxFactors];
  __shared__ int level[16];
  __shared__ alignas(16) float2 mid[kMatMid];  // read two entries at a time
  const int t = threadIdx.x;
  for (int i = t; i < nf * static_cast<int>(sizeof(StepFactor) / 8); i += blockDim.x)
    reinterpret_cast<float2*>(fs)[TQS_IX(i, int(sizeof(fs) / 8))] =
        reinterpret_cast<const float2*>(factors)[i];
  if (t < 16) level[t] = ((idle >> t) & 1) ? kLevelIdle : kLevelCopy;
  __syncthreads();
  if (t < nf) level[31 - __clz(factor_qubits(fs[t]))] = t;
  __syncthreads();
  // 2^rq rows of 2^(n-3) mid entries in the block, from row r0
  const int mq = n - 3, rq = 11 - mq;
  const uint32_t r0 = blockIdx.x << rq;
  {
    // one product over the lowest n - 6 qubits, expanded by the next 3
    const int lq = n - 6;
    const uint32_t row = static_cast<uint32_t>(t) >> lq, c = static_cast<uint32_t>(t) & ((1u << lq) - 1);
    const uint32_t r = r0 + row;
    float2 x = make_float2(((r ^ c) & idle & ((1u << lq) - 1)) ? 0.f : 1.f, 0.f);
    for (int q = 0; q < lq; ++q)
      if (level[q] >= 0) x = step_cmul(x, custom_entry(fs[level[q]], r, c));
    float2 o[8];
    expand3(fs, level, lq, r, c, x, o);
#pragma unroll
    for (int i = 0; i < 8; ++i)
      mid[TQS_IX((row << mq) | (static_cast<uint32_t>(i) << lq) | c, kMatMid)] = o[i];
  }
  __syncthreads();
  const size_t NN = size_t(1) << (2 * n);
#pragma unroll 1
  for (int e = t; e < kMatMid / 2; e += kMatThreads) {
    const uint32_t row = static_cast<uint32_t>(2 * e) >> mq, c = static_cast<uint32_t>(2 * e) & ((1u << mq) - 1);
    const uint32_t r = r0 + row;
    const float4 m = reinterpret_cast<const float4*>(mid)[TQS_IX(e, kMatMid / 2)];
    float2 a[8], b[8];
    expand3(fs, level, mq, r, c, make_float2(m.x, m.y), a);
    expand3(fs, level, mq, r, c + 1, make_float2(m.z, m.w), b);
    float2* out = S + (static_cast<size_t>(r) << n) + c;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      (void)TQS_IX((static_cast<size_t>(r) << n) + c + (static_cast<size_t>(i) << mq) + 1, NN);
      __stcs(reinterpret_cast<float4*>(out + (static_cast<size_t>(i) << mq)),
             make_float4(a[i].x, a[i].y, b[i].x, b[i].y));
    }
  }
}

// y = S x: one warp per row, float4 (two amplitudes) per lane per iteration.
constexpr int kMvWarps = 8;

__global__ void __launch_bounds__(kMvWarps * 32)
    matvec_kernel(const float2* __restrict__ S, const float2* __restrict__ x,
                  float2* __restrict__ y, int n) {
  const int64_t N = int64_t(1) << n;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t row = int64_t(blockIdx.x) * kMvWarps + warp;
  if (row >= N) return;
  const float4* srow = reinterpret_cast<const float4*>(S) + TQS_IX(row, N) * (N >> 1);
  const float4* x4 = reinterpret_cast<const float4*>(x);
  float re = 0.f, im = 0.f;
  for (int64_t k = lane; k < (N >> 1); k += 32) {
    const float4 s = __ldcs(srow + TQS_IX(k, N >> 1));
    const float4 v = __ldg(x4 + TQS_IX(k, N >> 1));
    re = fmaf(s.x, v.x, re);
    re = fmaf(-s.y, v.y, re);
    re = fmaf(s.z, v.z, re);
    re = fmaf(-s.w, v.w, re);
    im = fmaf(s.x, v.y, im);
    im = fmaf(s.y, v.x, im);
    im = fmaf(s.z, v.w, im);
    im = fmaf(s.w, v.z, im);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, o);
    im += __shfl_xor_sync(0xffffffffu, im, o);
  }
  if (lane == 0) y[row] = make_float2(re, im);
}

}  // namespace

TQS_DEFINE_VIOLATIONS(violations_plain)

namespace {

int sm_count() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  return sms;
}

}  // namespace

cudaError_t launch_materialize(const StepFactor* d_factors, StepDesc step, int n, float2* d_S,
                               cudaStream_t s) {
  if (step.f_count > kMaxFactors) return cudaErrorInvalidValue;
  if (expansion_pays(n, step.f_count)) {
    materialize_kernel<<<1 << (2 * n - 14), kMatThreads, 0, s>>>(d_factors + step.f_begin, step.f_count,
                                                                 step.idle, n, d_S);
    count_launches(1);
    return cudaGetLastError();
  }
  const int64_t N = int64_t(1) << n;
  const int64_t pairs = (N * N) >> 1;
  int64_t blocks = (pairs + kMatThreads - 1) / kMatThreads;
  const int64_t cap = int64_t(sm_count()) * 8;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  materialize_small_kernel<<<static_cast<int>(blocks), kMatThreads, 0, s>>>(
      d_factors + step.f_begin, step.f_count, step.idle, n, d_S);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_matvec(const float2* d_S, const float2* d_x, float2* d_y, int n,
                          cudaStream_t s) {
  const int64_t N = int64_t(1) << n;
  const int64_t blocks = (N + kMvWarps - 1) / kMvWarps;
  matvec_kernel<<<static_cast<int>(blocks), kMvWarps * 32, 0, s>>>(d_S, d_x, d_y, n);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace tqs
