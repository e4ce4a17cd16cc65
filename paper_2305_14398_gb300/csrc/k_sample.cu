// Inverse-CDF sampling of outcomes from probabilities (sm_103a): the collapse
// of simulateAndCollapse (Sec. 5.2), drawn according to p_i = |psi_i|^2
// (Sec. 2.1, eq. 2).
//
// A "segment" is one state's probability vector (one for tqs_sample, one per
// circuit for a batch), cut into blocks of 256 entries, each block into 32
// chunks of 8 consecutive entries.  The cumulative sums are defined by this
// file's summation order (FP64 on the global path; exact 64-bit fixed point,
// where the order does not matter, on the shared-memory path):
//   * chunk total: the chunk's 8 entries added in index order;
//   * chunk prefix in its block: exclusive warp scan of the 32 chunk totals
//     (Hillis-Steele, fixed order); the block total is the inclusive value of
//     the last chunk;
//   * block prefix: each thread of a CTA sums a contiguous run of block
//     totals, the runs are combined in order (warp scan, then warp totals);
//   * chunk base cbase_{b,l} = bpre_b + cpre_{b,l};
//   * C_i = cbase_{b,l} + p_{first of chunk} + ... + p_i.
// A shot with uniform u and target u T (T: the segment total) takes the last
// block b with bpre_b <= target, the last chunk l of it with cbase_{b,l} <=
// target, and the first entry i of that chunk with p_i > 0 and target <
// C_i.  If there is none (rounding, or u T >= T), the last index at or before
// that point with p_i > 0; -1 when every probability is 0.
//
// GB300's FP64 rate is about 1/64 of its FP32 rate, so the design keeps FP64
// operations few: on the global path the tables cost about 15 warp-wide FP64
// additions per 256 entries (the chunk bases bpre_b + cpre_{b,l} are stored
// absolute), and a shot is one multiply, binary searches that compare the FP64
// bit patterns as integers (the order of non-negative doubles), and at most 8
// adds; the shared-memory path needs one FP64 multiply per shot and nothing else.
// Two paths: segments of up to 2^13 entries are read by one CTA each, which
// builds exact tables in shared memory and runs every shot of the segment
// there; larger segments use three kernels over global memory (block tables,
// block prefix, shots).
#include "checked.h"
#include "tqs_internal.h"

namespace tqs {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kThreads = 256;
constexpr int kChunks = kSampleBlk / kSampleChunk;  // 32: one per lane
static_assert(kChunks == 32, "one chunk per lane");

// Non-negative FP64 values compared by their bit patterns (the same order).
__device__ __forceinline__ bool le_val(double a, double b) {
  return __double_as_longlong(a) <= __double_as_longlong(b);
}
__device__ __forceinline__ bool pos_val(double a) { return __double_as_longlong(a) > 0; }

template <class V>
__device__ __forceinline__ V warp_incl_scan(V x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const V y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

__device__ __forceinline__ int seg_of_block(const SampleSeg* segs, int nseg, int64_t gb) {
  int lo = 0, hi = nseg - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (segs[mid].blk_off <= gb) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Block b's tables (whole warp, lane = chunk): cpre[lane] = exclusive chunk
// prefix; returns the block total (same value in every lane).  `p` may be
// global or shared memory; entries past len count as 0.
template <class V>
__device__ __forceinline__ V block_tables(const V* p, int64_t len, int64_t b, int lane, V* cpre) {
  const int64_t i0 = b * kSampleBlk + int64_t(lane) * kSampleChunk;
  V t = V(0);
#pragma unroll
  for (int j = 0; j < kSampleChunk; ++j) t += (i0 + j < len) ? p[TQS_IX(i0 + j, len)] : V(0);
  const V incl = warp_incl_scan(t, lane);
  const V up = __shfl_up_sync(kFull, incl, 1);
  cpre[lane] = lane > 0 ? up : V(0);
  return __shfl_sync(kFull, incl, 31);
}

// Exclusive prefix bp[0..nb) of the block totals bs[0..nb) and their total
// *tot, by the kThreads threads of a CTA: thread t sums the contiguous run of
// ceil(nb / kThreads) blocks starting at t * that, the runs are combined by a
// warp scan and the warp totals in order, then each thread writes its run.
template <class V>
__device__ void block_prefix_cta(const V* bs, V* bp, int64_t nb, V* tot, V* wtot, V* wpre) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t chunk = (nb + kThreads - 1) / kThreads;
  const int64_t b0 = int64_t(t) * chunk;
  const int64_t b1 = b0 + chunk < nb ? b0 + chunk : nb;
  V s = V(0);
  for (int64_t b = b0; b < b1; ++b) s += bs[TQS_IX(b, nb)];
  const V incl = warp_incl_scan(s, lane);
  const V up = __shfl_up_sync(kFull, incl, 1);
  const V excl = lane > 0 ? up : V(0);
  if (lane == 31) wtot[TQS_IX(warp, kThreads / 32)] = incl;
  __syncthreads();
  if (t == 0) {
    V a = V(0);
    for (int w = 0; w < kThreads / 32; ++w) { wpre[w] = a; a += wtot[w]; }
  }
  __syncthreads();
  V acc = wpre[warp] + excl;
  for (int64_t b = b0; b < b1; ++b) {
    bp[TQS_IX(b, nb)] = acc;
    acc += bs[TQS_IX(b, nb)];
  }
  if (b0 < nb && b1 == nb) *tot = acc;
}

// Chunk prefixes of the blocks [0, nb) made absolute: cp[b * 32 + l] becomes
// bp[b] + cp[b * 32 + l] (whole CTA).
template <class V>
__device__ void absolute_chunks(const V* bp, V* cp, int64_t nb) {
  for (int64_t e = threadIdx.x; e < nb * kChunks; e += kThreads)
    cp[e] = bp[TQS_IX(e / kChunks, nb)] + cp[e];
}

// Last index <= i with p > 0, or -1 (one thread; reached only after rounding
// or for u T >= T).
template <class V>
__device__ int64_t last_nonzero_upto(const V* p, int64_t len, int64_t i) {
  for (; i >= 0; --i)
    if (pos_val(p[TQS_IX(i, len)])) return i;
  return -1;
}

// One shot (one thread).  p: the segment's entries; bp: its block prefix; cp:
// its absolute chunk bases (global or shared memory).
template <class V>
__device__ int64_t sample_shot(const V* p, int64_t len, const V* bp, const V* cp, int64_t nb, V T,
                               V target) {
  if (!(target < T)) return last_nonzero_upto(p, len, len - 1);
  int64_t lo = 0, hi = nb - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (le_val(bp[TQS_IX(mid, nb)], target)) lo = mid; else hi = mid - 1;
  }
  const int64_t b = lo;
  const V* cpb = cp + TQS_IX(b, nb) * kChunks;
  int l = 0, h = kChunks - 1;
  while (l < h) {
    const int mid = (l + h + 1) >> 1;
    if (le_val(cpb[TQS_IX(mid, kChunks)], target)) l = mid; else h = mid - 1;
  }
  const int64_t i0 = b * kSampleBlk + int64_t(l) * kSampleChunk;
  V c = cpb[TQS_IX(l, kChunks)];
  for (int j = 0; j < kSampleChunk && i0 + j < len; ++j) {
    const V x = p[TQS_IX(i0 + j, len)];
    c += x;
    if (pos_val(x) && !le_val(c, target)) return i0 + j;
  }
  const int64_t end = i0 + kSampleChunk - 1 < len - 1 ? i0 + kSampleChunk - 1 : len - 1;
  return last_nonzero_upto(p, len, end);
}

// ------------------------------------------------------------ global path

__global__ void __launch_bounds__(kThreads)
    block_tables_kernel(const SampleLaunch L) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = int64_t(gridDim.x) * (kThreads / 32);
  for (int64_t gb = int64_t(blockIdx.x) * (kThreads / 32) + (threadIdx.x >> 5); gb < L.nblocks;
       gb += warps) {
    const SampleSeg sg = L.gsegs[TQS_IX(seg_of_block(L.gsegs, L.n_gseg, gb), L.n_gseg)];
    (void)TQS_IX(sg.p_off + (int64_t(1) << sg.n) - 1, L.probs_len);
    const double t = block_tables(L.probs + sg.p_off, int64_t(1) << sg.n, gb - sg.blk_off, lane,
                                  L.cpre + TQS_IX(gb, L.nblocks) * kChunks);
    if (lane == 0) L.bsum[TQS_IX(gb, L.nblocks)] = t;
  }
}

__global__ void __launch_bounds__(kThreads)
    block_prefix_kernel(const SampleLaunch L) {
  __shared__ double wtot[kThreads / 32], wpre[kThreads / 32];
  const SampleSeg sg = L.gsegs[TQS_IX(blockIdx.x, L.n_gseg)];
  (void)TQS_IX(sg.blk_off + sample_blocks(sg.n) - 1, L.nblocks);
  block_prefix_cta(L.bsum + sg.blk_off, L.bpre + sg.blk_off, sample_blocks(sg.n),
                   L.tot + blockIdx.x, wtot, wpre);
  __syncthreads();
  absolute_chunks(L.bpre + sg.blk_off, L.cpre + int64_t(sg.blk_off) * kChunks, sample_blocks(sg.n));
}

__global__ void __launch_bounds__(kThreads)
    shots_kernel(const SampleLaunch L) {
  const int64_t total = int64_t(L.n_gseg) * L.shots;
  for (int64_t k = int64_t(blockIdx.x) * kThreads + threadIdx.x; k < total;
       k += int64_t(gridDim.x) * kThreads) {
    const int g = static_cast<int>(k / L.shots);
    const SampleSeg sg = L.gsegs[TQS_IX(g, L.n_gseg)];
    const int64_t kk = TQS_IX(sg.index * L.shots + (k - int64_t(g) * L.shots), L.n_segs * L.shots);
    const double T = L.tot[g];
    L.out[kk] = sample_shot(L.probs + sg.p_off, int64_t(1) << sg.n, L.bpre + sg.blk_off,
                            L.cpre + int64_t(sg.blk_off) * kChunks, sample_blocks(sg.n), T,
                            L.u[kk] * T);
  }
}

// ------------------------------------------------------ shared-memory path
// One CTA per segment (n <= kSampleSmemMaxQ).  Dynamic shared memory holds the
// segment's entries, 9 words to a chunk of 8 (kChunkPad), then a base per chunk.
//
// Here the cumulative sums are exact: each probability p becomes the 64-bit
// integer floor(p 2^S), with S chosen from an FP32 estimate of the segment's
// total T so that T 2^S stays below 2^61 (each entry then loses less than
// 2^-60 T, all of them together less than 2^(n - 60) T: 4e-15 T at n = 13; a
// probability below 2^-S counts as 0); the sums are integer additions, the
// same in any order, and a shot's target is floor(u T 2^S).  The FP64 pipe
// (1/64 of the FP32 rate on this GPU) is left to one multiply per shot.

// p as FP32 (truncated; 0 below the FP32 range), from the FP64 bits with
// integer operations only: for the estimate of the total.
__device__ __forceinline__ float approx_f32(unsigned long long bits) {
  const int e = static_cast<int>((bits >> 52) & 0x7FF);
  if (e < 1023 - 126) return 0.f;
  if (e > 1023 + 127) return __int_as_float(0x7f800000);
  return __int_as_float(((e - 1023 + 127) << 23) | static_cast<int>((bits >> 29) & 0x7FFFFF));
}

// floor(p 2^S) for a non-negative FP64 p given by its bits; S such that the
// result stays below 2^62.
__device__ __forceinline__ unsigned long long to_fixed(unsigned long long bits, int S) {
  const int e = static_cast<int>((bits >> 52) & 0x7FF);
  unsigned long long m = bits & ((1ull << 52) - 1);
  int ex = e;
  if (e == 0) ex = 1;        // subnormal: no implicit bit
  else m |= 1ull << 52;
  const int sh = ex - 1075 + S;  // p = m 2^(ex - 1075)
  if (sh >= 0) return m << sh;
  if (sh <= -64) return 0ull;
  return m >> (-sh);
}

//
// A thread owns K consecutive chunks in registers: it loads them (64 bytes a
// chunk), converts them once S is known, and the chunk bases come from one
// scan over the threads, so the entries cross shared memory once (written,
// 9 words to a chunk of 8 so that neither the 64-bit stores nor a shot's
// reads collide) and the block meets at three barriers.  With the entries
// staged first, converted in place and summed in strides of 8 (16-way bank
// conflicts), 16384 states of 2^11 entries and 64 shots took 158 us; now
// 96 us (2.8 TB/s read), 16000 states of 2^5 and 10 shots 47 us, now 14 us.
constexpr int kChunkPad = kSampleChunk + 1;

// The last chunk whose base is at most the target, then the entry in it.
__device__ __forceinline__ int64_t sample_shot_smem(const unsigned long long* e, int len,
                                                    const unsigned long long* cb, int nc, unsigned long long T,
                                                    unsigned long long target) {
  auto entry = [&](int i) {
    return e[TQS_IX((i >> 3) * kChunkPad + (i & 7), nc * kChunkPad)];
  };
  int i = len - 1;  // target >= T: the last entry above 0
  if (target < T) {
    int lo = 0, hi = nc - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (cb[TQS_IX(mid, nc)] <= target) lo = mid; else hi = mid - 1;
    }
    unsigned long long c = cb[lo];
    const int i0 = lo * kSampleChunk;
#pragma unroll
    for (int j = 0; j < kSampleChunk; ++j) {
      const unsigned long long x = entry(i0 + j);  // 0 past len
      c += x;
      if (x > 0 && c > target) return i0 + j;
    }
    i = min(i0 + kSampleChunk, len) - 1;
  }
  for (; i >= 0; --i)
    if (entry(i) > 0) return i;
  return -1;
}

template <int K>
__global__ void __launch_bounds__(kThreads)
    segment_smem_kernel(const SampleLaunch L) {
  using U = unsigned long long;
  extern __shared__ U sm[];
  __shared__ U wtot[kThreads / 32];
  __shared__ int s_emax[kThreads / 32];
  __shared__ float s_fsum[kThreads / 32];
  const SampleSeg sg = L.ssegs[TQS_IX(blockIdx.x, L.n_sseg)];
  const int len = 1 << sg.n;
  const int nc = (len + kSampleChunk - 1) / kSampleChunk;  // chunks of this segment
  U* e = sm;
  U* cb = sm + nc * kChunkPad;
  const int t = threadIdx.x, T = blockDim.x, lane = t & 31, warp = t >> 5, nw = T >> 5;
  const int c0 = t * K;  // this thread's chunks: c0 .. c0 + K - 1
  (void)TQS_IX(sg.p_off + len - 1, L.probs_len);
  const double* ub = L.u + sg.index * L.shots;
  double u = t < L.shots ? __ldcs(ub + t) : 0.0;
  // the probabilities' bits, their largest exponent and an estimate of their sum
  const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(L.probs + sg.p_off);
  U v[K * kSampleChunk];
  int emax = 0;
  float fsum = 0.f;
#pragma unroll
  for (int j = 0; j < K * kSampleChunk / 2; ++j) {
    const int i = c0 * kSampleChunk + 2 * j;
    const ulonglong2 x = i < len ? __ldg(gp + (i >> 1)) : make_ulonglong2(0, 0);
    v[2 * j] = x.x;
    v[2 * j + 1] = x.y;
  }
#pragma unroll
  for (int j = 0; j < K * kSampleChunk; ++j) {
    emax = max(emax, static_cast<int>((v[j] >> 52) & 0x7FF));
    fsum += approx_f32(v[j]);
  }
  emax = __reduce_max_sync(kFull, emax);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) fsum += __shfl_xor_sync(kFull, fsum, o);
  if (lane == 0) {
    s_emax[warp] = emax;
    s_fsum[warp] = fsum;
  }
  __syncthreads();
  emax = 0;
  fsum = 0.f;
  for (int w = 0; w < nw; ++w) {
    emax = max(emax, s_emax[w]);
    fsum += s_fsum[w];
  }
  // T < 2^(ET + 1) (within the estimate's error), so T 2^S < 2^61 with
  // S = 60 - ET; entries below the FP32 range (no estimate) use the largest
  // exponent instead: every p < 2^(emax - 1022), 2^n of them below 2^62
  const int ET = (__float_as_int(fsum) >> 23) - 127;
  const int S = (fsum > 0.f && fsum < 3.0e38f) ? 60 - ET : 62 - sg.n - (max(emax, 1) - 1022);
  U own = 0;
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int j = 0; j < kSampleChunk; ++j) {
      const U x = to_fixed(v[k * kSampleChunk + j], S);
      own += x;
      v[k * kSampleChunk + j] = x;
      if (c0 + k < nc) e[TQS_IX((c0 + k) * kChunkPad + j, nc * kChunkPad)] = x;
    }
  // chunk bases: exclusive scan of the threads' sums (exact, so in any order)
  const U incl = warp_incl_scan(own, lane);
  if (lane == 31) wtot[warp] = incl;
  __syncthreads();
  U base = incl - own, total = 0;
  for (int w = 0; w < nw; ++w) {
    if (w < warp) base += wtot[w];
    total += wtot[w];
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (c0 + k < nc) cb[TQS_IX(c0 + k, nc)] = base;
#pragma unroll
    for (int j = 0; j < kSampleChunk; ++j) base += v[k * kSampleChunk + j];
  }
  __syncthreads();
  const double Tf = static_cast<double>(total);
  for (int64_t k = t; k < L.shots; k += T) {
    if (k != t) u = __ldcs(ub + k);
    const int64_t kk = TQS_IX(sg.index * L.shots + k, L.n_segs * L.shots);
    // floor(u T); u < 1 keeps it below T up to the rounding of the product
    const double x = u * Tf;
    const U target = x >= Tf ? total : static_cast<U>(x);
    L.out[kk] = sample_shot_smem(e, len, cb, nc, total, target);
  }
}

__global__ void set_basis_kernel(float2* st, int64_t len, const int64_t* idx) {
  const int64_t i0 = *idx;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < len;
       i += int64_t(gridDim.x) * blockDim.x)
    st[i] = make_float2(i == i0 ? 1.f : 0.f, 0.f);
}

int grid_for(int64_t items, int per_cta) {
  const int64_t ctas = (items + per_cta - 1) / per_cta;
  const int64_t cap = 152 * 8;
  return static_cast<int>(ctas < 1 ? 1 : (ctas < cap ? ctas : cap));
}

}  // namespace

TQS_DEFINE_VIOLATIONS(violations_sample)

cudaError_t launch_sample(const SampleLaunch& L, cudaStream_t s) {
  int k = 0;
  if (L.n_gseg > 0) {
    block_tables_kernel<<<grid_for(L.nblocks, kThreads / 32), kThreads, 0, s>>>(L);
    block_prefix_kernel<<<L.n_gseg, kThreads, 0, s>>>(L);
    k += 2;
    if (L.shots > 0) {
      shots_kernel<<<grid_for(int64_t(L.n_gseg) * L.shots, kThreads), kThreads, 0, s>>>(L);
      ++k;
    }
  }
  if (L.n_sseg > 0 && L.shots > 0) {
    // A thread per chunk of the largest segment, or per two shots (from 256 shots on
    // four, from 512 on more) where that is more, up to kThreads; from 2^12
    // entries on two or four chunks a thread.  With a thread per shot the blocks of
    // small segments hold more warps than their tables are worth: 16000 states
    // of 2^5, 64, 200 and 500 shots 24.7, 80 and 107 us, so 18.6, 49 and 76 us; 1000 states of
    // 2^6, 200 shots 10.3 and 7.2 us.
    const int nc = L.smem_q > 3 ? 1 << (L.smem_q - 3) : 1;
    int threads = 32;
    while (threads < kThreads && (threads < nc || (threads < 128 ? 2 : 4) * threads < L.shots)) threads *= 2;
    const int smem = nc * (kChunkPad + 1) * static_cast<int>(sizeof(double));
    static std::atomic<uint64_t> done[3];
    auto launch = [&](auto kernel, std::atomic<uint64_t>& d) -> cudaError_t {
      const cudaError_t e = allow_all_smem(reinterpret_cast<const void*>(kernel), d);
      if (e == cudaSuccess) kernel<<<L.n_sseg, threads, smem, s>>>(L);
      return e;
    };
    const cudaError_t e = nc <= threads       ? launch(segment_smem_kernel<1>, done[0])
                          : nc <= 2 * threads ? launch(segment_smem_kernel<2>, done[1])
                                              : launch(segment_smem_kernel<4>, done[2]);
    if (e != cudaSuccess) return e;
    ++k;
  }
  count_launches(k);
  return cudaGetLastError();
}

cudaError_t launch_set_basis(float2* d_state, int n, const int64_t* d_index, cudaStream_t s) {
  const int64_t len = int64_t(1) << n;
  set_basis_kernel<<<grid_for(len, kThreads), kThreads, 0, s>>>(d_state, len, d_index);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace tqs
