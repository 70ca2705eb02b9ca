// zmc_kernels.cu -- the kernels shared by every integrand family, and the
// host-side dispatch to the per-family sampling paths (zmc_fam_<family>.cu).
//
//   zmc_batched_kernel<FAM>  (one file per family) persistent work-list launch over
//                        (integrand, chunk) items: Philox4x32-10 -> map onto the
//                        box -> FP32 integrand -> per-lane shifted sums -> warp
//                        Chan merge -> one (mean, M2) record per chunk.  Direct MC
//                        per integrand is the paper's solution method (Sec.
//                        "Solution method"); many integrands of different form,
//                        dimension and box share one launch (Sec. "Summary of
//                        revisions", Eq. 1, Eq. 2).
//   zmc_merge_kernel     FP64 k-way Chan merge of an integrand's chunk records in a
//                        fixed order: mean, M2, estimate = V mean,
//                        stderr = V sqrt(M2 / (N (N-1))) (Fig. 1 caption: an estimate
//                        with its spread).
//   zmc_finish_kernel    for a launch whose last chunks were handed out by
//                        accumulation blocks: their records, then the same merge.
//   zmc_plain_fp64_kernel  (zmc_plain.cu) the plain form, one launch per integrand.
//   zmc_philox_rate_kernel  the generator alone (its throughput: the ceiling of
//                        any sampling kernel, which draws d / 5 blocks per sample).
//   zmc_philox_kernel, zmc_eval_kernel<FAM>   the generator and the per-sample
//                        integrand values of the sampling path, for parity tests.
//
// No tensor cores and no TMA: the path is integer and FP32 arithmetic on the FMA,
// ALU and MUFU pipes, with a few KB of descriptor reads and 8 bytes written per
// 160 * quints_per_lane samples.
#include <algorithm>
#include <atomic>

#include "zmc_device.cuh"

namespace zmc {
namespace {

// ---------------------------------------------------------------- split chunks
// Samples of a lane's steps [jb, je) in a chunk of nc samples.
__device__ __forceinline__ uint32_t lane_block_samples(uint32_t nc, uint32_t lane, uint32_t jb,
                                                       uint32_t je) {
  const uint32_t nq = nc / kQuint, rest = nc - kQuint * nq;  // whole quints, samples after them
  const uint32_t jl = nq > lane ? (nq - lane + 31u) / 32u : 0u;  // the lane's whole quints
  const uint32_t whole = jl <= jb ? 0u : (jl < je ? jl : je) - jb;
  const uint32_t j = nq / 32u;
  return kQuint * whole + (lane == nq % 32u && j >= jb && j < je ? rest : 0u);
}

// The record of a chunk from its blocks' lane summaries: the same steps, in the
// same order, as a warp that took the whole chunk.  Eight blocks (a chunk at the
// default Q = 104) are loaded at a time, so that their latencies overlap.
__device__ __forceinline__ void combine_blocks(const FnDev *__restrict__ fn, uint64_t chunk,
                                               uint32_t nc, uint32_t Q, uint32_t lane,
                                               const float2 *part) {
  float n = 0.0f, mean = 0.0f, m2 = 0.0f;
  for (uint32_t j0 = 0; j0 < Q && chunk_samples_of(j0) < nc; j0 += 8 * kBlockQuints) {
    uint32_t cnt[8];
    float2 b[8];
#pragma unroll
    for (uint32_t i = 0; i < 8; ++i) {
      const uint32_t jb = j0 + i * kBlockQuints;
      const uint32_t je = jb + kBlockQuints < Q ? jb + kBlockQuints : Q;
      cnt[i] = jb < Q ? lane_block_samples(nc, lane, jb, je) : 0u;
      if (cnt[i]) b[i] = __ldcg(part + 32u * (jb / kBlockQuints) + lane);
    }
#pragma unroll
    for (uint32_t i = 0; i < 8; ++i)
      if (cnt[i]) chan_step(n, mean, m2, static_cast<float>(cnt[i]), b[i].x, b[i].y);
  }
  __syncwarp();
  warp_chan_merge(n, mean, m2);
  if (lane == 0) fn->rec[chunk] = make_float2(mean, m2);
}

// ---------------------------------------------------------------- FP64 merge
// One warp per integrand.  With chunk summaries (n_c, m_c, M2_c):
//   mean = sum_c n_c m_c / N,  M2 = sum_c [M2_c + n_c (m_c - mean)^2]
// (Chan et al.'s combination of partial moments, all chunks at once), summed in a
// fixed lane / butterfly order, so the result depends only on the records.  Moments
// of earlier samples of the stream (prior_n > 0) are combined in last with the
// pairwise update, n = n_a + n_b, mean = mean_a + d n_b / n,
// M2 = M2_a + M2_b + d^2 n_a n_b / n, d = mean_b - mean_a.
// A chain of loads and FP64 steps, so bound by latency: the first kHeld records of a
// lane are loaded at once and held for the second pass (most rows have no more).
__device__ __forceinline__ void merge_row(const FnDev *__restrict__ fn, uint64_t chunk_samples,
                                          uint32_t lane) {
  constexpr uint32_t kHeld = 4;
  const uint64_t N = fn->n_samples;
  const uint64_t C = (N + chunk_samples - 1) / chunk_samples;
  const float2 *rec = fn->rec;  // perhaps written by this launch: read past the L1
  const auto weight = [&](uint64_t c) {
    const uint64_t left = N - c * chunk_samples;
    return static_cast<double>(left < chunk_samples ? left : chunk_samples);
  };
  float2 held[kHeld];
#pragma unroll
  for (uint32_t i = 0; i < kHeld; ++i)
    if (lane + 32 * i < C) held[i] = __ldcg(rec + lane + 32 * i);
  double s = 0.0;
#pragma unroll
  for (uint32_t i = 0; i < kHeld; ++i)
    if (lane + 32 * i < C) s = fma(weight(lane + 32 * i), static_cast<double>(held[i].x), s);
  for (uint64_t c = lane + 32 * kHeld; c < C; c += 32)
    s = fma(weight(c), static_cast<double>(__ldcg(rec + c).x), s);
  const double mean = N ? warp_sum_f64(s) / static_cast<double>(N) : 0.0;
  double m = 0.0;
  const auto spread = [&](uint64_t c, float2 rc) {
    const double dm = static_cast<double>(rc.x) - mean;
    m += fma(weight(c) * dm, dm, static_cast<double>(rc.y));
  };
#pragma unroll
  for (uint32_t i = 0; i < kHeld; ++i)
    if (lane + 32 * i < C) spread(lane + 32 * i, held[i]);
  for (uint64_t c = lane + 32 * kHeld; c < C; c += 32) spread(c, __ldcg(rec + c));
  const double inv = fn->inv_scale;
  double mu = mean * inv;
  double m2 = fmax(warp_sum_f64(m), 0.0) * inv * inv;
  uint64_t n_all = N;
  if (fn->prior_n > 0) {
    const double na = static_cast<double>(fn->prior_n), nb = static_cast<double>(N);
    const double nab = na + nb;
    const double d = mu - fn->prior_mean;
    mu = fn->prior_mean + d * (nb / nab);
    m2 = fn->prior_m2 + m2 + d * d * (na * nb / nab);
    n_all = fn->prior_n + N;
  }
  if (lane == 0) {
    const double nd = static_cast<double>(n_all);
    zmc_result res;
    if (fn->out_mode == 0) {
      res.estimate = fn->volume * mu;
      res.stderr_ = fn->volume * sqrt(m2 / (nd * (nd - 1.0)));
    } else {  // zmc_moments: unscaled mean and M2 of f over the samples
      res.estimate = mu;
      res.stderr_ = m2;
    }
    res.n = n_all;
    res.status = ZMC_OK;
    res.reserved = 0;
    *fn->out = res;
  }
}

// reset: the launch's counters go back to zero for its next run (the sampling
// kernels that drew from them have ended), which saves a memset per run.
__global__ void __launch_bounds__(256) zmc_merge_kernel(const FnDev *const *__restrict__ fns,
                                                        LaunchHdr *__restrict__ hdr, bool reset) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t nm = hdr->n_merge;
  const uint64_t chunk_samples = chunk_samples_of(hdr->quints_per_lane);
  if (reset && warp == 0 && lane < 4) hdr->counter[lane] = 0;
  for (uint32_t k = warp; k < nm; k += nwarps) merge_row(fns[k], chunk_samples, lane);
}

// The merge of a launch with split chunks, whose entries are its rows in some order:
// one warp per split chunk makes its record, and the warp that completes a row's
// count of split chunks merges the row; one warp per row without any merges it at
// once.  One kernel less than records and merge apart (~4 us of a small call).
// hdr->left: a count per entry, zero before the first run; it wraps to zero by itself.
// merge = false: the records alone, no result is written.
__global__ void __launch_bounds__(256) zmc_finish_kernel(const Entry *__restrict__ entries,
                                                         LaunchHdr *__restrict__ hdr, bool merge) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t Q = hdr->quints_per_lane;
  const uint32_t ne = hdr->n_entries;
  uint32_t total = 0;
  for (int f = 0; f < 4; ++f) total += hdr->split[f];
  uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w == 0 && lane < 4) hdr->counter[lane] = 0;
  for (; w < total + (merge ? ne : 0u); w += nwarps) {
    if (w < total) {
      int f = 0;
      uint32_t t = w;
      for (; t >= hdr->split[f]; ++f) t -= hdr->split[f];
      const uint64_t split0 = hdr->item_end[f] - hdr->split[f];  // the family's first split item
      const uint32_t e = find_entry(entries, ne, split0 + t, lane);
      const Entry en = entries[e];
      const uint64_t chunk = en.chunk_begin + (split0 + t - en.item_begin);
      combine_blocks(en.fn, chunk, samples_of(en.fn, chunk, Q), Q, lane,
                     hdr->part[f] + static_cast<size_t>(t) * 32u * chunk_blocks(Q));
      if (!merge) continue;
      const uint64_t next = e + 1 < ne ? entries[e + 1].item_begin : hdr->item_end[f];
      const uint64_t end = next < hdr->item_end[f] ? next : hdr->item_end[f];
      const uint32_t last =
          static_cast<uint32_t>(end - (en.item_begin > split0 ? en.item_begin : split0)) - 1;
      uint32_t before = 0;
      if (lane == 0)  // after this lane's record
        asm volatile("atom.acq_rel.gpu.global.inc.u32 %0, [%1], %2;"
                     : "=r"(before)
                     : "l"(hdr->left + e), "r"(last)
                     : "memory");
      before = __shfl_sync(kFullMask, before, 0);
      if (before != last) continue;
      __syncwarp();  // the shuffle orders no memory: all lanes after lane 0's acquire
      merge_row(en.fn, chunk_samples_of(Q), lane);
    } else {
      const uint32_t e = w - total;
      const Entry en = entries[e];
      const uint32_t family = (en.fn->variant >> 4) & 0xFu;
      const uint32_t f = family < 4 ? family : 0;  // HdrSlot
      const uint64_t next = e + 1 < ne ? entries[e + 1].item_begin : hdr->item_end[f];
      const uint64_t end = next < hdr->item_end[f] ? next : hdr->item_end[f];
      if (end <= hdr->item_end[f] - hdr->split[f]) merge_row(en.fn, chunk_samples_of(Q), lane);
    }
  }
}

// ---------------------------------------------------------------- test kernels
__global__ void zmc_philox_kernel(const uint32_t *__restrict__ ctr,
                                  const uint32_t *__restrict__ key, uint32_t *__restrict__ out,
                                  size_t n) {
  for (size_t j = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; j < n;
       j += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const RoundKeys rk = make_round_keys(key[2 * j], key[2 * j + 1]);
    const uint4 o = philox(ctr[4 * j], ctr[4 * j + 1], ctr[4 * j + 2], ctr[4 * j + 3], rk);
    out[4 * j + 0] = o.x;
    out[4 * j + 1] = o.y;
    out[4 * j + 2] = o.z;
    out[4 * j + 3] = o.w;
  }
}

// Generator rate: every thread draws per_thread Philox4x32-10 blocks, four
// independent calls at a time, with the sampling kernels' counter layout and
// chunk prefix (block lo advancing; stream word, block hi and key the same for
// the whole warp) and their launch bound, and folds the words into one so that
// none is dead.
__global__ void __launch_bounds__(256, 2) zmc_philox_rate_kernel(uint32_t key0, uint32_t key1,
                                                                 uint32_t sid,
                                                                 uint32_t per_thread,
                                                                 uint32_t *__restrict__ out) {
  const StreamPrefix sp = make_stream_prefix(make_round_keys(key0, key1), sid, 0u);
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t base = t * per_thread;  // wraps on huge grids: a rate needs no distinct counters
  uint32_t acc = 0;
  for (uint32_t q = 0; q < per_thread; q += 4) {
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
      const uint4 o = philox_block(base + q + j, sp);
      acc ^= o.x ^ o.y ^ o.z ^ o.w;
    }
  }
  out[t] = acc;
}

const FamilyOps *ops_of(int family, int unroll = 1) {
  static const FamilyOps *const kOps[kMaxUnroll][4] = {
      {&kFamilyHarmonicU1, &kFamilyAbslinU1, &kFamilyGaussU1, &kFamilyPolyU1},
      {&kFamilyHarmonicU2, &kFamilyAbslinU2, &kFamilyGaussU2, &kFamilyPolyU2}};
  if (family < 0 || family > ZMC_POLY || unroll < 1 || unroll > kMaxUnroll) return nullptr;
  return kOps[unroll - 1][family];
}

}  // namespace

// ---------------------------------------------------------------- launch wrappers
cudaError_t launch_batched(int family, const Entry *entries, LaunchHdr *hdr, unsigned grid,
                           unsigned block, cudaStream_t stream, int unroll) {
  const FamilyOps *ops = ops_of(family, unroll);
  return ops ? ops->launch_batched(entries, hdr, grid, block, stream) : cudaErrorInvalidValue;
}

cudaError_t launch_merge(const FnDev *const *fns, LaunchHdr *hdr, unsigned grid,
                         cudaStream_t stream, bool reset) {
  zmc_merge_kernel<<<grid, 256, 0, stream>>>(fns, hdr, reset);
  return cudaGetLastError();
}

cudaError_t launch_finish(const Entry *entries, LaunchHdr *hdr, uint64_t warps, int sms,
                          cudaStream_t stream, bool merge) {
  const uint64_t blocks = std::min<uint64_t>((warps + 7) / 8, 16ull * static_cast<unsigned>(sms));
  zmc_finish_kernel<<<static_cast<unsigned>(blocks), 256, 0, stream>>>(entries, hdr, merge);
  return cudaGetLastError();
}

// Kept per kernel and block size: every device this library runs on is the same
// part, and the query is on the path of each blocking call.
int batched_max_blocks_per_sm(int family, int block, int unroll) {
  const FamilyOps *ops = ops_of(family, unroll);
  if (!ops || block < 32 || block > 1024) return 0;
  static std::atomic<int> known[kMaxUnroll][4][33];
  std::atomic<int> &k = known[unroll - 1][family][block / 32];
  int n = k.load(std::memory_order_relaxed);
  if (n == 0) {
    n = ops->max_blocks_per_sm(block);
    k.store(n, std::memory_order_relaxed);
  }
  return n;
}

int batched_regs_per_thread(int family, int unroll) {
  const FamilyOps *ops = ops_of(family, unroll);
  return ops ? ops->regs_per_thread() : 0;
}

cudaError_t launch_philox(const uint32_t *ctr, const uint32_t *key, uint32_t *out, size_t n,
                          cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  const size_t blocks = (n + 255) / 256;
  zmc_philox_kernel<<<static_cast<unsigned>(blocks < 4096 ? blocks : 4096), 256, 0, stream>>>(
      ctr, key, out, n);
  return cudaGetLastError();
}

cudaError_t launch_philox_rate(uint32_t per_thread, unsigned grid, uint32_t *out,
                               cudaStream_t stream) {
  zmc_philox_rate_kernel<<<grid, 256, 0, stream>>>(0x2104u, 0x10073u, 7u, per_thread, out);
  return cudaGetLastError();
}

cudaError_t launch_eval(int family, const FnDev *fn, uint64_t s_begin, uint32_t count,
                        float *out, cudaStream_t stream) {
  const FamilyOps *ops = ops_of(family);
  return ops ? ops->launch_eval(fn, s_begin, count, out, stream) : cudaErrorInvalidValue;
}

}  // namespace zmc
