// SimHash signatures of the window queries (Section 3.3 "Recall"; Algorithm 1 line 6 counts
// collisions against exactly these query buckets) in one kernel:
//
//   qsig_kernel - Q_win . P^T for one KV head's group of window queries and eight tables of
//                 hyperplanes on the tensor core (tcgen05, fp32 accumulation in TMEM); every
//                 thread owns a query row, packs the sign bits of each table into a bucket code,
//                 writes the codes and counts them into the tables' histograms (the number of
//                 window queries per bucket). Tables with a bit that came from a projection too
//                 small to trust are listed and settled by eight lanes each (fp64 accumulation of
//                 exact bf16 products; rare) before they are counted.
//                 The kernel also clears the call's collision counts and restarts the fix-up
//                 counters.
//
// Bucket code: hyperplane r*K + b0 sits at bit K-1-b0; bit = [projection >= 0].
#pragma once
#include "ptx.cuh"
#include "stream_gemm.cuh"
#include "aux_kernels.cuh"

namespace lkv {

// Two warpgroups, one per row block of 128 queries. The kernel is a chain of latencies (operands 2 us, MMA,
// tensor-memory loads, signs, histogram) on SMs that the pass beside it waits for: 7.6 us with 64 CTAs of 256
// queries and 10-bit tables (13.2 us with one warpgroup, fp64 sums by single threads and 2-byte stores).
constexpr int kQsigThreads = 256;
constexpr int kQsigTables = 8;             // tables per CTA: 8*K hyperplanes, a multiple of 16 for every K

struct QsigArgs {
  const uint16_t* Q;       // [batch][H_q][W][d] via strides (exact recomputation reads it directly)
  long long qs_b, qs_h, qs_w;
  const uint16_t* P;       // [L*K][128]
  uint16_t* hist;          // [batch][H_kv][L][2^K]
  uint16_t* qbuckets;      // [batch][H_kv][GW][L]
  int H_kv, G, W, GW;
  int q_rows_alloc;        // rows reserved per 64-column half for the query group (multiple of 128)
  int lsh_tables;
  uint4* zero_begin;       // the call's collision counts, cleared here (16-byte units)
  long long zero_n;
  int* counters;           // fix-up and changed counters, restarted here
  int* seg_counters;       // per-segment fix-up list lengths, restarted here
  int n_seg_counters;
  int* status;
  int n_real_tables;       // tables from this index on are padding: their histograms stay empty
  int q_w0;                // first window position of this pass; W and GW describe the pass
  int q_row0, q_rows_total;   // qbuckets rows: [bh][q_rows_total][L], this pass starts at row q_row0
  int first_part;          // nonzero: clear the counts, restart the counters, store the histogram;
                           // zero: a later part of a wide window: add to the histogram
  int release_next;        // nonzero: the next kernel in the stream was launched to start beside this one
  int* done_counter;       // every CTA adds one when its results are written: the projection pass, which may
                           // start while later kernels still run, is held back until all of them have
  int overlap_prev;        // nonzero: launched to start beside the kernel ahead in the stream
};

__host__ __device__ inline uint32_t qsig_smem_bytes(int q_rows_alloc, int kbits) {
  return 2u * q_rows_alloc * 128u + 2u * (kQsigTables * kbits) * 128u + kQsigTables * (4u << kbits) + 64u + 1024u;
}

// One CTA per (group of eight tables, KV head, sequence). A = the group's queries (row blocks of
// 128), B = the 8*K hyperplanes of the tables, D[query][hyperplane] in TMEM (one 128-column slot
// per row block).
template <int KBITS>
__global__ void __launch_bounds__(kQsigThreads, 1)
qsig_kernel(const __grid_constant__ CUtensorMap map_q,    // Q: (d, W, H_q, batch), box (64, W, G, 1)
            const __grid_constant__ CUtensorMap map_p,    // P: (d, L*K), box (64, 8*K)
            const QsigArgs a) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int N = kQsigTables * KBITS;           // hyperplanes of the CTA
  constexpr int LD = (N & -N) < 32 ? (N & -N) : 32;
  constexpr uint32_t nbins = 1u << KBITS;
  constexpr uint32_t bucket_mask = nbins - 1u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tg = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  // everything before this in the stream is complete, for this kernel and for the one it releases: the
  // log-sum-exp pass that follows needs nothing from this kernel and takes the SMs this small grid leaves free.
  // This CTA's tensor memory is not allocated yet, and a streaming CTA takes all of an SM's: the two never share an SM,
  // because their registers do not fit together (608 threads x 96 and 256 x 93 at least of 65,536). Kernels with
  // fewer would have to release behind the allocation, which costs a call 0.1 to 3 us (96 tiles in all, 32 tables of
  // 8 bits: 29.6 -> 32.9 us; 128 segments of 2048 keys 96.0 -> 96.5).
  grid_dependency_wait();
  if (a.release_next) allow_dependents();
  const int nmb = (a.GW + 127) / 128;
  const size_t bh = (size_t)b * a.H_kv + h;

  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* const gen_base = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t q_atom = a.q_rows_alloc * 128u;
  const uint32_t sm_q = base;
  const uint32_t sm_p = sm_q + 2u * q_atom;
  const uint32_t sm_bins = sm_p + 2u * N * 128u;
  const uint32_t sm_bars = sm_bins + kQsigTables * nbins * 4u;
  const uint32_t bar_load = sm_bars, bar_mma = sm_bars + 8, sm_slot = sm_bars + 16;
  int* n_items = reinterpret_cast<int*>(gen_base + (sm_bars + 20 - base));
  uint2* items = reinterpret_cast<uint2*>(gen_base);          // over the queries, which only the MMAs read: at most 256 x 8
  uint32_t* bins = reinterpret_cast<uint32_t*>(gen_base + (sm_bins - base));      // [8][2^K]
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gen_base + (sm_slot - base));

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&map_q);
    tma_prefetch_desc(&map_p);
    mbar_init(bar_load, 1);
    mbar_init(bar_mma, 1);
    fence_mbar_init();
    // the operands are on their way before the tensor memory is allocated
    mbar_expect_tx(bar_load, 2u * a.GW * 128u + 2u * N * 128u);
    tma_load_4d(sm_q, &map_q, bar_load, 0, a.q_w0, h * a.G, b);
    tma_load_4d(sm_q + q_atom, &map_q, bar_load, kAtomCols, a.q_w0, h * a.G, b);
    tma_load_2d(sm_p, &map_p, bar_load, 0, tg * N);
    tma_load_2d(sm_p + N * 128u, &map_p, bar_load, kAtomCols, tg * N);
    *n_items = 0;
  }
  const uint32_t tmem_cols = nmb == 2 ? 256u : 128u;   // one 128-column slot per row block
  if (warp == 0) { __syncwarp(); tmem_alloc(sm_slot, tmem_cols); tmem_relinquish(); }
  // while the operands fly: this CTA's share of the count array, and empty histograms
  {
    const long long cta = ((long long)b * gridDim.y + h) * gridDim.x + tg;
    const long long nctas = (long long)gridDim.x * gridDim.y * gridDim.z;
    const long long per = (a.zero_n + nctas - 1) / nctas;
    const long long z0 = cta * per, z1 = min(a.zero_n, z0 + per);
    if (a.first_part) {
      for (long long i = z0 + threadIdx.x; i < z1; i += kQsigThreads) a.zero_begin[i] = make_uint4(0u, 0u, 0u, 0u);
      if (cta == 0 && threadIdx.x < 2) a.counters[threadIdx.x] = 0;
      if (cta == nctas - 1)
        for (int i = threadIdx.x; i < a.n_seg_counters; i += kQsigThreads) a.seg_counters[i] = 0;
    }
    for (uint32_t i = threadIdx.x; i < kQsigTables * nbins / 4; i += kQsigThreads)
      reinterpret_cast<uint4*>(bins)[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  bool ok = true;
  if (warp == 0) {
    ok = mbar_wait_spin(bar_load, 0);
    tc_fence_after();
    if (ok && elect_one()) {
      const uint32_t idesc = umma_idesc_bf16(128, N);
      const uint32_t q_lo = umma_sdesc_lo(sm_q), p_lo = umma_sdesc_lo(sm_p);
#pragma unroll
      for (int mb = 0; mb < 2; ++mb) {
        if (mb < nmb) {
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint32_t qk = q_lo + (k >> 2) * (q_atom >> 4) + (k & 3) * 2 + mb * ((128 * 128) >> 4);
            const uint32_t pk = p_lo + (k >> 2) * ((N * 128) >> 4) + (k & 3) * 2;
            umma_bf16_lo(tmem_base + mb * 128, qk, pk, idesc, k > 0);
          }
        }
      }
      umma_commit(bar_mma);
    }
    __syncwarp();
  }
  // every thread: its query row of its warpgroup's row block
  if (ok) ok = mbar_wait(bar_mma, 0);
  const int mb = warp >> 2, q = threadIdx.x;
  if (ok && mb < nmb) {
    tc_fence_after();
    const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    uint32_t v[N];
#pragma unroll
    for (int j = 0; j < N / LD; ++j) tmem_ld_cols<LD>(t_lane + mb * 128 + j * LD, v + j * LD);
    tmem_wait_ld();
    reg_fence<N>(v);
    if (q < a.GW) {
      float amax = 0.f;
#pragma unroll
      for (int k = 0; k < 16; k += 2) amax = max3_abs(__uint_as_float(v[k]), __uint_as_float(v[k + 1]), amax);
      const float tau = amax * (1.0f / 32768.0f);
      uint32_t codes[kQsigTables];
#pragma unroll
      for (int t = 0; t < kQsigTables; ++t) {
        uint32_t neg = 0;
        float mn = INFINITY;
#pragma unroll
        for (int k = 0; k < KBITS; k += 2) {
          const uint32_t x0 = v[t * KBITS + k], x1 = v[t * KBITS + k + 1];
          neg = __funnelshift_l(x0, neg, 1);
          neg = __funnelshift_l(x1, neg, 1);
          mn = min3_abs_nan(__uint_as_float(x0), __uint_as_float(x1), mn);   // a NaN is doubtful too
        }
        codes[t] = (~neg) & bucket_mask;
        if (!(mn >= tau)) {                         // rare: counted once its signs are settled
          uint32_t doubt = 0;
#pragma unroll
          for (int k = 0; k < KBITS; ++k)
            if (!(fabsf(__uint_as_float(v[t * KBITS + k])) >= tau)) doubt |= 1u << (KBITS - 1 - k);
          items[atomicAdd(n_items, 1)] = make_uint2((uint32_t)q | ((uint32_t)t << 16), codes[t] | (doubt << 16));
        } else if (tg * kQsigTables + t < a.n_real_tables) {
          atomicAdd(&bins[t * nbins + codes[t]], 1u);
        }
      }
      // eight consecutive tables: one 16-byte store (L is a multiple of 8)
      uint4 packed;
      packed.x = codes[0] | (codes[1] << 16);
      packed.y = codes[2] | (codes[3] << 16);
      packed.z = codes[4] | (codes[5] << 16);
      packed.w = codes[6] | (codes[7] << 16);
      *reinterpret_cast<uint4*>(a.qbuckets + (bh * a.q_rows_total + a.q_row0 + q) * a.lsh_tables + tg * kQsigTables) = packed;
    }
  }
  if (!ok) record_status(a.status, kStatusTimeout);
  tc_fence_before();
  ok = __syncthreads_and(ok);
  if (ok) {
    const int n = *n_items, sl = lane & 7;
    const uint32_t gmask = 0xFFu << (lane & 24);
    for (int it = (int)(threadIdx.x >> 3); it < n; it += kQsigThreads >> 3) {
      const uint2 item = items[it];
      const int qi = (int)(item.x & 0xFFFFu), t = (int)(item.x >> 16);
      uint32_t mask = item.y >> 16, code = item.y & 0xFFFFu;
      const uint16_t* row = a.Q + b * a.qs_b + (long long)(h * a.G + qi / a.W) * a.qs_h + (a.q_w0 + qi % a.W) * a.qs_w + sl * 16;
      while (mask) {
        const int pos = 31 - __clz(mask);           // code bit; hyperplane r*K + (K-1-pos)
        mask &= ~(1u << pos);
        double acc = exact_dot<16>(row, a.P + ((size_t)(tg * kQsigTables + t) * KBITS + (KBITS - 1 - pos)) * 128 + sl * 16);
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) acc += __shfl_xor_sync(gmask, acc, off);
        code = (code & ~(1u << pos)) | ((acc >= 0.0 ? 1u : 0u) << pos);
      }
      if (sl == 0) {
        if (tg * kQsigTables + t < a.n_real_tables) atomicAdd(&bins[t * nbins + code], 1u);
        a.qbuckets[(bh * a.q_rows_total + a.q_row0 + qi) * a.lsh_tables + tg * kQsigTables + t] = (uint16_t)code;
      }
    }
    __syncthreads();
    uint4* out = reinterpret_cast<uint4*>(a.hist + (bh * a.lsh_tables + (size_t)tg * kQsigTables) * nbins);
    for (uint32_t i = threadIdx.x; i < kQsigTables * nbins / 8; i += kQsigThreads) {
      const uint4 lo = reinterpret_cast<const uint4*>(bins)[2 * i], hi = reinterpret_cast<const uint4*>(bins)[2 * i + 1];
      uint4 w = make_uint4(lo.x | (lo.y << 16), lo.z | (lo.w << 16), hi.x | (hi.y << 16), hi.z | (hi.w << 16));
      if (!a.first_part) {                          // 16-bit counts of at most 1024 queries: no carry between halves
        const uint4 o = out[i];
        w.x += o.x; w.y += o.y; w.z += o.z; w.w += o.w;
      }
      out[i] = w;
    }
  }
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, tmem_cols);
  }
  if (a.done_counter) {
    __syncthreads();                                   // the CTA's histograms, codes and zeros are written ...
    if (threadIdx.x == 0) {
      __threadfence();                                 // ... and visible before the count goes up
      atomicAdd(a.done_counter, 1);
    }
  }
}

}  // namespace lkv
