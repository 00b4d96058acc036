// The non-GEMM kernels of the selection path:
//   select_kernel  - Algorithm 1 lines 4-8: two-stage top-k per (sequence, KV head, block) by radix
//                    selection on registers, ties to the lower index, ascending output.
//   append_kernel  - gather of the kept K/V rows into the append-only cache (16-byte vectors).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "ptx.cuh"

namespace lkv {

// ------------------------------------------------------------------------------------------------
// Two-stage top-k. One CTA of T threads per segment; thread t owns the keys t, t + T, t + 2T, ... and
// holds their values of the running stage in registers, its candidate / kept flags as bit masks.
//
// Bound by barriers and by histogram atomics in shared memory, not by bytes (64 KB per segment of
// 8192 keys). A radix round bins the values that are still undecided by the eleven highest bits in
// which they can differ: the first round subtracts the smallest candidate, so that scores that share
// their exponent bits do not pile up in a few bins (atomics of a warp on one bin go one by one), and
// the k-th largest of 8192 scores is usually alone in its bin after two rounds, a count after one.
// A round takes three barriers. Against 8-bit rounds over values and flags in shared memory (both with the
// doubtful signs settled in front): 512 segments of 4096 keys 62 -> 29 us, 128 of 8192 25.2 -> 20.3 us, 8 of
// 8192 22.2 -> 16.5 us; 80 of 1864 without signs 7.5 -> 4.7 us. Since the projection pass settles the
// signs the first three take 24.7, 12.8 and 10.6 us.
// ------------------------------------------------------------------------------------------------
constexpr int kSelBins = 2048;
constexpr int kSelBinBits = 11;
constexpr int kSelMaxKeys = 24 * 1024;   // a block of 16384 keys and the 8192 that look-back may hold back

__device__ __forceinline__ uint32_t orderable_f32(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

template <int T, int NI>
struct SelShared {
  static constexpr int kWarps = T / 32;
  int hist[kSelBins];              // all zero between rounds
  int chunk_sum[kWarps];
  int found[3];                    // bin, elements still needed from it, elements in it
  uint32_t range[4][kWarps];       // per warp: smallest and largest score, smallest and largest count
  int before[2][kWarps * NI];      // ordered_ranks: tie break, compaction
};

// For every row i of the CTA (keys i*T .. i*T + T - 1): how many keys of smaller index than the
// calling warp's part of the row have their bit set in `mask` (bit i of a thread's mask: its key of
// row i). Lane i of the warp receives the number for row i. Two barriers.
template <int T, int NI>
__device__ __forceinline__ int ordered_ranks(uint32_t mask, int* before) {
  constexpr int NW = T / 32, E = NW * NI, PER = (E + 31) / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int mine = 0;
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    const int n = __popc(__ballot_sync(0xffffffffu, (mask >> i) & 1u));
    if (lane == i) mine = n;
  }
  if (lane < NI) before[lane * NW + warp] = mine;
  __syncthreads();
  if (warp == 0) {
    int v[PER], sum = 0;
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      v[p] = (lane * PER + p < E) ? before[lane * PER + p] : 0;
      sum += v[p];
    }
    int incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += n;
    }
    int run = incl - sum;
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      if (lane * PER + p < E) before[lane * PER + p] = run;
      run += v[p];
    }
  }
  __syncthreads();
  return lane < NI ? before[lane * NW + warp] : 0;
}

// Moves the k largest values among the candidates (bit i of `cand`: v[i] takes part) from `cand` to
// `kept`; equal values: lower index first. lo and hi bound the candidates' values; there are at
// least k candidates.
template <int T, int NI>
__device__ __forceinline__ void take_topk(const uint32_t (&v)[NI], uint32_t& cand, uint32_t& kept, int k, uint32_t lo,
                                          uint32_t hi, SelShared<T, NI>& sh) {
  if (k <= 0) return;                    // uniform across the CTA
  constexpr int NW = T / 32;
  constexpr int PER = kSelBins / T;      // bins a thread sums up
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t in = cand, base = lo;         // still undecided; the smallest value they can have
  int need = k, shift = 32 - __clz(hi - lo) - kSelBinBits;
  if (shift < 0) shift = 0;
  for (;;) {
#pragma unroll
    for (int i = 0; i < NI; ++i)
      if ((in >> i) & 1u) atomicAdd(&sh.hist[(v[i] - base) >> shift], 1);
    __syncthreads();
    // warp w sums the w-th highest run of 32 * PER bins; the lanes go from high bins to low ones
    const int b0 = kSelBins - (warp * 32 + lane + 1) * PER;
    int c[PER], sum = 0;
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      c[p] = sh.hist[b0 + PER - 1 - p];
      sh.hist[b0 + PER - 1 - p] = 0;
      sum += c[p];
    }
    const int wsum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) sh.chunk_sum[warp] = wsum;
    __syncthreads();
    {
      const int x = lane < NW ? sh.chunk_sum[lane] : 0;
      int incl = x;
#pragma unroll
      for (int off = 1; off < NW; off <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += n;
      }
      const int owner = __ffs(__ballot_sync(0xffffffffu, need <= incl)) - 1;
      if (warp == owner) {               // this warp's bins hold the k-th value
        int run = __shfl_sync(0xffffffffu, incl - x, owner);
        int in_warp = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int n = __shfl_up_sync(0xffffffffu, in_warp, off);
          if (lane >= off) in_warp += n;
        }
        run += in_warp - sum;            // elements in higher bins than this lane's
#pragma unroll
        for (int p = 0; p < PER; ++p) {
          if (run < need && need <= run + c[p]) {
            sh.found[0] = b0 + PER - 1 - p;
            sh.found[1] = need - run;
            sh.found[2] = c[p];
          }
          run += c[p];
        }
      }
    }
    __syncthreads();
    const uint32_t bin = (uint32_t)sh.found[0];
    need = sh.found[1];
    const int held = sh.found[2];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const uint32_t d = (v[i] - base) >> shift, bit = in & (1u << i);
      if (d != bin) in &= ~bit;
      if (d > bin) kept |= bit;
    }
    if (need == held) {                  // the whole bin
      kept |= in;
      break;
    }
    if (shift == 0) {                    // equal values: the ones of lowest index
      const int rank0 = ordered_ranks<T, NI>(in, sh.before[0]);
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const uint32_t row = __ballot_sync(0xffffffffu, (in >> i) & 1u);
        const int rank = __shfl_sync(0xffffffffu, rank0, i) + __popc(row & ((1u << lane) - 1u));
        if (rank < need) kept |= in & (1u << i);
      }
      break;
    }
    base += bin << shift;
    shift = shift > kSelBinBits ? shift - kSelBinBits : 0;
  }
  cand &= ~kept;
}

// The S scored keys of a segment fall into three classes: kept whatever their scores (two index
// ranges: Section 3.1's anchors and local window), excluded (one range: a tail that is held back
// for the next block under look-back, Section 3.2), and candidates (everything else).
struct SelectArgs {
  const float* s_exact;     // [n_seg][S]
  const uint32_t* counts;   // [n_seg][S]
  int32_t* idx;             // [n_seg][B], B = kept + k_exact + k_lsh
  int S, k_exact, k_lsh;
  int keep_a_lo, keep_a_hi, keep_b_lo, keep_b_hi;   // kept ranges [lo, hi); empty when lo >= hi
  int excl_lo, excl_hi;                             // excluded range
};

template <int T, int NI>
__global__ void __launch_bounds__(T, 1024 / T) select_kernel(const SelectArgs a) {
  extern __shared__ uint8_t smem_sel[];
  uint32_t* ucnt = reinterpret_cast<uint32_t*>(smem_sel);     // [S]
  __shared__ SelShared<T, NI> sh;
  const int seg = blockIdx.x, S = a.S;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int B = max(0, a.keep_a_hi - a.keep_a_lo) + max(0, a.keep_b_hi - a.keep_b_lo) + a.k_exact + a.k_lsh;
  const float* s_seg = a.s_exact + (size_t)seg * S;
  const uint32_t* c_seg = a.counts + (size_t)seg * S;
  uint32_t v[NI], cand = 0, kept = 0;
  // starts beside the projection pass: only the launch and this are ahead of the wait for its results
  for (int i = threadIdx.x; i < kSelBins; i += T) sh.hist[i] = 0;
  grid_dependency_wait();
  allow_dependents();
  {
    float x[NI];
    uint32_t n[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int j = i * T + (int)threadIdx.x;
      x[i] = j < S ? s_seg[j] : 0.f;
      n[i] = j < S ? c_seg[j] : 0u;
    }
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int j = i * T + (int)threadIdx.x;
      v[i] = orderable_f32(x[i]);
      if (j < S) {
        ucnt[j] = n[i];
        const bool keep = (j >= a.keep_a_lo && j < a.keep_a_hi) || (j >= a.keep_b_lo && j < a.keep_b_hi);
        if (keep) kept |= 1u << i;
        else if (!(j >= a.excl_lo && j < a.excl_hi)) cand |= 1u << i;
      }
    }
  }
  // the candidates' range of scores and of counts
  uint32_t lo = 0xffffffffu, hi = 0u, clo = 0xffffffffu, chi = 0u;
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    if ((cand >> i) & 1u) {
      const uint32_t n = ucnt[i * T + (int)threadIdx.x];
      lo = min(lo, v[i]); hi = max(hi, v[i]);
      clo = min(clo, n); chi = max(chi, n);
    }
  }
  lo = __reduce_min_sync(0xffffffffu, lo); hi = __reduce_max_sync(0xffffffffu, hi);
  clo = __reduce_min_sync(0xffffffffu, clo); chi = __reduce_max_sync(0xffffffffu, chi);
  if (lane == 0) { sh.range[0][warp] = lo; sh.range[1][warp] = hi; sh.range[2][warp] = clo; sh.range[3][warp] = chi; }
  __syncthreads();
  {
    const int w = lane & (T / 32 - 1);
    lo = __reduce_min_sync(0xffffffffu, sh.range[0][w]); hi = __reduce_max_sync(0xffffffffu, sh.range[1][w]);
    clo = __reduce_min_sync(0xffffffffu, sh.range[2][w]); chi = __reduce_max_sync(0xffffffffu, sh.range[3][w]);
  }
  take_topk<T, NI>(v, cand, kept, a.k_exact, lo, hi, sh);            // K_exact
  if (a.k_lsh > 0) {
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int j = i * T + (int)threadIdx.x;
      v[i] = j < S ? ucnt[j] : 0u;
    }
    take_topk<T, NI>(v, cand, kept, a.k_lsh, clo, chi, sh);          // K_lsh from the residual
  }
  // ordered compaction of all kept indices
  const int rank0 = ordered_ranks<T, NI>(kept, sh.before[1]);
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    const bool keep = (kept >> i) & 1u;
    const uint32_t row = __ballot_sync(0xffffffffu, keep);
    const int out = __shfl_sync(0xffffffffu, rank0, i) + __popc(row & ((1u << lane) - 1u));
    if (keep && out < B) a.idx[(size_t)seg * B + out] = i * T + (int)threadIdx.x;
  }
}

// ------------------------------------------------------------------------------------------------
// Gather + append. 16 threads move one 256-byte row of K and of V as 16-byte vectors; a thread has the
// vectors of four rows under way together. Large calls are bound by HBM (128 segments of 3855 rows: 77 us
// either way, 0.95 of the copy rate). Small ones are a chain of round trips (index, row, store), four times over when
// a thread took its rows one after the other: sixteen calls of one block of 8192 tokens 1022 -> 1011 us in
// all, calls of two blocks of 4096 298 -> 288 us, and 979 and 277 us when the kernel is also started
// beside the selection.
// ------------------------------------------------------------------------------------------------
struct AppendArgs {
  const uint16_t* K;
  const uint16_t* V;
  long long ks_b, ks_h, ks_t;   // source strides (elements): batch, head, token
  int H_kv, nb;
  int S_stride;                 // source rows between the first rows of consecutive blocks
  int B;                        // entries per segment
  const int32_t* idx;           // [batch][H_kv][nb][B]; NULL: entry i is source row i
  uint16_t* Kc;
  uint16_t* Vc;
  int32_t* pos;
  long long c_seg_stride;       // elements between (batch, head) cache slabs
  long long pos_seg_stride;
  long long dst_off0;           // first destination entry of block t = 0
  int pos_base0;                // absolute position of token 0 of block t = 0
  int n_src_rows;               // rows of a source segment: an index outside [0, n_src_rows) is not read
  int* status;                  // receives kAppendBadIndex when an index was out of range
};

constexpr int kAppendRowsPerCta = 64;
// Up to this many indices the first CTA looks them all over by itself and stores the status word, so that
// the caller's word needs no launch of its own to be cleared (one index set gathered head by head: a memset
// of 1.5 us and its launch in front of every 5 us gather). Above it the scan would outlast the gather.
constexpr int kAppendOwnStatusMax = 16384;
constexpr int kAppendBadIndex = 1;   // LASER_KV_ERR_INVALID_ARG

__device__ __forceinline__ uint4 ld_nc_v4(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

template <bool OWN_STATUS>
__global__ void __launch_bounds__(256, 4) append_kernel(const AppendArgs a) {
  allow_dependents();                              // the next call's first kernel waits for this one before it does anything
  const int seg = blockIdx.y;                      // (b*H_kv + h)*nb + t
  const int t = seg % a.nb;
  const int bh = seg / a.nb;
  const int h = bh % a.H_kv, b = bh / a.H_kv;
  const int part = threadIdx.x & 15;
  const int i0 = blockIdx.x * kAppendRowsPerCta + (threadIdx.x >> 4);
  const int i_end = min(a.B, (int)(blockIdx.x + 1) * kAppendRowsPerCta);
  const long long src_base = b * a.ks_b + h * a.ks_h + (long long)t * a.S_stride * a.ks_t;
  const long long dst_base = bh * a.c_seg_stride + (a.dst_off0 + (long long)t * a.B) * 128;
  int32_t* pos = a.pos + bh * a.pos_seg_stride + a.dst_off0 + (long long)t * a.B;
  const int32_t* idx = a.idx ? a.idx + (size_t)seg * a.B : nullptr;
  // launched beside the selection: nothing is read or written before that is complete
  grid_dependency_wait();
  constexpr int N = kAppendRowsPerCta / 16;        // rows of a thread, all under way together
  int src[N];
  uint4 kv[N], vv[N];
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int i = i0 + 16 * j;
    src[j] = i < i_end ? (idx ? idx[i] : i) : -1;
  }
#pragma unroll
  for (int j = 0; j < N; ++j) {
    if ((unsigned)src[j] < (unsigned)a.n_src_rows) {          // never read outside the segment
      const long long so = src_base + (long long)src[j] * a.ks_t + part * 8;
      kv[j] = ld_nc_v4(a.K + so);
      vv[j] = ld_nc_v4(a.V + so);
    }
  }
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int i = i0 + 16 * j;
    if ((unsigned)src[j] < (unsigned)a.n_src_rows) {
      const long long dof = dst_base + (long long)i * 128 + part * 8;
      *reinterpret_cast<uint4*>(a.Kc + dof) = kv[j];
      *reinterpret_cast<uint4*>(a.Vc + dof) = vv[j];
      if (part == 0) pos[i] = a.pos_base0 + t * a.S_stride + src[j];
    } else if (!OWN_STATUS && part == 0 && i < i_end) {
      atomicCAS(a.status, 0, kAppendBadIndex);
    }
  }
  if (OWN_STATUS && blockIdx.x == 0 && blockIdx.y == 0) {
    const int n = (int)gridDim.y * a.B;
    int bad = 0;
    for (int i = threadIdx.x; i < n; i += 256) bad |= (unsigned)a.idx[i] >= (unsigned)a.n_src_rows;
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) *a.status = bad ? kAppendBadIndex : 0;
  }
}

// ------------------------------------------------------------------------------------------------
// Consensus aggregation: the paper's Algorithm 1 line 3 scores a candidate with the attention it
// receives from all heads (and layers). For every sequence b and position i of the call's blocks,
// adds the scores and the collision counts of the H KV heads and either stores the sums or adds
// them to sums carried over from other layers.
// ------------------------------------------------------------------------------------------------
struct ConsensusArgs {
  const float4* s;        // [batch][H][n4]  (n4 = n_blocks * S / 4)
  const uint4* c;         // [batch][H][n4]
  float4* s_acc;          // [batch][n4]
  uint4* c_acc;           // [batch][n4]
  long long n4;
  int batch, H;
  int carry;              // 0: overwrite the sums, 1: add to them
};

__global__ void __launch_bounds__(256) consensus_kernel(const ConsensusArgs a) {
  const long long total = (long long)a.batch * a.n4;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const long long b = i / a.n4, j = i - b * a.n4;
    float4 fs = a.carry ? a.s_acc[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    uint4 cs = a.carry ? a.c_acc[i] : make_uint4(0u, 0u, 0u, 0u);
    for (int h = 0; h < a.H; ++h) {              // fixed order: deterministic sums
      const float4 x = a.s[(b * a.H + h) * a.n4 + j];
      const uint4 y = a.c[(b * a.H + h) * a.n4 + j];
      fs.x += x.x; fs.y += x.y; fs.z += x.z; fs.w += x.w;
      cs.x += y.x; cs.y += y.y; cs.z += y.z; cs.w += y.w;
    }
    a.s_acc[i] = fs;
    a.c_acc[i] = cs;
  }
}

}  // namespace lkv
