// How calls are cut into CTAs: rules on sizes alone, in plain C++ (tests/test_launch_rules.py compiles them for the host).
#pragma once

#ifdef __CUDACC__
#define LKV_HOST_DEVICE __host__ __device__
#else
#define LKV_HOST_DEVICE
#endif

namespace lkv {

constexpr int kDecTile = 64;            // cache rows per stage of the decode kernel
constexpr int kDecCtasPerSm = 2;
constexpr int kDecMaxSplit = 512;
constexpr int kDecMaxCluster = 16;

// Splits per (sequence, KV head) of a decode call whose partials go through memory: as many as fill the GPU's resident CTAs
// once, but at most eight of up to 24 tiles and a third of the tiles above: a tile costs a CTA 0.3 us, a split's partials cost
// the CTA that merges them about as much. us per layer in a captured graph, one tile per split against
// three: 26 tiles x 8 heads 7.2 / 6.9, 52 x 8 9.2 / 8.2, 103 x 8 11.2 / 10.9, 52 x 4 heads of seven queries
// 12.0 / 8.0; four tiles 5.0 / 5.3, hence the eight (short caches come here where clusters do not fit, see below). `heads`:
// sequences x KV heads.
inline int decode_splits(int num_sms, long long heads, long long len) {
  long long n = (long long)num_sms * kDecCtasPerSm / heads;
  const long long tiles = (len + kDecTile - 1) / kDecTile;
  const long long most = tiles <= 8 ? tiles : tiles <= 24 ? 8 : (tiles + 2) / 3;
  if (n > most) n = most;
  if (n > kDecMaxSplit) n = kDecMaxSplit;
  return n < 1 ? 1 : (int)n;
}

// Splits per (sequence, KV head) that merge inside a thread-block cluster (0: n_split of them by way of global memory, where
// a partial goes to memory, is counted there and comes back to the CTA that merges). us per layer in a captured graph, by way of
// memory against a cluster of at most eight: 8 heads of four queries and 4 tiles 5.2 / 3.5, 13 5.9 / 4.5, 26 7.2 / 6.3, 64 9.3 /
// 8.5, 103 10.8 / 10.9; 4 heads of seven queries and 26 tiles 7.4 / 5.4. A cluster has to find room on one part of the GPU:
// up to 256 CTAs in all do (264 of them 10.3 against 10.7, 280 14.3 against 10.8).
// With few heads eight CTAs of more than six tiles each fall behind splits that have an SM each; a cluster of sixteen does not:
// 4 heads of one query and 64 tiles 6.3 by way of memory / 7.0 eight / 6.4 sixteen, of four 6.7 / 7.2 / 6.5, 2 heads of two
// and 50 tiles 6.4 / 6.6 / 6.2, 6 heads of eight and 64 0.79 / 0.72 of the time by way of memory. From 8 heads on clusters of
// sixteen share SMs and are slower (8 heads of one, 50 tiles 6.5 / 6.7 / 7.2); with 7, of one over 56 tiles, 6.4 / 6.6 / 6.4
// over four layers' caches, but 7.7 / 7.5 / 7.7 over 24, which come from memory.
// Longer caches of few heads with many queries: the general path's merge costs as much as its partials are large, a cluster
// of sixteen reads the cache with fewer CTAs (one head of eight, 512 tiles 28.4 / 18.5; 4 heads of seven, 160 15.5 / 10.7, 512
// 24.4 / 21.2, 1024 35.1 / 36.2; 8 heads of four, 80 8.3 / 8.5, 255 16.8 / 16.7, 512 27.0 / 27.4; 4 heads of two, 80 6.4 / 6.5).
// The inequality is where the two cross for 1 to 9 heads and twelve lengths of 70 to 1024 tiles over four layers' caches. Where the
// caches of more layers come from memory in turn, clusters gain more: 16 layers, 8 heads of four, 66 tiles 9.0 / 8.7, 98 10.4 / 10.0, 160
// 13.2 / 12.4; 8 of five, 130 13.2 / 11.6; 9 of four, 80 9.9 / 9.2; 5 of three, 160 the same. Two layers, which the L2 cache holds,
// are up to 17 % slower of three to five queries (8 heads of four, 98 tiles 8.3 / 9.3): not what a model's decoding looks like. The
// results are 2.1e-7 instead of 2.7e-7 to 4e-7 from fp64 (normal keys, values and queries).
// `room(n)`: how many clusters of n (up to kDecMaxCluster) the device holds at once; asked only of a size about to be used. Only
// sizes of which it holds all the call's are used; a device, or a part of one, that holds none of a size would refuse the
// launch. The B200's 148 SMs hold 33 of eight, 14 of sixteen.
template <typename Room>
inline int decode_cluster(int num_sms, long long heads, int group, long long len, int n_split, Room&& room) {
  const long long tiles = (len + kDecTile - 1) / kDecTile;
  if (tiles <= 64) {
    if (tiles > 48 && heads <= 6 && 16 * heads <= num_sms && heads <= room(16)) return 16;
    long long n = (long long)num_sms * kDecCtasPerSm / heads;
    if (n > 8) n = 8;
    if (n > tiles) n = tiles;
    if (n <= 1) return 1;
    return n * heads <= 256 && heads <= room((int)n) ? (int)n : 0;
  }
  return 16 * heads <= num_sms && 3 * ((long long)group * n_split - 60) > tiles * (heads < 5 ? 6 - heads : 1) && heads <= room(16) ? 16 : 0;
}

// Whether the append of a select call (`ctas` CTAs, four of which an SM holds) is launched beside the selection, which hides its
// launch: its CTAs then start on the SMs that the selection's leave free. Up to half of the SMs in use by the selection,
// sixteen CTAs per SM: 24 segments of 2048 keys 42.7 -> 42.3 us a call, 16 of 8192 66.6 -> 65.6, 64 of 4096 (12 per SM) 94.7 ->
// 95.5 with 10-bit tables and 79.5 either way with 8-bit ones. With more segments the early CTAs crowd onto few SMs: up to eight
// per SM gain or lose 1 % (128 segments of 1024 keys 53.7 -> 53.3), more lose (80 of 4096, 15 per SM, 113.5 -> 115.5; 128,
// 11 per SM, 130.0 -> 133.3; 7808 CTAs 447 -> 469, four sequences of 128k tokens 628 -> 654). More segments than SMs: the selection itself
// starts in waves, and the append is released with the last of them, when there is nothing left to hide.
inline bool append_beside(int num_sms, int nseg, long long ctas) {
  return nseg <= num_sms && ctas <= (2 * nseg <= num_sms ? 16ll : 8ll) * num_sms;
}

// Score pass: log-sum-exp partials of a column that a warp fetches at a time. A segment with more is shared by a group's four warps.
constexpr int kLseBatch = 5;
LKV_HOST_DEVICE inline bool lse_split(int partials) { return partials > kLseBatch; }

// Slices of the projection pass of a select call. The SMs that held a query-signature CTA come 5 to 7 us later to the log-sum-exp
// pass, and every SM goes from pass to pass as it is done, so the last CTAs of the projection pass start that much later and
// the selection waited for them. They get fewer tiles, about 5 us less of them (eight of 160 columns), but not less than 55 %:
// sixteen calls of one block of 8192 tokens 978 -> 953 us (at least 50 %: 959, 60 %: 961, 70 %: 969), 64k in one call
// 203 -> 198, 32k 101.8 -> 98.8.
// With several chunks of hyperplanes the keys are read once for each, and the slices of the chunks lie abreast: CTAs with the same keys
// and different chunks stay together. One behind the other, unequal slices took a 128k layer from 399 to 432 us in a burst; abreast
// they leave it as it was (four sequences of 128k tokens 622 -> 614 us, 64k 179 -> 176). Keys that stay in the L2 cache lose less:
// 64 MiB 114.1 one behind the other, 113.1 abreast (four chunks), 48 MiB 79.9 / 79.0 (two), 32 MiB 63.7 / 63.2. 16 MiB in segments of 1024
// keys are better one behind the other, 40.5 / 40.8 and 47.7 / 48.0, hence the line between. Chunks that do not divide the grid
// cannot lie abreast: up to 64 MiB their slices are unequal one behind the other, above they are equal.
constexpr long long kProjAbreastBytes = 24ll << 20, kProjUnequalBytes = 64ll << 20;
struct ProjSlices {
  int n_late, w_late, w_early;   // the last n_late CTAs' slices are to the others' as w_late to w_early; all 0: equal slices
  int abreast;                   // > 1: the sequence is cut into that many equal parts, CTAs c, c + 1, ... at the same place of each
};

// `grid` CTAs over the tiles of `chunks` passes over keys of seg_tiles tiles, stat_rows columns each, behind a log-sum-exp pass of lse_ctas CTAs that started beside qsig_ctas of the
// query-signature kernel. Late are only the log-sum-exp CTAs that found no SM free: with few tiles in all, weights for every SM
// with a signature CTA gave some CTAs a second tile for nothing (64 tiles of one head 34.1 us a call with equal slices, 34.9 so
// weighted; 128 tiles of 16 segments 25.3 / 26.5, of 2 heads 28.4 / 29.9). A window scored in parts has an ordinary launch between the
// parts, behind which all CTAs start alike (144 segments of 1016 keys, 320 queries a head, 106.8 / 108.6).
inline ProjSlices proj_slices(int num_sms, int grid, long long seg_tiles, int chunks, int stat_rows, int lse_ctas, long long qsig_ctas,
                              int window_parts) {
  const long long key_bytes = seg_tiles * 128 * 256, n_tiles = seg_tiles * chunks;
  const bool divides = grid % chunks == 0;
  long long late = lse_ctas + qsig_ctas - num_sms;
  if (late > qsig_ctas) late = qsig_ctas;
  if (window_parts > 1 || late <= 0 || late >= grid || (!divides && key_bytes > kProjUnequalBytes)) return ProjSlices{0, 0, 0, 0};
  const long long per = 1000 * n_tiles / grid, less = 1000ll * 8 * 160 / stat_rows;      // thousandths of a tile
  ProjSlices s;
  s.abreast = divides && key_bytes > kProjAbreastBytes ? chunks : 1;
  s.n_late = (int)late;
  s.w_early = (int)(per < 1000000 ? per : 1000000);
  const long long w_less = less * s.w_early / per, most = s.w_early * 45ll / 100;
  s.w_late = s.w_early - (int)(w_less < most ? w_less : most);
  return s;
}

// First tile of the c-th of n slices of `part` tiles, of which the last are those of the CTAs that start late.
LKV_HOST_DEVICE inline long long weighted_begin(long long part, int c, int n, const ProjSlices& s) {
  const int early = n - (s.n_late + s.abreast - 1) / s.abreast;
  const long long w = (long long)(c < early ? c : early) * s.w_early + (long long)(c > early ? c - early : 0) * s.w_late;
  return part * w / ((long long)early * s.w_early + (long long)(n - early) * s.w_late);
}

}  // namespace lkv
