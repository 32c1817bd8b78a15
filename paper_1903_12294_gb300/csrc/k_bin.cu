// The §3.1 preprocessing index on sm_103a: which voxel every point sample lies in, and per
// (voxel, timestep) the sample count and the attribute aggregates.
//
// Determinism: attributes are summed as int64 fixed point, q = round_half_even(v * 2^k) with
// k = 62 - e - b (max|v| < 2^e, 2^b >= P*T + 1), so sums are exact and independent of order;
// the fp32 mean is a fixed sequence of IEEE fp32 operations on that sum. The paper's own GPU
// scheme keeps float running averages with atomics (§3.4), whose result depends on the order
// of arrival. No per-sample or per-voxel work touches the fp64 units.
//
// Schedule: a counting sort of the samples by voxel range ("bucket" of R consecutive voxels),
// so that the per-voxel sums are formed in shared memory rather than with global atomics
// (scattered L2 atomics run at a fixed rate that would bound the whole pass):
//   k_bin_keys     one thread per 4 samples of one point step: key[j][p], and per block (at least
//                  eight samples per bucket) a shared-memory histogram of buckets, added into
//                  hist[field step][bucket]
//   scan           offsets = exclusive prefix of hist (every bucket's slot range)
//   k_bin_place    one CTA per 8192 samples of one point step: each sample, read in order, takes
//                  its bucket's next slot (one global cursor per bucket) and is stored there as a
//                  (voxel, attributes) record; also the largest finite |v| per attribute
//
// Point samples may come on a finer time grid than the field (point step j falls in field step
// fstep[j]); the records of all point steps of a field step go to that step's buckets.
//   k_bin_reduce   one CTA per (bucket, field step): its records arrive by bulk copy while the
//                  counters are cleared and go to registers; counts by shared-memory atomics; the
//                  means form in shared memory, one thread per record, and every voxel's count
//                  and means are stored once; the voxel pairs of the records in their order, for
//                  the trajectory joins
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <atomic>

#include "msf_internal.cuh"

namespace msf {

constexpr int kBinPer = 4;             // samples per thread in the per-sample passes
constexpr int kBinNT = 512;            // threads per CTA of the sort and reduce passes
constexpr int kHistSmem = 8192;        // buckets counted in shared memory (else global atomics)

struct BinArgs {
  int nx, ny, nz, A, T;
  int Tp;                       // point steps; point step j falls in field step fstep[j]
  const int32_t* fstep;         // [Tp]
  const int32_t* pj0;           // [T + 1] first point step of each field step
  int64_t V, P;
  int64_t scale_n;              // point samples the fixed-point scale counts (P * Tp, or a
                                // whole dataset's when binning one slab of it)
  int logR, nb;                 // bucket = voxel >> logR; nb buckets
  int nblk;                     // sample blocks per point step of the keys pass
  int64_t chunk;                // samples per block of the keys pass
  int jbase;                    // keys and place passes: first point step of the launch
  const float* pos;             // [T][3][P]
  const float* attr;            // [T][A][P]
  int32_t* key;                 // [T][P]
  uint32_t* hist;               // [T][nb] samples per (field step, bucket)
  uint32_t* offs;               // [T][nb + 1] slot ranges: the step's record region (from
                                // pj0[t] * P) split by the exclusive prefix of hist; [t][nb]
                                // ends the step's records
  uint32_t* cursor;             // [T][nb] next free slot, from offs, one per kCurStride words
  char* pairs;                  // a uint2 per sample, every pair_bytes: its voxel, and the same
  uint32_t pair_bytes;          // point's voxel at the next point step (-1 at the last or outside
                                // the grid), side by side; or, where memory is short, the records'
                                // own pairs, which the reduce then writes once more as they are
  uint32_t* rec;                // [P*Tp][rec_words(A)] attribute values and the same voxel pair
  unsigned* err;                // bounded waits that gave up
  uint32_t* ovf;                // items (t * nb + bucket) left to the wide reduce
  uint32_t* novf;               // their number
  long long wait_cycles;        // limit of those waits (SM cycles)
  int pf_ahead;                 // reduce: items ahead whose records a block prefetches to L2
  unsigned* absmax;             // [A] float bits of max finite |v|
  unsigned long long* outside;  // [T]
  int32_t* count;               // [T][V]
  float* mean;                  // [A][T][V]
  long long* sumq;              // [A][T][V] or null
};

// k = 62 - e - b from the fp32 bits of max|v| (e: frexp exponent, 0 for zero) and the sample
// count (b: smallest with 2^b >= n + 1).
__host__ __device__ __forceinline__ int scale_exponent_bits(unsigned mbits, long long n) {
  int e = 0;
  if (mbits != 0u && mbits < 0x7F800000u) {
    const int E = (int)(mbits >> 23);
    if (E) {
      e = E - 126;
    } else {
#ifdef __CUDA_ARCH__
      const int L = 32 - __clz((int)mbits);
#else
      int L = 0;
      for (unsigned m = mbits; m; m >>= 1) ++L;
#endif
      e = L - 149;
    }
  }
  // b = the bit length of n (n >= 0): the smallest b with 2^b > n
#ifdef __CUDA_ARCH__
  const int b = n > 0 ? 64 - __clzll(n) : 0;
#else
  int b = 0;
  while (((long long)1 << b) < n + 1) ++b;
#endif
  return 62 - e - b;
}


// int64 -> fp32, round to nearest-even, with integer operations only (the hardware conversion
// of 64-bit integers issues on the fp64 pipe, which is narrow on this part). |s| < 2^62.
// The top 24 significant bits convert exactly; rounding adds one unit to the fp32 bit pattern
// (a carry out of the mantissa moves into the exponent, as it must); the exponent then rises by
// the number of dropped bits.
__device__ __forceinline__ float i64_to_f32_rn(long long s) {
  const unsigned long long u = s < 0 ? (unsigned long long)(-s) : (unsigned long long)s;
  const int lz = __clzll(u);
  uint32_t bits;
  if (lz >= 40) {
    bits = __float_as_uint(__uint2float_rn((uint32_t)u));  // < 2^24: exact
  } else {
    const int sh = 40 - lz;                                // dropped bits, 1..40
    const uint32_t m = (uint32_t)(u >> sh);                // 24 significant bits
    const unsigned long long rem = u << (64 - sh);         // dropped bits, left-aligned
    const uint32_t up = (rem > 0x8000000000000000ull) ||
                        (rem == 0x8000000000000000ull && (m & 1u));
    bits = __float_as_uint(__uint2float_rn(m)) + up + ((uint32_t)sh << 23);
  }
  return __uint_as_float(bits | (s < 0 ? 0x80000000u : 0u));
}

// Exact fp32 quotient x / c (IEEE round to nearest): a power-of-two count is an exact scaling,
// anything else takes the IEEE division. Both give the correctly rounded quotient.
__device__ __forceinline__ float div_count(float x, int c) {
  if ((c & (c - 1)) == 0) return __fmul_rn(x, pow2f(-(__ffs(c) - 1)));
  return __fdiv_rn(x, __int2float_rn(c));
}

// ---------------------------------------------------------------------------------------------
// pass 1: keys and the per-block bucket histograms
// ---------------------------------------------------------------------------------------------
// Block blk of point step j owns samples [blk * chunk, (blk + 1) * chunk). Its histogram is added
// into hist[fstep[j]][bucket] (one atomic per non-empty bucket), so that one exclusive scan
// yields every bucket's slot range, all point steps of a field step together.
template <bool SMEM>
__global__ void __launch_bounds__(256) k_bin_keys(const __grid_constant__ BinArgs b) {
  __shared__ uint32_t s_hist[SMEM ? kHistSmem : 1];
  const int t = b.jbase + blockIdx.y, blk = blockIdx.x;  // t: the point step
  uint32_t* hrow = b.hist + (int64_t)__ldg(b.fstep + t) * b.nb;
  if (SMEM) {
    for (int i = threadIdx.x; i < b.nb; i += 256) s_hist[i] = 0u;
    __syncthreads();
  }
  const int64_t pbeg = (int64_t)blk * b.chunk;
  const int64_t pend = min(pbeg + b.chunk, b.P);
  const float* pt = b.pos + (int64_t)t * 3 * b.P;
  int out = 0;
  for (int64_t q0 = pbeg + threadIdx.x; q0 < pend; q0 += 256 * kBinPer) {
    float px[kBinPer], py[kBinPer], pz[kBinPer];
#pragma unroll
    for (int j = 0; j < kBinPer; ++j) {
      const int64_t p = q0 + j * 256;
      const bool in = p < pend;
      px[j] = in ? __ldcs(pt + p) : NAN;
      py[j] = in ? __ldcs(pt + b.P + p) : NAN;
      pz[j] = in ? __ldcs(pt + 2 * b.P + p) : NAN;
    }
#pragma unroll
    for (int j = 0; j < kBinPer; ++j) {
      const int64_t p = q0 + j * 256;
      if (p >= pend) continue;
      const int32_t k = voxel_of(px[j], py[j], pz[j], b.nx, b.ny, b.nz);
      __stcs(b.key + (int64_t)t * b.P + p, k);
      if (k < 0) {
        ++out;
      } else if (SMEM) {
        atomicAdd(s_hist + (k >> b.logR), 1u);
      } else {
        atomicAdd(hrow + (k >> b.logR), 1u);
      }
    }
  }
  const int tot = __reduce_add_sync(0xFFFFFFFFu, out);
  if ((threadIdx.x & 31) == 0 && tot) atomicAdd(b.outside + t, (unsigned long long)tot);
  if (SMEM) {
    __syncthreads();
    for (int i = threadIdx.x; i < b.nb; i += 256)
      if (s_hist[i]) atomicAdd(hrow + i, s_hist[i]);
  }
}

// ---------------------------------------------------------------------------------------------
// pass 2: records in bucket order (and the attribute maxima)
// ---------------------------------------------------------------------------------------------
// A record is the sample's attributes, its voxel and the same point's voxel at the next point step
// (what a trajectory link joins), in one, two or three 16-byte units so that it is written by one
// store (of 16 or 32 bytes; three for seven or eight attributes). The block reads its samples in
// order (coalesced keys and attributes, several per thread in flight) and sends each to the next
// free slot of its bucket, taken from one global cursor per (field step, bucket). The pass is
// bound by its scattered requests to L2, half of which cross to the other die: a slot atomic and
// a store per sample (voxel pair and attributes stored apart, 8M particles x 24 steps, A = 4: 4.59
// ms; together 2.80 ms, although a record then has 32 bytes instead of 24). Records thus fill
// every bucket's range front to back in the order they arrive from all blocks, so a partly
// written sector is completed within microseconds while it is still in L2 (per-block slot
// ranges would leave one partial sector per block and bucket open for a block's whole life and
// push them out to DRAM half-written: ranks from the keys pass instead of the slot atomics took
// 7.6 ms). The order within a bucket changes nothing downstream: counts and fixed-point sums are
// exact.
__host__ __device__ constexpr int rec_words(int A) { return A <= 2 ? 4 : A <= 6 ? 8 : 12; }
// first word of the voxel pair (the attributes come first)
__host__ __device__ constexpr int rec_pair(int A) { return A <= 2 ? 2 : A <= 4 ? 4 : A <= 6 ? 6 : 8; }

constexpr int kPlaceNT = 512;                  // threads per block of the place pass
constexpr int kPlacePer = 4;                   // samples per thread in flight
constexpr int kPlaceChunk = 8192;              // samples per block of the place pass
constexpr int kChunkMax = 65536;               // samples per block of the keys pass, at most
constexpr int kCurStride = 32;                 // words between two buckets' cursors: one per
                                               // 128-byte line, so that the slot atomics of
                                               // neighbouring buckets do not queue on one line

__device__ __forceinline__ void store32(uint32_t* p, const uint32_t (&w)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]),
               "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}

template <int A>
__device__ __forceinline__ void put_record(const BinArgs& b, uint32_t slot, int32_t k, int32_t kn,
                                           const float (&av)[A > 0 ? A : 1]) {
  constexpr int RW = rec_words(A), VO = rec_pair(A);
  uint32_t w[RW];
#pragma unroll
  for (int i = 0; i < RW; ++i) w[i] = i < A ? __float_as_uint(av[i < A ? i : 0]) : 0u;
  w[VO] = (uint32_t)k;
  w[VO + 1] = (uint32_t)kn;
  uint32_t* dst = b.rec + (size_t)slot * RW;
  if constexpr (RW == 8) {
    store32(dst, w);
  } else {
#pragma unroll
    for (int i = 0; i < RW; i += 4)
      *reinterpret_cast<uint4*>(dst + i) = make_uint4(w[i], w[i + 1], w[i + 2], w[i + 3]);
  }
}

// One block per field step t of [t0, t0 + gridDim.x): the step's records take the region that
// starts at pj0[t] * P (room for all of its point steps' samples), so that field steps bin
// independently of each other; the exclusive prefix of its bucket counts splits the region into
// the buckets' slot ranges (offs[t][nb]: the end of its records), and the slot cursors start
// there.
constexpr int kScanNT = 1024;

__global__ void __launch_bounds__(kScanNT) k_bin_scan_steps(const __grid_constant__ BinArgs b,
                                                             int t0) {
  __shared__ uint32_t s_w[kScanNT / 32];
  const int t = t0 + (int)blockIdx.x;
  const uint32_t* h = b.hist + (int64_t)t * b.nb;
  uint32_t* o = b.offs + (int64_t)t * (b.nb + 1);
  uint32_t* c = b.cursor + (int64_t)t * b.nb * kCurStride;
  const uint32_t base = (uint32_t)((int64_t)__ldg(b.pj0 + t) * b.P);
  const int per = (b.nb + kScanNT - 1) / kScanNT;
  const int lo = min((int)threadIdx.x * per, b.nb), hi = min(lo + per, b.nb);
  uint32_t sum = 0;
  for (int i = lo; i < hi; ++i) sum += h[i];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t x = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) s_w[w] = x;
  __syncthreads();
  if (w == 0) {
    uint32_t y = s_w[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t z = __shfl_up_sync(0xFFFFFFFFu, y, d);
      if (lane >= d) y += z;
    }
    s_w[lane] = y;
  }
  __syncthreads();
  uint32_t run = base + (x - sum) + (w ? s_w[w - 1] : 0u);
  for (int i = lo; i < hi; ++i) {
    o[i] = run;
    c[(int64_t)i * kCurStride] = run;
    run += h[i];
  }
  if (threadIdx.x == kScanNT - 1) o[b.nb] = base + s_w[kScanNT / 32 - 1];
}

template <int A>
__global__ void __launch_bounds__(kPlaceNT) k_bin_place(const __grid_constant__ BinArgs b) {
  __shared__ unsigned s_max[A > 0 ? A : 1];
  const int j = b.jbase + blockIdx.y, blk = blockIdx.x;  // j: the point step
  uint32_t* crow = b.cursor + (int64_t)__ldg(b.fstep + j) * b.nb * kCurStride;
  if ((int)threadIdx.x < A) s_max[threadIdx.x] = 0u;
  __syncthreads();
  const int64_t pbeg = (int64_t)blk * kPlaceChunk;
  const int64_t pend = min(pbeg + kPlaceChunk, b.P);
  const int32_t* krow = b.key + (int64_t)j * b.P;
  const bool nxt = j + 1 < b.Tp;  // the next point step's keys follow this step's row
  const float* arow = b.attr + (int64_t)j * A * b.P;
  unsigned lmax[A > 0 ? A : 1];
#pragma unroll
  for (int a = 0; a < (A > 0 ? A : 1); ++a) lmax[a] = 0u;
  for (int64_t q0 = pbeg + threadIdx.x; q0 < pend; q0 += (int64_t)kPlaceNT * kPlacePer) {
    int32_t k[kPlacePer], kn[kPlacePer];
    float av[kPlacePer][A > 0 ? A : 1];
#pragma unroll
    for (int u = 0; u < kPlacePer; ++u) {
      const int64_t p = q0 + (int64_t)u * kPlaceNT;
      const bool in = p < pend;
      k[u] = in ? __ldcs(krow + p) : -1;
      kn[u] = (in && nxt) ? __ldg(krow + b.P + p) : -1;
#pragma unroll
      for (int a = 0; a < (A > 0 ? A : 1); ++a)
        av[u][a] = (in && A > 0) ? __ldcs(arow + (int64_t)a * b.P + p) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kPlacePer; ++u) {
#pragma unroll
      for (int a = 0; a < A; ++a)
        if (isfinite(av[u][a])) lmax[a] = max(lmax[a], __float_as_uint(fabsf(av[u][a])));
      if (k[u] < 0) continue;
      const uint32_t slot = atomicAdd(crow + (k[u] >> b.logR) * kCurStride, 1u);
      put_record<A>(b, slot, k[u], kn[u], av[u]);
    }
  }
#pragma unroll
  for (int a = 0; a < A; ++a) {
    const unsigned m = __reduce_max_sync(0xFFFFFFFFu, lmax[a]);
    if ((threadIdx.x & 31) == 0 && m) atomicMax(s_max + a, m);
  }
  __syncthreads();
  if ((int)threadIdx.x < A && s_max[threadIdx.x]) atomicMax(b.absmax + threadIdx.x, s_max[threadIdx.x]);
}

// ---------------------------------------------------------------------------------------------
// pass 3: per (bucket, timestep) counts, sums, means
// ---------------------------------------------------------------------------------------------
// Bulk copy of records [a0, a0 + n) into a staging area (a record is whole 16-byte units).
template <int A>
__device__ __forceinline__ void reduce_issue(const BinArgs& b, uint32_t a0, uint32_t n,
                                             uint32_t* s_st, uint64_t* bar) {
  constexpr int RW = rec_words(A);
  mbar_expect_tx(bar, 4u * n * RW);
  bulk_g2s(s_st, b.rec + (size_t)a0 * RW, 4u * n * RW, bar);
}

__device__ __forceinline__ uint2* pair_at(const BinArgs& b, uint32_t r) {
  return reinterpret_cast<uint2*>(b.pairs + (size_t)r * b.pair_bytes);
}

// record range [r0, r1) of the item (field step t, bucket): the slots of its point steps
__device__ __forceinline__ void item_range(const BinArgs& b, int t, int bucket, uint32_t& r0,
                                           uint32_t& r1) {
  r0 = r1 = 0u;
  if (b.P == 0) return;
  const int64_t h = (int64_t)t * (b.nb + 1) + bucket;
  r0 = __ldg(b.offs + h);
  r1 = __ldg(b.offs + h + 1);
}

// the fixed-point exponent of attribute a and the two exact factors of 2^-k
__device__ __forceinline__ void item_scale(const BinArgs& b, int a, int* s_k, float* s_f1,
                                           float* s_f2) {
  const int k = scale_exponent_bits(b.absmax[a], (long long)b.scale_n);
  s_k[a] = k;
  s_f1[a] = pow2f(-(k / 2));
  s_f2[a] = pow2f(-(k - k / 2));
}

// The staged record q: attribute values and the voxel pair.
template <int A>
__device__ __forceinline__ uint2 staged_record(const uint32_t* s_st, int q,
                                               float (&v)[A > 0 ? A : 1]) {
  constexpr int RW = rec_words(A), VO = rec_pair(A);
  uint32_t w[RW];
#pragma unroll
  for (int i = 0; i < RW; i += 4) {
    const uint4 x = reinterpret_cast<const uint4*>(s_st)[(q * RW + i) / 4];
    w[i] = x.x, w[i + 1] = x.y, w[i + 2] = x.z, w[i + 3] = x.w;
  }
#pragma unroll
  for (int a = 0; a < A; ++a) v[a] = __uint_as_float(w[a]);
  return make_uint2(w[VO], w[VO + 1]);
}

// One block per item (field step t, bucket): the bucket's records (at most red_stage(A) of them,
// a few per thread) arrive by bulk copy while the voxel counters are cleared and go to registers,
// their attributes quantised; the staging area then becomes the bucket's means. A record's
// shared-memory atomic on its voxel's counter (two 16-bit counters per word) counts the voxel's
// records and gives the record its place among them. What a voxel needs depends on its count:
//   1   the record's thread forms the mean: (float)sum / 1 is the quantised value itself;
//   2   the second record leaves its quantised values in the voxel's mean, the first adds its
//       own: both are exact in fp32, so one fp32 addition rounds their exact sum once, as
//       converting the int64 sum does;
//   3+  exact int64 sums in a compact list of such voxels (two 32-bit atomics with the carry),
//       then the fp32 mean chain, one thread per voxel.
// Then the block streams counts and means out, four voxels per thread with 16-byte stores, NaN
// where there are no records (storing NaN everywhere and the means over it, one 4-byte store per
// non-empty voxel and attribute, issued twice the stores; sorting the records by voxel first and
// quantising in the divergent parts made it 16,000 instructions a bucket). 8M records x 24 steps,
// 256^3 voxels, A = 4: 4.17 ms before, 3.50 ms now. A bucket with more records than the staging
// area holds is listed for k_bin_reduce_wide and left to it.
__host__ __device__ constexpr int red_stage(int A) { return A <= 6 ? 2048 : 1536; }

// The quantised value of v as fp32, q = round_half_even(v * 2^k): exact (a 24-bit mantissa shifted
// left, or an integer below 2^24), so it is formed in fp32: v * 2^k is exact (two power-of-two
// factors u1, u2; a product too small for a normal fp32 is below one half either way), rounding
// it to an integer (half to even) is the quantisation, and adding +0 turns a negative zero into
// the positive zero the integer path gives. Non-finite v gives 0.
__device__ __forceinline__ float quantised(float v, float u1, float u2) {
  return isfinite(v) ? __fadd_rn(rintf(__fmul_rn(__fmul_rn(v, u1), u2)), 0.0f) : 0.0f;
}

// an integer held in fp32, as int64 (integer operations: the hardware conversion issues on the
// narrow fp64 pipe)
__device__ __forceinline__ long long exact_ll(float q) {
  const uint32_t b = __float_as_uint(q);
  const int e = (int)((b >> 23) & 0xFFu) - 150;
  if (e < -23) return 0;  // zero
  const long long m = (long long)((b & 0x7FFFFFu) | 0x800000u);
  const long long u = e >= 0 ? m << e : m >> -e;
  return (b >> 31) ? -u : u;
}

template <int A, bool KEEP>
__global__ void __launch_bounds__(kBinNT, A <= 4 ? 3 : 2) k_bin_reduce(const __grid_constant__ BinArgs b) {
  constexpr int A1 = A > 0 ? A : 1;
  constexpr int SS = red_stage(A), PER = SS / kBinNT, MANY = SS / 3;
  extern __shared__ __align__(16) uint32_t s_red[];
  const int R = 1 << b.logR;
  uint32_t* s_cnt = s_red;                              // [R] 16-bit counters, two per word
  uint32_t* s_area = s_red + R / 2;                     // staged records, then
  float* s_mean = reinterpret_cast<float*>(s_area);     // [A][R] and
  uint32_t* s_sum = s_area + A * R;                     // [MANY][A] low, high
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ uint16_t s_many[MANY];
  __shared__ int s_nmany;
  __shared__ float4 s_sc[A1];  // 2^k as two factors, 2^-k as two factors
  const int bucket = blockIdx.x, t = blockIdx.y;  // t: the field step
  uint32_t r0, r1;
  item_range(b, t, bucket, r0, r1);
  if (r1 - r0 > (uint32_t)SS) {  // too many records to stage: the wide pass takes it
    if (threadIdx.x == 0) b.ovf[atomicAdd(b.novf, 1u)] = (uint32_t)t * (uint32_t)b.nb + bucket;
    return;
  }
  const int n = (int)(r1 - r0);
  if (threadIdx.x == 0) {
    mbar_init(&s_bar, 1);
    if (n) reduce_issue<A>(b, r0, (uint32_t)n, s_area, &s_bar);
    // the records of the item one wave of blocks later, into L2 (its block then copies from
    // there instead of from DRAM)
    const int64_t nxt = (int64_t)t * b.nb + bucket + b.pf_ahead;
    if (nxt < (int64_t)b.T * b.nb) {
      uint32_t q0, q1;
      item_range(b, (int)(nxt / b.nb), (int)(nxt % b.nb), q0, q1);
      if (q1 > q0 && q1 - q0 <= (uint32_t)SS)
        prefetch_l2(b.rec + (size_t)q0 * rec_words(A), 4u * rec_words(A) * (q1 - q0));
    }
    s_nmany = 0;
  }
  if ((int)threadIdx.x < A) {
    const int k = scale_exponent_bits(b.absmax[threadIdx.x], (long long)b.scale_n);
    s_sc[threadIdx.x] = make_float4(pow2f(k / 2), pow2f(k - k / 2), pow2f(-(k / 2)),
                                    pow2f(-(k - k / 2)));
  }
  for (int q = threadIdx.x; q < R / 8; q += kBinNT)
    reinterpret_cast<uint4*>(s_cnt)[q] = make_uint4(0u, 0u, 0u, 0u);
  const int64_t vbase = (int64_t)bucket << b.logR;
  const int nv = (int)min((int64_t)R, b.V - vbase);
  auto keep = [&](int a, int v, long long sum) {  // the int64 sum of a non-empty voxel
    if (KEEP) b.sumq[((int64_t)a * b.T + t) * b.V + vbase + v] = sum;
  };
  if (KEEP)  // zero sums; those of the non-empty voxels are stored over them behind a barrier
    for (int a = 0; a < A; ++a)
      for (int q = threadIdx.x; q < nv; q += kBinNT) keep(a, q, 0ll);
  __syncthreads();
  if (n) {
    const bool ok = mbar_wait(&s_bar, 0, b.wait_cycles);
    if (__syncthreads_or(!ok)) {  // the copy did not arrive in time
      if (threadIdx.x == 0) {
        atomicAdd(b.err, 1u);
        mbar_wait(&s_bar, 0);      // let it land before the block exits
      }
      return;
    }
    int v[PER], place[PER];
    float x[PER][A1];  // quantised attributes
    char* pair = reinterpret_cast<char*>(pair_at(b, r0 + threadIdx.x));
    const uint32_t pair_step = kBinNT * b.pair_bytes;
#pragma unroll
    for (int i = 0; i < PER; ++i, pair += pair_step) {
      const int q = (int)threadIdx.x + kBinNT * i;
      v[i] = -1;
      place[i] = 0;
      if (q < n) {
        const uint2 vn = staged_record<A>(s_area, q, x[i]);
        __stcs(reinterpret_cast<uint2*>(pair), vn);
        v[i] = (int)(vn.x & (uint32_t)(R - 1));
        const int sh = (v[i] & 1) << 4;
        place[i] = (int)((atomicAdd(s_cnt + (v[i] >> 1), 1u << sh) >> sh) & 0xFFFFu);
#pragma unroll
        for (int a = 0; a < A; ++a) {
          const float2 up = *reinterpret_cast<const float2*>(&s_sc[a]);
          x[i][a] = quantised(x[i][a], up.x, up.y);
        }
      }
    }
    __syncthreads();  // the counts are complete, the staging area is read
    if constexpr (A > 0) {
      auto mean_of = [&](int a, float m) { return __fmul_rn(__fmul_rn(m, s_sc[a].z), s_sc[a].w); };
      int c[PER];
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        c[i] = 0;
        if (v[i] < 0) continue;
        c[i] = (int)((s_cnt[v[i] >> 1] >> ((v[i] & 1) << 4)) & 0xFFFFu);
        if (c[i] <= 2 && place[i] == c[i] - 1) {
#pragma unroll
          for (int a = 0; a < A; ++a) {
            s_mean[a * R + v[i]] = c[i] == 1 ? mean_of(a, x[i][a]) : x[i][a];
            if (c[i] == 1) keep(a, v[i], exact_ll(x[i][a]));
          }
        } else if (c[i] > 2 && place[i] == 0) {
          const int slot = atomicAdd(&s_nmany, 1);
          s_many[slot] = (uint16_t)v[i];
          s_mean[v[i]] = __int_as_float(slot);
#pragma unroll
          for (int a = 0; a < A; ++a)
            *reinterpret_cast<uint2*>(s_sum + 2 * (slot * A + a)) = make_uint2(0u, 0u);
        }
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        if (c[i] == 2 && place[i] == 0) {
#pragma unroll
          for (int a = 0; a < A; ++a) {
            const float q1 = s_mean[a * R + v[i]];
            s_mean[a * R + v[i]] = mean_of(a, __fmul_rn(__fadd_rn(x[i][a], q1), 0.5f));
            keep(a, v[i], exact_ll(x[i][a]) + exact_ll(q1));
          }
        } else if (c[i] > 2) {
          const int slot = __float_as_int(s_mean[v[i]]);
#pragma unroll
          for (int a = 0; a < A; ++a) {
            const unsigned long long q = (unsigned long long)exact_ll(x[i][a]);
            uint32_t* p = s_sum + 2 * (slot * A + a);
            const uint32_t lo = (uint32_t)q, old = atomicAdd(p, lo);
            atomicAdd(p + 1, (uint32_t)(q >> 32) + (old + lo < old ? 1u : 0u));
          }
        }
      }
      __syncthreads();
      for (int i = threadIdx.x; i < s_nmany; i += kBinNT) {
        const int u = s_many[i];
        const int m = (int)((s_cnt[u >> 1] >> ((u & 1) << 4)) & 0xFFFFu);
#pragma unroll
        for (int a = 0; a < A; ++a) {
          const uint2 w = *reinterpret_cast<const uint2*>(s_sum + 2 * (i * A + a));
          const long long sum = (long long)(((unsigned long long)w.y << 32) | w.x);
          s_mean[a * R + u] = mean_of(a, div_count(i64_to_f32_rn(sum), m));
          keep(a, u, sum);
        }
      }
      __syncthreads();
    }
  }
  const float qnan = __int_as_float(0x7fc00000);
  for (int q = 4 * (int)threadIdx.x; q < nv; q += 4 * kBinNT) {
    const uint2 w = *reinterpret_cast<const uint2*>(s_cnt + q / 2);
    const uint4 c4 = make_uint4(w.x & 0xFFFFu, w.x >> 16, w.y & 0xFFFFu, w.y >> 16);
    const int64_t o = (int64_t)t * b.V + vbase + q;
    if ((b.V & 3) == 0) {  // nv is then a multiple of four
      __stcs(reinterpret_cast<uint4*>(b.count + o), c4);
#pragma unroll
      for (int a = 0; a < A; ++a) {
        const float4 m4 = *reinterpret_cast<const float4*>(s_mean + a * R + q);
        __stcs(reinterpret_cast<float4*>(b.mean + (int64_t)a * b.T * b.V + o),
               make_float4(c4.x ? m4.x : qnan, c4.y ? m4.y : qnan, c4.z ? m4.z : qnan,
                           c4.w ? m4.w : qnan));
      }
    } else {
      const uint32_t cc[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (q + e >= nv) break;
        __stcs(b.count + o + e, (int)cc[e]);
#pragma unroll
        for (int a = 0; a < A; ++a)
          __stcs(b.mean + (int64_t)a * b.T * b.V + o + e, cc[e] ? s_mean[a * R + q + e] : qnan);
      }
    }
  }
}

// Buckets with more records than k_bin_reduce stages (listed by it): the records arrive in
// pieces of wide_piece; counts and fixed-point sums accumulate in shared memory (sums [A][R] u64,
// counts [R] u32, then the staging buffer, reused for the means [A][R] f32 and the non-empty
// lists once the records are in). After the records, every warp owns 128 voxels (four
// per lane): it lists its non-empty ones, forms their means and stores its outputs. Blocks take
// listed items in turn. A piece of seven or eight attributes is what the means need anyway (1024
// records a piece, 1M x 4 samples on 6 x 6 x 6 voxels, A = 8: 1.69 ms, so 1.52).
__host__ __device__ constexpr int wide_piece(int A) { return A <= 6 ? 2048 : 1536; }

template <int A, bool KEEP>
__global__ void __launch_bounds__(kBinNT, 1) k_bin_reduce_wide(const __grid_constant__ BinArgs b) {
  constexpr uint32_t PW = wide_piece(A);
  extern __shared__ __align__(16) unsigned long long s_dyn64[];
  const int R = 1 << b.logR;
  unsigned long long* s_sum = s_dyn64;                                    // [A][R]
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_dyn64 + (size_t)A * R);  // [R]
  uint32_t* s_st = s_cnt + R;                                             // [PW] records
  float* s_mean = reinterpret_cast<float*>(s_st);                         // after the records
  uint32_t* s_list = s_st + (size_t)A * R;
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ int s_k[A > 0 ? A : 1];
  __shared__ float s_f1[A > 0 ? A : 1], s_f2[A > 0 ? A : 1];
  if (threadIdx.x == 0) mbar_init(&s_bar, 1);
  if ((int)threadIdx.x < A) item_scale(b, threadIdx.x, s_k, s_f1, s_f2);
  uint32_t phase = 0;  // copies this block has waited for (the mbarrier's phase)
  const uint32_t nwide = *b.novf;
  for (uint32_t it = blockIdx.x; it < nwide; it += gridDim.x) {
  __syncthreads();  // the previous item's reads of shared memory are done
  const uint32_t itm = b.ovf[it];
  const int bucket = (int)(itm % (uint32_t)b.nb), t = (int)(itm / (uint32_t)b.nb);
  uint32_t r0, r1;
  item_range(b, t, bucket, r0, r1);
  const int npiece = (int)((r1 - r0 + PW - 1) / PW);
  if (threadIdx.x == 0 && npiece) {
    fence_proxy_async_smem();
    reduce_issue<A>(b, r0, min(PW, r1 - r0), s_st, &s_bar);
  }
  {
    uint4* z = reinterpret_cast<uint4*>(s_dyn64);
    const int n16 = (int)(((size_t)A * R * 8 + (size_t)R * 4) / 16);
    for (int q = threadIdx.x; q < n16; q += kBinNT) z[q] = make_uint4(0, 0, 0, 0);
  }
  __syncthreads();
  for (int piece = 0; piece < npiece; ++piece, ++phase) {
    const bool ok = mbar_wait(&s_bar, phase & 1u, b.wait_cycles);
    if (__syncthreads_or(!ok)) {  // the copy did not arrive in time
      if (threadIdx.x == 0) {
        atomicAdd(b.err, 1u);
        mbar_wait(&s_bar, phase & 1u);  // let it land before the block exits
      }
      return;
    }
    const uint32_t a0 = r0 + (uint32_t)piece * PW;
    const int m = (int)min(PW, r1 - a0);
    for (int q = threadIdx.x; q < m; q += kBinNT) {
      float vv[A > 0 ? A : 1];
      const uint2 vn = staged_record<A>(s_st, q, vv);
      __stcs(pair_at(b, a0 + q), vn);
      const uint32_t v = vn.x & (uint32_t)(R - 1);  // voxel within the bucket
      atomicAdd(s_cnt + v, 1u);
#pragma unroll
      for (int a = 0; a < A; ++a)
        atomicAdd(s_sum + (size_t)a * R + v, (unsigned long long)quantise(vv[a], s_k[a]));
    }
    __syncthreads();
    if (piece + 1 < npiece && threadIdx.x == 0) {
      fence_proxy_async_smem();  // the reads above before the next copy overwrites them
      const uint32_t a1 = a0 + PW;
      reduce_issue<A>(b, a1, min(PW, r1 - a1), s_st, &s_bar);
    }
  }
  const float qnan = __int_as_float(0x7fc00000);
  const int lane = threadIdx.x & 31;
  const int wq = threadIdx.x & ~31;  // first thread of this warp
  const int64_t vbase = (int64_t)bucket << b.logR;
  const int nv = (int)min((int64_t)R, b.V - vbase);
  for (int i0 = 0; i0 < R; i0 += 4 * kBinNT) {
    const int wbase = i0 + 4 * wq;  // this warp's voxels [wbase, wbase + 128)
    if (wbase >= R) break;          // warp-uniform
    const int q = wbase + 4 * lane;
    uint4 c4 = make_uint4(0u, 0u, 0u, 0u);
    if (q < R) c4 = *reinterpret_cast<const uint4*>(s_cnt + q);
    // this warp's non-empty voxels, listed in order
    const int nz = (c4.x != 0u) + (c4.y != 0u) + (c4.z != 0u) + (c4.w != 0u);
    int x = nz;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= o) x += y;
    }
    const int nw = __shfl_sync(0xFFFFFFFFu, x, 31);
    if (A > 0 && nw) {
      int pos = wbase + x - nz;
      if (c4.x) s_list[pos++] = (uint32_t)q;
      if (c4.y) s_list[pos++] = (uint32_t)(q + 1);
      if (c4.z) s_list[pos++] = (uint32_t)(q + 2);
      if (c4.w) s_list[pos] = (uint32_t)(q + 3);
      __syncwarp();
      for (int j = lane; j < nw; j += 32) {
        const int u = (int)s_list[wbase + j];
        const int c = (int)s_cnt[u];
#pragma unroll
        for (int a = 0; a < A; ++a)
          s_mean[(size_t)a * R + u] = __fmul_rn(
              __fmul_rn(div_count(i64_to_f32_rn((long long)s_sum[(size_t)a * R + u]), c),
                        s_f1[a]),
              s_f2[a]);
      }
      __syncwarp();
    }
    if (q >= nv) continue;
    const int64_t v = vbase + q;
    if ((b.V & 3) == 0) {  // nv is then a multiple of four
      __stcs(reinterpret_cast<uint4*>(b.count + (int64_t)t * b.V + v), c4);
#pragma unroll
      for (int a = 0; a < A; ++a) {
        const int64_t o = ((int64_t)a * b.T + t) * b.V + v;
        const float4 m4 = *reinterpret_cast<const float4*>(s_mean + (size_t)a * R + q);
        __stcs(reinterpret_cast<float4*>(b.mean + o),
               make_float4(c4.x ? m4.x : qnan, c4.y ? m4.y : qnan, c4.z ? m4.z : qnan,
                           c4.w ? m4.w : qnan));
        if (KEEP) {
          const unsigned long long* sq = s_sum + (size_t)a * R + q;
          __stcs(reinterpret_cast<longlong2*>(b.sumq + o),
                 make_longlong2((long long)sq[0], (long long)sq[1]));
          __stcs(reinterpret_cast<longlong2*>(b.sumq + o + 2),
                 make_longlong2((long long)sq[2], (long long)sq[3]));
        }
      }
    } else {
      const uint32_t cc[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (q + e >= nv) break;
        __stcs(b.count + (int64_t)t * b.V + v + e, (int)cc[e]);
#pragma unroll
        for (int a = 0; a < A; ++a) {
          const int64_t o = ((int64_t)a * b.T + t) * b.V + v + e;
          __stcs(b.mean + o, cc[e] ? s_mean[(size_t)a * R + q + e] : qnan);
          if (KEEP) __stcs(b.sumq + o, (long long)s_sum[(size_t)a * R + q + e]);
        }
      }
    }
  }
  }  // items
}

// Bucket width: 2048 voxels, wider when the grid has more buckets than the shared-memory
// histograms hold and the wide pass's sums still fit.
static size_t reduce_smem(int A, int logR) {
  const size_t R = (size_t)1 << logR, SS = red_stage(A);
  const size_t staged = 4 * SS * rec_words(A);
  const size_t means = 4 * R * A + 8 * (SS / 3) * A;  // and the int64 sums
  return 2 * R + std::max(staged, means);
}
static size_t reduce_wide_smem(int A, int logR) {
  const size_t R = (size_t)1 << logR;
  const size_t staged = 4 * (size_t)wide_piece(A) * rec_words(A);
  return R * (8 * (size_t)A + 4) + std::max(staged, 4 * R * A + 4 * R);
}

static int max_bucket_log2(int A) {
  return reduce_wide_smem(A, 12) <= (size_t)220 * 1024 ? 12 : 11;
}
static int bucket_log2(int A, int64_t V) {
  return ((V + 2047) >> 11) > kHistSmem ? max_bucket_log2(A) : 11;
}

// phase 0: keys of point steps [j0, j0 + nj); 1: their records; 2: every (bucket, field step);
// 3: the nj of them that phase 2 listed
template <int A>
static void launch_bin(msf_ctx* ctx, BinArgs b, bool keep, int phase, bool smem, cudaStream_t s,
                       int j0, int nj) {
  b.jbase = j0;
  const dim3 gs((unsigned)b.nblk, (unsigned)nj);  // (block, point step)
  const dim3 gp((unsigned)((b.P + kPlaceChunk - 1) / kPlaceChunk), (unsigned)nj);
  if (phase == 0) {
    ScopedKernel k(ctx, "k_bin_keys", s);
    if (smem) k_bin_keys<true><<<gs, 256, 0, s>>>(b);
    else k_bin_keys<false><<<gs, 256, 0, s>>>(b);
  } else if (phase == 1) {
    ScopedKernel k(ctx, "k_bin_place", s);
    k_bin_place<A><<<gp, kPlaceNT, 0, s>>>(b);
  } else if (phase == 2) {
    {
      ScopedKernel k(ctx, "k_bin_reduce", s);
      const size_t sm = reduce_smem(A, b.logR);
      const dim3 gr((unsigned)b.nb, (unsigned)b.T);
      if (keep) {
        static std::atomic<uint64_t> set{0};
        ensure_smem_attr(k_bin_reduce<A, true>, reduce_smem(A, max_bucket_log2(A)), set);
        k_bin_reduce<A, true><<<gr, kBinNT, sm, s>>>(b);
      } else {
        static std::atomic<uint64_t> set{0};
        ensure_smem_attr(k_bin_reduce<A, false>, reduce_smem(A, max_bucket_log2(A)), set);
        k_bin_reduce<A, false><<<gr, kBinNT, sm, s>>>(b);
      }
    }
  } else {
    {
      // the buckets k_bin_reduce listed (more records than it stages)
      ScopedKernel k(ctx, "k_bin_reduce_wide", s);
      const size_t sm = reduce_wide_smem(A, b.logR);
      const unsigned g = (unsigned)std::min<int64_t>(nj, (int64_t)ctx->sm_count * 2);
      if (keep) {
        static std::atomic<uint64_t> set{0};
        ensure_smem_attr(k_bin_reduce_wide<A, true>, reduce_wide_smem(A, max_bucket_log2(A)), set);
        k_bin_reduce_wide<A, true><<<g, kBinNT, sm, s>>>(b);
      } else {
        static std::atomic<uint64_t> set{0};
        ensure_smem_attr(k_bin_reduce_wide<A, false>, reduce_wide_smem(A, max_bucket_log2(A)), set);
        k_bin_reduce_wide<A, false><<<g, kBinNT, sm, s>>>(b);
      }
    }
  }
}

static void launch_bin_a(msf_ctx* ctx, const BinArgs& b, bool keep, int phase, bool smem,
                         cudaStream_t s, int j0 = 0, int nj = 0) {
  switch (b.A) {
    case 0: launch_bin<0>(ctx, b, keep, phase, smem, s, j0, nj); break;
    case 1: launch_bin<1>(ctx, b, keep, phase, smem, s, j0, nj); break;
    case 2: launch_bin<2>(ctx, b, keep, phase, smem, s, j0, nj); break;
    case 3: launch_bin<3>(ctx, b, keep, phase, smem, s, j0, nj); break;
    case 4: launch_bin<4>(ctx, b, keep, phase, smem, s, j0, nj); break;
    case 5: launch_bin<5>(ctx, b, keep, phase, smem, s, j0, nj); break;
    case 6: launch_bin<6>(ctx, b, keep, phase, smem, s, j0, nj); break;
    case 7: launch_bin<7>(ctx, b, keep, phase, smem, s, j0, nj); break;
    default: launch_bin<8>(ctx, b, keep, phase, smem, s, j0, nj); break;
  }
}

// The result words of a binning, behind its histogram: cleared with it and copied back at once.
struct BinWords {
  unsigned absmax[MSF_MAX_ATTR];
  uint32_t err, novf;             // bounded waits that gave up, buckets left to the wide pass
  unsigned long long outside[1];  // [Tp]
};

int bin_run(msf_ctx* ctx, unsigned flags) {
  Dataset& d = ctx->ds;
  const bool keep = flags & MSF_BIN_KEEP_SUMQ;
  cudaStream_t s = ctx->stream;
  BinScratch& S = ctx->bin;
  BinArgs b{};
  b.nx = d.nx;
  b.ny = d.ny;
  b.nz = d.nz;
  b.A = d.A;
  b.T = d.T;
  b.Tp = d.Tp;
  b.fstep = d.fstep.as<int32_t>();
  b.pj0 = d.pj0.as<int32_t>();
  b.V = d.V;
  b.P = d.P;
  b.scale_n = d.scale_fixed ? d.scale_samples : d.P * (int64_t)d.Tp;
  b.logR = bucket_log2(d.A, d.V);
  b.nb = (int)((d.V + ((int64_t)1 << b.logR) - 1) >> b.logR);
  // Samples per block of the keys pass: at least eight per bucket on average (each block adds
  // its shared-memory histogram into the global one, one atomic per bucket), from 4096 up to
  // kChunkMax. With more buckets than shared memory holds, every sample adds to the global
  // histogram directly.
  const bool smem = b.nb <= kHistSmem;
  b.chunk = 4096;
  while (b.chunk < kChunkMax && b.chunk < 8 * (int64_t)b.nb) b.chunk <<= 1;
  b.nblk = (int)std::max<int64_t>(1, (d.P + b.chunk - 1) / b.chunk);
  const int64_t TB = (int64_t)d.T * b.nb;
  const int64_t NR = d.P * (int64_t)d.Tp;
  const int Af = d.A > 0 ? d.A : 1;
  const int RW = rec_words(d.A);
  if (NR >= ((int64_t)1 << 32) || TB >= ((int64_t)1 << 31) ||
      (d.P + kPlaceChunk - 1) / kPlaceChunk > 0x7FFFFFFF)
    return MSF_ERR_TOO_LARGE;
  const size_t hist_bytes = (sizeof(uint32_t) * (size_t)TB + 7) & ~size_t(7);
  const size_t word_bytes = offsetof(BinWords, outside) + sizeof(unsigned long long) * d.Tp;
  MSF_TRY(S.hist.ensure(hist_bytes + word_bytes));
  MSF_TRY(ctx_result(ctx, word_bytes));
  MSF_TRY(S.offs.ensure(sizeof(uint32_t) * (TB + d.T)));
  MSF_TRY(S.cursor.ensure(sizeof(uint32_t) * kCurStride * TB));
  MSF_TRY(S.rec.ensure(sizeof(uint32_t) * RW * std::max<int64_t>(NR, 1)));
  MSF_TRY(S.ovf.ensure(sizeof(uint32_t) * (size_t)d.T * (size_t)b.nb));
  MSF_TRY(d.key.ensure(sizeof(int32_t) * ((int64_t)d.Tp * d.P + 4)));  // slack: bulk copies
  MSF_TRY(d.count.ensure(sizeof(int32_t) * d.T * d.V));
  MSF_TRY(d.mean.ensure(sizeof(float) * d.T * d.V * Af));
  if (keep) MSF_TRY(d.sumq.ensure(sizeof(int64_t) * d.T * d.V * Af));
  // the pairs a second time, where memory allows (after everything that a binning needs)
  if (S.rec_vn.ensure(sizeof(uint2) * std::max<int64_t>(NR, 1)) != MSF_OK) S.rec_vn.release();
  b.pos = d.pos.as<float>();
  b.attr = d.attr.as<float>();
  b.key = d.key.as<int32_t>();
  b.hist = S.hist.as<uint32_t>();
  b.offs = S.offs.as<uint32_t>();
  b.cursor = S.cursor.as<uint32_t>();
  b.rec = S.rec.as<uint32_t>();
  b.pairs = S.rec_vn.p ? S.rec_vn.as<char>() : S.rec.as<char>() + sizeof(uint32_t) * rec_pair(d.A);
  b.pair_bytes = (uint32_t)(S.rec_vn.p ? sizeof(uint2) : sizeof(uint32_t) * RW);
  b.wait_cycles = ctx->wait_cycles;
  b.pf_ahead = ctx->sm_count * (d.A <= 4 ? 3 : 2);  // resident reduce blocks
  BinWords* dw = reinterpret_cast<BinWords*>(S.hist.as<char>() + hist_bytes);
  b.err = &dw->err;
  b.novf = &dw->novf;
  b.ovf = S.ovf.as<uint32_t>();
  b.absmax = dw->absmax;
  b.outside = dw->outside;
  b.count = d.count.as<int32_t>();
  b.mean = d.mean.as<float>();
  b.sumq = keep ? d.sumq.as<long long>() : nullptr;
  // Points still coming in from the host (msf_load_timesteps with host pointers): the field
  // steps are binned chunk by chunk as their point steps arrive. Every field step's records own
  // the region from pj0[t] * P, so the steps' histograms, slot ranges and records are
  // independent of each other; a chunk's records need the keys of the next chunk's first point
  // step (the next-step voxel), so keys run one chunk ahead of the records.
  std::vector<int> ct = {0, d.T};
  const bool piped = ctx->points_pending && d.P > 0;
  if (piped) ct = ctx->chunk_t;
  ctx->points_pending = false;
  MSF_CUDA_TRY(cudaMemsetAsync(b.hist, 0, hist_bytes + word_bytes, s));
  if (d.scale_fixed)  // the whole dataset's maxima: a slab's can only be smaller
    MSF_CUDA_TRY(cudaMemcpyAsync(b.absmax, d.scale_absmax, sizeof(unsigned) * MSF_MAX_ATTR,
                                 cudaMemcpyHostToDevice, s));
  if (d.P > 0) {
    const int G = (int)ct.size() - 1;
    auto keys = [&](int g) -> int {
      if (piped) MSF_CUDA_TRY(cudaStreamWaitEvent(s, ctx->ev_chunk[g], 0));
      const int j0 = d.h_pj0[ct[g]], j1 = d.h_pj0[ct[g + 1]];
      if (j1 > j0) launch_bin_a(ctx, b, keep, 0, smem, s, j0, j1 - j0);
      MSF_CUDA_TRY(cudaGetLastError());
      return MSF_OK;
    };
    MSF_TRY(keys(0));
    for (int g = 0; g < G; ++g) {
      if (g + 1 < G) MSF_TRY(keys(g + 1));
      {
        ScopedKernel k(ctx, "k_bin_scan_steps", s);
        k_bin_scan_steps<<<(unsigned)(ct[g + 1] - ct[g]), kScanNT, 0, s>>>(b, ct[g]);
      }
      const int j0 = d.h_pj0[ct[g]], j1 = d.h_pj0[ct[g + 1]];
      if (j1 > j0) launch_bin_a(ctx, b, keep, 1, smem, s, j0, j1 - j0);
      MSF_CUDA_TRY(cudaGetLastError());
    }
  }
  launch_bin_a(ctx, b, keep, 2, smem, s);
  MSF_CUDA_TRY(cudaGetLastError());
  const BinWords* hw = static_cast<const BinWords*>(ctx->res);
  MSF_CUDA_TRY(cudaMemcpyAsync(ctx->res, dw, word_bytes, cudaMemcpyDeviceToHost, s));
  S.rec_valid = false;
  MSF_CUDA_TRY(cudaStreamSynchronize(s));
  if (hw->novf && !hw->err) {  // crowded buckets (rare): the wide pass, now that they are known
    launch_bin_a(ctx, b, keep, 3, smem, s, 0, (int)hw->novf);
    MSF_CUDA_TRY(cudaGetLastError());
    MSF_CUDA_TRY(cudaMemcpyAsync(ctx->res, dw, word_bytes, cudaMemcpyDeviceToHost, s));
    MSF_CUDA_TRY(cudaStreamSynchronize(s));
  }
  ctx->timer.flush();
  if (hw->err) {
    d.binned = false;
    return MSF_ERR_TIMEOUT;
  }
  const unsigned* hmax = hw->absmax;
  S.rec_valid = d.P > 0;
  S.rec_logR = b.logR;
  S.rec_nb = b.nb;
  S.rec_words = RW;
  S.rec_pair = rec_pair(d.A);
  for (int a = 0; a < d.A; ++a) {
    float m;
    memcpy(&m, &hmax[a], sizeof(float));
    d.max_abs[a] = m;
    d.kscale[a] = scale_exponent_bits(hmax[a], (long long)b.scale_n);
  }
  int64_t o = 0;
  for (int j = 0; j < d.Tp; ++j) o += (int64_t)hw->outside[j];
  d.out_of_domain = o;
  d.in_domain = d.P * (int64_t)d.Tp - o;
  d.binned = true;
  d.has_sumq = keep;
  return MSF_OK;
}

}  // namespace msf
