// sparse.cu -- cosine of sparse composition vectors, the comparison of the
// bioinformatics application (Sec. V-B: "essentially the dot product between
// two sparse vectors"):
//
//   c(i,j) = sum_k a_ik a_jk / sqrt(sum_k a_ik^2 sum_k a_jk^2)
//
// Rows are CSR (strictly increasing int32 codes, FP32 values) over an index
// space of `dim` codes (20^k k-mers), cut into chunks of kSparseChunk codes.
// A pair's sum needs only the codes that both rows hold, which for a code in
// p of the n rows is p (p - 1) / 2 products.  Each chunk takes the cheapest of
// three ways, decided at creation from its codes' counts:
//
//   join    few rows per code: one CTA sorts the chunk's entries by code in
//           shared memory (count, scan, scatter) and adds every pair of
//           entries of a code into the FP64 output, one product each;
//   gather  more: tiles of 128 x 128 rows, 64 codes at a time; block J is
//           scattered dense into shared memory straight from its CSR rows, and
//           each entry of block I multiplies the 128 values of its code;
//   dense   about a fifth of the rows per code and more: both blocks dense, 32 codes
//           at a time, and an FP32 Gram of them.
//
// Tiles keep FP32 sums over one chunk (or a part of one) and add them into the
// FP64 output.  A last pass scales by the norms.  (Before, every chunk was made
// dense for 8 rows at a time in tiles of 32 x 64 rows, one product per entry of
// row j and row i whether row i held the code or not: 256 rows of 20^6 codes,
// 1e5 to 1.8e6 entries each, took 255 ms, 20 CTAs' work; 10.5 with join and dense
// alone, now 8.5.)
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "ap_internal.h"

namespace ap {

namespace {

constexpr int W = kSparseChunk;

// ---------------------------------------------------------------------------
// join
// ---------------------------------------------------------------------------
// Bound by the FP64 additions at L2 (one per product, 1.8e11 a second) where
// many rows share codes, by the latency of the two passes over the entries
// where few do (15 ps an entry over the GPU: 122 million entries and as many
// products in 2.3 ms, 256 rows of 20^6 codes).  Two CTAs per SM.
constexpr int kJoinThreads = 512;
constexpr int kJoinCap = 9216;             // entries sorted at a time
constexpr size_t kJoinSmem = (size_t)(W + 1) * 4 + 12 + (size_t)kJoinCap * 10;

// f(row, entry index in the CSR arrays) for the entries of chunk c: eight
// lanes on consecutive entries of a row (a chunk of a composition vector
// holds a few dozen), a whole warp where there are fewer rows than octets
template <class F>
__device__ __forceinline__ void for_entries(const int64_t *__restrict__ off,
                                            const int32_t *__restrict__ cptr, int64_t n, int64_t c,
                                            F f) {
  const int lpr = n * 8 >= blockDim.x ? 8 : 32;
  const int sub = threadIdx.x & (lpr - 1);
  for (int64_t r = threadIdx.x / lpr; r < n; r += blockDim.x / lpr) {
    const int e1 = cptr[(c + 1) * n + r];
    const int64_t b = off[r];
#pragma unroll 4
    for (int e = cptr[c * n + r] + sub; e < e1; e += lpr) f((int32_t)r, b + e);
  }
}

// exclusive scan of s[0, W) in place, s[W] = total (kJoinThreads threads)
__device__ __forceinline__ void scan_counts(int32_t *s, int32_t *wsum) {
  constexpr int PER = W / kJoinThreads;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t v[PER], sum = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    v[q] = s[threadIdx.x * PER + q];
    sum += v[q];
  }
  int32_t inc = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t x = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += x;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  int32_t before = 0;
  for (int w = 0; w < warp; ++w) before += wsum[w];
  int32_t at = before + inc - sum;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    s[threadIdx.x * PER + q] = at;
    at += v[q];
  }
  if (threadIdx.x == kJoinThreads - 1) s[W] = at;
  __syncthreads();
}

__global__ void __launch_bounds__(kJoinThreads, 2)
sparse_join_kernel(const int64_t *__restrict__ off, const int32_t *__restrict__ idx,
                   const float *__restrict__ val, const int32_t *__restrict__ cptr, int64_t n,
                   const int32_t *__restrict__ chunks, int32_t n_chunks,
                   unsigned long long *queue, double *__restrict__ out) {
  extern __shared__ __align__(16) uint8_t smem[];
  int32_t *s_at = reinterpret_cast<int32_t *>(smem);              // [W + 1] code starts
  int32_t *s_row = s_at + W + 4;                                  // [kJoinCap]
  float *s_val = reinterpret_cast<float *>(s_row + kJoinCap);     // [kJoinCap]
  uint16_t *s_code = reinterpret_cast<uint16_t *>(s_val + kJoinCap);
  __shared__ int32_t s_wsum[kJoinThreads / 32];
  __shared__ unsigned long long s_unit;
  for (;;) {
    if (threadIdx.x == 0) s_unit = atomicAdd(queue, 1ull);
    for (int k = threadIdx.x; k < W; k += kJoinThreads) s_at[k] = 0;
    __syncthreads();
    const int64_t u = (int64_t)s_unit;
    if (u >= n_chunks) break;
    const int64_t c = chunks[u];
    const int32_t code0 = (int32_t)(c * W);
    for_entries(off, cptr, n, c, [&](int32_t, int64_t e) { atomicAdd(&s_at[idx[e] - code0], 1); });
    __syncthreads();
    scan_counts(s_at, s_wsum);
    const int32_t total = s_at[W];
    // codes [a, b) hold at most kJoinCap entries: usually the whole chunk (no
    // code alone holds more, or the chunk would be a dense one)
    for (int a = 0; a < W;) {
      const int32_t first = s_at[a];
      if (first == total) break;
      int b = W, lo = a + 1;
      if (total - first > kJoinCap) {
        for (int hi = W; lo < hi;) {                // last b with s_at[b] - first <= kJoinCap
          const int mid = (lo + hi + 1) >> 1;
          if (s_at[mid] - first <= kJoinCap) lo = mid;
          else hi = mid - 1;
        }
        b = lo;
      }
      const int32_t count = s_at[b] - first;
      __syncthreads();                              // every thread has read the starts
      for_entries(off, cptr, n, c, [&](int32_t row, int64_t e) {
        const int k = idx[e] - code0;
        if (k < a || k >= b) return;
        const int32_t at = atomicAdd(&s_at[k], 1) - first;   // s_at[k] becomes the code's end
        s_row[at] = row;
        s_val[at] = val[e];
        s_code[at] = (uint16_t)k;
      });
      __syncthreads();
      for (int e = threadIdx.x; e < count; e += kJoinThreads) {
        const int end = s_at[s_code[e]] - first;
        const int64_t r = s_row[e];
        const float v = s_val[e];
        for (int f = e + 1; f < end; ++f) {
          const int64_t q = s_row[f];
          const int64_t i = r < q ? r : q, j = r < q ? q : r;
          atomicAdd(out + pair_index(i, j, n), widen(__fmul_rn(v, s_val[f])));
        }
      }
      __syncthreads();                              // before the entries are replaced
      a = b;
    }
    __syncthreads();
  }
}

// per chunk: {most entries of one code, entries, products}, at creation
struct ChunkCount { int32_t most, pad; int64_t entries, products; };
__global__ void __launch_bounds__(kJoinThreads)
sparse_count_kernel(const int64_t *__restrict__ off, const int32_t *__restrict__ idx,
                    const int32_t *__restrict__ cptr, int64_t n, int64_t n_chunks,
                    ChunkCount *__restrict__ out) {
  __shared__ int32_t s_cnt[W];
  __shared__ int32_t s_most;
  __shared__ unsigned long long s_sum[2];
  for (int64_t c = blockIdx.x; c < n_chunks; c += gridDim.x) {
    for (int k = threadIdx.x; k < W; k += kJoinThreads) s_cnt[k] = 0;
    if (threadIdx.x == 0) { s_most = 0; s_sum[0] = s_sum[1] = 0; }
    __syncthreads();
    const int32_t code0 = (int32_t)(c * W);
    for_entries(off, cptr, n, c, [&](int32_t, int64_t e) {
      const uint32_t k = (uint32_t)(idx[e] - code0);
      if (k < (uint32_t)W) atomicAdd(&s_cnt[k], 1);        // (rows not yet known to be in order)
    });
    __syncthreads();
    int32_t most = 0;
    unsigned long long ent = 0, prod = 0;
    for (int k = threadIdx.x; k < W; k += kJoinThreads) {
      const int64_t p = s_cnt[k];
      most = max(most, s_cnt[k]);
      ent += (unsigned long long)p;
      prod += (unsigned long long)(p * (p - 1) / 2);
    }
    for (int o = 16; o > 0; o >>= 1) {
      most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
      ent += __shfl_xor_sync(0xffffffffu, ent, o);
      prod += __shfl_xor_sync(0xffffffffu, prod, o);
    }
    if ((threadIdx.x & 31) == 0) {
      atomicMax(&s_most, most);
      atomicAdd(&s_sum[0], ent);
      atomicAdd(&s_sum[1], prod);
    }
    __syncthreads();
    if (threadIdx.x == 0) out[c] = {s_most, 0, (int64_t)s_sum[0], (int64_t)s_sum[1]};
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// dense
// ---------------------------------------------------------------------------
// Units (tile of 128 x 128 rows, dense chunk or a part of one), a part's tiles
// in a row so that they read its entries from L2.  256 threads, 8 x 8 outputs each as in
// the FP32 Gram of dense vectors, two CTAs per SM; the FMA pipe is busy 0.53
// of the time, the rest goes into bringing a stage in between two barriers (976
// chunks of 256 rows of which a code is in 31: 8.3 ms; joining them takes 11).
// Each warp brings in 32 of the 256 rows: eight lanes read the next eight
// entries of a row (one or two sectors), so a warp load covers four rows.
constexpr int kDenseTile = 128;
constexpr int kDenseStage = 32;                       // codes per stage
constexpr int kDenseLd = kDenseTile + 4;
constexpr int kDenseBuf = kDenseStage * kDenseLd;     // floats of one operand's stage
constexpr int kDenseAhead = 8;                        // entries of a row staged at a time
constexpr size_t kDenseSmem = (size_t)4 * kDenseBuf * 4 + 256 * (4 + 4 + 8) +
                              (size_t)256 * kDenseAhead * 8;

// asynchronous 4-byte copy global -> shared
__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}

template <int COVER>
__global__ void __launch_bounds__(256, 2)
sparse_dense_kernel(const int64_t *__restrict__ off, const int32_t *__restrict__ idx,
                    const float *__restrict__ val, const int32_t *__restrict__ cptr, int64_t n,
                    const int32_t *__restrict__ chunks, int32_t n_chunks,
                    int32_t split, const int32_t *__restrict__ tiles, int64_t n_tiles,
                    unsigned long long *queue, void *out) {
  extern __shared__ __align__(16) float dsm[];
  float *s_buf = dsm;                                              // [2][A, B][stage][ld]
  int64_t *s_base = reinterpret_cast<int64_t *>(dsm + 4 * kDenseBuf);   // [256] rows A, rows B
  int32_t *s_ptr = reinterpret_cast<int32_t *>(s_base + 256);      // next entry
  int32_t *s_end = s_ptr + 256;
  int32_t *s_code = s_end + 256;                                   // [256][kDenseAhead]
  float *s_val = reinterpret_cast<float *>(s_code + 256 * kDenseAhead);
  __shared__ unsigned long long s_unit;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int warp = tid >> 5, lane = tid & 31, sub = lane & 7;

  for (;;) {
    if (tid == 0) s_unit = atomicAdd(queue, 1ull);
    __syncthreads();
    const int64_t u = (int64_t)s_unit;
    __syncthreads();
    if (u >= n_tiles * split * n_chunks) break;
    const int64_t part = u / n_tiles, t = u - part * n_tiles;   // part of a chunk, tile
    const int64_t i0 = (int64_t)tiles[2 * t] * kDenseTile;
    const int64_t j0 = (int64_t)tiles[2 * t + 1] * kDenseTile;
    const bool diag = i0 == j0;
    float2 acc[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = make_float2(0.f, 0.f);

    if (!COVER) {
      const int64_t c = chunks[part / split];
      const int stages = W / kDenseStage / split;
      const int32_t code0 = (int32_t)(c * W + (part % split) * (W / split));
      {
        const int64_t row = tid < kDenseTile ? i0 + tid : j0 + tid - kDenseTile;
        const bool in = row < n;
        s_base[tid] = in ? off[row] : 0;
        int32_t lo = in ? cptr[c * n + row] : 0, hi = in ? cptr[(c + 1) * n + row] : 0;
        s_end[tid] = hi;
        if (split > 1)                              // first entry of this part
          while (lo < hi) {
            const int32_t mid = lo + ((hi - lo) >> 1);
            if (idx[s_base[tid] + mid] < code0) lo = mid + 1;
            else hi = mid;
          }
        s_ptr[tid] = lo;
      }
      __syncthreads();
      // the warps share the rows, four to a load (rr0 + 4 q, q < nq); a
      // diagonal tile's rows B are its rows A, and one operand serves both
      const int nq = diag ? 4 : 8, rr0 = warp * 4 * nq + (lane >> 3);
      // the next eight entries of a row of this lane's into the staging area
      auto load = [&](int q) {
        const int rr = rr0 + 4 * q, p = s_ptr[rr] + sub;
        if (p < s_end[rr]) {
          const int64_t e = s_base[rr] + p;
          cp_async4(&s_code[rr * kDenseAhead + sub], idx + e);
          cp_async4(&s_val[rr * kDenseAhead + sub], val + e);
        } else {
          s_code[rr * kDenseAhead + sub] = -1;
        }
      };
      // those of the stage's codes into its buffer; more while a row has them
      // (each lane reads what it staged itself)
      auto scatter = [&](int buf, int32_t k0) {
        float *dst = s_buf + (2 * buf + (rr0 >> 7)) * kDenseBuf;
        asm volatile("cp.async.wait_all;" ::: "memory");
        auto place = [&](int q) -> bool {          // whether some row may have more
          const int rr = rr0 + 4 * q, at = rr * kDenseAhead + sub;
          const int32_t code = s_code[at];
          const bool in = (uint32_t)(code - k0) < (uint32_t)kDenseStage;   // codes come in order
          if (in) dst[(code - k0) * kDenseLd + (rr & 127)] = s_val[at];
          const uint32_t m = __ballot_sync(0xffffffffu, in);
          const int taken = __popc((m >> (lane & 24)) & 0xffu);
          if (sub == 0 && taken) s_ptr[rr] += taken;
          return __any_sync(0xffffffffu, taken == 8);
        };
        uint32_t more = 0;
#pragma unroll 4
        for (int q = 0; q < nq; ++q) more |= place(q) ? 1u << q : 0u;
        for (; more; more &= more - 1) {
          const int q = __ffs(more) - 1;
          do {
            __syncwarp();
            load(q);
            asm volatile("cp.async.wait_all;" ::: "memory");
          } while (place(q));
        }
      };
      auto zero = [&](int buf) {
        float4 *z = reinterpret_cast<float4 *>(s_buf + 2 * buf * kDenseBuf);
        for (int k = tid; k < 2 * kDenseBuf / 4; k += 256) z[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      };
      auto load_all = [&]() {
#pragma unroll 4
        for (int q = 0; q < nq; ++q) load(q);
      };
      // outputs (a, b) of one code; SKIP: a diagonal tile has no pair among
      // the rows 64.. and columns ..63
      auto product = [&](const float *As, const float *Bs, auto skip) {
        constexpr bool SKIP = decltype(skip)::value;
#pragma unroll 8
        for (int k = 0; k < kDenseStage; ++k) {
          const float4 a0 = *reinterpret_cast<const float4 *>(As + k * kDenseLd + ty * 4);
          const float4 a1 = *reinterpret_cast<const float4 *>(As + k * kDenseLd + 64 + ty * 4);
          const float4 b0 = *reinterpret_cast<const float4 *>(Bs + k * kDenseLd + tx * 4);
          const float4 b1 = *reinterpret_cast<const float4 *>(Bs + k * kDenseLd + 64 + tx * 4);
          const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
          const float2 bv[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w),
                                make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
          for (int a = 0; a < 8; ++a) {
            const float2 aa = make_float2(av[a], av[a]);
#pragma unroll
            for (int b = SKIP && a >= 4 ? 2 : 0; b < 4; ++b)
              acc[a][b] = __ffma2_rn(aa, bv[b], acc[a][b]);
          }
        }
      };
      load_all();
      zero(0);
      __syncthreads();
      scatter(0, code0);
      __syncthreads();
      for (int st = 0; st < stages; ++st) {
        const int buf = st & 1;
        const bool more = st + 1 < stages;
        if (more) {
          load_all();
          zero(buf ^ 1);
        }
        const float *As = s_buf + 2 * buf * kDenseBuf;
        if (diag) product(As, As, std::true_type());
        else product(As, As + kDenseBuf, std::false_type());
        __syncthreads();                            // the other buffer is clear
        if (more) scatter(buf ^ 1, code0 + (st + 1) * kDenseStage);
        __syncthreads();
      }
    }

    const int ni = (int)(n - i0 < kDenseTile ? n - i0 : kDenseTile);
    const int nj = (int)(n - j0 < kDenseTile ? n - j0 : kDenseTile);
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int il = (a < 4 ? a : 60 + a) + ty * 4;
      if (il < ni) {
        const int64_t i = i0 + il;
        const int first = (int)(i - j0) + 1;        // pairs need j0 + jl > i
        const int64_t p0 = pair_index(i, j0, n);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          const int jl = (b < 4 ? b : 60 + b) + tx * 4;
          if (jl >= nj || jl < first) continue;
          if (COVER) atomicAdd(reinterpret_cast<int32_t *>(out) + p0 + jl, 1);
          else
            atomicAdd(reinterpret_cast<double *>(out) + p0 + jl,
                      widen((b & 1) ? acc[a][b >> 1].y : acc[a][b >> 1].x));
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// gather
// ---------------------------------------------------------------------------
// Units as the dense kernel's, but only rows B are made dense: 64 codes at a
// time of the 128 rows of block J, a code's values side by side.  Each entry of
// a row A takes one 512-byte read of its code's values (4 columns per lane) and
// four FMAs per lane, so the work falls with the density of the rows A.  A warp
// holds the 16 x 128 sums of its 16 rows A; rows that hold more of a stage's
// codes than are staged at a time take more turns over the 16.
// Bound by shared memory, busy 0.71 of the time: 4.5 wavefronts an entry (half a
// read of two entries, four of values), as many again to bring the stages in.
// 976 chunks of 256 rows of which a code is in 31: 6.2 ms, dense 8.3; with 8% of
// the rows in a code 0.96 ms (joins 1.26), 12% 1.23 (dense 1.55), 20% 2.23
// (2.25), 30% 3.27 (2.92).  The first form, with the further turns inside the
// unrolled rows, fetched instructions a quarter of the time (8.2 ms).
constexpr int kGatherStage = 64;                      // codes per stage
constexpr int kGatherAhead = 16;                      // entries of a row staged at a time
constexpr int kGatherBuf = (kGatherStage + 1) * kDenseLd;   // and a code of zeros
constexpr size_t kGatherSmem =
    (size_t)2 * kGatherBuf * 4 + 256 * 16 + (size_t)256 * kGatherAhead * 8;

struct __align__(16) Row {
  int64_t base;                          // of its entries in the CSR arrays
  int32_t next, end;                     // relative to base
};

__global__ void __launch_bounds__(256, 2)
sparse_gather_kernel(const int64_t *__restrict__ off, const int32_t *__restrict__ idx,
                     const float *__restrict__ val, const int32_t *__restrict__ cptr, int64_t n,
                     const int32_t *__restrict__ chunks, int32_t n_chunks, int32_t split,
                     const int32_t *__restrict__ tiles, int64_t n_tiles,
                     unsigned long long *queue, double *__restrict__ out) {
  extern __shared__ __align__(16) float dsm[];
  float *s_buf = dsm;                                              // [2][stage + 1][ld]
  int2 *s_ent = reinterpret_cast<int2 *>(dsm + 2 * kGatherBuf);    // [256][kGatherAhead]
  Row *s_row = reinterpret_cast<Row *>(s_ent + 256 * kGatherAhead);   // rows A, rows B
  __shared__ unsigned long long s_unit;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int half = lane >> 4, sub = lane & 15;        // two rows per warp load
  const int a0 = warp * 16, b0 = kDenseTile + warp * 16;   // this warp's rows

  for (;;) {
    if (tid == 0) s_unit = atomicAdd(queue, 1ull);
    __syncthreads();
    const int64_t u = (int64_t)s_unit;
    __syncthreads();
    if (u >= n_tiles * split * n_chunks) break;
    const int64_t part = u / n_tiles, t = u - part * n_tiles;   // part of a chunk, tile
    const int64_t i0 = (int64_t)tiles[2 * t] * kDenseTile;
    const int64_t j0 = (int64_t)tiles[2 * t + 1] * kDenseTile;
    const bool diag = i0 == j0;
    const int64_t c = chunks[part / split];
    const int stages = W / kGatherStage / split;
    const int32_t code0 = (int32_t)(c * W + (part % split) * (W / split));
    {
      const int64_t row = tid < kDenseTile ? i0 + tid : j0 + tid - kDenseTile;
      const bool in = row < n;
      const int64_t base = in ? off[row] : 0;
      int32_t lo = in ? cptr[c * n + row] : 0, hi = in ? cptr[(c + 1) * n + row] : 0;
      const int32_t end = hi;
      if (split > 1)                              // first entry of this part
        while (lo < hi) {
          const int32_t mid = lo + ((hi - lo) >> 1);
          if (idx[base + mid] < code0) lo = mid + 1;
          else hi = mid;
        }
      s_row[tid] = {base, lo, end};
    }
    __syncthreads();
    float2 acc[16][2];
#pragma unroll
    for (int r = 0; r < 16; ++r) acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);

    // the next entries of a row into its staging area, one a lane
    auto load = [&](int rr) {
      const int4 w = *reinterpret_cast<const int4 *>(s_row + rr);
      const int64_t base = (int64_t)(((uint64_t)(uint32_t)w.y << 32) | (uint32_t)w.x);
      const int p = w.z + sub;
      int2 *dst = s_ent + rr * kGatherAhead + sub;
      if (p < w.w) {
        cp_async4(&dst->x, idx + base + p);
        cp_async4(&dst->y, val + base + p);
      } else {
        dst->x = -1;
      }
    };
    auto load16 = [&](int first) {
#pragma unroll 4
      for (int q = 0; q < 8; ++q) load(first + 2 * q + half);
    };
    auto arrived = [] { asm volatile("cp.async.wait_all;" ::: "memory"); };
    auto zero = [&](int buf) {
      float4 *z = reinterpret_cast<float4 *>(s_buf + buf * kGatherBuf);
      for (int k = tid; k < kGatherBuf / 4; k += 256) z[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    };
    // the rows B's staged entries of the stage's codes into its buffer; more
    // while a row has them (each lane reads what it staged itself)
    auto scatter = [&](int buf, int32_t k0) {
      float *dst = s_buf + buf * kGatherBuf;
      auto place = [&](int q) -> bool {
        const int rr = b0 + 2 * q + half;
        const int2 e = s_ent[rr * kGatherAhead + sub];
        const bool in = (uint32_t)(e.x - k0) < (uint32_t)kGatherStage;   // codes come in order
        if (in) dst[(e.x - k0) * kDenseLd + rr - kDenseTile] = __int_as_float(e.y);
        const uint32_t m = __ballot_sync(0xffffffffu, in);
        const int taken = __popc((m >> (16 * half)) & 0xffffu);
        if (sub == 0 && taken) s_row[rr].next += taken;
        return __any_sync(0xffffffffu, taken == kGatherAhead);
      };
      uint32_t more = 0;
#pragma unroll 4
      for (int q = 0; q < 8; ++q) more |= place(q) ? 1u << q : 0u;
      for (; more; more &= more - 1) {
        const int q = __ffs(more) - 1;
        do {
          __syncwarp();
          load(b0 + 2 * q + half);
          arrived();
        } while (place(q));
      }
    };
    // Staged entries of rows A, two rows at once: {code in the stage, value},
    // {the code of zeros, 0} past the stage's; returns which lanes' are the stage's
    auto ready = [&](int rr, int32_t k0) -> uint32_t {
      int2 *at = s_ent + rr * kGatherAhead + sub;
      const int2 e = *at;
      const bool in = (uint32_t)(e.x - k0) < (uint32_t)kGatherStage;
      *at = in ? make_int2(e.x - k0, e.y) : make_int2(kGatherStage, 0);
      const uint32_t m = __ballot_sync(0xffffffffu, in);
      const int taken = __popc((m >> (16 * half)) & 0xffffu);
      if (sub == 0 && taken) s_row[rr].next += taken;
      return m;
    };
    // whether some row may have more of the stage's codes
    uint32_t have[8];
    auto ready16 = [&](int32_t k0) -> bool {
      bool full = false;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        have[q] = ready(a0 + 2 * q + half, k0);
        full |= (have[q] & 0xffffu) == 0xffffu || have[q] >> 16 == 0xffffu;
      }
      __syncwarp();
      return full;
    };

    load16(a0);
    load16(b0);
    zero(0);
    zero(1);
    __syncthreads();
    arrived();
    scatter(0, code0);
    bool full = ready16(code0);
    __syncthreads();
    for (int st = 0; st < stages; ++st) {
      const int buf = st & 1;
      const int32_t k0 = code0 + st * kGatherStage;
      const bool more = st + 1 < stages;
      if (more) {
        load16(b0);
        if (st > 0) zero(buf ^ 1);
      }
      const float *Bs = s_buf + buf * kGatherBuf + 4 * lane;
      for (;;) {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
          // a diagonal tile has no pair of a row with those before it
          const bool on = !diag || 4 * lane + 3 > a0 + r;
          const int4 *ent = reinterpret_cast<const int4 *>(s_ent + (a0 + r) * kGatherAhead);
          const int cnt = __popc((have[r >> 1] >> (16 * (r & 1))) & 0xffffu);
          int4 two = ent[0];
#pragma unroll 1
          for (int e = 0; e < cnt; e += 2) {
            const int4 now = two;
            two = ent[e / 2 + 1];                 // (past a row's last: not used)
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
            if (on) {
              x = *reinterpret_cast<const float4 *>(Bs + now.x * kDenseLd);
              y = *reinterpret_cast<const float4 *>(Bs + now.z * kDenseLd);
            }
            const float v = __int_as_float(now.y), w = __int_as_float(now.w);
            acc[r][0] = __ffma2_rn(make_float2(v, v), make_float2(x.x, x.y), acc[r][0]);
            acc[r][1] = __ffma2_rn(make_float2(v, v), make_float2(x.z, x.w), acc[r][1]);
            acc[r][0] = __ffma2_rn(make_float2(w, w), make_float2(y.x, y.y), acc[r][0]);
            acc[r][1] = __ffma2_rn(make_float2(w, w), make_float2(y.z, y.w), acc[r][1]);
          }
        }
        __syncwarp();
        if (!full) break;
        load16(a0);
        arrived();
        full = ready16(k0);
      }
      if (more) load16(a0);
      __syncthreads();                            // the other buffer is clear
      if (more) {
        arrived();
        scatter(buf ^ 1, k0 + kGatherStage);
        full = ready16(k0 + kGatherStage);
      }
      __syncthreads();
    }

    const int ni = (int)(n - i0 < kDenseTile ? n - i0 : kDenseTile);
    const int nj = (int)(n - j0 < kDenseTile ? n - j0 : kDenseTile);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const int il = a0 + r;
      if (il >= ni) continue;
      const int64_t i = i0 + il;
      const int first = (int)(i - j0) + 1;        // pairs need j0 + jl > i
      double *dst = out + pair_index(i, j0, n);
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int jl = 4 * lane + b;
        if (jl >= nj || jl < first) continue;
        atomicAdd(dst + jl, widen((b & 1) ? acc[r][b >> 1].y : acc[r][b >> 1].x));
      }
    }
  }
}

// out[p] *= rs_i rs_j over the packed triangle
__global__ void sparse_scale_kernel(double *__restrict__ out, const double *__restrict__ rs,
                                    int64_t n) {
  for (int64_t i = blockIdx.x; i < n - 1; i += gridDim.x) {
    const double ri = rs[i];
    const int64_t p0 = pair_index(i, i + 1, n);
    for (int64_t j = i + 1 + threadIdx.x; j < n; j += blockDim.x)
      out[p0 + (j - i - 1)] *= ri * rs[j];
  }
}

// Picoseconds of the whole GPU, measured on a GB300 (see the kernels); of a
// gather, 0.7e6 a tile with hardly an entry and 23-26 an entry from sets of 2 to
// 33% density.
constexpr double kJoinProductPs = 5.6, kJoinEntryPs = 15.0;
constexpr double kDenseTilePs = 2.6e6;
constexpr double kGatherTilePs = 0.7e6, kGatherEntryPs = 23.0;
constexpr double kJoinAlone = 0.4, kLaunchPs = 5e6;
constexpr double kGatherUnitPs = 12e6, kGatherStagePs = 3.3e6;   // of a CTA's time

// parts of a gather's chunks such that the rounds of units take least time
struct GatherFit {
  int32_t split;
  double ps;
};
GatherFit gather_fit(int64_t chunks, int64_t n_tiles) {
  GatherFit best{1, INFINITY};
  const int64_t slots = 2 * (int64_t)num_sms();
  for (int32_t split = 1; split <= 32; split *= 2) {
    const int64_t rounds = (chunks * n_tiles * split + slots - 1) / slots;
    const double ps = (double)rounds *
                      (kGatherUnitPs + kGatherStagePs * (double)(W / kGatherStage / split));
    if (ps < best.ps) best = {split, ps};
  }
  return best;
}

// row checks (strictly increasing codes in [0, dim)), FP64 squared norms
constexpr int kRowThreads = 512;
__global__ void __launch_bounds__(kRowThreads)
sparse_rows_kernel(const int64_t *__restrict__ off, const int32_t *__restrict__ idx,
                   const float *__restrict__ val, int64_t n, int64_t dim, double *__restrict__ rs,
                   int32_t *bad) {
  __shared__ double red[kRowThreads / 32];
  for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
    double s = 0.0;
#pragma unroll 4
    for (int64_t e = off[i] + threadIdx.x; e < off[i + 1]; e += blockDim.x) {
      const int32_t k = idx[e];
      if (k < 0 || k >= dim || (e > off[i] && idx[e - 1] >= k)) atomicExch(bad, 1);
      s += (double)val[e] * (double)val[e];
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
      rs[i] = t > 0.0 ? 1.0 / sqrt(t) : __longlong_as_double(0x7ff8000000000000ll);
    }
    __syncthreads();
  }
}

// cptr[c][i] = lower bound of c * W in row i's codes, relative to the row
__global__ void sparse_cptr_kernel(const int64_t *__restrict__ off, const int32_t *__restrict__ idx,
                                   int64_t n, int64_t n_chunks, int32_t *__restrict__ cptr) {
  const int64_t total = (n_chunks + 1) * n;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = q / n, i = q - c * n;
    const int64_t lo0 = off[i], hi0 = off[i + 1];
    const int64_t key = c * (int64_t)W;
    int64_t lo = lo0, hi = hi0;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if ((int64_t)idx[mid] < key) lo = mid + 1;
      else hi = mid;
    }
    cptr[q] = (int32_t)(lo - lo0);
  }
}

}  // namespace

void free_sparse(SparseStore &sp) {
  dfree(sp.d_off);
  dfree(sp.d_idx);
  dfree(sp.d_val);
  dfree(sp.d_cptr);
  dfree(sp.d_rs);
  dfree(sp.d_tiles);
  dfree(sp.d_chunks);
  dfree(sp.d_heads);
}

ap_status create_sparse(const ap_items_desc *d, ap_items *it, cudaStream_t s) {
  SparseStore &sp = it->sp;
  const int64_t *off = d->offsets;
  if (!off || off[0] != 0 || d->dim < 1 || d->dim > INT32_MAX) return AP_ERR_INVALID_ARG;
  sp.n = d->n_items;
  sp.dim = d->dim;
  for (int64_t i = 0; i < sp.n; ++i) {
    if (off[i + 1] < off[i]) return AP_ERR_INVALID_ARG;
    if (off[i + 1] - off[i] > d->dim) return AP_ERR_INVALID_ARG;   // more entries than codes
  }
  sp.nnz = off[sp.n];
  if (sp.nnz > 0 && (!d->indices || !d->data)) return AP_ERR_INVALID_ARG;
  sp.n_chunks = (sp.dim + kSparseChunk - 1) / kSparseChunk;
  AP_TRY(dmalloc(&sp.d_off, (size_t)sp.n + 1));
  AP_TRY(dmalloc(&sp.d_idx, (size_t)std::max<int64_t>(sp.nnz, 1)));
  AP_TRY(dmalloc(&sp.d_val, (size_t)std::max<int64_t>(sp.nnz, 1)));
  AP_TRY(dmalloc(&sp.d_cptr, (size_t)(sp.n_chunks + 1) * std::max<int64_t>(sp.n, 1)));
  AP_TRY(dmalloc(&sp.d_rs, (size_t)std::max<int64_t>(sp.n, 1)));
  AP_TRY(cudaMemcpyAsync(sp.d_off, off, (size_t)(sp.n + 1) * 8, cudaMemcpyHostToDevice, s));
  const cudaMemcpyKind kind = d->data_on_host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  if (sp.nnz > 0) {
    AP_TRY(cudaMemcpyAsync(sp.d_idx, d->indices, (size_t)sp.nnz * 4, kind, s));
    AP_TRY(cudaMemcpyAsync(sp.d_val, d->data, (size_t)sp.nnz * 4, kind, s));
  }
  int32_t *d_bad = it->d_queue + 2;              // scratch word of the handle
  AP_TRY(cudaMemsetAsync(d_bad, 0, 4, s));
  if (sp.n > 0) {
    const int g = (int)std::min<int64_t>(sp.n, 65535);
    sparse_rows_kernel<<<g, kRowThreads, 0, s>>>(sp.d_off, sp.d_idx, sp.d_val, sp.n, sp.dim, sp.d_rs,
                                         d_bad);
    AP_TRY(cudaGetLastError());
    const int64_t total = (sp.n_chunks + 1) * sp.n;
    const int g2 = (int)std::min<int64_t>((total + 255) / 256, 65535);
    sparse_cptr_kernel<<<g2, 256, 0, s>>>(sp.d_off, sp.d_idx, sp.n, sp.n_chunks, sp.d_cptr);
    AP_TRY(cudaGetLastError());
  }
  // what each chunk holds, read back with the verdict on the rows
  std::vector<ChunkCount> count((size_t)(sp.n > 0 ? sp.n_chunks : 0));
  ChunkCount *d_count = nullptr;
  if (!count.empty()) {
    AP_TRY(dmalloc(&d_count, count.size()));
    const int g = (int)std::min<int64_t>(sp.n_chunks, (int64_t)num_sms() * 4);
    sparse_count_kernel<<<g, kJoinThreads, 0, s>>>(sp.d_off, sp.d_idx, sp.d_cptr, sp.n,
                                                   sp.n_chunks, d_count);
  }
  int32_t bad = 0;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(&bad, d_bad, 4, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && !count.empty())
    e = cudaMemcpyAsync(count.data(), d_count, count.size() * sizeof(ChunkCount),
                        cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  dfree(d_count);
  if (e != cudaSuccess) return from_cuda(e);
  if (bad) return AP_ERR_INVALID_ARG;

  std::vector<int32_t> tiles;
  dc_block_pairs((sp.n + kDenseTile - 1) / kDenseTile, tiles);
  sp.n_tiles = (int64_t)tiles.size() / 2;
  // Each chunk by the cheapest way (picoseconds of the whole GPU): a join adds
  // kJoinProductPs per product and kJoinEntryPs per entry; a gather kGatherTilePs
  // per tile and kGatherEntryPs per entry and tile that has its row in block I
  // (half the blocks, and its own); a dense chunk kDenseTilePs per tile whatever
  // it holds.  A code in more rows than a join sorts at a time rules that out.
  std::vector<int32_t> join, gather, dense;
  const double blocks = (double)((sp.n + kDenseTile - 1) / kDenseTile);
  auto way_join = [&](int32_t c) {
    return count[c].most > kJoinCap ? INFINITY
                                    : kJoinProductPs * (double)count[c].products +
                                          kJoinEntryPs * (double)count[c].entries;
  };
  auto way_gather = [&](int32_t c) {
    return kGatherTilePs * (double)sp.n_tiles +
           kGatherEntryPs * (double)count[c].entries * 0.5 * (blocks + 1.0);
  };
  const double way_dense = kDenseTilePs * (double)sp.n_tiles;
  for (int32_t c = 0; c < (int32_t)count.size(); ++c) {
    if (count[c].products == 0) continue;        // no code in two rows
    const double wj = way_join(c), wg = way_gather(c);
    (wj <= std::min(wg, way_dense) ? join : wg <= way_dense ? gather : dense).push_back(c);
  }
  // heaviest joins first: their times differ, and the queue ends with a tail
  std::stable_sort(join.begin(), join.end(), [&](int32_t a, int32_t b) {
    return count[a].products + count[a].entries > count[b].products + count[b].entries;
  });
  // A join is one CTA's work, which alone takes kJoinAlone of its share of the
  // GPU's time on every CTA slot, so a few heavy ones outlast the rest: as many
  // of them go in tiles instead, by the gather's parts, as make the two
  // kernels' time least (600 rows of 2e6 codes: one join took 3.3 of 4.8 ms,
  // the chunk in which the frequent codes end).
  const double slots = 2.0 * num_sms();
  double join_sum = 0.0, gather_sum = 0.0;
  for (int32_t c : join) join_sum += way_join(c);
  for (int32_t c : gather) gather_sum += way_gather(c);
  size_t moved = 0;
  double least = INFINITY;
  for (size_t m = 0; m <= join.size(); ++m) {
    const int64_t g = (int64_t)(gather.size() + m);
    const double alone = m < join.size() ? kJoinAlone * slots * way_join(join[m]) : 0.0;
    const double t = std::max(join_sum, alone) +
                     (g ? std::max(gather_sum, gather_fit(g, sp.n_tiles).ps) + kLaunchPs : 0.0);
    if (m == 0 || t < 0.9 * least) {             // (a tenth, or it is not worth the change)
      least = t;
      moved = m;
    }
    if (m == join.size() || gather_sum > least) break;
    join_sum -= way_join(join[m]);
    gather_sum += way_gather(join[m]);
  }
  gather.insert(gather.end(), join.begin(), join.begin() + moved);
  join.erase(join.begin(), join.begin() + moved);
  sp.n_join = (int64_t)join.size();
  sp.n_gather = (int64_t)gather.size();
  sp.n_dense = (int64_t)dense.size();
  join.insert(join.end(), gather.begin(), gather.end());
  join.insert(join.end(), dense.begin(), dense.end());
  AP_TRY(dmalloc(&sp.d_chunks, std::max<size_t>(join.size(), 1)));
  AP_TRY(dmalloc(&sp.d_tiles, std::max<size_t>(tiles.size(), 2)));
  AP_TRY(dmalloc(&sp.d_heads, 3));
  if (!join.empty())
    AP_TRY(cudaMemcpyAsync(sp.d_chunks, join.data(), join.size() * 4, cudaMemcpyHostToDevice, s));
  if (!tiles.empty())
    AP_TRY(cudaMemcpyAsync(sp.d_tiles, tiles.data(), tiles.size() * 4, cudaMemcpyHostToDevice, s));
  it->stats.tiles = sp.n_tiles;
  it->stats.tile_m = it->stats.tile_n = kSparseBlock;
  return AP_OK;
}

cudaError_t launch_sparse_cosine(const SparseStore &sp, void *out, int coverage, cudaStream_t s) {
  if (sp.n_tiles <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(sp.d_heads, 0, 3 * sizeof(*sp.d_heads), s);
  if (e != cudaSuccess) return e;
  const int64_t slots = 2 * (int64_t)num_sms();      // two CTAs per SM, both kernels
  if (coverage) {
    sparse_dense_kernel<1><<<(int)std::min(slots, sp.n_tiles), 256, 0, s>>>(
        sp.d_off, sp.d_idx, sp.d_val, sp.d_cptr, sp.n, sp.d_chunks, 1, 1, sp.d_tiles, sp.n_tiles,
        sp.d_heads, out);
    return cudaGetLastError();
  }
  double *o = reinterpret_cast<double *>(out);
  e = cudaMemsetAsync(o, 0, (size_t)(sp.n * (sp.n - 1) / 2) * sizeof(double), s);
  if (e != cudaSuccess) return e;
  if (sp.n_gather > 0) {
    e = cudaFuncSetAttribute(sparse_gather_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kGatherSmem);
    if (e != cudaSuccess) return e;
    const int32_t split = gather_fit(sp.n_gather, sp.n_tiles).split;
    const int64_t units = sp.n_gather * sp.n_tiles * split;
    sparse_gather_kernel<<<(int)std::min(slots, units), 256, kGatherSmem, s>>>(
        sp.d_off, sp.d_idx, sp.d_val, sp.d_cptr, sp.n, sp.d_chunks + sp.n_join,
        (int32_t)sp.n_gather, split, sp.d_tiles, sp.n_tiles, sp.d_heads + 2, o);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (sp.n_dense > 0) {
    e = cudaFuncSetAttribute(sparse_dense_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kDenseSmem);
    if (e != cudaSuccess) return e;
    // parts of a chunk where whole ones leave SMs idle (at least 4 stages each)
    int32_t split = 1;
    while (split < 32 && sp.n_dense * sp.n_tiles * split < slots) split *= 2;
    const int64_t units = sp.n_dense * sp.n_tiles * split;
    sparse_dense_kernel<0><<<(int)std::min(slots, units), 256, kDenseSmem, s>>>(
        sp.d_off, sp.d_idx, sp.d_val, sp.d_cptr, sp.n, sp.d_chunks + sp.n_join + sp.n_gather,
        (int32_t)sp.n_dense, split, sp.d_tiles, sp.n_tiles, sp.d_heads, out);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (sp.n_join > 0) {
    e = cudaFuncSetAttribute(sparse_join_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kJoinSmem);
    if (e != cudaSuccess) return e;
    sparse_join_kernel<<<(int)std::min(slots, sp.n_join), kJoinThreads, kJoinSmem, s>>>(
        sp.d_off, sp.d_idx, sp.d_val, sp.d_cptr, sp.n, sp.d_chunks, (int32_t)sp.n_join,
        sp.d_heads + 1, o);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  const int grid = (int)std::min<int64_t>(sp.n - 1, 65535);
  sparse_scale_kernel<<<grid, 256, 0, s>>>(o, sp.d_rs, sp.n);
  return cudaGetLastError();
}

}  // namespace ap
