// factor.cu -- numeric block factorization A' = L D U' on the pattern P'.
//
// 1. Backfill (Algorithm 5 steps 3-4): every slot of the factor buffer
//    [L | D | U] gathers its A block, or zero for a fill position.
// 2. Block ILU(0) on A' (Algorithm 4), one warp per block row, rows claimed in
//    ascending order through an atomic ticket.  Row i walks its pivots p < i
//    in ascending order, waiting (bounded, acquire) until row p is finished,
//    and does
//        A_ip <- A_ip D_p^{-1}
//        A_ij <- A_ij - A_ip U_pj   for every j > p with (p,j) and (i,j) in P'
//    where U_pj is row p's final, still unscaled upper block.  The j updates of
//    one pivot are independent, so the warp spreads (block, element) pairs
//    over its lanes; each element is a b-term dot product.
//    Then D_i = A_ii is inverted in the warp (Gauss-Jordan with partial
//    pivoting inside the b x b block, one lane per column of [D_i | I]),
//    D_i^{-1} overwrites the D slot, and row i is released (fence + release
//    store of its ready flag).  Row i depends only on rows of smaller tickets,
//    which are held by running warps, so the schedule always progresses.
// 3. Eq. 5: U'_ij = D_i^{-1} U_ij for every upper block, once all rows are
//    done (later rows need the unscaled U_pj).
// A zero or non-finite pivot block records BILU_ERR_SINGULAR and the smallest
// such row; the row is still released so that no warp waits forever.
#include <cuda_runtime.h>

#include <algorithm>

#include "device_common.cuh"
#include "launch_cache.h"

namespace bilu {
namespace {


template <typename TV>
__global__ void backfill_kernel(long long total, int bb, const int32_t* __restrict__ slot_src,
                                const double* __restrict__ a, TV* __restrict__ f) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += stride) {
    const long long slot = q / bb;
    const int e = (int)(q - slot * bb);
    const int32_t src = __ldg(slot_src + slot);
    f[q] = src >= 0 ? (TV)__ldg(a + (size_t)src * bb + e) : TV(0);
  }
}

__global__ void factor_init_kernel(int32_t* header, int32_t* done, int32_t n) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride) done[q] = 0;
  if (blockIdx.x == 0 && threadIdx.x < kHeaderWords)
    header[threadIdx.x] = (threadIdx.x == kBadRow) ? 0x7fffffff : 0;
}

// Row storage of the factor kernel: rows of up to RC blocks are staged in
// shared memory (per warp); longer rows are worked on in place in global memory
// through the same slot interface.  A warp takes a row's pivots in batches of
// up to lc entries of their U rows, whose matches in the row are listed before
// anything is waited for.  8 warps per CTA: twice the chunks in flight of one
// 16-warp CTA for the same warps (measured 4-13 % faster with 256-row chunk
// targets).
// lc (LCMIN to LCMAX, batch_entries): a 27-point ILU(1) row has 25 entries; a batch
// below that takes each pivot in slices (b = 5 FP32 128x16x8 27-point with 16 / 42
// entries: 12.2 / 9.6 ms; b = 3 FP32 160x40x20 with 48 / 96: 11.2 / 9.2; b = 1 FP64
// 12x60x60 with 64 / 128: 18.0 / 15.6; with 256, 7-point b = 1 2.30 / 2.54).
// MINB: CTAs per SM the registers are cut for, 0 the compiler's choice (80 registers
// and 9 to 20 words spilled for FP64 b = 2 and FP32 b = 3 and 5, three CTAs): FP32 b =
// 2 and 4 otherwise take 80 and 94 (96x96x48 ILU(0) 1.40 / 1.27 and 2.29 / 1.92 ms),
// and FP64 b >= 6 does better with the 128 there are (160x20x20 27-point b = 6 36.6 /
// 34.7).
template <int B, typename TV>
struct FactorCap {
  static constexpr bool kSingle = sizeof(TV) == 4;
  static constexpr int W = 8;  // warps per CTA
  static constexpr int RC = B <= 4 ? 64 : (B <= 6 ? 32 : 24);
  static constexpr int LCMAX = B == 1 ? 128
                               : B <= 3 ? (B == 3 && !kSingle ? 64 : 96)
                               : B == 4 ? (kSingle ? 64 : 32)
                               : B <= 6 ? (kSingle ? 42 : 28)
                                        : 28;
  static constexpr int LCMIN = B <= 4 || (B == 5 && kSingle) ? LCMAX : B <= 6 ? 16 : 12;
  static constexpr int MINB = kSingle ? (B == 2 ? 4 : B == 4 ? 3 : 0) : (B >= 6 ? 2 : 0);
  static constexpr int KC = B <= 4 ? 16 : 6;  // pivot blocks D_p^{-1} held at once
  static constexpr int WVAL = (KC + 1) * B * B;  // values per warp beside the staged row and the batch
  static constexpr int WINT = 2 * 34;            // ints per warp beside the row's columns and the batch
};

int device_sms() {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

template <int B, typename TV>
size_t factor_smem_bytes(int chunk, int rc, int lc) {
  return (size_t)FactorCap<B, TV>::W * (FactorCap<B, TV>::WVAL + (rc + lc) * B * B) * sizeof(TV) +
         ((size_t)2 * chunk + (size_t)FactorCap<B, TV>::W * (FactorCap<B, TV>::WINT + 2 * lc + rc)) * sizeof(int);
}

// CTAs that fit into an SM's shared memory (228 KB, 1 KB of it kept per CTA); 0 for
// more than a CTA may ask for.
template <int B, typename TV>
int ctas_by_smem(int chunk, int rc, int lc) {
  const size_t bytes = factor_smem_bytes<B, TV>(chunk, rc, lc);
  return bytes > (size_t)kMaxDynamicSmem ? 0 : (int)(228 * 1024 / (bytes + 1024));
}

// rc: rows of up to rc blocks are staged (at most RC; the widest row of the
// pattern if that is less).  For b >= 5 none are where the mean row is longer than
// RC: the buffer would cost a CTA per SM and hold boundary rows only (FP64 b = 8
// 128x16x8 27-point 28.7 / 25.7 ms).  Nor are any for b >= 7 in FP64 where one CTA
// fits with the buffer and two without, and one leaves lines waiting: more rows per
// level than lines resident (b = 8, staged / in place: ILU(2) 96x96x48 78.9 / 58.4 ms,
// 64x64x32 25.7 / 22.0, ILU(1) 64x64x32 12.3 / 11.1; 280 rows per level, 304 lines
// resident: 50x45x30 ILU(1) 7.4 / 8.0).
template <int B, typename TV>
int staged_rows(const bilu_pattern* p) {
  using Cap = FactorCap<B, TV>;
  if (B >= 5 && p->cnt_p > (long long)p->n * Cap::RC) return 0;
  const int rc = std::min(Cap::RC, p->max_l + 1 + p->max_u), chunk = p->fact.max_len;
  const int lines = p->line_len > 0 ? std::max(1, chunk / p->line_len) : 1;
  if (B >= 7 && !Cap::kSingle && ctas_by_smem<B, TV>(chunk, rc, Cap::LCMIN) < 2 &&
      ctas_by_smem<B, TV>(chunk, 0, Cap::LCMIN) >= 2 && p->n > (long long)lines * device_sms() * p->nlev_l)
    return 0;
  return rc;
}

// lc: as long as LCMAX where that leaves as many CTAs per SM as LCMIN does
// (96x96x48 b = 6 FP64 ILU(2), one CTA with 28 entries 48.5 ms, two with fewer 32.2;
// b = 8 ILU(0) 22.2 / 16.7).
template <int B, typename TV>
int batch_entries(int chunk, int rc) {
  using Cap = FactorCap<B, TV>;
  const int want = std::min(ctas_by_smem<B, TV>(chunk, rc, Cap::LCMIN), Cap::kSingle ? 3 : 2);
  int lc = Cap::LCMIN;
  while (lc < Cap::LCMAX && ctas_by_smem<B, TV>(chunk, rc, lc + 1) >= want) ++lc;
  return lc;
}

// Whether a value is finite, and the order of magnitudes, on the integer pipes
// (an FP64 comparison takes the FP64 pipe).
__device__ __forceinline__ unsigned long long magnitude(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ unsigned magnitude(float v) { return __float_as_uint(v) & 0x7fffffffu; }
__device__ __forceinline__ bool finite_bits(double v) { return magnitude(v) < 0x7ff0000000000000ull; }
__device__ __forceinline__ bool finite_bits(float v) { return magnitude(v) < 0x7f800000u; }

// D^{-1} by Gauss-Jordan with partial pivoting on [D | I]: lane c < 2B holds
// column c in registers (the lanes above hold zeros).
// False if a pivot or the result is zero or not finite.
template <int B, typename TV>
__device__ __forceinline__ bool invert_columns(TV (&col)[B], int lane) {
  bool bad = false;
#pragma unroll
  for (int r = 0; r < B; ++r) bad |= lane < B && !finite_bits(col[r]);
  if (__any_sync(kFull, bad)) return false;
#pragma unroll
  for (int c = 0; c < B; ++c) {
    // the pivot row, from column c
    int pr = c;
    auto best = magnitude(__shfl_sync(kFull, col[c], c));
    TV piv = __shfl_sync(kFull, col[c], c);
#pragma unroll
    for (int r = c + 1; r < B; ++r) {
      const TV v = __shfl_sync(kFull, col[r], c);
      if (magnitude(v) > best) {
        best = magnitude(v);
        pr = r;
        piv = v;
      }
    }
    if (best == 0) return false;
    const TV top = col[c];
#pragma unroll
    for (int r = c + 1; r < B; ++r)
      if (pr == r) {
        col[c] = col[r];
        col[r] = top;
      }
    col[c] = col[c] / piv;
    TV fr[B];
#pragma unroll
    for (int r = 0; r < B; ++r) fr[r] = __shfl_sync(kFull, col[r], c);
#pragma unroll
    for (int r = 0; r < B; ++r)
      if (r != c && magnitude(fr[r]) != 0) col[r] = fma(-fr[r], col[c], col[r]);
  }
  bad = false;
#pragma unroll
  for (int r = 0; r < B; ++r) bad |= lane >= B && lane < 2 * B && !finite_bits(col[r]);
  return !__any_sync(kFull, bad);
}

// Measured before / after (backfill to U' = D^{-1} U, same chunks): 96x96x48
// ILU(1) b = 3 FP64 6.20 / 5.56 ms, 61x47x33 ILU(2) b = 4 FP32 5.64 / 4.23 ms (with
// chunks of one line 2.10); per row 37 k cycles, of which 10 k the inverse, 9 k the
// pivots, 5 k staging.
// What bounds it: the FP64 pipe (19 cycles per warp instruction and SM whatever
// the active lanes) and the chain of dependent rows.  So a row's work is cut to
// the matching entries of its pivots' U rows, packed over the lanes, with
// comparisons on the integer pipes and the b x b inverse in registers; and the
// blocks of all pivots that are finished are fetched in one round trip, with
// only what depends on the last pivots left once those arrive.
template <int B, typename TV>
__global__ void __launch_bounds__(FactorCap<B, TV>::W * 32, FactorCap<B, TV>::MINB) factor_kernel(
    int32_t n, int32_t chunk, int32_t rc, int32_t lc_arg, int32_t nchunks, const int32_t* __restrict__ bnd,
    const int32_t* __restrict__ ord, const int32_t* __restrict__ tick,
    const int32_t* __restrict__ lrp, const int32_t* __restrict__ lci,
    const int32_t* __restrict__ urp, const int32_t* __restrict__ uci, TV* f, long long nnz_l,
    int32_t* header, int32_t* done, long long spin_ns) {
  using Cap = FactorCap<B, TV>;
  constexpr int BB = B * B;
  constexpr int H = (BB + 31) / 32;
  constexpr int KC = Cap::KC;
  const int lc = Cap::LCMIN == Cap::LCMAX ? Cap::LCMAX : lc_arg;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wvals = Cap::WVAL + (rc + lc) * BB;
  TV* rowv = reinterpret_cast<TV*>(smem_raw) + (size_t)warp * wvals;  // the row being factored
  TV* ub = rowv + rc * BB;  // U_pj of the batch's matches
  TV* db = ub + lc * BB;    // D_p^{-1}
  TV* aip = db + KC * BB;   // scaled A_ip
  int* fl = reinterpret_cast<int*>(reinterpret_cast<TV*>(smem_raw) + (size_t)Cap::W * wvals);  // ready flags (value =
                                                                                               // chunk id)
  int* s_i = fl + chunk;  // rows of the chunk in local-level order
  int* cols = s_i + chunk + warp * (Cap::WINT + 2 * lc + rc);  // column of each staged slot
  int* msrc = cols + rc;    // the batch's matches: U entry,
  int* mdst = msrc + lc;    // slot in the row
  int* moff = mdst + lc;    // first match of each pivot of the batch (33)
  int* coff = moff + 34;    // first candidate of each pivot of the batch (33)
  __shared__ int s_c;
  TV* L = f;
  TV* D = f + (size_t)nnz_l * BB;
  TV* U = D + (size_t)n * BB;
  for (int q = tid; q < chunk; q += blockDim.x) fl[q] = -1;
  Waiter w{header, spin_ns, 0, nullptr};
  bool dead = false;
  for (;;) {
    __syncthreads();
    if (tid == 0) {
      int cc = atomicAdd(header + kTicketF, 1);
      if (ld_volatile_s32(header + kAbort)) cc = nchunks;
      s_c = cc < nchunks ? tick[cc] : nchunks;
    }
    __syncthreads();
    const int c = s_c;
    if (c >= nchunks) return;
    const int lo = bnd[c], hi = bnd[c + 1];  // at most `chunk` rows
    const int len = hi - lo;
    for (int q = tid; q < len; q += blockDim.x) s_i[q] = ord[lo + q];
    __syncthreads();
    // first and end entry of a row in L and U
    auto extent = [&](int pos) {
      const int i = s_i[min(pos, len - 1)];
      return make_int4(lrp[i], lrp[i + 1], urp[i], urp[i + 1]);
    };
    int4 next = extent(warp);
    for (int pos = warp; pos < len && !dead; pos += Cap::W) {
      const int i = s_i[pos];
      const int lb = next.x, nl = next.y - lb;
      const int ub0 = next.z, nu = next.w - ub0;
      next = extent(pos + Cap::W);
      const int nrow = nl + 1 + nu;
      const bool staged = nrow <= rc;
      // slot k of row i: L blocks (k < nl), the pivot block (k == nl), U blocks
      auto blk = [&](int k) -> TV* {
        if (staged) return rowv + k * BB;
        if (k < nl) return L + (size_t)(lb + k) * BB;
        if (k == nl) return D + (size_t)i * BB;
        return U + (size_t)(ub0 + k - nl - 1) * BB;
      };
      auto colk = [&](int k) -> int {
        if (staged) return cols[k];
        if (k < nl) return lci[lb + k];
        if (k == nl) return i;
        return uci[ub0 + k - nl - 1];
      };
      if (staged) {
        for (int k = lane; k < nrow; k += 32)
          cols[k] = k < nl ? lci[lb + k] : (k == nl ? i : uci[ub0 + k - nl - 1]);
        for (int q = lane; q < nl * BB; q += 32) rowv[q] = L[(size_t)lb * BB + q];
        for (int q = lane; q < BB; q += 32) rowv[nl * BB + q] = D[(size_t)i * BB + q];
        for (int q = lane; q < nu * BB; q += 32) rowv[(nl + 1) * BB + q] = U[(size_t)ub0 * BB + q];
      }
      __syncwarp();
      int k0 = 0, s0 = 0;  // the next batch starts with entry s0 of pivot k0's U row
      while (k0 < nl && !dead) {
        // ---- the batch: whole pivots while their U rows hold at most lc
        // entries (lane x: pivot k0 + x); of a longer one, lc entries of it
        const int np = min(32, nl - k0);
        int p = -1, pb = 0, plen = 0;
        if (lane < np) {
          p = colk(k0 + lane);
          pb = urp[p] + (lane == 0 ? s0 : 0);
          plen = urp[p + 1] - pb;
        }
        int upto = plen;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int v = __shfl_up_sync(kFull, upto, d);
          if (lane >= d) upto += v;
        }
        const unsigned fits = __ballot_sync(kFull, lane < np && upto <= lc);
        int nfit = __popc(fits), next_s0 = 0;
        const bool slice = nfit == 0;
        if (slice) {
          nfit = 1;
          next_s0 = s0 + lc;
          if (lane == 0) upto = plen = lc;
        }
        const int cands = __shfl_sync(kFull, upto, nfit - 1);
        __syncwarp();
        coff[lane] = upto - plen;
        moff[lane] = 0;
        if (lane == 0) moff[32] = 0;
        __syncwarp();
        // ---- its matches: entries (p, j) with (i, j) in the row, j > p
        int nm = 0;
        for (int q0 = 0; q0 < cands; q0 += 32) {
          const int q = q0 + lane;
          int x = 0, dst = -1, src = 0;
          {
            int z = nfit;  // the last pivot whose first candidate is <= q
            while (z - x > 1) {
              const int mid = (x + z) >> 1;
              if (coff[mid] <= q) x = mid;
              else z = mid;
            }
          }
          const int first = __shfl_sync(kFull, pb, x);
          if (q < cands) {
            src = first + q - coff[x];
            const int j = uci[src];
            int a = k0 + x + 1, z = nrow;
            while (a < z) {
              const int mid = (a + z) >> 1;
              const int v = colk(mid);
              if (v == j) {
                dst = mid;
                break;
              }
              if (v < j) a = mid + 1;
              else z = mid;
            }
          }
          const unsigned m = __ballot_sync(kFull, dst >= 0);
          if (dst >= 0) {
            const int at = nm + __popc(m & ((1u << lane) - 1u));
            msrc[at] = src;
            mdst[at] = dst;
            if (cands > 32) atomicAdd(&moff[x + 1], 1);
          }
          nm += __popc(m);
          if (cands <= 32 && lane < nfit)  // all in one go: the matches before each pivot's end
            moff[lane + 1] = __popc(m & (upto >= 32 ? ~0u : (1u << upto) - 1u));
        }
        __syncwarp();
        if (cands > 32) {
          int upm = lane < nfit ? moff[lane + 1] : 0;
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(kFull, upm, d);
            if (lane >= d) upm += v;
          }
          __syncwarp();
          if (lane < nfit) moff[lane + 1] = upm;
          __syncwarp();
        }
        // the warp's next row: into L2 while this one waits (b = 1: its few bytes are
        // in lines its neighbours fetch; 96x96x48 ILU(1) FP32 1.87 / 1.74 ms without)
        if (B > 1 && k0 == 0 && s0 == 0) {
          auto pull = [&](const void* first, size_t bytes) {
            for (size_t o = (size_t)lane * 128; o < bytes; o += 32 * 128)
              asm volatile("prefetch.global.L2 [%0];" ::"l"((const char*)first + o));
          };
          pull(lci + next.x, (size_t)(next.y - next.x) * sizeof(int32_t));
          pull(uci + next.z, (size_t)(next.w - next.z) * sizeof(int32_t));
          pull(L + (size_t)next.x * BB, (size_t)(next.y - next.x) * BB * sizeof(TV));
          pull(U + (size_t)next.z * BB, (size_t)(next.w - next.z) * BB * sizeof(TV));
        }
        // ---- the pivots, as far as their rows are finished
        const bool local = p >= lo && p < hi;
        bool have = false;
        for (int x = 0; x < nfit && !dead;) {
          int run = 0;
          w.t0 = 0;
          for (unsigned it = 1;; ++it) {
            if (lane >= x && lane < nfit && !have)
              have = local ? ld_acquire_cta_shared_s32(fl + (p - lo)) == c : ld_acquire_s32(done + p) != 0;
            run = __ffs(~(__ballot_sync(kFull, have && lane < nfit) >> x)) - 1;
            if (run != 0) break;
            if (__any_sync(kFull, w.give_up(it))) {
              dead = true;
              break;
            }
          }
          if (dead) break;
          __syncwarp();
          if (run < 0) run = 32;
          run = min(min(run, nfit - x), KC);
          // their D_p^{-1} and matching U_pj, all loads in flight together
          const int m0 = moff[x], mv = (moff[x + run] - m0) * BB, dv = run * BB;
          constexpr int NB = (KC * BB + 31) / 32 < 5 ? (KC * BB + 31) / 32 : 5;
          for (int e0 = 0; e0 < dv || e0 < mv; e0 += 32 * NB) {
            TV tu[NB], td[NB];
#pragma unroll
            for (int h = 0; h < NB; ++h) {
              const int e = e0 + lane + 32 * h;
              if (e < dv) {
                const int y = e / BB;
                td[h] = D[(size_t)colk(k0 + x + y) * BB + (e - y * BB)];
              }
              if (e < mv) {
                const int y = e / BB;
                tu[h] = U[(size_t)msrc[m0 + y] * BB + (e - y * BB)];
              }
            }
#pragma unroll
            for (int h = 0; h < NB; ++h) {
              const int e = e0 + lane + 32 * h;
              if (e < dv) db[e] = td[h];
              if (e < mv) ub[e] = tu[h];
            }
          }
          __syncwarp();
          for (int y = 0; y < run; ++y) {
            const int k = k0 + x + y;
            // A_ip <- A_ip D_p^{-1} (once: with the first slice of a long U row)
            TV* const a = blk(k);
            if (x + y > 0 || s0 == 0) {
              const TV* const dp = db + y * BB;
              TV nv[H];
#pragma unroll
              for (int h = 0; h < H; ++h) {
                const int e = lane + 32 * h;
                if (e < BB) {
                  const int r = e % B, cc = e / B;
                  TV s = TV(0);
#pragma unroll
                  for (int m = 0; m < B; ++m) s = fma(a[m * B + r], dp[cc * B + m], s);
                  nv[h] = s;
                }
              }
              __syncwarp();
#pragma unroll
              for (int h = 0; h < H; ++h) {
                const int e = lane + 32 * h;
                if (e < BB) {
                  a[e] = nv[h];
                  aip[e] = nv[h];
                }
              }
              __syncwarp();
            }
            // A_ij <- A_ij - A_ip U_pj
            const int mb = moff[x + y], cnt = (moff[x + y + 1] - mb) * BB;
            auto term = [&](int sidx, int e) {
              const int r = e % B, cc = e / B;
              const TV* const upj = ub + (mb - m0 + sidx) * BB + cc * B;
              TV s = TV(0);
#pragma unroll
              for (int m = 0; m < B; ++m) s = fma(aip[m * B + r], upj[m], s);
              return s;
            };
            if (B >= 7 && !staged) {
              // in place: two elements a lane at a time, both read before either is
              // written (a pivot's matches are different blocks); one at a time is a
              // chain of round trips (b = 7 FP32 160x20x20 27-point 34.4 / 27.6 ms)
              for (int w0 = lane; w0 < cnt; w0 += 64) {
                const int w1 = w0 + 32;
                const int s0i = w0 / BB, e0 = w0 - s0i * BB;
                TV* const at0 = blk(mdst[mb + s0i]) + e0;
                const TV was0 = *at0;
                if (w1 < cnt) {
                  const int s1i = w1 / BB, e1 = w1 - s1i * BB;
                  TV* const at1 = blk(mdst[mb + s1i]) + e1;
                  const TV was1 = *at1;
                  const TV t0 = term(s0i, e0), t1 = term(s1i, e1);
                  *at0 = was0 - t0;
                  *at1 = was1 - t1;
                } else {
                  *at0 = was0 - term(s0i, e0);
                }
              }
            } else {
              for (int wk = lane; wk < cnt; wk += 32) {
                const int sidx = wk / BB, e = wk - sidx * BB;
                const TV s = term(sidx, e);
                blk(mdst[mb + sidx])[e] -= s;
              }
            }
            __syncwarp();
          }
          x += run;
        }
        if (slice) {
          s0 = next_s0;
        } else {
          k0 += nfit;
          s0 = 0;
        }
      }
      if (dead) break;
      // the row's U is final; later rows read it
      if (staged)
        for (int q = lane; q < nu * BB; q += 32) U[(size_t)ub0 * BB + q] = rowv[(nl + 1) * BB + q];
      TV col[B];
      {
        const TV* const di = blk(nl);
#pragma unroll
        for (int r = 0; r < B; ++r)
          col[r] = lane < B ? di[lane * B + r] : (lane < 2 * B && r == lane - B ? TV(1) : TV(0));
      }
      const bool bad = !invert_columns<B, TV>(col, lane);
      if (lane >= B && lane < 2 * B) {
#pragma unroll
        for (int r = 0; r < B; ++r) D[(size_t)i * BB + (lane - B) * B + r] = col[r];
      }
      if (bad && lane == 0) {
        atomicMin(header + kBadRow, i);
        atomicCAS(header + kErr, 0, (int)BILU_ERR_SINGULAR);
      }
      // rows of this chunk first: their flag needs no device-wide fence
      __threadfence_block();
      __syncwarp();
      if (lane == 0) st_release_cta_shared_s32(fl + (i - lo), c);
      __threadfence();
      __syncwarp();
      if (lane == 0) st_release_s32(done + i, 1);
      if (staged)
        for (int q = lane; q < nl * BB; q += 32) L[(size_t)lb * BB + q] = rowv[q];
      __syncwarp();
    }
  }
}

// Eq. 5: U'_ij = D_i^{-1} U_ij, one warp per block row; lane q of the row's
// (block, column) pairs reads one column of U_ij, forms that column of
// D_i^{-1} U_ij (b x b FMAs) and writes it back in place.  Columns are
// independent, so no lane waits on another.
template <int B, typename TV>
__global__ void __launch_bounds__(256) scale_upper_kernel(int32_t n, const int32_t* __restrict__ urp,
                                                          const TV* __restrict__ dinv,
                                                          TV* __restrict__ u) {
  constexpr int BB = B * B;
  const int lane = threadIdx.x & 31;
  const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long i = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += nw) {
    const int ub = urp[i], cnt = (urp[i + 1] - ub) * B;
    if (cnt == 0) continue;
    TV d[BB];  // D_i^{-1}, column-major
#pragma unroll
    for (int e = 0; e < BB; ++e) d[e] = __ldg(dinv + (size_t)i * BB + e);
    for (int q = lane; q < cnt; q += 32) {
      TV* col = u + ((size_t)ub + q / B) * BB + (q % B) * B;
      TV x[B];
#pragma unroll
      for (int m = 0; m < B; ++m) x[m] = col[m];
#pragma unroll
      for (int r = 0; r < B; ++r) {
        TV acc = TV(0);
#pragma unroll
        for (int m = 0; m < B; ++m) acc = fma(d[m * B + r], x[m], acc);
        col[r] = acc;
      }
    }
  }
}

template <typename TV>
int launch_backfill_t(const bilu_pattern* p, int32_t b, const double* a_vals, TV* f, void* stream) {
  const long long total = p->nslots() * (long long)b * b;
  if (total == 0) return 0;
  const int blocks = (int)std::min<long long>((total + 255) / 256, (long long)device_sms() * 16);
  ProfScope ps(BILU_PROF_BACKFILL, stream);
  backfill_kernel<TV><<<blocks, 256, 0, (cudaStream_t)stream>>>(total, b * b, p->d_slot_src, a_vals, f);
  return (int)cudaGetLastError();
}

template <typename TV>
int launch_factor_t(const bilu_pattern* p, int32_t b, TV* f, int32_t* header, int32_t* done,
                    void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  const int32_t n = p->n;
  const int sms = device_sms();
  {
    ProfScope ps0(BILU_PROF_FACTOR_INIT, stream);
    factor_init_kernel<<<std::max(1, std::min((n + 255) / 256, sms * 4)), 256, 0, s>>>(header, done, n);
  }
  if (n == 0) return (int)cudaGetLastError();
  if (p->fact.chunk <= 0 || !p->fact.d_mem) return (int)cudaErrorInvalidValue;
  const int chunk = p->fact.max_len;  // shared-memory rows per CTA
  const int nchunks = p->fact.nchunks;
  const long long spin = trisolve_config().spin_ns;
  BILU_DISPATCH_B(b, {
    const int rc = staged_rows<B, TV>(p);
    const int lc = batch_entries<B, TV>(chunk, rc);
    const size_t smem = factor_smem_bytes<B, TV>(chunk, rc, lc);
    static LaunchCache cache;
    const int per_sm = cache.ctas_per_sm(current_device(), smem, [](size_t bytes) {
      cudaFuncSetAttribute(factor_kernel<B, TV>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynamicSmem);
      int q = 0;
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, factor_kernel<B, TV>, FactorCap<B, TV>::W * 32, bytes);
      return q;
    });
    const int grid = std::max(1, std::min(nchunks, per_sm * sms));
    ProfScope ps(BILU_PROF_FACTOR, stream);
    factor_kernel<B, TV><<<grid, FactorCap<B, TV>::W * 32, smem, s>>>(n, chunk, rc, lc, nchunks, p->fact.d_bnd, p->fact.d_ord_l, p->fact.d_tick_l, p->d_lrp, p->d_lci,
                                                            p->d_urp, p->d_uci, f, p->nnz_l(), header, done,
                                                            spin);
  });
  return (int)cudaGetLastError();
}

template <typename TV>
int launch_scale_upper_t(const bilu_pattern* p, int32_t b, TV* f, void* stream) {
  const int32_t n = p->n;
  if (n == 0 || p->nnz_u() == 0) return 0;
  const size_t bb = (size_t)b * b;
  const TV* dinv = f + (size_t)p->nnz_l() * bb;
  TV* u = f + ((size_t)p->nnz_l() + n) * bb;
  const int grid = std::max(1, std::min((n + 7) / 8, device_sms() * 8));
  BILU_DISPATCH_B(b, {
    ProfScope ps(BILU_PROF_SCALE_UPPER, stream);
    scale_upper_kernel<B, TV><<<grid, 256, 0, (cudaStream_t)stream>>>(n, p->d_urp, dinv, u);
  });
  return (int)cudaGetLastError();
}

}  // namespace

int launch_backfill(const bilu_pattern* p, int32_t b, const double* a_vals, double* f, void* stream) {
  return launch_backfill_t<double>(p, b, a_vals, f, stream);
}
int launch_factor(const bilu_pattern* p, int32_t b, double* f, int32_t* header, int32_t* done, void* stream) {
  return launch_factor_t<double>(p, b, f, header, done, stream);
}
int launch_scale_upper(const bilu_pattern* p, int32_t b, double* f, void* stream) {
  return launch_scale_upper_t<double>(p, b, f, stream);
}
int launch_backfill_f32(const bilu_pattern* p, int32_t b, const double* a_vals, float* f, void* stream) {
  return launch_backfill_t<float>(p, b, a_vals, f, stream);
}
int launch_factor_f32(const bilu_pattern* p, int32_t b, float* f, int32_t* header, int32_t* done, void* stream) {
  return launch_factor_t<float>(p, b, f, header, done, stream);
}
int launch_scale_upper_f32(const bilu_pattern* p, int32_t b, float* f, void* stream) {
  return launch_scale_upper_t<float>(p, b, f, stream);
}

}  // namespace bilu
