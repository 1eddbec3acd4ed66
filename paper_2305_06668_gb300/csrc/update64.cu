// FP64 block updates out_t = base_t + alpha in_t U (X = V u_x with AX = AV u_x and the residual
// norms, P = V u_p, W - Y C, W L^{-T}) on the 5th-generation tensor cores: the rows of in_t and the
// columns of U are cut into FP16 digits (slices.cuh) whose products the tensor core sums exactly.
//
// What bounds it.  As FP64 FMAs (2 per clock and SM) the pair X, AX of 10^6 rows, 63 columns to 21,
// takes 5 ms, in double-float on the FP32 pipes 2.4 ms; its bytes take 0.2 ms and its digit products
// 0.12 ms of tensor time.  What is left to pay is the cutting into digits and the joining of the sums, on
// the integer pipe (60% busy at 200,000 rows; tensor pipe 13%, DRAM 18%): a call of that pair with norms
// went from 2,890 (double-float) to 800 us, 910 with the test of spread below.  Four epilogue warps instead
// of eight took 1,480, stores by row instead of turned ones and residuals exchanged behind barriers 868.
//
// Scaling.  Column l of V and row l of U are scaled against each other by the power of two above
// max_j |alpha U_lj|, so an entry of a row counts by the most it contributes to any output; then every
// row of V has one exponent and every column of U one.  A row's entries are held to 2^-56 of its
// largest contribution, digit sums are exact, each product is rounded to FP64 once and the base is
// added in FP64.  That is a bound against the row's norm; SPREAD finds the rows with an output whose own
// terms are far below it.
//
// One persistent CTA per SM takes a contiguous range of 128-row tiles:
//   * warps 0..15, splitters: warp w owns rows 8 w .. 8 w + 7 of the tile.  Its lane 0 copies them
//     (1-D TMA bulk copies, one per segment) into the warp's own raw slot, the next tile's as soon
//     as this tile's are in registers.  A lane holds 8 columns of one row per 32-column chunk; the
//     row's exponent comes from two shuffles; a chunk's digits go to a tile buffer as K-major core
//     matrices, 128 bytes per quarter warp without bank conflicts.
//   * warp 24, one thread: the MMA issuer.  Digit i of V against digits j, j + 1, .. of U writes TMEM
//     columns 32 (i + j), ..: region t of an accumulator sums the products with i + j = t, at most
//     7 * 96 * 2^14 < 2^24, exact.
//   * warps 16..23, epilogue: two threads per row, which take the groups of four columns in turn.  The
//     eight regions of an element are joined into FP64 with integer operations and turned inside the warp
//     to four lanes per row, which add the base, store 32-byte pieces of rows and, from the pair's two
//     elements, keep the sum of squares and the maximum of the residuals of their column.
// Rows with an infinity, a NaN or an exponent outside 2^+-400 (and all rows when U has one), and with
// SPREAD rows with an output far below the rest, are formed by their epilogue warp with FP64 FMAs.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "slices.cuh"
#include "umma.cuh"

namespace lobpcg {
namespace {

using namespace umma;
using namespace slices;

constexpr int kTile = 128;      // rows per tile
constexpr int kQ = 32;          // output columns, padded
constexpr int kKC = 32;         // columns of V per chunk
constexpr int kMaxTS = 2;       // chunk buffers: two where shared memory holds them, else one
constexpr int kRing = 8;        // row-exponent ring (a splitter is at most 4 products ahead)
constexpr int kSplitWarps = 16, kEpi0 = 16, kEpiWarps = 8, kMma = 24;
constexpr int kThreads = 32 * 25;
constexpr uint32_t kLBO = 128, kSBO = kKC / 8 * 128;
constexpr uint32_t kSlice = kTile / 8 * kSBO;  // bytes of one digit of a chunk of V
constexpr uint32_t kBuf = kSlices * kSlice;
constexpr int kAcc = kDiags * kQ;              // TMEM columns of one accumulator
constexpr int kBad = -1;
constexpr size_t kStatic = 14 * 1024;  // static shared memory, at most
constexpr size_t kSmemBudget = 227 * 1024;

// bytes of U's digits: kSlices slices of kQ columns x KP rows
__host__ __device__ constexpr uint32_t u_slice(int kp) { return (uint32_t)(kQ * kp * 2); }

// What the digits of a row may drop is 2^-56 of its largest contribution to any output, and an output
// may consist of smaller ones (columns of V of different length met by equal rows of U).  With 2^E and
// 2^C the powers of two at row i's largest |V_il| g_l and at column j's largest |U_lj| / g_l (g_l: row l
// of alpha U, at most), an entry l whose factors are both within 3 binades of those gives
// sum |V||alpha U| at least 2^-6 2^(E+C), one whose U is within 6 binades 2^-9.  An output is safe
// where that comes to 2^-6 2^(E+C) per 32 entries of the row: the digits' rounding, 2^-57.8 sqrt(s)
// 2^(E+C+2) in the mean, is then below double-float's 2^-48 of the sum.
constexpr int kNear = 3, kMid = 6;
__device__ __forceinline__ bool output_safe(int near, int mid, int s32) { return 7 * near + mid >= 8 * s32; }

// The scaling of U, by all threads of a CTA; us: alpha U (s x q, column-major).
struct UScale {
  int16_t up[kMaxS];         // exponent of row l of U: V's column l is scaled by 2^up; -4000: a zero row
  int col_exp[kQ];           // exponent of column j over its scaled entries
  uint32_t near[kQ][kMaxS / 32], mid[kQ][kMaxS / 32];  // bit l: (l, j) within kNear, kMid binades of 2^col_exp
  uint32_t nonzero;          // columns with any non-zero entry
  int small;                 // most entries of a non-zero column that are not in `mid`
  int bad;                   // a row or column outside the digits' range
};
__device__ __forceinline__ void scale_u(UScale& u, const double* us, int s, int q) {
  if (threadIdx.x == 0) u.bad = 0, u.nonzero = 0u, u.small = 0;
  __syncthreads();
  for (int l = threadIdx.x; l < kMaxS; l += blockDim.x) {
    uint32_t key = 0u;
    if (l < s)
      for (int j = 0; j < q; ++j) key = max(key, exp_key(us[l + j * s]));
    const int e = group_exp(key);
    if (e < 0) u.bad = 1;
    u.up[l] = key ? (int16_t)(e - 1022) : (int16_t)-4000;  // a zero row of U: no contribution
  }
  __syncthreads();
  // U's entry (l, j) scaled by 2^-up: below 1 in magnitude.  A warp per column.
  const int lane = threadIdx.x & 31;
  for (int j = threadIdx.x >> 5; j < kQ; j += blockDim.x >> 5) {
    int e[kMaxS / 32], E = 0;
    bool any = false;
#pragma unroll
    for (int c = 0; c < kMaxS / 32; ++c) {
      const int l = 32 * c + lane;
      const uint32_t key = j < q && l < s ? exp_key(us[l + j * s]) : 0u;
      any |= key != 0u;
      e[c] = key >> 20 ? (int)(key >> 20) - u.up[l] : -10000;
      E = max(E, e[c]);
    }
    E = __reduce_max_sync(0xffffffffu, E);
    any = __any_sync(0xffffffffu, any);
    int in = 0;
#pragma unroll
    for (int c = 0; c < kMaxS / 32; ++c) {
      const uint32_t near = __ballot_sync(0xffffffffu, e[c] >= E - kNear);
      const uint32_t mid = __ballot_sync(0xffffffffu, e[c] >= E - kMid);
      if (lane == 0) u.near[j][c] = near, u.mid[j][c] = mid;
      in += __popc(mid);
    }
    if (lane) continue;
    if (any && E < kExpMin) u.bad = 1;  // a column of numbers far below their rows'
    u.col_exp[j] = any ? E : kExpOne;
    if (any) atomicOr(&u.nonzero, 1u << j), atomicMax(&u.small, s - in);
  }
  __syncthreads();
}

// NC: 32-column chunks of V (ceil(s / 32)).  SPREAD: rows too far apart are found and formed with FMAs.
template <int NC, bool NORM, bool SPREAD>
__global__ void __launch_bounds__(kThreads, 1)
    update64_kernel(int64_t n, UpdateJob<double> job, const double* __restrict__ U, int s, int q, double alpha,
                    const double* __restrict__ lam, double* __restrict__ norm_part, int64_t tiles_per_cta,
                    int ts, int* __restrict__ err) {
  constexpr int KP = NC * kKC;
  constexpr uint32_t kSliceU = u_slice(KP), kSBOU = KP / 8 * 128;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ uint64_t raw_full[kSplitWarps], tile_full[kMaxTS], tile_empty[kMaxTS], acc_full[2], acc_empty[2], exp_full[kRing];
  __shared__ uint64_t rows_read[4];  // both epilogue warps of a lane quadrant have read their rows
  __shared__ int16_t row_exp[kRing][kTile];
  __shared__ __align__(16) UScale us_;
  int16_t* const up = us_.up;
  int* const col_exp = us_.col_exp;
  __shared__ double nred[2][kEpiWarps][NORM ? kQ / 2 : 1];  // a warp's sums and maxima of its columns
  __shared__ double lam_s[kQ];
  __shared__ double stage[kEpiWarps][32][4];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nseg = job.in[0].nseg, nprod = job.nprod;
  int raw_row = 0;  // doubles of one row of all segments
  for (int g = 0; g < nseg; ++g) raw_row += job.in[0].ld[g];
  unsigned char* tiles = smem;                                            // [ts][kBuf]
  unsigned char* udig = smem + (uint32_t)ts * kBuf;                       // [kSlices][kSliceU]
  double* raw = reinterpret_cast<double*>(udig + kSlices * kSliceU);      // [kSplitWarps][segment][8][ld]

  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < kSplitWarps; ++i) mbar_init(&raw_full[i], 1);
    for (int i = 0; i < kMaxTS; ++i) mbar_init(&tile_full[i], kSplitWarps), mbar_init(&tile_empty[i], 1);
    for (int i = 0; i < 2; ++i) mbar_init(&acc_full[i], 1), mbar_init(&acc_empty[i], kEpiWarps);
    for (int i = 0; i < kRing; ++i) mbar_init(&exp_full[i], kSplitWarps);
    for (int i = 0; i < 4; ++i) mbar_init(&rows_read[i], 2);
    fence_barrier_init();
  }
  for (uint32_t e = tid; e < kSlices * kSliceU / 16; e += kThreads) reinterpret_cast<uint4*>(udig)[e] = make_uint4(0, 0, 0, 0);
  // alpha U, staged in the first tile buffer (s x q column-major, at most 24 KB of its 56)
  double* us = reinterpret_cast<double*>(tiles);
  for (int e = tid; e < s * q; e += kThreads) us[e] = alpha * U[e];
  if (NORM)
    for (int j = tid; j < kQ; j += kThreads) lam_s[j] = j < q ? lam[j] : 0.0;
  scale_u(us_, us, s, q);
  for (int e = tid; e < s * q; e += kThreads) {
    const int l = e % s, j = e / s;
    // digits() takes the exponent in the entry's own scale; entries far below their column shift out
    const uint64_t w = up[l] > -4000 ? digits(us[e], col_exp[j] + up[l]) : digits(0.0, kExpOne);
    unsigned char* o = udig + (uint32_t)(j >> 3) * kSBOU + (uint32_t)(l >> 3) * kLBO + 16u * (j & 7) + 2u * (l & 7);
    uint32_t d[kSlices];
    digit_pairs(w, w, d);
#pragma unroll
    for (int k = 0; k < kSlices; ++k) *reinterpret_cast<uint16_t*>(o + k * kSliceU) = (uint16_t)d[k];
  }
  __syncwarp();
  if (warp == kMma) tmem_alloc(&tmem_slot, 2 * kAcc);
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const bool all_bad = us_.bad != 0;

  const int64_t t_begin = (int64_t)blockIdx.x * tiles_per_cta;
  const int64_t r_begin = t_begin * kTile, r_end = min(n, r_begin + tiles_per_cta * kTile);
  const int ntiles = r_end > r_begin ? (int)((r_end - r_begin + kTile - 1) / kTile) : 0;
  const int nT = ntiles * nprod;  // tile-products, in the order tile, product
  int copied = 0, committed = 0;  // splitter lane 0 / MMA thread

  if (warp < kSplitWarps) {
    const int r = lane & 7, k8 = lane >> 3;  // row within the warp's eight; group of 8 columns within a chunk
    double* slot = raw + (size_t)warp * 8 * raw_row;
    auto copy = [&](int T) {
      const Cols<double>& c = job.in[T % nprod];
      const int64_t r0 = r_begin + (int64_t)(T / nprod) * kTile + 8 * warp;
      const int rows = (int)min((int64_t)8, r_end - r0);
      if (rows <= 0) {  // no row of this warp in the last tile
        mbar_arrive(&raw_full[warp]);
        return;
      }
      uint32_t total = 0;  // a segment's last row is copied up to its used columns
      for (int g = 0; g < nseg; ++g) total += (uint32_t)((rows - 1) * c.ld[g] + (c.w[g] + 1) / 2 * 2) * 8u;
      mbar_expect_tx(&raw_full[warp], total);
      double* d = slot;
      for (int g = 0; g < nseg; ++g) {
        bulk_g2s(d, c.p[g] + r0 * c.ld[g], (uint32_t)((rows - 1) * c.ld[g] + (c.w[g] + 1) / 2 * 2) * 8u, &raw_full[warp]);
        d += 8 * c.ld[g];
      }
    };
    // column l of row r in the slot: base_g + l with the segment's base
    const int w0 = job.in[0].w[0], w1 = nseg > 1 ? w0 + job.in[0].w[1] : INT_MAX;
    const int b0 = r * job.in[0].ld[0];
    const int b1 = nseg > 1 ? 8 * job.in[0].ld[0] + r * job.in[0].ld[1] - w0 : 0;
    const int b2 = nseg > 2 ? 8 * (job.in[0].ld[0] + job.in[0].ld[1]) + r * job.in[0].ld[2] - w1 : 0;
    if (lane == 0 && nT > 0) copy(0), copied = 1;
    int buf = 0;
    uint32_t tph = 1;  // parity of the tile_empty phase to wait for (the first ts chunks do not wait)
    int chunk = 0;
    for (int T = 0; T < nT; ++T) {
      if (!__all_sync(0xffffffffu, wait_bar(&raw_full[warp], (uint32_t)T & 1u, &abort_flag, err, 1))) break;
      const bool live = r_begin + (int64_t)(T / nprod) * kTile + 8 * warp + r < r_end;
      double x[NC][8];
      int E = 0;
      bool bad = false;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int4 u4 = *reinterpret_cast<const int4*>(&up[c * kKC + 8 * k8]);
        const int us4[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int l = c * kKC + 8 * k8 + i;
          x[c][i] = live && l < s ? slot[(l < w0 ? b0 : l < w1 ? b1 : b2) + l] : 0.0;
          const int e = (__double2hiint(x[c][i]) >> 20) & 0x7ff;
          const int v = i & 1 ? us4[i >> 1] >> 16 : (int)(int16_t)us4[i >> 1];
          bad |= e == 0x7ff;
          if (e > 0) E = max(E, e + v);
        }
      }
      __syncwarp();  // the warp's slot is in registers: refill it
      if (lane == 0 && T + 1 < nT) copy(T + 1), copied = T + 2;
      E = max(E, __shfl_xor_sync(0xffffffffu, E, 8));
      E = max(E, __shfl_xor_sync(0xffffffffu, E, 16));
      const uint32_t badm = __ballot_sync(0xffffffffu, bad);
      bad = (badm & (0x01010101u << r)) != 0u || (E > 0 && (E < kExpMin || E > kExpMax));
      if (__any_sync(0xffffffffu, E <= 0)) {  // no contribution of normal size: a row of zeros, or too small
        bool some = false;
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
          for (int i = 0; i < 8; ++i) some |= up[c * kKC + 8 * k8 + i] > -4000 && x[c][i] != 0.0;
        const uint32_t somem = __ballot_sync(0xffffffffu, some);
        bad |= E <= 0 && (somem & (0x01010101u << r)) != 0u;
      }
      const bool judge = SPREAD && E > 0 && !bad;
      if (E <= 0 || bad) E = kExpOne;
      uint32_t near[NC];  // entries of the row within kNear binades of 2^E, this lane's in its byte
#pragma unroll
      for (int c = 0; c < NC; ++c) near[c] = 0u;
      bool done = true;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (chunk >= ts && !__all_sync(0xffffffffu, wait_bar(&tile_empty[buf], tph, &abort_flag, err, 2))) {
          done = false;
          break;
        }
        const int4 u4 = *reinterpret_cast<const int4*>(&up[c * kKC + 8 * k8]);
        const int us4[4] = {u4.x, u4.y, u4.z, u4.w};
        uint64_t w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int v = i & 1 ? us4[i >> 1] >> 16 : (int)(int16_t)us4[i >> 1];
          // the row's exponent in the entry's own scale; a bad row's digits are not used
          w[i] = digits(bad ? 0.0 : x[c][i], v > -4000 ? E - v : 4 * kExpOne);
        }
        if constexpr (SPREAD) {
          // |leading digit| >= 9: at least 2^51 of the 2^54 that 2^E is
#pragma unroll
          for (int i = 0; i < 8; ++i)
            near[c] |= (((uint32_t)(w[i] >> 48) & 0xffu) - 120u > 16u ? 1u : 0u) << (8 * k8 + i);
        }
        unsigned char* o = tiles + (uint32_t)buf * kBuf + (uint32_t)warp * kSBO + (uint32_t)k8 * kLBO + 16u * r;
        put_digits(w, o, kSlice);
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tile_full[buf]);
        ++chunk;
        if (++buf == ts) buf = 0, tph ^= 1u;
      }
      if (!done) break;
      if constexpr (SPREAD) {
        int count = 0;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          near[c] |= __shfl_xor_sync(0xffffffffu, near[c], 8);
          near[c] |= __shfl_xor_sync(0xffffffffu, near[c], 16);
          count += __popc(near[c]);
        }
        // enough of them for every output, whichever the column's small entries are; else output by output
        const bool unsure = judge && count - us_.small < 8 * NC;
        if (__any_sync(0xffffffffu, unsure)) {
          bool apart = false;
          for (int j = k8; j < q; j += 4) {
            int nn = 0, nm = 0;
#pragma unroll
            for (int c = 0; c < NC; ++c)
              nn += __popc(near[c] & us_.near[j][c]), nm += __popc(near[c] & us_.mid[j][c]);
            apart |= unsure && !output_safe(nn, nm, NC) && (us_.nonzero >> j & 1u) != 0u;
          }
          const uint32_t apartm = __ballot_sync(0xffffffffu, apart);
          bad |= (apartm & (0x01010101u << r)) != 0u;
        }
      }
      if (lane < 8) row_exp[T & (kRing - 1)][8 * warp + lane] = (int16_t)(bad ? kBad : E);
      __syncwarp();
      if (lane == 0) mbar_arrive(&exp_full[T & (kRing - 1)]);
    }
  } else if (warp == kMma) {
    if (lane == 0) {
      const uint64_t dA = desc_kmajor(smem_addr(tiles), kLBO, kSBO);
      const uint64_t dB = desc_kmajor(smem_addr(udig), kLBO, kSBOU);
      const int ksteps = (s + 15) / 16;
      int buf = 0;
      uint32_t tph = 0, aph = 0;
      bool ok = true;
      for (int T = 0; T < nT && ok; ++T) {
        const int a = T & 1;
        if (T >= 2 && !wait_bar(&acc_empty[a], aph ^ 1u, &abort_flag, err, 3)) break;
        const uint32_t d = tmem + (uint32_t)(a * kAcc);
        for (int c = 0; c < NC; ++c) {
          if (!wait_bar(&tile_full[buf], tph, &abort_flag, err, 3)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t bo = dA + (uint64_t)((uint32_t)buf * kBuf >> 4);
          for (int kk = 0; kk < kKC / 16 && 2 * c + kk < ksteps; ++kk) {
            const uint32_t acc = c > 0 || kk > 0 ? 1u : 0u;
            const uint64_t ka = bo + (uint64_t)(kk * 16), kb = dB + (uint64_t)((2 * c + kk) * 16);
            auto mma = [&](int i, int j, int cnt, uint32_t ac) {
              mma_f16(d + (uint32_t)(kQ * (i + j)), ka + (uint64_t)(i * (kSlice >> 4)),
                      kb + (uint64_t)(j * (kSliceU >> 4)), idesc_f16(kTile, (uint32_t)(kQ * cnt)), ac);
            };
            mma(0, 0, 7, acc);  // regions 0..6
            mma(1, 0, 6, 1u);
            mma(1, 6, 1, acc);  // region 7, overwriting what an earlier product left
#pragma unroll
            for (int i = 2; i < kSlices; ++i) mma(i, 0, kDiags - i, 1u);
          }
          mma_commit(&tile_empty[buf]);
          if (++buf == ts) buf = 0, tph ^= 1u;
        }
        if (ok) {
          mma_commit(&acc_full[a]);
          committed = T + 1;
          if (a == 1) aph ^= 1u;
        }
      }
    }
  } else {
    const int quad = warp & 3, half = (warp - kEpi0) >> 2, row = 32 * quad + lane;
    double nsum[kQ / 8], nmax[kQ / 8];
#pragma unroll
    for (int g = 0; g < kQ / 8; ++g) nsum[g] = 0.0, nmax[g] = 0.0;
    bool ok = true;
    uint32_t rph = 0;  // parity of the next rows_read phase
    for (int it = 0; it < ntiles && ok; ++it) {
      const bool live = r_begin + (int64_t)it * kTile + row < r_end;
      int er[2] = {kExpOne, kExpOne};
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        if (t >= nprod) break;
        const int T = it * nprod + t;
        ok = ok && __all_sync(0xffffffffu, wait_bar(&exp_full[T & (kRing - 1)], (uint32_t)(T / kRing) & 1u, &abort_flag, err, 2));
        ok = ok && __all_sync(0xffffffffu, wait_bar(&acc_full[T & 1], (uint32_t)(T / 2) & 1u, &abort_flag, err, 2));
        if (ok) er[t] = all_bad ? kBad : row_exp[T & (kRing - 1)][row];
      }
      if (!ok) break;
      tc_fence_after();
      // rows outside the digits' range or too far apart: FP64 FMAs from global memory, a row at a time by the
      // whole warp (eight lanes a column, four columns at once), all of this warp's elements before any store
      const int64_t row0 = r_begin + (int64_t)it * kTile + 32 * quad;  // rows of this warp
      const int nrows = (int)max((int64_t)0, min((int64_t)32, r_end - row0));
      double slow[2][kQ / 8][4];
#pragma unroll 1
      for (int t = 0; t < nprod; ++t) {
        for (uint32_t m = __ballot_sync(0xffffffffu, live && er[t] == kBad); m; m &= m - 1u) {
          const int rr = __ffs(m) - 1;
#pragma unroll 1
          for (int gh = 0; gh < kQ / 8; ++gh) {
            const int j = 4 * (2 * gh + half) + (lane & 3);
            if (j - (lane & 3) >= q) break;
            double a = 0.0;
            if (j < q) {
              const double* u = U + j * s;
#pragma unroll 1
              for (int g = 0; g < nseg; ++g) {
                const double* v = job.in[t].p[g] + (row0 + rr) * job.in[t].ld[g];
                for (int i = lane >> 2; i < job.in[t].w[g]; i += 8) a = fma(v[i], u[i], a);
                u += job.in[t].w[g];
              }
            }
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const double x = __shfl_sync(0xffffffffu, a, k);
              if (lane == rr) slow[t][gh][k] = alpha * x;
            }
          }
        }
      }
      int se[2];  // element: (sum_t v_t 256^(7-t)) 2^(40 - 110) 2^(er - 1022) 2^(col_exp - 1022)
#pragma unroll
      for (int t = 0; t < 2; ++t) se[t] = (er[t] == kBad ? kExpOne : er[t]) - 2 * 1022 - 70;
      // both threads of a row have read it before either stores (the two warps see the same rows, so both
      // or neither come here); bounded like every wait, for the partner may have given up
      const bool any_bad = __any_sync(0xffffffffu, er[0] == kBad || er[1] == kBad);
      if (any_bad) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&rows_read[quad]);
        ok = __all_sync(0xffffffffu, wait_bar(&rows_read[quad], rph, &abort_flag, err, 4));
        rph ^= 1u;
        if (!ok) break;
      }
#pragma unroll
      for (int gh = 0; gh < kQ / 8; ++gh) {
        const int g = 2 * gh + half;
        if (4 * g >= q) break;
        double xs[4];  // NORM: the pair's X elements of this lane's rows and column
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          if (t >= nprod) break;
          const int a = (it * nprod + t) & 1;
          float v[kDiags][4];
#pragma unroll
          for (int d = 0; d < kDiags; ++d)
            tmem_ld4(tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(a * kAcc + kQ * d + 4 * g), v[d]);
          tmem_wait_ld(v);
          double o[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int j = 4 * g + i;
            float w[kDiags];
#pragma unroll
            for (int d = 0; d < kDiags; ++d) w[d] = v[d][i];
            o[i] = join(w, se[t] + col_exp[j]);
          }
          if (any_bad && er[t] == kBad)
#pragma unroll
            for (int i = 0; i < 4; ++i) o[i] = slow[t][gh][i];
          // to the warp's stage (columns turned by row / 4: no bank conflicts either way), then four lanes per
          // row: whole 32-byte pieces of eight rows a store
#pragma unroll
          for (int i = 0; i < 4; ++i) stage[warp - kEpi0][lane][(i + (lane >> 2)) & 3] = o[i];
          __syncwarp();
          const int j = 4 * g + (lane & 3);
          double* out = job.out[t] + (row0 + (lane >> 2)) * job.ld_out[t] + j;
          const double* base = NORM || !job.base[t] ? nullptr : job.base[t] + (row0 + (lane >> 2)) * job.ld_base[t] + j;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int rr = 8 * k + (lane >> 2);
            double x = stage[warp - kEpi0][rr][((lane & 3) + (rr >> 2)) & 3];
            const bool mine = rr < nrows && j < q;
            if (mine) {
              if (!NORM && base) x = base[(int64_t)(8 * k) * job.ld_base[t]] + x;
              out[(int64_t)(8 * k) * job.ld_out[t]] = x;
            }
            if constexpr (NORM) {
              if (t == 0) {
                xs[k] = x;
              } else if (mine) {
                const double res = fma(-lam_s[j], xs[k], x);  // AX - lam X, one rounding
                nsum[gh] = fma(res, res, nsum[gh]);
                // max of magnitudes by their bits (a NaN does not count, as in fmax)
                const long long ax = __double_as_longlong(res) & 0x7fffffffffffffffll;
                if (ax > __double_as_longlong(nmax[gh]) && ax <= 0x7ff0000000000000ll) nmax[gh] = __longlong_as_double(ax);
              }
            }
          }
          __syncwarp();
        }
      }
      tc_fence_before();
      __syncwarp();
#pragma unroll
      for (int t = 0; t < 2; ++t)
        if (t < nprod && lane == 0) mbar_arrive(&acc_empty[(it * nprod + t) & 1]);
    }
    if constexpr (NORM) {
      // lanes of one column, then the four warps of one half, in a fixed order
#pragma unroll
      for (int gh = 0; gh < kQ / 8; ++gh) {
        double s2 = nsum[gh], mx = nmax[gh];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
          s2 += __shfl_xor_sync(0xffffffffu, s2, o);
          mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        if (lane < 4) nred[0][warp - kEpi0][4 * gh + lane] = s2, nred[1][warp - kEpi0][4 * gh + lane] = mx;
      }
      asm volatile("bar.sync 3, 256;\n" ::: "memory");  // the eight epilogue warps
      const int j = tid - 32 * kEpi0;
      if (j < q) {
        const int h = (j >> 2) & 1, c = 4 * (j >> 3) + (j & 3);  // half and column within it
        double s2 = 0.0, mx = 0.0;
        for (int u = 0; u < 4; ++u) s2 += nred[0][4 * h + u][c], mx = fmax(mx, nred[1][4 * h + u][c]);
        norm_part[(int64_t)blockIdx.x * 2 * q + j] = s2;
        norm_part[(int64_t)blockIdx.x * 2 * q + q + j] = mx;
      }
    }
  }
  __syncthreads();
  if (abort_flag) {
    if (warp < kSplitWarps && lane == 0 && copied > 0) mbar_wait(&raw_full[warp], (uint32_t)(copied - 1) & 1u, kWaitCycles);
    if (warp == kMma && lane == 0 && committed > 0)
      mbar_wait(&acc_full[(committed - 1) & 1], (uint32_t)((committed - 1) / 2) & 1u, kWaitCycles);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMma) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 2 * kAcc);
  }
}

// *count += the rows among `samples` evenly spaced ones that update64_kernel would form with FMAs for
// their spread.  A warp per row, a lane per entry.
__global__ void __launch_bounds__(256) update64_sample_kernel(int64_t n, UpdateJob<double> job, const double* __restrict__ U,
                                                              int s, int q, double alpha, int samples,
                                                              int* __restrict__ count) {
  __shared__ UScale u;
  extern __shared__ double us[];
  for (int e = threadIdx.x; e < s * q; e += blockDim.x) us[e] = alpha * U[e];
  __syncthreads();
  scale_u(u, us, s, q);
  if (u.bad) return;  // every row takes the FMAs, none for its spread
  const int lane = threadIdx.x & 31, warps = gridDim.x * (blockDim.x >> 5);
  int total = 0;
  for (int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < samples; i += warps) {
    const int64_t row = (int64_t)i * n / samples;
    bool apart = false;
    for (int t = 0; t < job.nprod; ++t) {
      int e[kMaxS / 32], E = 0;
#pragma unroll
      for (int c = 0; c < kMaxS / 32; ++c) {
        int l = 32 * c + lane, g = 0;
        e[c] = -10000;
        if (l < s) {
          const int up = u.up[l];
          while (l >= job.in[t].w[g]) l -= job.in[t].w[g], ++g;
          const int x = (__double2hiint(job.in[t].p[g][row * job.in[t].ld[g] + l]) >> 20) & 0x7ff;
          if (x != 0 && x != 0x7ff) e[c] = x + up;
        }
        E = max(E, e[c]);
      }
      E = __reduce_max_sync(0xffffffffu, E);
      if (E <= 0) continue;
      int nn = 0, nm = 0;
#pragma unroll
      for (int c = 0; c < kMaxS / 32; ++c) {
        const uint32_t near = __ballot_sync(0xffffffffu, e[c] >= E - kNear);
        nn += __popc(near & u.near[lane][c]), nm += __popc(near & u.mid[lane][c]);  // lane: an output
      }
      apart |= __any_sync(0xffffffffu, !output_safe(nn, nm, (s + 31) / 32) && (u.nonzero >> lane & 1u) != 0u);
    }
    total += apart ? 1 : 0;
  }
  if (lane == 0 && total) atomicAdd(count, total);
}

template <int NC, bool NORM, bool SPREAD>
int update64_launch(int64_t n, const UpdateJob<double>& job, const double* U, int s, int q, double alpha,
                    const double* lam, double* norm_part, int max_ctas, size_t smem, int ts, int* err,
                    cudaStream_t st) {
  static const bool attr = [&] {
    LB_CUDA(cudaFuncSetAttribute(update64_kernel<NC, NORM, SPREAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kSmemBudget - kStatic)));
    return true;
  }();
  (void)attr;
  int dev = 0, sms = 152;
  LB_CUDA(cudaGetDevice(&dev));
  LB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t tiles = ceil_div(n, kTile);
  const int64_t per = ceil_div(tiles, std::min<int64_t>(std::min<int64_t>(max_ctas, sms), tiles));
  const int64_t ctas = ceil_div(tiles, per);
  update64_kernel<NC, NORM, SPREAD><<<(unsigned)ctas, kThreads, smem, st>>>(n, job, U, s, q, alpha, lam, norm_part, per,
                                                                    ts, err);
  LB_LAUNCH_CHECK();
  return (int)ctas;
}

}  // namespace

// The block update through digit products; returns 0 without launching where the blocks do not fit
// (unaligned or odd row strides, products of different layout, more shared memory than a CTA has).
int launch_update_digits(int64_t n, const UpdateJob<double>& job, const double* U, int s, int q, double alpha,
                         const double* lam, double* norm_part, int max_ctas, bool spread, int* err,
                         cudaStream_t st) {
  if (n <= 0 || q < 1 || q > kQ || s < 1 || s > kMaxS || job.in[0].nseg < 1) return 0;
  if (norm_part && (job.nprod != 2 || job.base[0] || job.base[1])) return 0;
  size_t raw = 0;
  for (int t = 0; t < job.nprod; ++t) {
    const Cols<double>& c = job.in[t];
    if (c.nseg != job.in[0].nseg) return 0;
    for (int g = 0; g < c.nseg; ++g) {
      if ((c.ld[g] & 1) || c.w[g] > c.ld[g] || (reinterpret_cast<uintptr_t>(c.p[g]) & 15)) return 0;
      if (c.w[g] != job.in[0].w[g] || c.ld[g] != job.in[0].ld[g]) return 0;
      if (t == 0) raw += (size_t)kTile * c.ld[g] * 8;
    }
  }
  const int nc = (s + kKC - 1) / kKC;
  const size_t fixed = kSlices * (size_t)u_slice(nc * kKC) + raw;
  const int ts = fixed + 2 * (size_t)kBuf <= kSmemBudget - kStatic ? 2 : 1;
  const size_t smem = fixed + (size_t)ts * kBuf;
  if (smem > kSmemBudget - kStatic) return 0;
#define LB_UPDATE64_(NC, NORM, SPREAD) \
  return update64_launch<NC, NORM, SPREAD>(n, job, U, s, q, alpha, lam, norm_part, max_ctas, smem, ts, err, st)
#define LB_UPDATE64(NC)                                \
  {                                                    \
    if (norm_part && spread) LB_UPDATE64_(NC, true, true);   \
    if (norm_part) LB_UPDATE64_(NC, true, false);      \
    if (spread) LB_UPDATE64_(NC, false, true);         \
    LB_UPDATE64_(NC, false, false);                    \
  }
  if (nc == 1) LB_UPDATE64(1)
  if (nc == 2) LB_UPDATE64(2)
  LB_UPDATE64(3)
#undef LB_UPDATE64_
#undef LB_UPDATE64
}

int update64_sample(int64_t n, const UpdateJob<double>& job, const double* U, int s, int q, double alpha, int* count,
                    cudaStream_t st) {
  const int samples = (int)std::min<int64_t>(n, 152 * 8);  // one row a warp
  LB_CUDA(cudaMemsetAsync(count, 0, sizeof(int), st));
  update64_sample_kernel<<<(unsigned)((samples + 7) / 8), 256, (size_t)s * q * sizeof(double), st>>>(
      n, job, U, s, q, alpha, samples, count);
  LB_LAUNCH_CHECK();
  return samples;
}

}  // namespace lobpcg
