// FP64 Gram matrices C = A^T B (V^T AV, Y^T W, W^T W) on the 5th-generation tensor cores: the
// columns are cut into FP16 digits (slices.cuh) whose products the tensor core sums exactly.
//
// What bounds it.  The FP64 pipe of this part does 2 FMA per clock and SM: a 63 x 63 Gram of 10^6
// rows takes it 7.2 ms, 50 times the time its bytes take.  34 digit products of the same Gram are
// 0.28 TFLOP of FP16, which the tensor cores do in 0.15 ms, so what is left to pay is the cutting
// into digits (about 30 integer instructions per element) and reading the blocks.
//
// Accuracy.  Each column has its own exponent in every block of 256 rows (kGroupRows): its
// entries are held to 2^-56 of the column's largest magnitude there, digit sums are exact, and each
// block's sum is rounded to FP64 once and added in FP64.
//
// Two kernels.  exp_kernel reads the blocks once and writes the exponents.  gram64_kernel is one
// persistent CTA per SM with the roles of the FP32 Gram (umma.cu): a producer thread (1-D TMA bulk
// copies of KC rows of every row-major block into a raw ring), eight splitter warps in two groups
// (raw FP64 -> digit tiles, K-major core matrices), one MMA thread, eight epilogue warps.
//   * The tile buffer holds A's digits as eight slices of 64 columns (the eighth zero), so slices i
//     and i + 1 (i even) are one M = 128 operand, and B's seven slices of NB columns back to back,
//     so consecutive slices are one operand of N = NB, 2 NB, ... columns.  The MMA of A pair i and
//     B slices j, j + 1, .. writes TMEM columns NB (i + j), ..: TMEM lanes 0..63 of region t sum the
//     products with i + j = t (i even) and lanes 64..127 those with i + j = t + 1 (i odd).
//   * At most four digit products per row meet in one accumulator: 4 * 256 * 2^14 = 2^24, exact.
//   * After 256 rows the epilogue joins the eight regions of every element into one FP64 number
//     with integer operations and adds it to its running sum (one FP64 add).
// A flag set by exp_kernel (a column's block with an infinity, a NaN or an exponent outside
// 2^+-400) makes gram64_kernel return at once; the caller's general kernel, launched behind it on
// the same flag, then forms the partials.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "slices.cuh"
#include "umma.cuh"

namespace lobpcg {
namespace {

using namespace umma;
using namespace slices;

constexpr int kGroupRows = 256;               // rows that share a column's exponent
constexpr int kKC = 32;                       // rows per chunk
constexpr int kChunks = kGroupRows / kKC;     // chunks per group
constexpr int kTS = 2;                        // tile buffers
constexpr int kMaxRS = 6;                     // raw ring stages, chosen at launch
constexpr int kMaxU = 6;
constexpr int kCB = 64;                       // columns of A and B per launch
constexpr int kEpi0 = 2, kEpiWarps = 8;
constexpr int kSplit0 = kEpi0 + kEpiWarps, kSplitWarps = 8, kSplitGroups = 2;
constexpr int kThreads = 32 * (kSplit0 + kSplitWarps);
constexpr uint32_t kLBO = 128, kSBO = kKC / 8 * 128;  // bytes between core matrices along K and M / N
constexpr uint32_t kSliceA = kCB / 8 * kSBO;          // bytes of one A slice
constexpr long long kWaitCycles = 1ll << 31;
constexpr size_t kSmemBudget = 220 * 1024;

__device__ int g_gram64_err = 0;

__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int code) {
  const long long t0 = clock64();
  for (uint32_t i = 0;; ++i) {
    if (mbar_try(bar, parity)) return true;
    if ((i & 15u) == 15u) {
      if (*abort_flag) return false;
      if (clock64() - t0 > kWaitCycles) break;
    }
  }
  *abort_flag = 1;
  atomicExch(&g_gram64_err, code);
  return false;
}

// exps[g * stride + j]: biased exponent of column j (A's columns, then B's) over the rows of group
// g, one CTA per group.  A thread keeps one 16-byte pair of columns and strides over the rows with
// eight loads in flight.
__global__ void __launch_bounds__(256) exp_kernel(int64_t n, Cols<double> A, Cols<double> B, int ld, int same,
                                                  int* __restrict__ exps, int stride, int* __restrict__ flag) {
  __shared__ uint32_t key[2 * kMaxS];
  const int64_t r0 = (int64_t)blockIdx.x * kGroupRows;
  const int rows = (int)min((int64_t)kGroupRows, n - r0);
  const int pa = A.width(), total = pa + (same ? 0 : B.width());
  for (int j = threadIdx.x; j < 2 * kMaxS; j += blockDim.x) key[j] = 0u;
  __syncthreads();
  int base = 0;
  for (int o = 0; o < (same ? 1 : 2); ++o) {
    const Cols<double>& c = o == 0 ? A : B;
    for (int s = 0; s < c.nseg; ++s) {
      const int w = c.w[s], vec = (w + 1) / 2, groups = blockDim.x / vec;
      const int grp = threadIdx.x / vec, v = threadIdx.x - grp * vec;
      if (grp < groups) {
        const double2* p = reinterpret_cast<const double2*>(c.p[s] + r0 * ld) + v;
        const int64_t step = ld / 2;
        uint32_t k0 = 0u, k1 = 0u;
        int r = grp;
        for (; r + 7 * groups < rows; r += 8 * groups) {
          double2 x[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) x[u] = __ldg(p + (r + u * groups) * step);
#pragma unroll
          for (int u = 0; u < 8; ++u) k0 = max(k0, exp_key(x[u].x)), k1 = max(k1, exp_key(x[u].y));
        }
        for (; r < rows; r += groups) {
          const double2 x = __ldg(p + r * step);
          k0 = max(k0, exp_key(x.x)), k1 = max(k1, exp_key(x.y));
        }
        atomicMax(&key[base + 2 * v], k0);
        if (2 * v + 1 < w) atomicMax(&key[base + 2 * v + 1], k1);
      }
      base += w;
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < total; j += blockDim.x) {
    const int e = group_exp(key[j]);
    if (e < 0) *flag = 1;
    exps[(int64_t)blockIdx.x * stride + j] = e;
  }
}

// Columns [a0, a0 + pa) of A and [b0, b0 + pb) of B; NB: B columns per slice (>= pb).
template <int NB>
__global__ void __launch_bounds__(kThreads, 1)
    gram64_kernel(int64_t n, Cols<double> A, Cols<double> B, int ld, int a0, int pa, int b0, int pb, int upper,
                  int same, int rs, const int* __restrict__ exps, int estride, int eb0,
                  const int* __restrict__ flag, double* __restrict__ part, int64_t groups_per_cta) {
  constexpr int kAS = NB <= 32 ? 2 : 1;  // accumulators (of kDiags * NB TMEM columns)
  constexpr int kAcc = kDiags * NB;
  constexpr uint32_t kSliceB = NB / 8 * kSBO;
  constexpr int kEW = NB / 2;  // columns per epilogue warp (two warps per lane quadrant)
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ uint64_t raw_full[kMaxRS], raw_empty[kMaxRS], tile_full[kTS], tile_empty[kTS];
  __shared__ uint64_t acc_full[2], acc_empty[2];
  __shared__ const double* useg[kMaxU];
  __shared__ int ucopy[kMaxU];
  __shared__ int colofs[2][kCB];
  __shared__ int nu_s;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;

  if (*flag) return;  // written by an earlier kernel: the same for every thread
  const int ta = A.width(), tb = B.width();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int seg = kKC * ld;
  if (tid == 0) {
    int nu = 0;
    for (int o = 0; o < (same ? 1 : 2); ++o) {
      const Cols<double>& c = o == 0 ? A : B;
      const int lo = o == 0 ? a0 : b0, hi = lo + (o == 0 ? pa : pb);
      int base = 0;
      for (int g = 0; g < c.nseg; base += c.w[g], ++g) {
        if (base >= hi || base + c.w[g] <= lo) continue;  // no column of this launch
        int u = 0;
        while (u < nu && useg[u] != c.p[g]) ++u;
        if (u == nu) useg[nu] = c.p[g], ucopy[nu] = 0, ++nu;
        ucopy[u] = max(ucopy[u], (c.w[g] + 1) / 2 * 2);
      }
    }
    nu_s = nu;
    abort_flag = 0;
    for (int s = 0; s < kMaxRS; ++s) mbar_init(&raw_full[s], 1), mbar_init(&raw_empty[s], kSplitWarps / kSplitGroups);
    for (int s = 0; s < kTS; ++s) mbar_init(&tile_full[s], kSplitWarps / kSplitGroups), mbar_init(&tile_empty[s], 1);
    for (int s = 0; s < 2; ++s) mbar_init(&acc_full[s], 1), mbar_init(&acc_empty[s], kEpiWarps);
    fence_barrier_init();
  }
  __syncthreads();
  const int nu = nu_s;
  for (int i = tid; i < 2 * kCB; i += blockDim.x) {
    const int o = i / kCB, m = i % kCB;
    const Cols<double>& c = o == 0 ? A : B;
    int off = -1;
    if (m < (o == 0 ? pa : pb) && !(o == 1 && same)) {
      const int col = m + (o == 0 ? a0 : b0);
      int base = 0, g = 0;
      while (col >= base + c.w[g]) base += c.w[g], ++g;
      int u = 0;
      while (useg[u] != c.p[g]) ++u;
      off = u * seg + (col - base);
    }
    colofs[o][m] = off;
  }
  const size_t raw_bytes = ((size_t)rs * nu * seg * 8 + 127) / 128 * 128;
  double* raw = reinterpret_cast<double*>(smem);  // [rs][nu][kKC][ld]
  unsigned char* tiles = smem + raw_bytes;
  const uint32_t oB = same ? 0u : 8u * kSliceA;
  const uint32_t tbuf = 8u * kSliceA + (same ? 0u : (uint32_t)kSlices * kSliceB);
  for (uint32_t e = tid; e < kTS * tbuf / 16; e += blockDim.x) reinterpret_cast<uint4*>(tiles)[e] = make_uint4(0, 0, 0, 0);
  __syncwarp();
  if (warp == 1) tmem_alloc(&tmem_slot, kAS * kAcc);
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  const int64_t g_begin = (int64_t)blockIdx.x * groups_per_cta;
  const int64_t r_begin = g_begin * kGroupRows;
  const int64_t r_end = min(n, r_begin + groups_per_cta * kGroupRows);
  const int nchunks = r_end > r_begin ? (int)((r_end - r_begin + kKC - 1) / kKC) : 0;
  const int ngroups = (nchunks + kChunks - 1) / kChunks;
  int issued = 0, committed = 0;  // producer thread; MMA thread (groups)
  if (warp == 0) {
    if (lane == 0) {
      int st = 0;
      uint32_t ph = 0;
      for (int c = 0; c < nchunks; ++c) {
        if (c >= rs && !wait_bar(&raw_empty[st], ph ^ 1u, &abort_flag, 3)) break;
        const int64_t r0 = r_begin + (int64_t)c * kKC;
        const int rows = (int)min((int64_t)kKC, r_end - r0);
        uint32_t total = 0;  // the last row's copy stops at the used columns
        for (int u = 0; u < nu; ++u) total += (uint32_t)((rows - 1) * ld + ucopy[u]) * 8u;
        mbar_expect_tx(&raw_full[st], total);
        for (int u = 0; u < nu; ++u)
          bulk_g2s(raw + ((size_t)st * nu + u) * seg, useg[u] + r0 * ld, (uint32_t)((rows - 1) * ld + ucopy[u]) * 8u,
                   &raw_full[st]);
        issued = c + 1;
        if (++st == rs) st = 0, ph ^= 1u;
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint64_t dA = desc_kmajor(smem_addr(tiles), kLBO, kSBO);
      const uint64_t dB = desc_kmajor(smem_addr(tiles) + oB, kLBO, kSBO);
      int buf = 0, r = 0;
      uint32_t tph = 0, aph = 0;
      for (int c = 0; c < nchunks; ++c) {
        const int in_group = c % kChunks;
        if (!wait_bar(&tile_full[buf], tph, &abort_flag, 3)) break;
        if (in_group == 0 && c / kChunks >= kAS && !wait_bar(&acc_empty[r], aph ^ 1u, &abort_flag, 3)) break;
        tc_fence_after();
        const uint64_t bo = (uint64_t)((uint32_t)buf * tbuf >> 4);
        const uint32_t d = tmem + (uint32_t)(r * kAcc);
        // A pair i against B slices [j, j + cnt), into regions i + j ..
        auto mma = [&](int kk, int i, int j, int cnt, uint32_t acc) {
          const uint64_t ko = bo + (uint64_t)(kk * 16);  // two core matrices (256 bytes) per 16 rows
          mma_f16(d + (uint32_t)(NB * (i + j)), dA + ko + (uint64_t)(i * (kSliceA >> 4)),
                  dB + ko + (uint64_t)(j * (kSliceB >> 4)), idesc_f16(128, (uint32_t)(NB * cnt)), acc);
        };
        constexpr int W = 256 / NB;  // slices per MMA
#pragma unroll
        for (int kk = 0; kk < kKC / 16; ++kk) {
          const uint32_t acc = in_group > 0 || kk > 0 ? 1u : 0u;
          // regions 0..6
#pragma unroll
          for (int j = 0; j < kSlices; j += W) mma(kk, 0, j, min(W, kSlices - j), acc);
          // regions 2..6, then 7, whose first product overwrites what an earlier group left
#pragma unroll
          for (int j = 0; j < 5; j += W) mma(kk, 2, j, min(W, 5 - j), 1u);
          mma(kk, 2, 5, 1, acc);
          mma(kk, 4, 0, 4, 1u);
          mma(kk, 6, 0, 2, 1u);
        }
        mma_commit(&tile_empty[buf]);
        if (in_group == kChunks - 1 || c == nchunks - 1) {
          mma_commit(&acc_full[r]);
          committed = c / kChunks + 1;
          if (++r == kAS) r = 0, aph ^= 1u;
        }
        if (++buf == kTS) buf = 0, tph ^= 1u;
      }
    }
  } else if (warp < kSplit0) {
    // epilogue: warp w reads TMEM lanes 32 (w mod 4) .. + 31, columns [kEW half, + kEW) of each region
    const int quad = warp & 3, half = (warp - kEpi0) >> 2;
    const int row = (32 * quad + lane) & 63;  // column of A
    const bool odd = quad >= 2;               // regions hold i + j = t + 1
    double acc[kEW];
#pragma unroll
    for (int j = 0; j < kEW; ++j) acc[j] = 0.0;
    int r = 0, g = 0;
    uint32_t aph = 0;
    for (; g < ngroups; ++g) {
      const int* ge = exps + (g_begin + g) * estride;
      const int ea = row < pa ? __ldg(ge + a0 + row) : kExpOne;
      if (!__all_sync(0xffffffffu, wait_bar(&acc_full[r], aph, &abort_flag, 2))) break;
      tc_fence_after();
      const uint32_t t0 = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(r * kAcc + kEW * half);
      // element: (sum_t v_t 256^(7-t)) 2^(40 - 110) 2^(ea - 1022) 2^(eb - 1022), / 256 in lanes 64..127
      const int sa = ea - 1022 - 70 - (odd ? 8 : 0);
#pragma unroll
      for (int j0 = 0; j0 < kEW; j0 += 4) {
        if (kEW * half + j0 < pb) {  // warp-uniform
          float v[kDiags][4];
#pragma unroll
          for (int t = 0; t < kDiags; ++t) tmem_ld4(t0 + (uint32_t)(NB * t + j0), v[t]);
          tmem_wait_ld(v);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int j = kEW * half + j0 + i;
            const int eb = j < pb ? __ldg(ge + eb0 + b0 + j) : kExpOne;
            float w[kDiags];
#pragma unroll
            for (int t = 0; t < kDiags; ++t) w[t] = v[t][i];
            acc[j0 + i] += join(w, sa + eb - 1022);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[r]);
      if (++r == kAS) r = 0, aph ^= 1u;
    }
    // every group's MMAs done means every copy and tile is done with: lanes 64..127 hand their
    // sums to lanes 0..63 through the raw ring's memory
    const bool done = g == ngroups;
    double* red = reinterpret_cast<double*>(smem);
    if (odd && done)
#pragma unroll
      for (int j = 0; j < kEW; ++j) red[(kEW * half + j) * 64 + row] = acc[j];
    asm volatile("bar.sync 3, 256;\n" ::: "memory");  // the eight epilogue warps
    if (!odd && row < pa) {
      const bool ok = done && !abort_flag;
      double* out = part + (int64_t)blockIdx.x * ta * tb;
#pragma unroll
      for (int j = 0; j < kEW; ++j) {
        const int col = kEW * half + j;
        if (col < pb && (!upper || a0 + row <= b0 + col))
          out[(a0 + row) + (int64_t)(b0 + col) * ta] = ok ? acc[j] + red[col * 64 + row] : 0.0;
      }
    }
  } else {
    // splitters: two groups of four warps take the chunks in turn; the units (32 columns x 8 rows
    // of one operand) of a warp are the same in every chunk
    constexpr int wpg = kSplitWarps / kSplitGroups, K8 = kKC / 8, kMaxUW = 4 * K8 / wpg;
    const int sw = warp - kSplit0, g = sw / wpg, sg = sw % wpg;
    const int gA = (pa + 31) / 32, gB = same ? 0 : (pb + 31) / 32;
    const int units = (gA + gB) * K8;
    int src[kMaxUW], ecol[kMaxUW], exp_[kMaxUW];
    uint32_t dst[kMaxUW], step[kMaxUW], k0[kMaxUW];
#pragma unroll
    for (int j = 0; j < kMaxUW; ++j) {
      const int u = sg + j * wpg;
      src[j] = -1, dst[j] = 0, step[j] = 0, ecol[j] = 0, exp_[j] = kExpOne, k0[j] = 0;
      if (u < units) {
        const bool isA = u < gA * K8;
        const int v = isA ? u : u - gA * K8;
        const int k8 = v % K8, m = v / K8 * 32 + lane;
        const int off = colofs[isA ? 0 : 1][m];
        if (off >= 0) {
          src[j] = off + 8 * k8 * ld;
          k0[j] = 8 * k8;
          ecol[j] = isA ? a0 + m : eb0 + b0 + m;
          dst[j] = (isA ? 0u : oB) + (uint32_t)(m >> 3) * kSBO + (uint32_t)k8 * kLBO + 16u * (m & 7);
          step[j] = isA ? kSliceA : kSliceB;
        }
      }
    }
    int st = g % rs, buf = g % kTS, cur = -1;
    uint32_t ph = 0, tph = 0;
    for (int c = g; c < nchunks; c += kSplitGroups) {
      if (c / kChunks != cur) {
        cur = c / kChunks;
#pragma unroll
        for (int j = 0; j < kMaxUW; ++j)
          if (src[j] >= 0) exp_[j] = __ldg(exps + (g_begin + cur) * estride + ecol[j]);
      }
      if (!__all_sync(0xffffffffu, wait_bar(&raw_full[st], ph, &abort_flag, 1))) break;
      if (c >= kTS && !__all_sync(0xffffffffu, wait_bar(&tile_empty[buf], tph ^ 1u, &abort_flag, 2))) break;
      const int rows = (int)min((int64_t)kKC, r_end - (r_begin + (int64_t)c * kKC));
      const double* rsb = raw + (size_t)st * nu * seg;
      unsigned char* tb_ = tiles + (uint32_t)buf * tbuf;
#pragma unroll
      for (int j = 0; j < kMaxUW; ++j) {
        if (src[j] < 0) continue;
        double x[8];
        if (rows == kKC) {
#pragma unroll
          for (int i = 0; i < 8; ++i) x[i] = rsb[src[j] + i * ld];
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) x[i] = (int)k0[j] + i < rows ? rsb[src[j] + i * ld] : 0.0;
        }
        uint64_t w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = digits(x[i], exp_[j]);
        unsigned char* o = tb_ + dst[j];
        auto put = [&](auto k) {
          constexpr int K = decltype(k)::value;
          *reinterpret_cast<uint4*>(o + K * step[j]) =
              make_uint4(digit_pair<K>(w[0], w[1]), digit_pair<K>(w[2], w[3]), digit_pair<K>(w[4], w[5]),
                         digit_pair<K>(w[6], w[7]));
        };
        put(std::integral_constant<int, 0>{});
        put(std::integral_constant<int, 1>{});
        put(std::integral_constant<int, 2>{});
        put(std::integral_constant<int, 3>{});
        put(std::integral_constant<int, 4>{});
        put(std::integral_constant<int, 5>{});
        put(std::integral_constant<int, 6>{});
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&raw_empty[st]);
        mbar_arrive(&tile_full[buf]);
      }
      if ((st += kSplitGroups) >= rs) st -= rs, ph ^= 1u;
      if ((buf += kSplitGroups) >= kTS) buf -= kTS, tph ^= 1u;
    }
  }
  __syncthreads();
  if (abort_flag) {
    // bounded waits for the copies and MMAs in flight before the memory they use goes
    if (warp == 0 && lane == 0)
      for (int c = max(0, issued - rs); c < issued; ++c) mbar_wait(&raw_full[c % rs], (uint32_t)(c / rs) & 1u, kWaitCycles);
    if (warp == 1 && lane == 0 && committed > 0)
      mbar_wait(&acc_full[(committed - 1) % kAS], (uint32_t)((committed - 1) / kAS) & 1u, kWaitCycles);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, kAS * kAcc);
  }
}

__global__ void gram64_err_reset_kernel() { g_gram64_err = 0; }

bool same_cols(const Cols<double>& a, const Cols<double>& b) {
  bool same = a.nseg == b.nseg;
  for (int g = 0; same && g < a.nseg; ++g) same = a.p[g] == b.p[g] && a.w[g] == b.w[g];
  return same;
}

int count_blocks(const Cols<double>& a, const Cols<double>& b) {
  const double* u[kMaxU];
  int nu = 0;
  for (int o = 0; o < 2; ++o) {
    const Cols<double>& c = o == 0 ? a : b;
    for (int g = 0; g < c.nseg; ++g) {
      int i = 0;
      while (i < nu && u[i] != c.p[g]) ++i;
      if (i == nu) u[nu++] = c.p[g];
    }
  }
  return nu;
}

int sm_count() {
  int dev = 0, sms = 152;
  LB_CUDA(cudaGetDevice(&dev));
  LB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  return sms;
}

template <int NB>
void gram64_launch(int64_t n, const Cols<double>& a, const Cols<double>& b, int ld, int a0, int pa, int b0, int pb,
                   bool upper, bool same, int rs, size_t smem, const int* exps, int estride, int eb0,
                   const int* flag, double* part, int ctas, int64_t gpc, cudaStream_t st) {
  static const bool attr = [&] {
    LB_CUDA(cudaFuncSetAttribute(gram64_kernel<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget));
    return true;
  }();
  (void)attr;
  gram64_kernel<NB><<<(unsigned)ctas, kThreads, smem, st>>>(n, a, b, ld, a0, pa, b0, pb, upper ? 1 : 0, same ? 1 : 0,
                                                           rs, exps, estride, eb0, flag, part, gpc);
  LB_LAUNCH_CHECK();
}

}  // namespace

size_t gram64_scratch_ints(int64_t n) { return (size_t)ceil_div(n, kGroupRows) * 2 * kMaxS + 4; }

// Gram partials through digit products; returns 0 without launching where the operands do not share
// one 16-byte aligned row stride or need more shared memory than a CTA has.  scratch:
// gram64_scratch_ints(n) ints; its first word is the flag: when the launched kernels leave it at 1
// the partials are not written, and the caller's general kernel (launched on the same flag) forms
// them over the same number of CTAs.
int gram_partials_digits(int64_t n, const Cols<double>& a, const Cols<double>& b, bool upper, double* part,
                         int max_ctas, int* scratch, cudaStream_t st) {
  if (a.nseg == 0 || b.nseg == 0 || n <= 0) return 0;
  const int ld = a.ld[0];
  if (ld & 1) return 0;
  for (int o = 0; o < 2; ++o) {
    const Cols<double>& c = o == 0 ? a : b;
    for (int g = 0; g < c.nseg; ++g)
      if (c.ld[g] != ld || c.w[g] > ld || c.w[g] < 1 || (reinterpret_cast<uintptr_t>(c.p[g]) & 15)) return 0;
  }
  const int pa = a.width(), pb = b.width();
  if (pa > kMaxS || pb > kMaxS) return 0;
  const bool same = same_cols(a, b);
  const int na = (pa + kCB - 1) / kCB, nb = (pb + kCB - 1) / kCB;  // column blocks, of equal widths
  const int wa = (pa + na - 1) / na, wb = (pb + nb - 1) / nb;
  const int nbw = wb <= 32 ? 32 : 64;
  const size_t stage = (size_t)kKC * count_blocks(a, b) * ld * 8;
  const size_t tiles = (size_t)kTS * (8 * kSliceA + kSlices * (size_t)(nbw / 8) * kSBO);
  if (tiles + 2 * stage + 128 > kSmemBudget) return 0;
  const int rs = (int)std::min<size_t>(kMaxRS, (kSmemBudget - tiles - 128) / stage);
  // the raw ring also holds the epilogue's exchange
  const size_t smem = std::max((rs * stage + 127) / 128 * 128, (size_t)64 * nbw * 8) + tiles;
  if (smem > kSmemBudget) return 0;
  const int64_t ngroups = ceil_div(n, kGroupRows);
  int64_t ctas = std::min<int64_t>(std::min<int64_t>(max_ctas, sm_count()), ngroups);
  const int64_t gpc = ceil_div(ngroups, ctas);
  ctas = ceil_div(ngroups, gpc);
  int* flag = scratch;
  int* exps = scratch + 4;
  const int estride = pa + (same ? 0 : pb), eb0 = same ? 0 : pa;
  LB_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), st));
  exp_kernel<<<(unsigned)ngroups, 256, 0, st>>>(n, a, b, ld, same ? 1 : 0, exps, estride, flag);
  LB_LAUNCH_CHECK();
  for (int ia = 0; ia < na; ++ia)
    for (int ib = 0; ib < nb; ++ib) {
      const int a0 = ia * wa, b0 = ib * wb;
      const int ca = std::min(wa, pa - a0), cb = std::min(wb, pb - b0);
      if (upper && a0 > b0 + cb - 1) continue;
      // B can read A's tiles where its slices have A's width
      const bool diag = same && ia == ib && nbw == kCB;
      if (nbw == 32)
        gram64_launch<32>(n, a, b, ld, a0, ca, b0, cb, upper, diag, rs, smem, exps, estride, eb0, flag, part,
                          (int)ctas, gpc, st);
      else
        gram64_launch<64>(n, a, b, ld, a0, ca, b0, cb, upper, diag, rs, smem, exps, estride, eb0, flag, part,
                          (int)ctas, gpc, st);
    }
  return (int)ctas;
}

// Reads and clears the give-up flag (synchronises the stream); throws when a CTA gave up waiting.
void gram64_check(cudaStream_t st) {
  int err = 0;
  LB_CUDA(cudaMemcpyFromSymbolAsync(&err, g_gram64_err, sizeof(int), 0, cudaMemcpyDeviceToHost, st));
  LB_CUDA(cudaStreamSynchronize(st));
  if (err) {
    gram64_err_reset_kernel<<<1, 1, 0, st>>>();
    LB_LAUNCH_CHECK();
    LB_CUDA(cudaStreamSynchronize(st));
    throw CudaError("tensor-core FP64 Gram: a pipeline stage did not complete in time");
  }
}

}  // namespace lobpcg
