// FP64 Gram matrices C = A^T B (V^T AV, Y^T W, W^T W) on the 5th-generation tensor cores: the
// columns are cut into FP16 digits (slices.cuh) whose products the tensor core sums exactly.
//
// What bounds it.  The FP64 pipe of this part does 2 FMA per clock and SM: a 63 x 63 Gram of 10^6
// rows takes it 7.2 ms, 50 times the time its bytes take.  34 digit products of the same Gram are
// 0.28 TFLOP of FP16, which the tensor cores do in 0.15 ms, so what is left to pay is the cutting
// into digits (about 25 integer instructions per element, at half the rate of FMAs), the joining of the
// sums, and reading the blocks.  A call of that Gram went from 7,230 to 660 us (exponents 165, products
// 450) and takes 750 with the test of spread below; its bytes take 150.  Counters at 200,000 rows: integer
// pipe 47%, tensor pipe 27%, DRAM 24%.  Clocks of the roles at 63 columns: the MMA thread issues about 40%
// of the time and waits for tiles 35%, for the joins 25%; at 21 columns it issues 85%.
//
// Accuracy.  Each column has its own exponent in every block of 256 rows (kGroupRows): its
// entries are held to 2^-56 of the column's largest magnitude there, digit sums are exact, and each
// block's sum is rounded to FP64 once and added in FP64.  So an entry of the product is off by at most
// 256 mx my 2^-53 per block, a bound against the columns' norms.  It is not one against the entry's own
// sum |x||y|, as an FMA chain has, where columns are large at different rows; callers that ask for that
// one have such columns found (kSpread) and formed by the older kernels.
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
//     A of at most 32 columns has slices of 32 (CA), four to an operand: five products of 608 TMEM columns
//     a K step become three of 352, and A and B of one block share their tiles.
//   * At most four digit products per row meet in one accumulator: 4 * 256 * 2^14 = 2^24, exact.
//   * After 256 rows the epilogue joins the eight regions of every element into one FP64 number
//     with integer operations and adds it to its running sum (one FP64 add).
// The dense symmetric product Y = A X (PANEL) is the same contraction with A's columns in memory order:
// a CTA owns 64 columns of A and a range of its rows and writes its 64 x p sums; ranges of rows split a
// matrix of few panels over the SMs.  The producer warp copies 32 rows of each column with cp.async, half a
// warp per column (256 bytes, at a 272-byte stride in shared memory, which keeps the splitters' reads of 8
// columns in different banks), as far ahead as the raw ring holds.  256-byte bulk copies took 70 clocks
// each, 4.5k per chunk (1078 us a product of n = 8192), loads by the splitters a chunk ahead left 16 KB in
// flight (899 us).  A row-major A (row_a) is copied by rows of 64 columns; it needs no transposed copy.
//
// A flag raised by exp_kernel (a column's block with an infinity, a NaN or an exponent outside 2^+-400,
// or columns too far apart) makes gram64_kernel return at once; the caller's general kernel, launched
// behind it on the same flag, then forms the partials.
#include <algorithm>
#include <climits>

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
constexpr size_t kSmemBudget = 220 * 1024;

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
// Arrive on the barrier when this thread's cp.async copies so far have landed.
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(smem_addr(bar)) : "memory");
}

// Two columns are close enough in a group where at least kSpreadRows of its rows hold entries of both
// within kSpreadBits binades of the column's largest there.  With 2^a <= mx < 2^(a+1) and my likewise,
// those rows alone give sum |x||y| >= 32 2^-6 2^(a+b), and the digits' error is at most
// 256 mx my 2^-53 <= 2^11 2^-53 of that sum: below the bound of a chain of FMAs over 2^11 rows, and in
// the mean below their error.  Gaussian columns share 97 rows or more of 256 in the mean.
constexpr int kSpreadBits = 3, kSpreadRows = 32;
constexpr int kMaskWords = kGroupRows / 32;
constexpr int kOutOfRange = 1, kSpread = 2;  // bits of the flag

// exps[g * stride + j]: biased exponent of column j (A's columns, then B's) over the rows of group
// g, one CTA per group.  A thread keeps one 16-byte pair of columns and strides over the rows with
// eight loads in flight.
// CHECK (one segment an operand): also raises kSpread where two columns are too far apart.  The
// exponents of the group stay in shared memory (two bytes an entry), each column becomes 256 bits, and a
// pair of columns is the population count of two of those.  The rows of a last, incomplete group are
// judged with those before them, by a CTA of its own over the last 256.
template <bool CHECK>
__global__ void __launch_bounds__(256) exp_kernel(int64_t n, Cols<double> A, Cols<double> B, int ld, int same,
                                                  int* __restrict__ exps, int stride, int* __restrict__ flag) {
  extern __shared__ uint32_t ex2[];  // CHECK: [kGroupRows][pairs] exponents of two columns
  __shared__ uint32_t key[2 * kMaxS];
  const bool window = CHECK && (int64_t)blockIdx.x * kGroupRows >= n;
  const int64_t r0 = window ? n - kGroupRows : (int64_t)blockIdx.x * kGroupRows;
  const int rows = (int)min((int64_t)kGroupRows, n - r0);
  const int pa = A.width(), total = pa + (same ? 0 : B.width());
  const int va = (pa + 1) / 2, pairs = va + (same ? 0 : (B.width() + 1) / 2);
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
        auto take = [&](const double2& x, int r) {
          k0 = max(k0, exp_key(x.x)), k1 = max(k1, exp_key(x.y));
          if (CHECK)
            ex2[r * pairs + (o ? va : 0) + v] = (((uint32_t)__double2hiint(x.x) >> 20) & 0x7ffu) |
                                                ((((uint32_t)__double2hiint(x.y) >> 20) & 0x7ffu) << 16);
        };
        int r = grp;
        for (; r + 7 * groups < rows; r += 8 * groups) {
          double2 x[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) x[u] = __ldg(p + (r + u * groups) * step);
#pragma unroll
          for (int u = 0; u < 8; ++u) take(x[u], r + u * groups);
        }
        for (; r < rows; r += groups) take(__ldg(p + r * step), r);
        atomicMax(&key[base + 2 * v], k0);
        if (2 * v + 1 < w) atomicMax(&key[base + 2 * v + 1], k1);
      }
      base += w;
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < total; j += blockDim.x) {
    const int e = group_exp(key[j]);
    if (e < 0) atomicOr(flag, kOutOfRange);
    if (!window) exps[(int64_t)blockIdx.x * stride + j] = e;
  }
  if constexpr (CHECK) {
    if (rows < kGroupRows) return;
    __shared__ __align__(16) uint32_t mask[2 * kMaxS][kMaskWords];
    for (int u = threadIdx.x; u < pairs * kMaskWords; u += blockDim.x) {
      const int v = u % pairs, k = u / pairs;
      const bool ofB = v >= va;
      const int c = ofB ? pa + 2 * (v - va) : 2 * v, end = ofB ? total : pa;  // the pair's columns c, c + 1
      const uint32_t t0 = (key[c] >> 20) - min(key[c] >> 20, (uint32_t)kSpreadBits);
      const uint32_t k1 = c + 1 < end ? key[c + 1] >> 20 : 0u;
      const uint32_t t1 = k1 - min(k1, (uint32_t)kSpreadBits);
      uint32_t m0 = 0u, m1 = 0u;
#pragma unroll 8
      for (int r = 0; r < 32; ++r) {
        const uint32_t e = ex2[(32 * k + r) * pairs + v];
        m0 |= ((e & 0xffffu) >= t0 ? 1u : 0u) << r;
        m1 |= ((e >> 16) >= t1 ? 1u : 0u) << r;
      }
      mask[c][k] = m0;
      if (c + 1 < end) mask[c + 1][k] = m1;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, pb = same ? pa : B.width(), b0 = same ? 0 : pa;
    bool apart = false;
    for (int i = lane; i < pa; i += 32) {
      uint32_t m[kMaskWords];
#pragma unroll
      for (int k = 0; k < kMaskWords; ++k) m[k] = mask[i][k];
      for (int j = threadIdx.x >> 5; j < pb; j += blockDim.x / 32) {
        int shared_rows = 0;
#pragma unroll
        for (int k = 0; k < kMaskWords; ++k) shared_rows += __popc(m[k] & mask[b0 + j][k]);
        apart |= shared_rows < kSpreadRows && key[i] != 0u && key[b0 + j] != 0u;
      }
    }
    if (apart) atomicOr(flag, kSpread);
  }
}

// The dense product asks the same of every column of A and of X, the diagonal of A left out: it has its
// own place in the sums, for one large entry per column would take the others' digits.
// Bit l of word 2 u + h of a mask is row 64 u + 2 l + h of the group, the order in which a warp reads a
// column of A by 16-byte pairs.  xmask: per group 32 columns of X, kMaskWords each, then a word of the
// columns that are not zero; the last group's are those of the last 256 rows where it is incomplete.
constexpr int kXMask = 32 * kMaskWords + 1;
__device__ __forceinline__ uint32_t near_limit(uint32_t key) {  // smallest exponent that counts as near
  return (key >> 20) - min(key >> 20, (uint32_t)kSpreadBits);
}
__device__ __forceinline__ uint32_t exp_of(double x) { return ((uint32_t)__double2hiint(x) >> 20) & 0x7ffu; }
// Whether a column with mask m and any of the p <= 32 of X in the group share too few rows (j, j + step, ..).
__device__ __forceinline__ bool far_from_x(const uint32_t (&m)[kMaskWords], const uint32_t* __restrict__ xm, int p, int j,
                                           int step) {
  const uint32_t nonzero = __ldg(xm + 32 * kMaskWords);
  bool apart = false;
  for (; j < p; j += step) {
    int both = 0;
#pragma unroll
    for (int k = 0; k < kMaskWords; ++k) both += __popc(m[k] & __ldg(xm + j * kMaskWords + k));
    apart |= both < kSpreadRows && (nonzero >> j & 1u) != 0u;
  }
  return apart;
}
// First row of block y of the groups, one more than there are for the last 256 rows.
__device__ __forceinline__ int64_t group_row(int64_t n, bool& window) {
  window = (int64_t)blockIdx.y * kGroupRows >= n;
  return window ? n - kGroupRows : (int64_t)blockIdx.y * kGroupRows;
}

// Exponents of a dense column-major A (n x n, lda): one warp per column and group of kGroupRows rows.
template <bool CHECK>
__global__ void __launch_bounds__(256) exp_dense_kernel(int64_t n, const double* __restrict__ A, int64_t lda,
                                                        int* __restrict__ exps, int64_t stride, int p,
                                                        const uint32_t* __restrict__ xmask, int* __restrict__ flag) {
  const int64_t col = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (col >= n) return;
  bool window;
  const int64_t r0 = group_row(n, window);
  const int rows = (int)min((int64_t)kGroupRows, n - r0);
  const double2* a = reinterpret_cast<const double2*>(A + col * lda + r0);
  double2 x[kGroupRows / 64];
#pragma unroll
  for (int u = 0; u < kGroupRows / 64; ++u)
    x[u] = 2 * (lane + 32 * u) < rows ? __ldg(a + lane + 32 * u) : make_double2(0.0, 0.0);  // rows is even
  uint32_t k = 0u;
#pragma unroll
  for (int u = 0; u < kGroupRows / 64; ++u) {
    const int64_t r = r0 + 2 * (lane + 32 * u);
    if (r == col) x[u].x = 0.0;
    if (r + 1 == col) x[u].y = 0.0;
    k = max(k, max(exp_key(x[u].x), exp_key(x[u].y)));
  }
  k = __reduce_max_sync(0xffffffffu, k);
  if constexpr (CHECK) {
    if (rows == kGroupRows && k != 0u) {
      const uint32_t limit = near_limit(k);
      uint32_t m[kMaskWords];
#pragma unroll
      for (int u = 0; u < kGroupRows / 64; ++u) {
        m[2 * u] = __ballot_sync(0xffffffffu, exp_of(x[u].x) >= limit);
        m[2 * u + 1] = __ballot_sync(0xffffffffu, exp_of(x[u].y) >= limit);
      }
      const uint32_t* xm = xmask + (int64_t)blockIdx.y * kXMask;
      if (__any_sync(0xffffffffu, far_from_x(m, xm, p, lane, 32)) && lane == 0) atomicOr(flag, kSpread);
    }
  }
  if (lane) return;
  const int e = group_exp(k);
  if (e < 0) atomicOr(flag, kOutOfRange);
  if (!window) exps[blockIdx.y * stride + col] = e;
}

// The same of a row-major A: one CTA per group and 64 columns, a lane per 16-byte pair of columns.
template <bool CHECK>
__global__ void __launch_bounds__(256) exp_dense_rows_kernel(int64_t n, const double* __restrict__ A, int64_t lda,
                                                             int* __restrict__ exps, int64_t stride, int p,
                                                             const uint32_t* __restrict__ xmask, int* __restrict__ flag) {
  __shared__ uint32_t key[64];
  __shared__ uint32_t ex2[CHECK ? kGroupRows : 1][32];  // exponents of a pair of columns
  if (threadIdx.x < 64) key[threadIdx.x] = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  bool window;
  const int64_t c = (int64_t)blockIdx.x * 64 + 2 * lane, r0 = group_row(n, window);
  const int rows = (int)min((int64_t)kGroupRows, n - r0);
  uint32_t k0 = 0u, k1 = 0u;
  if (c < n) {  // n is even
    const double* a = A + r0 * lda + c;
#pragma unroll 8
    for (int r = w; r < rows; r += 8) {
      double2 x = __ldg(reinterpret_cast<const double2*>(a + r * lda));
      if (r0 + r == c) x.x = 0.0;
      if (r0 + r == c + 1) x.y = 0.0;
      k0 = max(k0, exp_key(x.x)), k1 = max(k1, exp_key(x.y));
      if (CHECK) ex2[r][lane] = exp_of(x.x) | exp_of(x.y) << 16;
    }
  }
  atomicMax(&key[2 * lane], k0);
  atomicMax(&key[2 * lane + 1], k1);
  __syncthreads();
  const int64_t col = (int64_t)blockIdx.x * 64 + (threadIdx.x & 63);
  if constexpr (CHECK) {
    if (rows == kGroupRows) {
      __shared__ uint32_t mask[64][kMaskWords];
      const int cc = threadIdx.x & 63, q = threadIdx.x >> 6;
      const uint32_t limit = near_limit(key[cc]);
      for (int k = q; k < kMaskWords; k += 4) {
        uint32_t m = 0u;
#pragma unroll 8
        for (int l = 0; l < 32; ++l)
          m |= ((ex2[64 * (k >> 1) + 2 * l + (k & 1)][cc >> 1] >> (16 * (cc & 1)) & 0xffffu) >= limit ? 1u : 0u) << l;
        mask[cc][k] = m;
      }
      __syncthreads();
      if (col < n && key[cc] != 0u) {
        uint32_t m[kMaskWords];
#pragma unroll
        for (int k = 0; k < kMaskWords; ++k) m[k] = mask[cc][k];
        if (far_from_x(m, xmask + (int64_t)blockIdx.y * kXMask, p, q, 4)) atomicOr(flag, kSpread);
      }
    }
  }
  if (threadIdx.x < 64 && col < n) {
    const int e = group_exp(key[threadIdx.x]);
    if (e < 0) atomicOr(flag, kOutOfRange);
    if (!window) exps[blockIdx.y * stride + col] = e;
  }
}

// Exponents of a row-major block of p <= 32 columns (any row stride), one CTA per group; CHECK: and xmask.
template <bool CHECK>
__global__ void __launch_bounds__(256) exp_rows_kernel(int64_t n, int p, const double* __restrict__ X, int ldx,
                                                       int* __restrict__ exps, int64_t stride,
                                                       uint32_t* __restrict__ xmask, int* __restrict__ flag) {
  __shared__ uint32_t key[32];
  __shared__ uint16_t ex[CHECK ? kGroupRows : 1][32];
  if (threadIdx.x < 32) key[threadIdx.x] = 0u;
  __syncthreads();
  bool window;
  const int64_t r0 = group_row(n, window);
  const int rows = (int)min((int64_t)kGroupRows, n - r0), j = threadIdx.x & 31;
  uint32_t k = 0u;
  if (j < p)
    for (int r = threadIdx.x >> 5; r < rows; r += 8) {
      const double x = __ldg(X + (r0 + r) * ldx + j);
      k = max(k, exp_key(x));
      if (CHECK) ex[r][j] = (uint16_t)exp_of(x);
    }
  atomicMax(&key[j], k);
  __syncthreads();
  if constexpr (CHECK) {
    if (rows == kGroupRows) {
      uint32_t* xm = xmask + (int64_t)blockIdx.y * kXMask;
      const int w = threadIdx.x >> 5;
      const uint32_t limit = near_limit(key[j]);
      uint32_t m = 0u;
      if (j < p)
        for (int l = 0; l < 32; ++l) m |= (ex[64 * (w >> 1) + 2 * l + (w & 1)][j] >= limit ? 1u : 0u) << l;
      xm[j * kMaskWords + w] = m;
      const uint32_t nonzero = __ballot_sync(0xffffffffu, key[j] != 0u);
      if (threadIdx.x == 0) xm[32 * kMaskWords] = nonzero;
    }
  }
  if (threadIdx.x < p) {
    const int e = group_exp(key[threadIdx.x]);
    if (e < 0) atomicOr(flag, kOutOfRange);
    if (!window) exps[blockIdx.y * stride + threadIdx.x] = e;
  }
}

// Columns [a0, a0 + pa) of A and [b0, b0 + pb) of B; NB: B columns per slice (>= pb).  PANEL: A and B
// hold one dense column-major A (ld: its leading dimension) and one row-major block; the CTA's a0 and
// rows follow from its index, and element (row, j) goes to part[split][row * pb + j].
// CA: columns of an A slice (32 or 64; >= pa).
template <int CA, int NB, bool PANEL>
__global__ void __launch_bounds__(kThreads, 1)
    gram64_kernel(int64_t n, Cols<double> A, Cols<double> B, int ld, int a0, int pa, int b0, int pb, int upper,
                  int same, int rs, const int* __restrict__ exps, int estride, int eb0,
                  const int* __restrict__ flag, double* __restrict__ part, int64_t groups_per_cta, int npanels,
                  int row_a, int* __restrict__ err) {
  constexpr int kAS = NB <= 32 ? 2 : 1;  // accumulators (of kDiags * NB TMEM columns)
  constexpr int kAcc = kDiags * NB;
  constexpr uint32_t kSliceA = CA / 8 * kSBO, kSliceB = NB / 8 * kSBO;  // bytes of a slice
  constexpr int kColStride = kKC + 2;  // PANEL: doubles between the columns of a raw stage
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
  if constexpr (PANEL) {
    a0 = (int)(blockIdx.x % (unsigned)npanels) * kCB;
    pa = (int)min((int64_t)kCB, n - a0);
  }
  const int seg = kKC * ld;
  if (tid == 0) {
    int nu = 0;
    for (int o = 0; o < (PANEL ? 0 : same ? 1 : 2); ++o) {
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
    for (int s = 0; s < kMaxRS; ++s) mbar_init(&raw_full[s], PANEL ? 33 : 1), mbar_init(&raw_empty[s], kSplitWarps / kSplitGroups);
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
    if (PANEL) {
      if (m < (o == 0 ? pa : pb)) off = o == 0 ? m * (row_a ? 1 : kColStride) : kCB * kColStride + m;
    } else if (m < (o == 0 ? pa : pb) && !(o == 1 && same)) {
      const int col = m + (o == 0 ? a0 : b0);
      int base = 0, g = 0;
      while (col >= base + c.w[g]) base += c.w[g], ++g;
      int u = 0;
      while (useg[u] != c.p[g]) ++u;
      off = u * seg + (col - base);
    }
    colofs[o][m] = off;
  }
  // doubles of a raw stage: [nu][kKC][ld], or kCB columns of A and kKC rows of X
  const int stage = PANEL ? kCB * kColStride + kKC * B.ld[0] : nu * seg;
  const size_t raw_bytes = ((size_t)rs * stage * 8 + 127) / 128 * 128;
  double* raw = reinterpret_cast<double*>(smem);  // [rs][stage]
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

  const int64_t g_begin = (int64_t)(PANEL ? blockIdx.x / (unsigned)npanels : blockIdx.x) * groups_per_cta;
  const int64_t r_begin = g_begin * kGroupRows;
  const int64_t r_end = min(n, r_begin + groups_per_cta * kGroupRows);
  const int nchunks = r_end > r_begin ? (int)((r_end - r_begin + kKC - 1) / kKC) : 0;
  const int ngroups = (nchunks + kChunks - 1) / kChunks;
  int issued = 0, committed = 0;  // producer thread; MMA thread (groups)
  if (PANEL && warp == 0) {
    int st = 0;
    uint32_t ph = 0;
    for (int c = 0; c < nchunks; ++c) {
      if (c >= rs && !__all_sync(0xffffffffu, wait_bar(&raw_empty[st], ph ^ 1u, &abort_flag, err, 3))) break;
      const int64_t r0 = r_begin + (int64_t)c * kKC;
      const int rows = (int)min((int64_t)kKC, r_end - r0);  // even: n is
      double* raw_st = raw + (size_t)st * stage;
      if (lane == 0) {
        const uint32_t bytes = (uint32_t)((rows - 1) * B.ld[0] + pb + 1) / 2 * 16u;
        mbar_expect_tx(&raw_full[st], bytes);
        bulk_g2s(raw_st + kCB * kColStride, B.p[0] + r0 * B.ld[0], bytes, &raw_full[st]);
      }
      const int v = 2 * (lane & 15);
      if (row_a) {  // columns 2 lane, + 1 of every row
        if (2 * lane < pa) {
          const double* src = A.p[0] + r0 * ld + a0 + 2 * lane;
          for (int r = 0; r < rows; ++r, src += ld) cp_async16(raw_st + r * kCB + 2 * lane, src);
        }
      } else if (v < rows) {  // rows v, v + 1 of columns lane / 16, + 2, ..
        const double* src = A.p[0] + (int64_t)(a0 + (lane >> 4)) * ld + r0 + v;
        for (int m = lane >> 4; m < pa; m += 2, src += 2 * (int64_t)ld) cp_async16(raw_st + m * kColStride + v, src);
      }
      cp_async_arrive(&raw_full[st]);  // one arrival per lane, once its copies have landed
      issued = c + 1;
      if (++st == rs) st = 0, ph ^= 1u;
    }
  } else if (warp == 0) {
    if (lane == 0) {
      int st = 0;
      uint32_t ph = 0;
      for (int c = 0; c < nchunks; ++c) {
        if (c >= rs && !wait_bar(&raw_empty[st], ph ^ 1u, &abort_flag, err, 3)) break;
        const int64_t r0 = r_begin + (int64_t)c * kKC;
        const int rows = (int)min((int64_t)kKC, r_end - r0);
        uint32_t total = 0;  // the last row's copy stops at the used columns
        for (int u = 0; u < nu; ++u) total += (uint32_t)((rows - 1) * ld + ucopy[u]) * 8u;
        mbar_expect_tx(&raw_full[st], total);
        for (int u = 0; u < nu; ++u)
          bulk_g2s(raw + (size_t)st * stage + u * seg, useg[u] + r0 * ld, (uint32_t)((rows - 1) * ld + ucopy[u]) * 8u,
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
        if (!wait_bar(&tile_full[buf], tph, &abort_flag, err, 3)) break;
        if (in_group == 0 && c / kChunks >= kAS && !wait_bar(&acc_empty[r], aph ^ 1u, &abort_flag, err, 3)) break;
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
          if constexpr (CA == 32) {  // four A slices an operand: TMEM lanes 32 u .. hold i + j = t + u
            mma(kk, 0, 0, kSlices, acc);  // regions 0..6
            mma(kk, 4, 0, 3, 1u);
            mma(kk, 4, 3, 1, acc);  // region 7
          } else {
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
    const int row = (32 * quad + lane) & (CA - 1);  // column of A
    const int part_ = 32 * quad / CA;               // regions hold i + j = t + part_
    double acc[kEW];
#pragma unroll
    for (int j = 0; j < kEW; ++j) acc[j] = 0.0;
    int r = 0, g = 0;
    uint32_t aph = 0;
    for (; g < ngroups; ++g) {
      const int* ge = exps + (g_begin + g) * (int64_t)estride;
      // exponents of this lane's row and of column `lane` of this warp, before the wait
      const int ea = row < pa ? __ldg(ge + a0 + row) : kExpOne;
      const int ebl = lane < kEW && kEW * half + lane < pb ? __ldg(ge + eb0 + b0 + kEW * half + lane) : kExpOne;
      if (!__all_sync(0xffffffffu, wait_bar(&acc_full[r], aph, &abort_flag, err, 2))) break;
      tc_fence_after();
      const uint32_t t0 = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(r * kAcc + kEW * half);
      // element: (sum_t v_t 256^(7-t)) 2^(40 - 110) 2^(ea - 1022) 2^(eb - 1022) / 256^part_
      const int sa = ea - 1022 - 70 - 8 * part_;
#pragma unroll
      for (int j0 = 0; j0 < kEW; j0 += 4) {
        if (kEW * half + j0 < pb) {  // warp-uniform
          float v[kDiags][4];
#pragma unroll
          for (int t = 0; t < kDiags; ++t) tmem_ld4(t0 + (uint32_t)(NB * t + j0), v[t]);
          tmem_wait_ld(v);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int eb = __shfl_sync(0xffffffffu, ebl, j0 + i);
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
    // every group's MMAs done means every copy and tile is done with: the other parts hand their sums to
    // part 0 through the raw ring's memory
    const bool done = g == ngroups;
    double* red = reinterpret_cast<double*>(smem);
    if (part_ && done)
#pragma unroll
      for (int j = 0; j < kEW; ++j) red[((part_ - 1) * NB + kEW * half + j) * CA + row] = acc[j];
    asm volatile("bar.sync 3, 256;\n" ::: "memory");  // the eight epilogue warps
    if (!part_ && row < pa) {
      const bool ok = done && !abort_flag;
#pragma unroll
      for (int j = 0; j < kEW; ++j)
#pragma unroll
        for (int u = 0; u < 128 / CA - 1; ++u) acc[j] += red[(u * NB + kEW * half + j) * CA + row];
      double* out = part + (PANEL ? (int64_t)(blockIdx.x / (unsigned)npanels) * n * pb : (int64_t)blockIdx.x * ta * tb);
#pragma unroll
      for (int j = 0; j < kEW; ++j) {
        const int col = kEW * half + j;
        if constexpr (PANEL) {
          if (col < pb) out[(int64_t)(a0 + row) * pb + col] = ok ? acc[j] : 0.0;
        } else if (col < pb && (!upper || a0 + row <= b0 + col))
          out[(a0 + row) + (int64_t)(b0 + col) * ta] = ok ? acc[j] : 0.0;
      }
    }
  } else {
    // splitters: two groups of four warps take the chunks in turn; the units (32 columns x 8 rows
    // of one operand) of a warp are the same in every chunk
    constexpr int wpg = kSplitWarps / kSplitGroups, K8 = kKC / 8, kMaxUW = 4 * K8 / wpg;
    const int sw = warp - kSplit0, g = sw / wpg, sg = sw % wpg;
    const int gA = (pa + 31) / 32, gB = same ? 0 : (pb + 31) / 32;
    const int units = (gA + gB) * K8;
    int src[kMaxUW], ecol[kMaxUW], exp_[kMaxUW], rstep[kMaxUW];  // rstep: doubles between rows
    uint32_t dst[kMaxUW], step[kMaxUW], k0[kMaxUW];
#pragma unroll
    for (int j = 0; j < kMaxUW; ++j) {
      const int u = sg + j * wpg;
      src[j] = -1, dst[j] = 0, step[j] = 0, ecol[j] = 0, rstep[j] = ld, exp_[j] = kExpOne, k0[j] = 0;
      if (u < units) {
        const bool isA = u < gA * K8;
        const int v = isA ? u : u - gA * K8;
        const int k8 = v % K8, m = v / K8 * 32 + lane;
        const int off = colofs[isA ? 0 : 1][m];
        if (off >= 0) {
          if constexpr (PANEL) rstep[j] = isA ? (row_a ? kCB : 1) : B.ld[0];
          src[j] = off + 8 * k8 * rstep[j];
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
          if (src[j] >= 0) exp_[j] = __ldg(exps + (g_begin + cur) * (int64_t)estride + ecol[j]);
      }
      if (!__all_sync(0xffffffffu, wait_bar(&raw_full[st], ph, &abort_flag, err, 1))) break;
      if (c >= kTS && !__all_sync(0xffffffffu, wait_bar(&tile_empty[buf], tph ^ 1u, &abort_flag, err, 2))) break;
      const int rows = (int)min((int64_t)kKC, r_end - (r_begin + (int64_t)c * kKC));
      const double* rsb = raw + (size_t)st * stage;
      unsigned char* tb_ = tiles + (uint32_t)buf * tbuf;
#pragma unroll
      for (int j = 0; j < kMaxUW; ++j) {
        if (src[j] < 0) continue;
        double x[8];
        if (rows == kKC) {
#pragma unroll
          for (int i = 0; i < 8; ++i) x[i] = rsb[src[j] + i * rstep[j]];
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) x[i] = (int)k0[j] + i < rows ? rsb[src[j] + i * rstep[j]] : 0.0;
        }
        if constexpr (PANEL) {  // A's diagonal goes to the sums by itself
          const int64_t d = ecol[j] - (r_begin + (int64_t)c * kKC + k0[j]);
          if (ecol[j] < eb0 && d >= 0 && d < 8)
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = i == (int)d ? 0.0 : x[i];
        }
        uint64_t w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = digits(x[i], exp_[j]);
        unsigned char* o = tb_ + dst[j];
        put_digits(w, o, step[j]);
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
    if (warp == 0 && (PANEL || lane == 0))
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

template <int CA, int NB>
void gram64_launch(int64_t n, const Cols<double>& a, const Cols<double>& b, int ld, int a0, int pa, int b0, int pb,
                   bool upper, bool same, int rs, size_t smem, const int* exps, int estride, int eb0,
                   const int* flag, double* part, int ctas, int64_t gpc, int* err, cudaStream_t st) {
  static const bool attr = [&] {
    LB_CUDA(cudaFuncSetAttribute(gram64_kernel<CA, NB, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget));
    return true;
  }();
  (void)attr;
  gram64_kernel<CA, NB, false><<<(unsigned)ctas, kThreads, smem, st>>>(n, a, b, ld, a0, pa, b0, pb, upper ? 1 : 0, same ? 1 : 0,
                                                           rs, exps, estride, eb0, flag, part, gpc, 0, 0, err);
  LB_LAUNCH_CHECK();
}

}  // namespace

size_t gram64_scratch_ints(int64_t n) { return (size_t)ceil_div(n, kGroupRows) * 2 * kMaxS + 4; }

// Gram partials through digit products; returns 0 without launching where the operands do not share
// one 16-byte aligned row stride or need more shared memory than a CTA has.  scratch:
// gram64_scratch_ints(n) ints; its first word is the flag: where it is not zero the partials are not
// written, and the caller's general kernel (launched on the same flag) forms them.  spread: the flag is
// also raised where two columns of a group are too far apart.
int gram_partials_digits(int64_t n, const Cols<double>& a, const Cols<double>& b, bool upper, double* part,
                         int max_ctas, int* scratch, bool spread, int* err, cudaStream_t st) {
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
  const int nbw = wb <= 32 ? 32 : 64, caw = wa <= 32 && wb <= 32 ? 32 : 64;  // columns of B and A slices
  const size_t stage = (size_t)kKC * count_blocks(a, b) * ld * 8;
  const size_t tiles = (size_t)kTS * (8 * (size_t)(caw / 8) + kSlices * (size_t)(nbw / 8)) * kSBO;
  if (tiles + 2 * stage + 128 > kSmemBudget) return 0;
  const int rs = (int)std::min<size_t>(kMaxRS, (kSmemBudget - tiles - 128) / stage);
  // the raw ring also holds the epilogue's exchange
  const size_t smem = std::max((rs * stage + 127) / 128 * 128, (size_t)(128 - caw) * nbw * 8) + tiles;
  if (smem > kSmemBudget) return 0;
  const int64_t ngroups = ceil_div(n, kGroupRows);
  int64_t ctas = std::min<int64_t>(std::min<int64_t>(max_ctas, sm_count()), ngroups);
  const int64_t gpc = ceil_div(ngroups, ctas);
  ctas = ceil_div(ngroups, gpc);
  int* flag = scratch;
  int* exps = scratch + 4;
  const int estride = pa + (same ? 0 : pb), eb0 = same ? 0 : pa;
  LB_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), st));
  if (spread) {
    if (a.nseg != 1 || b.nseg != 1 || n < kGroupRows) return 0;
    static const bool attr = [&] {
      LB_CUDA(cudaFuncSetAttribute(exp_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   kGroupRows * kMaxS * (int)sizeof(uint32_t)));
      return true;
    }();
    (void)attr;
    const size_t bytes = (size_t)kGroupRows * ((pa + 1) / 2 + (same ? 0 : (pb + 1) / 2)) * sizeof(uint32_t);
    exp_kernel<true><<<(unsigned)(ngroups + (n % kGroupRows ? 1 : 0)), 256, bytes, st>>>(n, a, b, ld, same ? 1 : 0, exps,
                                                                                         estride, flag);
  } else {
    exp_kernel<false><<<(unsigned)ngroups, 256, 0, st>>>(n, a, b, ld, same ? 1 : 0, exps, estride, flag);
  }
  LB_LAUNCH_CHECK();
  for (int ia = 0; ia < na; ++ia)
    for (int ib = 0; ib < nb; ++ib) {
      const int a0 = ia * wa, b0 = ib * wb;
      const int ca = std::min(wa, pa - a0), cb = std::min(wb, pb - b0);
      if (upper && a0 > b0 + cb - 1) continue;
      // B can read A's tiles where its slices have A's width
      const bool diag = same && ia == ib && nbw == caw;
      if (caw == 32)
        gram64_launch<32, 32>(n, a, b, ld, a0, ca, b0, cb, upper, diag, rs, smem, exps, estride, eb0, flag, part,
                              (int)ctas, gpc, err, st);
      else if (nbw == 32)
        gram64_launch<64, 32>(n, a, b, ld, a0, ca, b0, cb, upper, diag, rs, smem, exps, estride, eb0, flag, part,
                          (int)ctas, gpc, err, st);
      else
        gram64_launch<64, 64>(n, a, b, ld, a0, ca, b0, cb, upper, diag, rs, smem, exps, estride, eb0, flag, part,
                          (int)ctas, gpc, err, st);
    }
  return (int)ctas;
}

namespace {
// Y[i][j] = sum over the splits, in order, then A's diagonal against X
__global__ void panel_reduce_kernel(int64_t n, int p, int splits, const double* __restrict__ part,
                                    const double* __restrict__ A, int64_t lda, const double* __restrict__ X, int ldx,
                                    double* __restrict__ Y, int ldy, const int* __restrict__ flag) {
  if (*flag) return;  // no sums were written
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * p; e += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int g = 0; g < splits; ++g) s += part[g * n * p + e];
    const int64_t i = e / p, j = e % p;
    Y[i * ldy + j] = fma(A[i * lda + i], X[i * ldx + j], s);
  }
}

constexpr int kMaxSplits = 8;
// Row ranges per panel: the count that fills whole waves of the SMs best (fewer where equal: every
// range pays the kernel's start).
int panel_splits(int64_t panels, int64_t groups, int sms) {
  int best = 1;
  double cost = 1e300;
  for (int k = 1; k <= kMaxSplits && k <= groups; ++k) {
    const int64_t per = ceil_div(groups, k), used = ceil_div(groups, per);
    // waves x (groups of a range + the start, about the time of two groups)
    const double c = (double)ceil_div(panels * used, sms) * ((double)per + 2.0);
    if (c < cost * 0.98) cost = c, best = (int)used;
  }
  return best;
}
}  // namespace

// Scratch of launch_spmm_dense_digits in bytes: flag, exponents, masks of X, partial sums.
static size_t dense64_exps_bytes(int64_t n, int p) {
  return ((size_t)ceil_div(n, kGroupRows) * (n + p) * sizeof(int) + 255) / 256 * 256;
}
static size_t dense64_mask_bytes(int64_t n) {
  return ((size_t)(ceil_div(n, kGroupRows) + 1) * kXMask * sizeof(uint32_t) + 255) / 256 * 256;
}
size_t dense64_scratch_bytes(int64_t n, int p) {
  return 256 + dense64_exps_bytes(n, p) + dense64_mask_bytes(n) + (size_t)kMaxSplits * n * p * sizeof(double);
}

// Y = A X (column i of the dense A against X; A column-major, or row-major with row_a) through digit products; false without
// launching where A or X do not fit (odd n or lda, unaligned).  *scratch is the flag, not zero when a
// number is outside the digits' range or, with `spread`, two columns of a group are too far apart: Y is
// then to be formed by launch_spmm_dense on that flag.
bool launch_spmm_dense_digits(int64_t n, const double* A, int64_t lda, int p, const double* X, int ldx, double* Y,
                              int ldy, void* scratch, bool row_a, bool spread, int* err, cudaStream_t st) {
  if (n < kGroupRows || (n & 1) || (lda & 1) || lda > INT_MAX || p < 1 || p > 32 || (reinterpret_cast<uintptr_t>(A) & 15) ||
      (reinterpret_cast<uintptr_t>(X) & 15))
    return false;
  constexpr int NB = 32;
  const size_t stage = ((size_t)kCB * (kKC + 2) + (size_t)kKC * ldx) * 8;
  const size_t tiles = (size_t)kTS * (8 * (size_t)(kCB / 8) + kSlices * (size_t)(NB / 8)) * kSBO;
  if (tiles + 2 * stage + 128 > kSmemBudget) return false;
  const int rs = (int)std::min<size_t>(kMaxRS, (kSmemBudget - tiles - 128) / stage);
  const size_t smem = std::max((rs * stage + 127) / 128 * 128, (size_t)64 * NB * 8) + tiles;
  static const bool attr = [&] {
    LB_CUDA(cudaFuncSetAttribute(gram64_kernel<kCB, NB, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget));
    return true;
  }();
  (void)attr;
  const int64_t groups = ceil_div(n, kGroupRows), panels = ceil_div(n, kCB);
  const int splits = panel_splits(panels, groups, sm_count());
  int* flag = static_cast<int*>(scratch);
  int* exps = flag + 64;
  const int64_t estride = n + p;
  uint32_t* xmask = reinterpret_cast<uint32_t*>(static_cast<char*>(scratch) + 256 + dense64_exps_bytes(n, p));
  double* part = reinterpret_cast<double*>(reinterpret_cast<char*>(xmask) + dense64_mask_bytes(n));
  LB_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), st));
  const unsigned gy = (unsigned)(groups + (spread && n % kGroupRows ? 1 : 0));
  if (spread) {
    exp_rows_kernel<true><<<dim3(1, gy), 256, 0, st>>>(n, p, X, ldx, exps + n, estride, xmask, flag);
    LB_LAUNCH_CHECK();
    if (row_a)
      exp_dense_rows_kernel<true><<<dim3((unsigned)panels, gy), 256, 0, st>>>(n, A, lda, exps, estride, p, xmask, flag);
    else
      exp_dense_kernel<true><<<dim3((unsigned)ceil_div(n, 8), gy), 256, 0, st>>>(n, A, lda, exps, estride, p, xmask, flag);
  } else {
    exp_rows_kernel<false><<<dim3(1, gy), 256, 0, st>>>(n, p, X, ldx, exps + n, estride, xmask, flag);
    LB_LAUNCH_CHECK();
    if (row_a)
      exp_dense_rows_kernel<false><<<dim3((unsigned)panels, gy), 256, 0, st>>>(n, A, lda, exps, estride, p, xmask, flag);
    else
      exp_dense_kernel<false><<<dim3((unsigned)ceil_div(n, 8), gy), 256, 0, st>>>(n, A, lda, exps, estride, p, xmask, flag);
  }
  LB_LAUNCH_CHECK();
  gram64_kernel<kCB, NB, true><<<(unsigned)(panels * splits), kThreads, smem, st>>>(
      n, cols1<double>(A, (int)lda, 1), cols1<double>(X, ldx, p), (int)lda, 0, 0, 0, p, 0, 0, rs, exps, (int)estride,
      (int)n, flag, part, ceil_div(groups, splits), (int)panels, row_a ? 1 : 0, err);
  LB_LAUNCH_CHECK();
  panel_reduce_kernel<<<(unsigned)std::min<int64_t>(ceil_div(n * p, 256), 4096), 256, 0, st>>>(n, p, splits, part, A,
                                                                                               lda, X, ldx, Y, ldy, flag);
  LB_LAUNCH_CHECK();
  return true;
}

}  // namespace lobpcg
