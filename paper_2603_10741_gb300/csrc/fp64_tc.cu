// FP64 principal-block x cell-vector products on the tensor cores, for the FP64 mode: the local part
// of K^-rom, Y[rows of cell s] = [G; Phi^T]_{key(s)} X_R^s, and the dual Schur complements of the
// interface preconditioner, over cells grouped by key.
//
// FP64 runs at 1.2 TFLOP/s on this GPU, 1/1500 of its BF16 tensor rate, and these products were 80 %
// of an FP64 3D solve.  They are formed without it, by an error-free splitting (the scheme of Ozaki,
// Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by using fast routines
// of matrix multiplication and its applications", 2012): each row of the matrix and each cell vector
// is scaled by a power of two and split into 12 signed base-128 digits,
//   x = 2^(e-6) sum_i s_i 2^(-7 i),  |s_i| <= 64   (|x| <= 2^e; the rest is below 2^(e-84)),
// digits are exact in BF16, products of digits are integers up to 2^12, and the tensor core adds
// them in FP32 exactly while a sum stays within 2^24.  The 78 digit products with i + j <= 11 go to
// twelve accumulators by i + j (at most 12 products of 2^12 per column: 336 columns may be summed),
// which the epilogue recombines as integers, four at a time, and converts to FP64.
//
// Precision.  What is left out (digits beyond the twelfth, products with i + j > 11) is less than
// 12.1 x 2^-82 of (row maximum) x (vector maximum) per term; the recombination and the sums over the
// CTAs of a cluster round ten times at most.  An FP64 sum rounds relative to sum |g| |x| instead, so the
// number of digits has to cover the spread of the operands as well: entries of either down to 2^-31 of
// their maximum keep all their bits.  Error of the product in the 2-norm, and the largest error of an
// entry against its sum |g| |x|, of the strut cell's dual Schur complement (1692 columns; its entries
// fall to 1e-24 of their row's largest), emulated; FP64 sums, then 8 digits (not enough on graded
// vectors) and 12:
//   uniform in [-1, 1]             1.4e-15 2.2e-15    8.3e-16 9.6e-16    4.5e-17 5.2e-17
//   magnitudes 1e-12 to 1          7.8e-16 3.2e-15    3.3e-15 2.4e-13    4.8e-17 9.1e-17
//   20 entries over 1e-6           9.8e-16 5.5e-15    5.0e-15 1.0e-10    3.7e-17 1.0e-16
//   one entry over 1e-8            7.5e-16 5.8e-15    1.3e-14 1.0e-07    6.5e-17 8.0e-16
//   one entry over 1e-12           4.1e-16 7.4e-15    5.4e-15 3.5e-04    4.3e-17 5.9e-12
// (G itself is denser: 1.0e-16 in every row of its dual block.)  What is left are results far below row
// maximum x vector maximum, whose terms may lie where the digits end: those below 2^-26 of it are summed
// again in FP64 from the matrix and vector themselves, by the CTA that holds them (k_oz_mm's last loop;
// cancellation alone takes few results that far).
//
// One tensor-memory tile is 128 rows x (12 accumulators of 16 cells): for digit i of the matrix one
// MMA multiplies the digits 0 .. 11-i of the 16 cells (N = 16 (12 - i), consecutive rows of the B
// panel) into the accumulators i .. 11, consecutive columns from 16 i on.  K is split over a cluster
// of CTAs (336 columns at most each while eight CTAs suffice, which the exactness needs) that add their
// FP64 tiles through distributed shared memory.  Bound by streaming the digits, 24 bytes per matrix
// entry: the strut cell's dual block (1716 x 1692) for 3 keys and 36 cells is 227 MB: 68 us with
// splitting the vectors (54 us with 8 digits) against 406 us on the FP64 pipe (175 us at its full rate).
#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace {

constexpr int ND = 12;                    // digits
constexpr int TM = 128, TK = 16, NC = kOzCells; // rows, K panel, cells of a tile
constexpr int A_SLICE = TM * TK;          // elements of one digit of an A panel
constexpr int A_ELEMS = ND * A_SLICE;     // 48 KiB
constexpr int B_ELEMS = ND * NC * TK;     // 6 KiB
constexpr int STAGE_BYTES = 2 * (A_ELEMS + B_ELEMS);
constexpr int STAGES = 2;                 // 108 KiB, two CTAs per SM
constexpr int TMEM_COLS = 256;            // ND * NC = 192, allocated in powers of two
constexpr int EXACT_PANELS = 336 / TK;    // panels one CTA sums exactly in every accumulator
constexpr int MAX_PANELS = 512 / TK;      // and in the accumulators 0 .. 7
constexpr int MAX_SPLIT = 8;              // portable cluster size
constexpr double kOzBytes = 24e9;         // most digits kept, a twelfth of the device's memory
constexpr int PART_LD = TM + 1;
constexpr uint32_t LBO = 128, SBO = (TK / 8) * 128;
constexpr size_t PART_BYTES = (size_t)NC * PART_LD * sizeof(double);   // the tile, then the list of small entries
static_assert(PART_BYTES + (size_t)NC * TM * sizeof(int) <= (size_t)STAGES * STAGE_BYTES, "both reuse the stages");
constexpr double SMALL = 0x1p-14;         // 2^-26 of row maximum x vector maximum, or up to four times that

__device__ __forceinline__ uint64_t desc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (uint64_t)(LBO >> 4) << 16 | (uint64_t)(SBO >> 4) << 32 | (uint64_t)1 << 46;
}

// element (row, k) of a K-major panel of TK columns
__host__ __device__ __forceinline__ int core_off(int r, int k) {
  return (r >> 3) * (TK / 8) * 64 + (k >> 3) * 64 + (r & 7) * 8 + (k & 7);
}

__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

// biased exponent of a magnitude's bits, subnormals with that of the smallest normal number
__device__ __forceinline__ int biased_exponent(unsigned long long mag) { return max(1, (int)(mag >> 52)); }
// e of a row or vector from the bits of its largest magnitude (every |x| <= 2^e), and the factor
// 2^(e-6) of its digits: 0 for an all-zero row, NaN when an entry is infinite or NaN
__device__ __forceinline__ int top_exponent(unsigned long long mx) { return biased_exponent(mx) - 1022; }
__device__ __forceinline__ double digit_scale(unsigned long long mx) {
  if (mx >= 0x7ff0000000000000ull) return __longlong_as_double(0x7ff8000000000000ll);
  if (mx == 0) return 0.0;
  return scalbn(1.0, top_exponent(mx) - 6);
}

// x 2^(P - e) for the top exponent e, P = BITS + 6 <= 83, rounded to a whole number hi 2^42 + lo of sign
// and magnitude, by integer operations (the FP64 pipe is the narrow one); 0 when the row is not finite
template <int BITS>
__device__ __forceinline__ void fixed_point(double x, unsigned long long mx, long long& hi, long long& lo) {
  constexpr unsigned long long low = (1ull << 42) - 1;
  const unsigned long long b = abs_bits(x);
  const unsigned long long m = (b & 0xfffffffffffffull) | (b >> 52 ? 0x10000000000000ull : 0);
  // x = m 2^(biased exponent - 1075)
  const int sh = biased_exponent(b) - 1022 - top_exponent(mx) + BITS - 47;   // at most BITS - 47
  unsigned long long vh = 0, vl = 0;
  if (mx < 0x7ff0000000000000ull) {
    if (sh >= 0) {
      vl = (m << sh) & low;
      vh = m >> (42 - sh);
    } else if (sh > -55) {
      const unsigned long long v = (m + (1ull << (-sh - 1))) >> -sh;
      vl = v & low;
      vh = v >> 42;
    }
  }
  const bool neg = __double_as_longlong(x) < 0;
  hi = neg ? -(long long)vh : (long long)vh;
  lo = neg ? -(long long)vl : (long long)vl;
}

// lowest balanced base-2^DB digit of q, taken off
template <int DB>
__device__ __forceinline__ int pop_digit(long long& q) {
  constexpr long long half = 1ll << (DB - 1), mask = (1ll << DB) - 1;
  const long long d = ((q + half) & mask) - half;
  q = (q - d) >> DB;
  return (int)d;
}

// digit panels of eight consecutive K entries of one row: dst + i * stride, 16 bytes per digit; lowest
// digit first, six from the low words, the rest from the high ones
__device__ __forceinline__ void store_digits(const double (&v)[8], unsigned long long mx, __nv_bfloat16* dst,
                                             int stride) {
  static_assert(ND == 12, "two words of six digits");
  long long hi[8], q[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) fixed_point<7 * (ND - 1)>(v[k], mx, hi[k], q[k]);
#pragma unroll
  for (int i = ND - 1; i >= 0; --i) {
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float f[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        long long& x = q[2 * k + u];
        if (i == 5) x += hi[2 * k + u];   // what is left of the low word is its carry
        f[u] = (float)(i ? pop_digit<7>(x) : (int)x);
      }
      const __nv_bfloat162 p = __floats2bfloat162_rn(f[0], f[1]);
      w[k] = *reinterpret_cast<const uint32_t*>(&p);
    }
    *reinterpret_cast<uint4*>(dst + (size_t)i * stride) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// Rows and columns of the tiled matrix: nI interior ones padded to MTI tiles / KI panels, then the
// others, so that the dual views start at a tile and a panel.
struct OzShape {
  int nI, MTI, KI;      // interior rows and columns (the same DOFs)
  int rows, cols;       // of the source matrix
  int MT, KP;           // row tiles and panels of the padded one
  __host__ __device__ int row(int tr) const {           // source row of padded row tr, or -1
    if (tr < MTI * TM) return tr < nI ? tr : -1;
    const int r = nI + tr - MTI * TM;
    return r < rows ? r : -1;
  }
  __host__ __device__ int col(int tk) const {
    if (tk < KI * TK) return tk < nI ? tk : -1;
    const int c = nI + tk - KI * TK;
    return c < cols ? c : -1;
  }
};

// largest magnitude of every source row (bits), a warp per (key, padded row); its factor
__global__ void __launch_bounds__(256)
    k_oz_rowmax(OzShape sh, int64_t n_rows, int ld, int64_t kstride, const double* __restrict__ G,
                unsigned long long* __restrict__ mx, double* __restrict__ scale) {
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= n_rows) return;
  const int per = sh.MT * TM;
  const int64_t key = t / per;
  const int r = sh.row((int)(t - key * per));
  unsigned long long m = 0;
  if (r >= 0)
    for (int k = lane; k < sh.cols; k += 32) m = max(m, abs_bits(G[key * kstride + (int64_t)r * ld + k]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) {
    mx[t] = m;
    scale[t] = digit_scale(m);
  }
}

// digits of the matrix: [key][row tile][panel][digit][core_off(row, k)], a thread per (row, 8 columns)
__global__ void __launch_bounds__(128)
    k_oz_tile(OzShape sh, int ld, int64_t kstride, const double* __restrict__ G,
              const unsigned long long* __restrict__ mx, __nv_bfloat16* __restrict__ T) {
  const int mt = blockIdx.x, k8 = blockIdx.y, r = threadIdx.x;   // padded columns [8 k8, 8 k8 + 8)
  const int64_t key = blockIdx.z;
  const int row = sh.row(mt * TM + r);
  double v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int c = sh.col(8 * k8 + q);
    v[q] = row >= 0 && c >= 0 ? G[key * kstride + (int64_t)row * ld + c] : 0.0;
  }
  const int kp = k8 / (TK / 8);
  __nv_bfloat16* dst = T + (((size_t)key * sh.MT + mt) * sh.KP + kp) * A_ELEMS + core_off(r, (k8 % (TK / 8)) * 8);
  store_digits(v, mx[(key * sh.MT + mt) * TM + r], dst, A_SLICE);
}

// largest magnitude of every cell vector of a tile over the view's columns (cleared before)
__global__ void __launch_bounds__(256)
    k_oz_cellmax(int n_cells, int n_K, const double* __restrict__ X, const int* __restrict__ rc,
                 const int* __restrict__ tile_seg, const int* __restrict__ tile_c0, const int* __restrict__ seg_ptr,
                 const int* __restrict__ perm, unsigned long long* __restrict__ mx) {
  __shared__ unsigned long long red[16][NC + 1];
  const int tile = blockIdx.x, c = threadIdx.x % NC, g = threadIdx.x / NC;
  const int pos = tile_c0[tile] + c;
  unsigned long long m = 0;
  if (pos < seg_ptr[tile_seg[tile] + 1]) {
    const int s = perm[pos];
#pragma unroll 4
    for (int k = blockIdx.y * 16 + g; k < n_K; k += gridDim.y * 16)
      m = max(m, abs_bits(X[(size_t)rc[k] * n_cells + s]));
  }
  red[g][c] = m;
  __syncthreads();
  if (g == 0) {
    for (int q = 1; q < 16; ++q) m = max(m, red[q][c]);
    atomicMax(mx + (size_t)tile * NC + c, m);
  }
}

// digits of the cell vectors: [tile][panel][core_off(digit * 16 + cell, k)], a thread per (cell, 8
// columns); the view's padded columns start at panel kp0
__global__ void __launch_bounds__(256)
    k_oz_pack(OzShape sh, int n_cells, int kp0, int npan, const double* __restrict__ X,
              const int* __restrict__ rdofs, const int* __restrict__ tile_seg, const int* __restrict__ tile_c0,
              const int* __restrict__ seg_ptr, const int* __restrict__ perm,
              const unsigned long long* __restrict__ mx, __nv_bfloat16* __restrict__ T) {
  const int tile = blockIdx.x, c = threadIdx.x % NC;
  const int k8 = blockIdx.y * 16 + threadIdx.x / NC;
  if (k8 >= npan * (TK / 8)) return;
  const int pos = tile_c0[tile] + c;
  const bool in = pos < seg_ptr[tile_seg[tile] + 1];
  const int s = in ? perm[pos] : 0;
  double v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = sh.col(kp0 * TK + 8 * k8 + q);
    v[q] = in && k >= 0 ? X[(size_t)rdofs[k] * n_cells + s] : 0.0;
  }
  const int kp = k8 / (TK / 8);
  __nv_bfloat16* dst = T + ((size_t)tile * npan + kp) * B_ELEMS + core_off(c, (k8 % (TK / 8)) * 8);
  store_digits(v, mx[(size_t)tile * NC + c], dst, NC * TK);
}

// integer sums of four digit accumulators (exact in FP32 up to 2^24), combined: below 2^50
template <int DB>
__device__ __forceinline__ double combine4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  const long long v = ((long long)__float2int_rn(__uint_as_float(a)) << (3 * DB)) +
                      ((long long)__float2int_rn(__uint_as_float(b)) << (2 * DB)) +
                      ((long long)__float2int_rn(__uint_as_float(c)) << DB) +
                      (long long)__float2int_rn(__uint_as_float(d));
  // |v| < 2^51 as a double: the bits of 1.5 2^52 plus v, one subtraction
  return __longlong_as_double(0x4338000000000000ll + v) - 6755399441055744.0;
}

__device__ __forceinline__ double ld_cluster(uint32_t addr, uint32_t rank) {
  uint32_t ra;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(ra) : "memory");
  return v;
}

__device__ __forceinline__ void tmem_ld4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

// Rows [128 (mt0 + mt), ...) of the tiled matrix x 16 cells; the cluster's S CTAs share the view's
// npan panels (from panel kp0 of the matrix), MAX_PANELS at most each.
__global__ void __launch_bounds__(128, 2)
    k_oz_mm(OzShape sh, int n_cells, int mt0, int kp0, int npan, int S, const __nv_bfloat16* __restrict__ GT,
            const double* __restrict__ rscale, const __nv_bfloat16* __restrict__ XT,
            const unsigned long long* __restrict__ cmax, const int* __restrict__ tile_seg,
            const int* __restrict__ tile_c0, const int* __restrict__ seg_ptr, const int* __restrict__ perm,
            const double* __restrict__ cscale, int n_R, int r_base, const int* __restrict__ rdofs,
            const int* __restrict__ pdofs, double* __restrict__ Y, int* __restrict__ err, int mul_scale,
            int polls, const double* __restrict__ G, int ld, int64_t kstride, const double* __restrict__ X, int lo_c,
            const uint8_t* __restrict__ fixed, const int2* __restrict__ lk) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], done;
  __shared__ uint32_t tmem_slot;
  __shared__ int fail, issued;   // a wait gave up; panels whose copies were issued
  __shared__ int cell[NC], n_small;
  __shared__ double cw[NC], cs1[NC], cs2[NC];   // a cell's factor; that times its digits' scale, and the scale
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = blockIdx.x % S, tile = blockIdx.x / S, mt = mt0 + blockIdx.y;
  const int key = tile_seg[tile];
  const int p0 = (int)((int64_t)npan * rank / S), np = (int)((int64_t)npan * (rank + 1) / S) - p0;
  const uint32_t s0 = smem_u32(smem);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full[s]));
      mbar_init(smem_u32(&empty[s]));
    }
    mbar_init(smem_u32(&done));
    fail = 0;
    n_small = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  if (tid == 0) {
    int n = 0;
    bool ok = true;
    for (int p = 0; p < np; ++p) {
      const int st = p % STAGES;
      if (p >= STAGES && !mbar_wait(smem_u32(&empty[st]), (uint32_t)((p / STAGES - 1) & 1), polls)) {
        ok = false;
        break;
      }
      const uint32_t bar = smem_u32(&full[st]), dst = s0 + (uint32_t)(st * STAGE_BYTES);
      expect_tx(bar, (uint32_t)STAGE_BYTES);
      bulk_copy(dst, GT + (((size_t)key * sh.MT + mt) * sh.KP + kp0 + p0 + p) * A_ELEMS, 2 * A_ELEMS, bar);
      bulk_copy(dst + 2 * A_ELEMS, XT + ((size_t)tile * npan + p0 + p) * B_ELEMS, 2 * B_ELEMS, bar);
      ++n;
    }
    if (!ok) fail = 1;
    issued = n;
  } else if (tid == 32) {
    bool ok = true;
    for (int p = 0; p < np; ++p) {
      const int st = p % STAGES;
      if (!mbar_wait(smem_u32(&full[st]), (uint32_t)((p / STAGES) & 1), polls)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sa = s0 + (uint32_t)(st * STAGE_BYTES), sb = sa + 2 * A_ELEMS;
#pragma unroll
      for (int i = 0; i < ND; ++i) {
        // kind::f16: D = F32, A = B = BF16, both K-major, N >> 3, M >> 4
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((ND - i) * NC >> 3) << 17) |
                               ((uint32_t)(TM >> 4) << 24);
        const uint32_t acc = (p > 0 || i > 0) ? 1u : 0u;   // digit 0 reaches every column first
        asm volatile(
            "{\n\t.reg .pred q;\n\t"
            "setp.ne.b32 q, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, q;\n\t}" ::"r"(tmem + (uint32_t)(i * NC)),
            "l"(desc(sa + (uint32_t)(2 * i * A_SLICE))), "l"(desc(sb)), "r"(idesc), "r"(acc)
            : "memory");
      }
      mma_commit(smem_u32(&empty[st]));
    }
    mma_commit(smem_u32(&done));
    ok = mbar_wait(smem_u32(&done), 0) && ok;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (!ok) fail = 1;
  } else if (warp >= 2 && tid - 64 < NC) {
    const int c = tid - 64, pos = tile_c0[tile] + c;
    const int s = pos < seg_ptr[key + 1] ? perm[pos] : -1;
    const double w = s >= 0 ? cscale[s] : 1.0, d = digit_scale(cmax[(size_t)tile * NC + c]);
    cell[c] = s;
    cw[c] = mul_scale ? w : 1.0 / w;          // c_s (S_DD rows) or 1 / c_s (G rows)
    cs1[c] = d * cw[c];
    cs2[c] = d;
  }
  __syncwarp();
  __syncthreads();
  const bool good = !fail;   // accumulators complete, every wait met
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!good && tid == 0) {
    atomicOr(err, kFlagProductWait);
    // copies in flight land (bounded) before the shared memory is released
    for (int q = max(0, issued - STAGES); q < issued; ++q)
      mbar_wait(smem_u32(&full[q % STAGES]), (uint32_t)((q / STAGES) & 1));
  }
  __syncwarp();
  // digit sums of the tile's row (this thread's) and each cell to one FP64 value, in shared memory
  double* part = reinterpret_cast<double*>(smem);   // [cell][129]
  int* small = reinterpret_cast<int*>(smem + PART_BYTES);
  if (good) {
    const uint32_t base = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
    for (int c = 0; c < NC; c += 4) {
      uint32_t r[ND][4];
#pragma unroll
      for (int g = 0; g < ND; ++g) tmem_ld4(base + (uint32_t)(g * NC + c), r[g]);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double hi = combine4<7>(r[0][q], r[1][q], r[2][q], r[3][q]);
        const double mid = combine4<7>(r[4][q], r[5][q], r[6][q], r[7][q]);
        const double lo = combine4<7>(r[8][q], r[9][q], r[10][q], r[11][q]);
        part[(c + q) * PART_LD + tid] = fma(hi, 0x1p-21, fma(mid, 0x1p-49, lo * 0x1p-77));
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (S > 1) cluster_sync();
  else __syncthreads();
  // cells rank, rank + S, ... of the tile: sums over the cluster in CTA order, a lane per row
  const int tr = mt * TM + tid, gi = sh.row(tr);
  const double rs = rscale[(size_t)key * sh.MT * TM + tr];
  const int o = gi < 0 ? -1 : r_base + gi < n_R ? rdofs[r_base + gi] : pdofs[r_base + gi - n_R];
  for (int c = rank; c < NC; c += S) {
    const uint32_t a = smem_u32(part + c * PART_LD + tid);
    double v = 0.0;
    if (S == 1) v = part[c * PART_LD + tid];
    else
      for (int q = 0; q < S; ++q) v += ld_cluster(a, (uint32_t)q);
    if (cell[c] >= 0 && o >= 0 && good) {
      const bool scaled = r_base + gi < n_R;
      Y[(size_t)o * n_cells + cell[c]] = v * rs * (scaled ? cs1[c] : cs2[c]);
      // an entry far below row maximum x vector maximum (v counts 2^-12 of their powers of two), unless it
      // is not read (Dirichlet rows; of S_DD those without a multiplier) or the vector has the smallest
      // exponent (its digits hold it whole; zero vectors alike)
      if (fabs(v) < SMALL && rs != 0.0 && !(cs2[c] <= 0x1p-1027) &&
          !(scaled && fixed[(size_t)o * n_cells + cell[c]])) {
        const int2 m = lk ? lk[(size_t)gi * n_cells + cell[c]] : make_int2(1, 0);
        if (m.x || m.y) small[atomicAdd(&n_small, 1)] = c * TM + tid;
      }
    }
  }
  if (S > 1) cluster_sync();   // peers have read this CTA's tile
  else __syncthreads();
  // those entries in FP64, a warp each: their terms may lie where the digits end
  for (int q = warp; q < n_small; q += 4) {
    const int c = small[q] / TM, gr = sh.row(mt * TM + small[q] % TM), s = cell[c];
    const double* g = G + key * kstride + (int64_t)gr * ld;
    double a = 0.0;
#pragma unroll 4
    for (int k = lo_c + lane; k < sh.cols; k += 32) a = fma(g[k], X[(size_t)rdofs[r_base + k] * n_cells + s], a);
    a = warp_sum(a);
    if (lane == 0) {
      const bool scaled = r_base + gr < n_R;
      Y[(size_t)(scaled ? rdofs[r_base + gr] : pdofs[r_base + gr - n_R]) * n_cells + s] = scaled ? a * cw[c] : a;
    }
  }
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

OzShape shape(int nI, int rows, int cols) {
  OzShape s{};
  s.nI = nI;
  s.MTI = div_up(nI, TM);
  s.KI = div_up(nI, TK);
  s.rows = rows;
  s.cols = cols;
  s.MT = s.MTI + div_up(rows - nI, TM);
  s.KP = s.KI + div_up(cols - nI, TK);
  return s;
}

OzShape g_shape(const lat_ctx* h) { return shape(h->n_I, h->n_R + h->n_P, h->n_R); }
OzShape s_shape(const lat_ctx* h) { return shape(0, h->n_R - h->n_I, h->n_R - h->n_I); }

void split_matrix(lat_ctx* h, const OzShape& sh, int ld, int64_t kstride, const double* G, DBuf<__nv_bfloat16>& T,
                  DBuf<double>& scale) {
  const int keys = h->n_keys;
  const int64_t rows = (int64_t)keys * sh.MT * TM;
  T.ensure((size_t)keys * sh.MT * sh.KP * A_ELEMS);
  scale.ensure((size_t)rows);
  h->oz_max.ensure(std::max((size_t)rows, (size_t)h->oz_tiles * NC));
  LAT_LAUNCH(h, k_oz_rowmax<<<div_up(rows * 32, 256), 256, 0, h->stream>>>(sh, rows, ld, kstride, G, h->oz_max.p,
                                                                          scale.p));
  LAT_LAUNCH(h, k_oz_tile<<<dim3(sh.MT, sh.KP * (TK / 8), keys), TM, 0, h->stream>>>(sh, ld, kstride, G, h->oz_max.p,
                                                                                    T.p));
  LAT_CHECK_LAUNCH();
}

void product(lat_ctx* h, const OzShape& sh, int mt0, int kp0, const DBuf<__nv_bfloat16>& T, const DBuf<double>& scale,
             const double* G, int ld, int64_t kstride, const int* rdofs, int r_base, const double* X, double* Y, int n_R,
             int mul_scale, const int2* lk) {
  const int npan = sh.KP - kp0, tiles = h->oz_tiles;
  const int lo_c = kp0 ? sh.nI : 0, n_K = sh.cols - lo_c;
  h->oz_X.ensure((size_t)tiles * npan * B_ELEMS);
  h->oz_max.ensure((size_t)tiles * NC);
  LAT_CUDA(cudaMemsetAsync(h->oz_max.p, 0, (size_t)tiles * NC * sizeof(unsigned long long), h->stream));
  const int* ts = h->tile_seg_oz.p;
  const int* tc = h->tile_c0_oz.p;
  LAT_LAUNCH(h, k_oz_cellmax<<<dim3(tiles, std::max(1, std::min(16, div_up(n_K, 64)))), 256, 0, h->stream>>>(
                    h->n_cells, n_K, X, rdofs + r_base + lo_c, ts, tc, h->seg_ptr.p, h->perm.p, h->oz_max.p));
  LAT_LAUNCH(h, k_oz_pack<<<dim3(tiles, div_up(npan * (TK / 8), 16)), 256, 0, h->stream>>>(
                    sh, h->n_cells, kp0, npan, X, rdofs + r_base, ts, tc, h->seg_ptr.p, h->perm.p, h->oz_max.p,
                    h->oz_X.p));
  const int S = std::min(MAX_SPLIT, (int)div_up(npan, EXACT_PANELS));
  const size_t shm = (size_t)STAGES * STAGE_BYTES;
  LAT_CUDA(cudaFuncSetAttribute(k_oz_mm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(S * tiles, sh.MT - mt0);
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = shm;
  cfg.stream = h->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = S;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  LAT_LAUNCH(h, LAT_CUDA(cudaLaunchKernelEx(&cfg, k_oz_mm, sh, h->n_cells, mt0, kp0, npan, S,
                                            (const __nv_bfloat16*)T.p, (const double*)scale.p,
                                            (const __nv_bfloat16*)h->oz_X.p, (const unsigned long long*)h->oz_max.p, ts,
                                            tc, (const int*)h->seg_ptr.p, (const int*)h->perm.p,
                                            (const double*)h->c_cell.p, n_R, r_base, rdofs, (const int*)h->pdofs.p, Y,
                                            h->flag.p, mul_scale, h->wait_polls, G, ld, kstride, X, lo_c,
                                            (const uint8_t*)h->loc_fixed.p, lk)));
  LAT_CHECK_LAUNCH();
}

}  // namespace

// Whether the FP64 mode's segmented products run on digits: blocks large enough that streaming 24
// bytes per entry and the launches that split the cell vectors cost less than the FP64 pipe does
// (36 cells of the strut cell's dual block 68 us against 406, 512 cells of the whole block 0.62 ms
// against 6.0; the ring cells' dual block is 56 columns, under 10 us either way), no more columns than
// the largest cluster sums exactly in the accumulators 0 .. 7 (in the others beyond 2688 columns a sum
// of like digits may round, at 2^-68 of row maximum x vector maximum), and at most kOzBytes of
// digits (95 keys of the strut cell).  Sizes alone decide, never the memory that happens to be free: the
// same call gives the same bits beside any other allocation.
bool oz_wanted(const lat_ctx* h) {
  if (h->prec != LAT_FP64 || (int64_t)h->n_keys * 8 > h->n_cells) return false;
  const OzShape g = g_shape(h), s = s_shape(h);
  if (h->n_R - h->n_I < 512 || g.KP > MAX_SPLIT * MAX_PANELS) return false;
  const double nG = (double)h->n_keys * A_ELEMS * g.MT * g.KP, nS = (double)h->n_keys * A_ELEMS * s.MT * s.KP;
  return 2 * (nG + nS) <= kOzBytes;
}

// digits of the augmented local matrices and of the dual Schur complements (after the inversions)
void run_oz_split(lat_ctx* h) {
  const int nR = h->n_R, nP = h->n_P, nD = nR - h->n_I;
  split_matrix(h, g_shape(h), nR, (int64_t)(nR + nP) * nR, h->G.p, h->oz_G, h->oz_Gs);
  split_matrix(h, s_shape(h), nD, (int64_t)nD * nD, h->SDD.p, h->oz_S, h->oz_Ss);
}

void run_local_oz(lat_ctx* h, const double* X, double* Y, KinvMode mode) {
  const OzShape g = g_shape(h);
  product(h, g, mode == KINV_DUAL ? g.MTI : 0, mode == KINV_FULL ? 0 : g.KI, h->oz_G, h->oz_Gs, h->G.p, h->n_R,
          (int64_t)(h->n_R + h->n_P) * h->n_R, h->rdofs.p, 0, X, Y, h->n_R, 0, nullptr);
}

void run_sdd_oz(lat_ctx* h, const double* X, double* Y) {
  const int nD = h->n_R - h->n_I;
  product(h, s_shape(h), 0, 0, h->oz_S, h->oz_Ss, h->SDD.p, nD, (int64_t)nD * nD, h->rdofs.p, h->n_I, X, Y, h->n_R, 1,
          h->dual_lk.p);
}

// ------------------------------------------------------------------------------------------------
// Large symmetric inversions (gj_invert) by sweeps of 128-column panels, the rank-128 updates on digits
// ------------------------------------------------------------------------------------------------
// The sweep of a panel p (see feti.cu): C = A_.p, Pi = A_pp^{-1} by sweeps of 32 columns, R = C Pi and
// A_ij -= C_i R_j^T on the lower triangle.  Both products run on digits: C as the A operand (a row's
// digits scaled by its own maximum), the rows of Pi (symmetric) and of R as the B operand, 128
// columns at most, so base-256 digits (|s| <= 128, products up to 2^14, 8 of them over 128 columns)
// still sum exactly and what is dropped is about 2^-62 of the row maxima; base-128 digits left
// inverses of the strut cell's blocks 2.4 times further off than FP64 sweeps do.  An entry below 2^-9 of
// its row's largest in the panel has fewer bits than in FP64; the inverse does not show it, because its
// error comes from the rounding of the diagonal.  Emulated on 12 local blocks of strut and solid cells
// with graded element sizes (624 and 1464 rows, condition 7e3 to 7e6), against FP64 sweeps of 32 columns:
// error 1.06 times theirs (geometric mean; FP64 panels of 128 columns 1.03, single blocks 0.4 to 2.7 for
// both), residual A A^-1 - I 0.58 times.  Rows and columns scaled by 2^-8 to 2^8 leave that unchanged.
// An entry of A takes four FP64 operations per panel instead of 128.  Per panel: the chain of the pivot block (four 32-column steps, 26 us each), two
// products and the splitting of C, Pi and R.  Three 2616 matrices: 9 ms against 53 ms.
namespace {

constexpr int SD = 8;                      // digits, base 256
constexpr int SW = kSweepPanel;
constexpr int SP = SW / TK;                // K panels
constexpr int SN = 32;                     // columns of a product's tile
constexpr int SA_ELEMS = SD * A_SLICE;     // 32 KiB
constexpr int SB_ELEMS = SD * SN * TK;     // 8 KiB
constexpr int SSTAGE_BYTES = 2 * (SA_ELEMS + SB_ELEMS);
constexpr int SSTAGES = 2;                 // 80 KiB, two CTAs per SM
constexpr int SCOLS = SD * SN;             // 256 tensor-memory columns

// digits of one row of a panel (128 values in shared memory, zero beyond the panel's width) by one
// warp: lane l takes the columns 4l .. 4l + 3; the row's largest magnitude goes to *mx.  base: the
// row's core-matrix position in the first panel; pstride / dstride: elements between panels / digits
__device__ __forceinline__ void row_digits(const double* v, int lane, __nv_bfloat16* base, int pstride, int dstride,
                                           unsigned long long* mx) {
  double x[4];
  unsigned long long m = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    x[q] = v[4 * lane + q];
    m = max(m, abs_bits(x[q]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) *mx = m;
  float s[4][SD];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    long long hi, lo;
    fixed_point<8 * (SD - 1)>(x[q], m, hi, lo);
    lo += hi * (1ll << 42);
#pragma unroll
    for (int i = SD - 1; i >= 0; --i) s[q][i] = (float)(i ? pop_digit<8>(lo) : (int)lo);
  }
  const int k = 4 * lane;
  __nv_bfloat16* d = base + (size_t)(k / TK) * pstride + core_off(0, k % TK);
#pragma unroll
  for (int i = 0; i < SD; ++i) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(s[0][i], s[1][i]), b = __floats2bfloat162_rn(s[2][i], s[3][i]);
    *reinterpret_cast<uint2*>(d + (size_t)i * dstride) =
        make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
  }
}

// C's digits [b][row tile][panel][digit][128 x 16] and row maxima, 32 rows per CTA (rows above the
// panel are read as columns of the lower triangle); the CTAs that hold panel rows also copy A_pp
__global__ void __launch_bounds__(256)
    k_sp_panel(int n, int64_t bs, int k0, int kw, int MT, const double* __restrict__ A, __nv_bfloat16* __restrict__ Cd,
               unsigned long long* __restrict__ cmax, double* __restrict__ P) {
  __shared__ double S[32][SW + 1];
  const int b = blockIdx.y, i0 = blockIdx.x * 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double* a = A + (size_t)b * bs;
  const bool above = i0 + 32 <= k0;
  for (int t = threadIdx.x; t < 32 * SW; t += 256) {
    const int r = above ? t % 32 : t / SW, c = above ? t / 32 : t % SW;
    const int i = i0 + r, k = k0 + c;
    const double v = i < n && c < kw ? a[(size_t)max(i, k) * n + min(i, k)] : 0.0;
    S[r][c] = v;
    if (i >= k0 && i < k0 + kw && c < kw) P[(size_t)b * SW * SW + (size_t)(i - k0) * kw + c] = v;
  }
  __syncthreads();
  for (int r = warp; r < 32; r += 8) {
    const int row = i0 + r;   // rows up to the padded tile's end have zero digits
    if (row >= MT * TM) continue;
    __nv_bfloat16* base = Cd + ((size_t)b * MT + row / TM) * SP * SA_ELEMS + core_off(row % TM, 0);
    row_digits(S[r], lane, base, SA_ELEMS, A_SLICE, cmax + (size_t)b * MT * TM + row);
  }
}

// digits of the rows of an [rows][ld] FP64 matrix (kw columns) as a B operand:
// [b][32-row tile][panel][core_off(digit * 32 + row, k)]
__global__ void __launch_bounds__(256)
    k_sp_rows(int rows, int ld, int64_t bs, int kw, int NT, const double* __restrict__ X, __nv_bfloat16* __restrict__ Xd,
              unsigned long long* __restrict__ xmax) {
  __shared__ double S[8][SW];
  const int b = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = blockIdx.x * 8 + warp;
  for (int c = lane; c < SW; c += 32) S[warp][c] = row < rows && c < kw ? X[(size_t)b * bs + (size_t)row * ld + c] : 0.0;
  __syncwarp();
  if (row >= NT * SN) return;
  __nv_bfloat16* base = Xd + ((size_t)b * NT + row / SN) * SP * SB_ELEMS + core_off(row % SN, 0);
  row_digits(S[warp], lane, base, SB_ELEMS, SN * TK, xmax + (size_t)b * NT * SN + row);
}

// One 128 x 32 tile of C B^T.  UPDATE: A_ij -= (C R^T)_ij on the lower triangle, A_ip = R_i, A_pp =
// -Pi; else: R = C Pi (B the rows of Pi).
template <bool UPDATE>
__global__ void __launch_bounds__(128, 2)
    k_sp_mm(int n, int64_t bs, int k0, int kw, int MT, int NT, const __nv_bfloat16* __restrict__ Cd,
            const unsigned long long* __restrict__ cmax, const __nv_bfloat16* __restrict__ Bd,
            const unsigned long long* __restrict__ bmax, const double* __restrict__ P, double* __restrict__ R,
            double* __restrict__ A, int* __restrict__ err, int polls) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[SSTAGES], empty[SSTAGES], done;
  __shared__ uint32_t tmem_slot;
  __shared__ int fail, issued;   // a wait gave up; panels whose copies were issued
  __shared__ double cs[SN];
  const int tid = threadIdx.x, warp = tid >> 5, b = blockIdx.y;
  int mt, nt;
  if (UPDATE) {   // lower tiles: 4 (mt + 1) column tiles per row tile
    mt = (int)((sqrtf(2.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
    while (2 * (mt + 1) * (mt + 2) <= (int)blockIdx.x) ++mt;
    while (2 * mt * (mt + 1) > (int)blockIdx.x) --mt;
    nt = (int)blockIdx.x - 2 * mt * (mt + 1);
  } else {
    mt = blockIdx.x / NT;
    nt = blockIdx.x % NT;
  }
  if (nt >= NT) return;
  const int np = (kw + TK - 1) / TK;
  const uint32_t s0 = smem_u32(smem);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(SCOLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int s = 0; s < SSTAGES; ++s) {
      mbar_init(smem_u32(&full[s]));
      mbar_init(smem_u32(&empty[s]));
    }
    mbar_init(smem_u32(&done));
    fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  if (tid == 0) {
    int n = 0;
    bool ok = true;
    for (int p = 0; p < np; ++p) {
      const int st = p % SSTAGES;
      if (p >= SSTAGES && !mbar_wait(smem_u32(&empty[st]), (uint32_t)((p / SSTAGES - 1) & 1), polls)) {
        ok = false;
        break;
      }
      const uint32_t bar = smem_u32(&full[st]), dst = s0 + (uint32_t)(st * SSTAGE_BYTES);
      expect_tx(bar, (uint32_t)SSTAGE_BYTES);
      bulk_copy(dst, Cd + (((size_t)b * MT + mt) * SP + p) * SA_ELEMS, 2 * SA_ELEMS, bar);
      bulk_copy(dst + 2 * SA_ELEMS, Bd + (((size_t)b * NT + nt) * SP + p) * SB_ELEMS, 2 * SB_ELEMS, bar);
      ++n;
    }
    if (!ok) fail = 1;
    issued = n;
  } else if (tid == 32) {
    bool ok = true;
    for (int p = 0; p < np; ++p) {
      const int st = p % SSTAGES;
      if (!mbar_wait(smem_u32(&full[st]), (uint32_t)((p / SSTAGES) & 1), polls)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sa = s0 + (uint32_t)(st * SSTAGE_BYTES), sb = sa + 2 * SA_ELEMS;
#pragma unroll
      for (int i = 0; i < SD; ++i) {
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((SD - i) * SN >> 3) << 17) |
                               ((uint32_t)(TM >> 4) << 24);
        const uint32_t acc = (p > 0 || i > 0) ? 1u : 0u;
        asm volatile(
            "{\n\t.reg .pred q;\n\t"
            "setp.ne.b32 q, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, q;\n\t}" ::"r"(tmem + (uint32_t)(i * SN)),
            "l"(desc(sa + (uint32_t)(2 * i * A_SLICE))), "l"(desc(sb)), "r"(idesc), "r"(acc)
            : "memory");
      }
      mma_commit(smem_u32(&empty[st]));
    }
    mma_commit(smem_u32(&done));
    ok = mbar_wait(smem_u32(&done), 0) && ok;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (!ok) fail = 1;
  } else if (tid >= 64 && tid < 64 + SN) {
    cs[tid - 64] = digit_scale(bmax[((size_t)b * NT + nt) * SN + tid - 64]) * 0x1p-24;
  }
  __syncwarp();
  __syncthreads();
  const bool good = !fail;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!good && tid == 0) {
    atomicOr(err, kFlagProductWait);
    // copies in flight land (bounded) before the shared memory is released
    for (int q = max(0, issued - SSTAGES); q < issued; ++q)
      mbar_wait(smem_u32(&full[q % SSTAGES]), (uint32_t)((q / SSTAGES) & 1));
  }
  __syncwarp();
  if (good) {
    const uint32_t base = tmem + ((uint32_t)(warp * 32) << 16);
    const int gi = mt * TM + tid, j0 = nt * SN;
    const double rs = digit_scale(cmax[((size_t)b * MT + mt) * TM + tid]);
    double* a = A + (size_t)b * bs;
    const double* Rb = R + (size_t)b * n * SW;
    const bool ip = gi >= k0 && gi < k0 + kw;
#pragma unroll 1
    for (int c = 0; c < SN; c += 4) {
      uint32_t r[SD][4];
#pragma unroll
      for (int g = 0; g < SD; ++g) tmem_ld4(base + (uint32_t)(g * SN + c), r[g]);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double hi = combine4<8>(r[0][q], r[1][q], r[2][q], r[3][q]);
        const double lo = combine4<8>(r[4][q], r[5][q], r[6][q], r[7][q]);
        const double v = fma(lo, 0x1p-32, hi), f = rs * cs[c + q];
        const int gj = j0 + c + q;
        if (!UPDATE) {
          if (gi < n && gj < SW) R[((size_t)b * n + gi) * SW + gj] = v * f;
        } else if (gi < n && gj <= gi) {
          const bool jp = gj >= k0 && gj < k0 + kw;
          double* dst = a + (size_t)gi * n + gj;
          if (ip) *dst = jp ? -P[(size_t)b * SW * SW + (size_t)(gi - k0) * kw + (gj - k0)] : Rb[(size_t)gj * SW + (gi - k0)];
          else if (jp) *dst = Rb[(size_t)gi * SW + (gj - k0)];
          else *dst = fma(-f, v, *dst);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(SCOLS) : "memory");
  }
}

}  // namespace

// matrices of one size whose panels' workspace (run_sweep_panel) stays within 2 GB
int sweep_panel_batch(int n) {
  const double per = 2.0 * div_up(n, TM) * SP * SA_ELEMS + 2.0 * (div_up(n, SN) + SW / SN) * SP * SB_ELEMS +
                     8.0 * n * SW + 8.0 * SW * SW;
  return std::max(1, (int)(2e9 / per));
}

// one panel [k0, k0 + kw) of the sweep of `batch` n x n matrices (lower triangles)
void run_sweep_panel(lat_ctx* h, double* A, int n, int batch, int64_t bs, int k0, int kw, int neg_bit) {
  const int MT = div_up(n, TM), NT = div_up(n, SN), PT = SW / SN;
  h->sp_C.ensure((size_t)batch * MT * SP * SA_ELEMS);
  h->sp_B.ensure((size_t)batch * (NT + PT) * SP * SB_ELEMS);
  h->sp_max.ensure((size_t)batch * (MT * TM + (NT + PT) * SN));
  h->sp_P.ensure((size_t)batch * SW * SW);
  h->sp_R.ensure((size_t)batch * n * SW);
  unsigned long long* cmax = h->sp_max.p;
  unsigned long long* rmax = cmax + (size_t)batch * MT * TM;
  unsigned long long* pmax = rmax + (size_t)batch * NT * SN;
  __nv_bfloat16* Rd = h->sp_B.p;
  __nv_bfloat16* Pd = Rd + (size_t)batch * NT * SP * SB_ELEMS;
  const size_t shm = (size_t)SSTAGES * SSTAGE_BYTES;
  LAT_CUDA(cudaFuncSetAttribute(k_sp_mm<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
  LAT_CUDA(cudaFuncSetAttribute(k_sp_mm<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
  {
    KernelTimer kt(h, "gj_pivot");
    LAT_LAUNCH(h, k_sp_panel<<<dim3(MT * TM / 32, batch), 256, 0, h->stream>>>(n, bs, k0, kw, MT, A, h->sp_C.p, cmax,
                                                                              h->sp_P.p));
  }
  sweep_small(h, h->sp_P.p, kw, batch, (int64_t)SW * SW, neg_bit);
  {
    KernelTimer kt(h, "gj_pivot");
    LAT_LAUNCH(h, k_sp_rows<<<dim3(SW / 8, batch), 256, 0, h->stream>>>(kw, kw, (int64_t)SW * SW, kw, PT, h->sp_P.p, Pd,
                                                                        pmax));
    LAT_LAUNCH(h, k_sp_mm<false><<<dim3(MT * PT, batch), 128, shm, h->stream>>>(
                      n, bs, k0, kw, MT, PT, h->sp_C.p, cmax, Pd, pmax, h->sp_P.p, h->sp_R.p, A, h->flag.p,
                      h->wait_polls));
    LAT_LAUNCH(h, k_sp_rows<<<dim3(NT * SN / 8, batch), 256, 0, h->stream>>>(n, SW, (int64_t)n * SW, kw, NT, h->sp_R.p,
                                                                            Rd, rmax));
  }
  {
    KernelTimer kt(h, "gj_update");
    LAT_LAUNCH(h, k_sp_mm<true><<<dim3(2 * MT * (MT + 1), batch), 128, shm, h->stream>>>(
                      n, bs, k0, kw, MT, NT, h->sp_C.p, cmax, Rd, rmax, h->sp_P.p, h->sp_R.p, A, h->flag.p,
                      h->wait_polls));
  }
  LAT_CHECK_LAUNCH();
}
