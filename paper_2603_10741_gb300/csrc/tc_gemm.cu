// Principal-block x cell-multivector product on the 5th-generation tensor cores (tcgen05) for the
// BF16 mixed mode: the local part of K^-rom (Eq. ifetidp_precond, Section 3.3.1) for all cells,
//   Y[rows of cell s] = [G; Phi^T]_{key(s)} X_R^s,   G = (K_RR^r)^{-1} of the cell's principal,
// as a segmented GEMM over cells grouped by key: one CTA computes a tile of 128 rows x TN cells of
// one key (TN = 128 in use) with A = rows of the key's augmented matrix and B = the cells'
// remaining values, accumulating in FP32 in tensor memory.  Each operand is a BF16 pair (high part and the BF16 rounding of the
// remainder) and three products G_hi X_hi + G_hi X_lo + G_lo X_hi accumulate into the same
// tile: ~16-bit operands, which the preconditioner needs on the ill-conditioned local problems
// of the corner-only primal set (one BF16 rounding stalls FGMRES near 1e-4 there).  The
// epilogue reads the accumulators with tcgen05.ld and applies the per-cell scale 1/c_s on the G
// rows.
//
// Operand staging.  Both operands are stored in global memory already tiled in the layout the
// tensor core reads from shared memory: the canonical no-swizzle K-major layout (8-row x 16-byte
// core matrices; K-adjacent core matrices 128 B apart, 8-row groups 512 B apart), one contiguous
// 16 KiB block per (key, 128-row tile, 32-wide K panel) for A, its BF16 high part followed by the
// low part, and one block per (cell tile, K panel) for B.  A K panel is then one bulk copy per
// operand (cp.async.bulk, completing on an mbarrier with its byte count), and its three products
// cost one load of each.  One thread issues the copies (three 32 KiB stages in flight, two CTAs
// per SM), another the MMAs (M = 128, N = TN, K = 16 per instruction), two warps meanwhile fetch
// the epilogue's row, cell and scale tables.  Every wait is bounded: on a timeout the kernel flags
// an error, gives outstanding work a bounded chance to finish, frees its tensor memory and returns.
//
// Split K.  A CTA is bound by what its SM takes in (the panels of 27 columns x 64 KiB took 50 us
// whether 42 or 126 CTAs ran), so few tiles are split along K over a cluster of 2 or 4 CTAs
// (split_k below): each accumulates its share of the panels, leaves the tile in shared memory, and
// after one cluster barrier sums its share of the columns over the cluster (distributed shared
// memory, in CTA order) and stores it.
#include "common.cuh"
#include "tc_ptx.cuh"

namespace {

constexpr int TM = 128;   // rows of an M tile (tensor-memory lanes)
constexpr int TK = 32;    // K panel
constexpr int TK8 = TK / 8;
constexpr int KSTEP = 16; // K per tcgen05.mma, kind::f16
constexpr int A_ELEMS = TM * TK;       // 4096 bf16 = 8 KiB per BF16 half of an M tile and K panel
constexpr int A_BYTES = A_ELEMS * 2;
constexpr uint32_t LBO = 128;              // K-adjacent core matrices
constexpr uint32_t SBO = (TK / 8) * 128;   // 8-row groups

// per-configuration sizes: TN cells per tile
template <int TN>
struct TcCfg {
  static constexpr int B_ELEMS = TN * TK;
  static constexpr int B_BYTES = B_ELEMS * 2;
  static constexpr int STAGE_BYTES = 2 * (A_BYTES + B_BYTES);   // both BF16 halves of A and of B
  static constexpr int STAGES = 3;                              // TN = 128: 96 KiB, two CTAs per SM
  static constexpr int PART_LD = TM + 1;                        // split tile in shared memory: [TN][129]
  static constexpr size_t SMEM_BYTES = (size_t)STAGES * STAGE_BYTES;
  static_assert((size_t)TN * PART_LD * sizeof(float) <= SMEM_BYTES, "the split tile reuses the stages");
  static constexpr int TMEM_COLS = TN;   // one accumulator of TN FP32 columns
  // instruction descriptor, kind::f16: D = F32, A = B = BF16, both K-major, N >> 3, M >> 4
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) |
                                    ((uint32_t)(TM >> 4) << 24);
};

// shared-memory matrix descriptor: start, leading (K) and stride (8-row group) byte offsets,
// version 1, no swizzle
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((LBO >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((SBO >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// element (row r, k) of a K-major panel with TK columns, in bf16 elements
__host__ __device__ __forceinline__ int core_off(int r, int k) {
  return (r >> 3) * (TK / 8) * 64 + (k >> 3) * 64 + (r & 7) * 8 + (k & 7);
}

// shared-memory float of CTA `rank` of the cluster at this CTA's shared address
__device__ __forceinline__ float ld_cluster(uint32_t addr, uint32_t rank) {
  uint32_t ra;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(ra) : "memory");
  return v;
}

// Tensor-core tile: rows [128 mt, 128 (mt + 1)) of the key's view of [G; Phi^T] times the TN cells
// of tile `tile` (key-ordered positions [c0, c0 + TN)), K panels shared by the cluster's CTAs along
// x.  GT: tiled pairs [key][mt][kp][high, low][4096], XT: tiled cell vectors [tile][kp][high,
// low][TN x 32].  The products G_hi X_hi, G_hi X_lo and G_lo X_hi of a panel accumulate into the
// same tensor-memory tile.
template <int TN>
__global__ void __launch_bounds__(128, 2)
    k_local_tc(int n_cells, int n_Kr, int n_P, int MT, int KP, const __nv_bfloat16* __restrict__ GT,
               const __nv_bfloat16* __restrict__ XT, const int* __restrict__ tile_seg,
               const int* __restrict__ tile_c0, const int* __restrict__ seg_ptr, const int* __restrict__ perm,
               const double* __restrict__ cscale, const int* __restrict__ rr, const int* __restrict__ pdofs,
               double* __restrict__ Y, int* __restrict__ err, int mul_scale, int S, int polls) {
  using C = TcCfg<TN>;
  constexpr int STAGES = C::STAGES;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], done;
  __shared__ uint32_t tmem_slot;
  __shared__ int fail, issued;   // a wait gave up; panels whose copies were issued
  __shared__ int cell[TN], orow[TM];       // cell of a column (-1: past the segment), local row of a tile row
  __shared__ double fac[TN];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = blockIdx.x % S, tile = blockIdx.x / S, mt = blockIdx.y;   // a cluster: S blocks along x
  const int key = tile_seg[tile];
  const int rows = n_Kr + n_P;
  const int p0 = (int)((int64_t)KP * rank / S), np = (int)((int64_t)KP * (rank + 1) / S) - p0;
  const uint32_t s0 = smem_u32(smem);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(C::TMEM_COLS)
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
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;

  if (tid == 0) {
    // producer: panel p goes to stage p % STAGES once that stage's previous MMAs have read it
    int n = 0;
    bool ok = true;
    for (int p = 0; p < np; ++p) {
      const int st = p % STAGES;
      if (p >= STAGES && !mbar_wait(smem_u32(&empty[st]), (uint32_t)((p / STAGES - 1) & 1), polls)) {
        ok = false;
        break;
      }
      const uint32_t bar = smem_u32(&full[st]), dst = s0 + (uint32_t)(st * C::STAGE_BYTES);
      expect_tx(bar, (uint32_t)C::STAGE_BYTES);
      bulk_copy(dst, GT + (((size_t)key * MT + mt) * KP + p0 + p) * 2 * A_ELEMS, 2 * A_BYTES, bar);
      bulk_copy(dst + 2 * A_BYTES, XT + ((size_t)tile * KP + p0 + p) * 2 * C::B_ELEMS, 2 * C::B_BYTES, bar);
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
      const uint32_t sa = s0 + (uint32_t)(st * C::STAGE_BYTES), sb = sa + 2 * A_BYTES;
#pragma unroll
      for (int ks = 0; ks < TK / KSTEP; ++ks) {
        // G_hi X_hi, G_hi X_lo, G_lo X_hi (the G_lo X_lo term is below the pairs' precision)
#pragma unroll
        for (int pass = 0; pass < 3; ++pass) {
          const uint64_t ad = make_desc(sa + (pass == 2 ? A_BYTES : 0) + ks * 2 * 128);
          const uint64_t bd = make_desc(sb + (pass == 1 ? C::B_BYTES : 0) + ks * 2 * 128);
          const uint32_t acc = (p > 0 || ks > 0 || pass > 0) ? 1u : 0u;
          asm volatile(
              "{\n\t.reg .pred q;\n\t"
              "setp.ne.b32 q, %4, 0;\n\t"
              "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, q;\n\t}" ::"r"(tmem),
              "l"(ad), "l"(bd), "r"(C::IDESC), "r"(acc)
              : "memory");
        }
      }
      mma_commit(smem_u32(&empty[st]));
    }
    mma_commit(smem_u32(&done));   // arrives when every MMA issued above has completed
    // the one thread that waits for it: the others wait in the CTA barrier below (lanes that poll
    // an mbarrier beside the issuing lane of their warp take its issue slots)
    ok = mbar_wait(smem_u32(&done), 0) && ok;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (!ok) fail = 1;
  } else if (warp >= 2) {
    // the epilogue's tables, off the critical path
    const int c0 = tile_c0[tile], c_end = seg_ptr[key + 1];
    for (int c = tid - 64; c < TN; c += 64) {
      const int s = c0 + c < c_end ? perm[c0 + c] : -1;
      const double cs = s >= 0 ? cscale[s] : 1.0;
      cell[c] = s;
      fac[c] = mul_scale ? cs : 1.0 / cs;   // c_s (S_DD rows) or 1 / c_s (G rows)
    }
    for (int r = tid - 64; r < TM; r += 64) {
      const int gi = mt * TM + r;
      orow[r] = gi < n_Kr ? rr[gi] : gi < rows ? pdofs[gi - n_Kr] : -1;
    }
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
  // accumulators to shared memory (the stages are idle), [column][row] with a row of 129 floats:
  // warp w holds accumulator lanes 32w..32w+31 (tile rows)
  float* part = reinterpret_cast<float*>(smem);
  if (good) {
#pragma unroll 1
    for (int cb = 0; cb < TN; cb += 32) {
      uint32_t r[32];
      const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)cb;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
          "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
            "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
            "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
            "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
          : "r"(taddr)
          : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int j = 0; j < 32; ++j) part[(cb + j) * C::PART_LD + warp * 32 + lane] = __uint_as_float(r[j]);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  const int cw = TN / S, cb0 = rank * cw;   // this CTA's share of the columns
  if (S > 1) {
    // sums over the cluster, in place (a share is read by its owner alone), a lane per row: remote
    // reads are whole 128-byte segments (a lane per column made each of them 32 packets and this
    // sum 40 us long)
    cluster_sync();
    float* const mine = part + warp * 32 + lane;
#pragma unroll 8
    for (int c = cb0; c < cb0 + cw; ++c) {
      const uint32_t a = smem_u32(mine + c * C::PART_LD);
      float v = ld_cluster(a, 0) + ld_cluster(a, 1);
      if (S == 4) v += ld_cluster(a, 2) + ld_cluster(a, 3);
      mine[c * C::PART_LD] = v;
    }
  }
  __syncthreads();
  // stores, a lane per column: a warp writes consecutive cells of a row
  for (int cb = cb0; cb < cb0 + cw; cb += 32) {
    const int col = cb + lane, s = cell[col];
    const double f = fac[col];
#pragma unroll 8
    for (int q = 0; q < 32; ++q) {
      const int r = warp * 32 + q, o = orow[r];
      const float v = part[col * C::PART_LD + r];
      if (s >= 0 && o >= 0 && good) Y[(size_t)o * n_cells + s] = mt * TM + r < n_Kr ? (double)v * f : (double)v;
    }
  }
  if (S > 1) cluster_sync();   // peers have read this CTA's tile
  else __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM_COLS) : "memory");
  }
}

// CTAs of a cluster that share a tile's K panels: as many of 1, 2, 4 as keep every CTA resident at
// once (two per SM), at least one panel each: a second wave would cost what the split saves.
// Measured on the strut cell's dual block (1716 x 1692, cold caches): 42 tiles 48 us with one CTA
// each, 23 us split over 4; 126 tiles 50 us and 37 us split over 2.
int split_k(const lat_ctx* h, int64_t tiles, int KP) {
  for (int S : {4, 2})
    if (tiles * S <= 2 * h->n_sm && KP >= S) return S;
  return 1;
}

// BF16 pairs of eight consecutive K entries of one cell: the high parts and the BF16 roundings of
// the remainders, as the two 16-byte core-matrix rows they are stored as
__device__ __forceinline__ void split8(const float (&v)[8], uint4& hi, uint4& lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
    const float2 f = __bfloat1622float2(a);
    const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * q] - f.x, v[2 * q + 1] - f.y);
    h[q] = *reinterpret_cast<const uint32_t*>(&a);
    l[q] = *reinterpret_cast<const uint32_t*>(&b);
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// Cell vectors of every tile, BF16 pairs in the tiled layout: XT[tile][kp][high, low][core_off(c, k)],
// cell c = position c0 + c of the tile's key segment (zero past the segment's end), column
// kp * 32 + k of the view (zero beyond n_K).  A thread owns
// one cell and eight consecutive columns, i.e. one 16-byte row of a core matrix: its eight reads
// are in flight together (a warp's are 32 consecutive cells of a row), eight neighbouring threads
// store one whole 128-byte core matrix, and nothing goes through shared memory.  Bound by the
// reads' latency and L2: with a CTA per (tile, panel) and the panel staged in shared memory there
// were 243 CTAs of dependent reads on the 10^3 strut lattice, 41 us per launch against 15 us.
template <int TN>
__global__ void __launch_bounds__(TN)
    k_pack_xt(int n_cells, int n_K, int KP, const double* __restrict__ X, const int* __restrict__ tile_seg,
              const int* __restrict__ tile_c0, const int* __restrict__ seg_ptr, const int* __restrict__ perm,
              const int* __restrict__ rc, __nv_bfloat16* __restrict__ XT) {
  constexpr int BE = TN * TK;
  const int tile = blockIdx.x, kp = blockIdx.y / TK8, c = threadIdx.x;
  const int g0 = blockIdx.y * 8;                               // first column of the eight
  const int pos = tile_c0[tile] + c;
  const bool in = pos < seg_ptr[tile_seg[tile] + 1];
  const int s = in ? perm[pos] : 0;
  float v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = in && g0 + q < n_K ? (float)X[(size_t)rc[g0 + q] * n_cells + s] : 0.f;
  uint4 hi, lo;
  split8(v, hi, lo);
  __nv_bfloat16* dst = XT + ((size_t)tile * KP + kp) * 2 * BE + core_off(c, (blockIdx.y % TK8) * 8);
  *reinterpret_cast<uint4*>(dst) = hi;
  *reinterpret_cast<uint4*>(dst + BE) = lo;
}

// the same tiles for an operand supported on the dual DOFs and given as B^T lambda (scaled by
// 1/multiplicity when lsc is given): each copy's value is formed from its multipliers through
// the per-(dual DOF, cell) table instead of being scattered into a zeroed local vector first.
// Formed in FP32 (the value is rounded to FP32 and split into a BF16 pair anyway): only the two
// multiplier reads convert from FP64, the FP64 pipe being the narrow one here.
template <int TN>
__global__ void __launch_bounds__(TN)
    k_pack_lam(int n_cells, int n_D, int KP, const double* __restrict__ lam, const int2* __restrict__ lk,
               const float* __restrict__ lsc, const int* __restrict__ tile_seg, const int* __restrict__ tile_c0,
               const int* __restrict__ seg_ptr, const int* __restrict__ perm, __nv_bfloat16* __restrict__ XT) {
  constexpr int BE = TN * TK;
  const int tile = blockIdx.x, kp = blockIdx.y / TK8, c = threadIdx.x;
  const int g0 = blockIdx.y * 8;
  const int pos = tile_c0[tile] + c;
  const bool in = pos < seg_ptr[tile_seg[tile] + 1];
  const int s = in ? perm[pos] : 0;
  int2 l[8];
  float sc[8], v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const bool ok = in && g0 + q < n_D;
    const size_t e = (size_t)(g0 + q) * n_cells + s;
    l[q] = ok ? lk[e] : make_int2(0, 0);
    sc[q] = ok && lsc ? lsc[e] : 1.f;
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    float a = 0.f;
    if (l[q].x) a = l[q].x > 0 ? __double2float_rn(lam[l[q].x - 1]) : -__double2float_rn(lam[-l[q].x - 1]);
    if (l[q].y) a += l[q].y > 0 ? __double2float_rn(lam[l[q].y - 1]) : -__double2float_rn(lam[-l[q].y - 1]);
    v[q] = a * sc[q];
  }
  uint4 hi, lo;
  split8(v, hi, lo);
  __nv_bfloat16* dst = XT + ((size_t)tile * KP + kp) * 2 * BE + core_off(c, (blockIdx.y % TK8) * 8);
  *reinterpret_cast<uint4*>(dst) = hi;
  *reinterpret_cast<uint4*>(dst + BE) = lo;
}

// a view of G (rows_v rows of n_K columns from (G, row stride ldsrc, key stride kstride)) as BF16
// pairs in the tiled layout: GT[key][mt][kp][high, low][core_off(r, k)], low part = the BF16
// rounding of G - hi; zero outside the view
__global__ void k_g_tile(int64_t keys, int rows_v, int n_K, int MT, int KP, int ldsrc, int64_t kstride,
                         const double* __restrict__ G, __nv_bfloat16* __restrict__ GT) {
  const int64_t n = keys * MT * KP * A_ELEMS;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int64_t blk = t / A_ELEMS;
  const int e = (int)(t % A_ELEMS);
  // invert core_off: e = (r >> 3) * 8 TK + (k >> 3) * 64 + (r & 7) * 8 + (k & 7)
  const int r = e / (8 * TK) * 8 + ((e >> 3) & 7);
  const int k = (e / 64) % TK8 * 8 + (e & 7);
  const int kp = (int)(blk % KP);
  const int64_t mk = blk / KP;
  const int mt = (int)(mk % MT);
  const int64_t key = mk / MT;
  const int gr = mt * TM + r, gk = kp * TK + k;
  const float v = (gr < rows_v && gk < n_K) ? (float)G[key * kstride + (int64_t)gr * ldsrc + gk] : 0.f;
  const __nv_bfloat16 h = __float2bfloat16(v);
  GT[blk * 2 * A_ELEMS + e] = h;
  GT[blk * 2 * A_ELEMS + A_ELEMS + e] = __float2bfloat16(v - __bfloat162float(h));
}

}  // namespace

// BF16 pairs of the augmented local matrices (after the FP64 Gauss-Jordan sweep) for the three
// views of the local products (whole; dual columns; trailing dual block), tiled for the bulk
// copies of the tensor-core kernel
void run_g_to_bf16(lat_ctx* h, size_t n) {
  const int nR = h->n_R, nP = h->n_P, nI = h->n_I;
  const int64_t keys = (int64_t)(n / ((size_t)(nR + nP) * nR));
  const int64_t kstride = (int64_t)(nR + nP) * nR;
  for (int mode = 0; mode < 3; ++mode) {
    const int lo_r = mode == KINV_DUAL ? nI : 0, lo_c = mode == KINV_FULL ? 0 : nI;
    const int nKr = nR - lo_r, nKc = nR - lo_c;
    const int MT = div_up(nKr + nP, TM), KP = std::max(1, div_up(nKc, TK));
    const int64_t cnt = keys * MT * KP * A_ELEMS;
    h->G16[mode].ensure((size_t)2 * cnt);   // high and low parts
    h->g16_ld[mode] = KP;
    LAT_LAUNCH(h, k_g_tile<<<div_up(cnt, 256), 256, 0, h->stream>>>(keys, nKr + nP, nKc, MT, KP, nR, kstride,
                                                                      h->G.p + (size_t)lo_r * nR + lo_c, h->G16[mode].p));
  }
  // the dual Schur complements S_DD [keys][n_D][n_D] of the Dirichlet interface preconditioner
  const int nD = nR - nI;
  if (nD > 0 && h->SDD.p) {
    const int MT = div_up(nD, TM), KP = std::max(1, div_up(nD, TK));
    const int64_t cnt = keys * MT * KP * A_ELEMS;
    h->G16[3].ensure((size_t)2 * cnt);
    h->g16_ld[3] = KP;
    LAT_LAUNCH(h, k_g_tile<<<div_up(cnt, 256), 256, 0, h->stream>>>(keys, nD, nD, MT, KP, nD, (int64_t)nD * nD,
                                                                      h->SDD.p, h->G16[3].p));
  }
  LAT_CHECK_LAUNCH();
}

namespace {

// the product of a tiled matrix (MT row tiles per key, KP panels) with the packed cell tiles
void launch_tc(lat_ctx* h, int n_Kr, int n_P, int MT, int KP, const __nv_bfloat16* G, const int* rr, double* Y,
               int mul_scale) {
  using C = TcCfg<kTcCells>;
  auto kern = k_local_tc<kTcCells>;
  LAT_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM_BYTES));
  const int S = split_k(h, (int64_t)h->max_tiles_tc * MT, KP);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(S * h->max_tiles_tc, MT);
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = C::SMEM_BYTES;
  cfg.stream = h->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = S;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  LAT_LAUNCH(h, LAT_CUDA(cudaLaunchKernelEx(&cfg, kern, h->n_cells, n_Kr, n_P, MT, KP, G,
                                            (const __nv_bfloat16*)h->Xb16.p, (const int*)h->tile_seg_tc.p,
                                            (const int*)h->tile_c0_tc.p, (const int*)h->seg_ptr.p,
                                            (const int*)h->perm.p, (const double*)h->c_cell.p, rr,
                                            (const int*)h->pdofs.p, Y, h->flag.p, mul_scale, S, h->wait_polls)));
  LAT_CHECK_LAUNCH();
}

// cell operand of a product with K columns from the remaining DOF position lo_c on: the local
// vector X, or B^T lam (scaled by lsc) on the dual DOFs
void pack_tc(lat_ctx* h, const double* X, const double* lam, const float* lsc, int lo_c, int KP) {
  const int n_K = h->n_R - lo_c;
  const int KPmax = std::max(1, div_up(h->n_R, TK));
  h->Xb16.ensure((size_t)h->max_tiles_tc * 2 * KPmax * TcCfg<kTcCells>::B_ELEMS);
  const dim3 grid(h->max_tiles_tc, KP * TK8);
  if (lam)
    LAT_LAUNCH(h, k_pack_lam<kTcCells><<<grid, kTcCells, 0, h->stream>>>(h->n_cells, n_K, KP, lam, h->dual_lk.p, lsc,
                                                                         h->tile_seg_tc.p, h->tile_c0_tc.p,
                                                                         h->seg_ptr.p, h->perm.p, h->Xb16.p));
  else
    LAT_LAUNCH(h, k_pack_xt<kTcCells><<<grid, kTcCells, 0, h->stream>>>(h->n_cells, n_K, KP, X, h->tile_seg_tc.p,
                                                                        h->tile_c0_tc.p, h->seg_ptr.p, h->perm.p,
                                                                        h->rdofs.p + lo_c, h->Xb16.p));
  LAT_CHECK_LAUNCH();
}

}  // namespace

// Y (rows of every cell, per the view: see KinvMode) = [G; Phi^T] X on the tensor cores, on
// 128-cell tiles of each key's cells; with lam the operand is B^T lam (mode KINV_DUAL: the view's
// columns are the dual DOFs)
void run_local_tc(lat_ctx* h, const double* X, double* Y, KinvMode mode, const double* lam) {
  const int lo_r = mode == KINV_DUAL ? h->n_I : 0, lo_c = mode == KINV_FULL ? 0 : h->n_I;
  const int nKr = h->n_R - lo_r;
  pack_tc(h, X, lam, nullptr, lo_c, h->g16_ld[mode]);
  static const char* const tg[3] = {"local_tc", "local_tc_dual", "local_tc_dual_in"};
  KernelTimer kt(h, tg[mode]);
  launch_tc(h, nKr, h->n_P, div_up(nKr + h->n_P, TM), h->g16_ld[mode], h->G16[mode].p, h->rdofs.p + lo_r, Y, 0);
}

// the Dirichlet interface preconditioner's local products y_D = c_s S_DD B_D^T lam on the same
// tiles (dual rows and columns, no corner rows, scaled by c_s)
void run_sdd_tc(lat_ctx* h, const double* lam, double* Y) {
  const int nD = h->n_R - h->n_I;
  pack_tc(h, nullptr, lam, h->dual_lsc.p, h->n_I, h->g16_ld[3]);
  KernelTimer kt(h, "dual_schur_tc");
  launch_tc(h, nD, 0, div_up(nD, TM), h->g16_ld[3], h->G16[3].p, h->rdofs.p + h->n_I, Y, 1);
}
