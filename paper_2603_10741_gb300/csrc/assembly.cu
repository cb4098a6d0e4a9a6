// Per-cell residual and tangent evaluation at quadrature points, the matrix-free exact tangent
// action, the mu-derivative of the internal force, the local-to-global scatter and FP64 norms.
//
// A cell's displacements are gathered into shared memory through the Boolean map A^s (Eq.
// residualvector).  All of it is FP64, and FP64 runs at two lanes per clock per SM, so the kernels
// are laid out to issue few FP64 instructions and none for idle lanes:
//   * residual and exact tangent action: a lane per quadrature point, the 2^d lanes of an element
//     exchanging values by shuffles.  Node and point share the lane's index bits, and the
//     displacement gradient and the nodal forces come from butterflies over those bits (the Q1
//     monomials), 54 + 72 FP64 operations per point in 3D instead of the 72 + 96 of sums over the
//     element's nodes.  Element forces are staged in shared memory and summed per node in element
//     order: no colours, no atomics, deterministic.
//   * tangent: kinematics once per point, then a lane per node pair a <= b (K_ab and its transpose),
//     element colour by colour, so that a colour's elements never touch the same node block.
//
// Kinematics and stress use the first Piola-Kirchhoff form of the neo-Hookean law of
// Eq. (sig_eq): with F = I + sum_a u_a (x) grad_X phi_a (Section 3.1.3), J = det F,
//   P = J sigma F^{-T} = mu (F - F^{-T}) + lam ln J F^{-T},
//   f_a = sum_q W_q P grad_X phi_a                 (Eq. internalloadvec pulled back, dx = J dX)
// and the tangent of Section 3.1.4 pulled back to the reference cell (Eq. stiffmatPulledback):
//   K_ab = sum_q W_q [ mu (g_a . g_b) I + lam h_a h_b^T + (mu - lam ln J) h_b h_a^T ],
//   g = grad_X phi, h = F^{-T} g = grad_x phi,
// which equals the contraction of D_ijkl = C_ikjl + delta_ij sigma_kl (Eq. const_eq) with
// grad_x phi_a (x) grad_x phi_b times J.
#include <cfloat>

#include "common.cuh"

namespace {

constexpr int kCellThreads = 256;

struct GeomArgs {
  const double* gradX;   // [n_el][nq][nen][D]
  const double* W;       // [n_el][nq]
  const int* elems;      // [n_el][nen]
  const int* color_elems;
  int nq;
  const double* gram;    // [n_el][pairs a <= b, a-major] sum_q W g_a.g_b
};

__device__ __forceinline__ void load_cell_u(const double* __restrict__ u_glob,
                                            const int* __restrict__ cnodes, int nn, int D,
                                            double* __restrict__ u_loc) {
  for (int k = threadIdx.x; k < nn * D; k += blockDim.x) {
    int a = k / D, i = k - a * D;
    u_loc[k] = u_glob[(int64_t)cnodes[a] * D + i];
  }
}

// --- Q1 butterflies over the lanes of an element -----------------------------------------------
// Lane bits (b_x, b_y[, b_z]) name both the node (b = 1: the + side) and the Gauss point (b = 1:
// +1/sqrt 3) of the lane.  With u(xi) = 2^-d sum_m c_m xi^m, m in {0,1}^d, c the Walsh-Hadamard
// transform of the nodal values, the reference derivatives at the point are sums of c_m over the
// bits other than the derivative's; the nodal forces are the transpose.  The factor 2^-d sits in
// the J0^{-1} table (an exact scaling).  Shuffles stay inside the 2^d lanes; every lane of the warp
// takes part.
template <int D>
struct LaneQ1 {
  bool b[D];
  double sg[D];   // +-1/sqrt 3 of the lane's point
  double sb[D];   // +1 (b = 0), -1 (b = 1)
  double sc[D];   // transpose: factor of the derivative's monomials, 0 where the lane has none
  __device__ __forceinline__ explicit LaneQ1(int lane) {
    const double g = 0.57735026918962576451;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      b[k] = (lane >> k) & 1;
      sg[k] = b[k] ? g : -g;
      sb[k] = b[k] ? -1.0 : 1.0;
    }
#pragma unroll
    for (int d = 0; d < D; ++d) {
      double v = b[d] ? 1.0 : 0.0;
#pragma unroll
      for (int k = 0; k < D; ++k)
        if (k != d && b[k]) v *= g;
      sc[d] = v;
    }
  }
  // local node of the lane in the element's order (counter-clockwise, bottom face then top face)
  __device__ __forceinline__ int node() const {
    int n = b[1] ? (b[0] ? 2 : 3) : (b[0] ? 1 : 0);
    if (D == 3) n += b[D - 1] ? 4 : 0;
    return n;
  }
  // nodal value of the lane's node -> the reference derivatives at the lane's point, times 2^d
  __device__ __forceinline__ void gradient(double v, int lane, double (&du)[D]) const {
#pragma unroll
    for (int k = 0; k < D; ++k) v = fma(sb[k], __shfl_xor_sync(0xffffffffu, v, 1 << k), v);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      double w = __shfl_sync(0xffffffffu, v, lane | (1 << d));
#pragma unroll
      for (int k = 0; k < D; ++k) {
        if (k == d) continue;
        const double p = __shfl_xor_sync(0xffffffffu, w, 1 << k);
        w = fma(sg[k], b[k] ? w : p, b[k] ? p : w);
      }
      du[d] = w;
    }
  }
  // coefficients of the reference derivatives at the lane's point -> force on the lane's node,
  // summed over the element's points, times 2^d
  __device__ __forceinline__ double force(const double (&q)[D]) const {
    double r = 0.0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      double t = q[d];
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const double p = __shfl_xor_sync(0xffffffffu, t, 1 << k);
        t = k == d ? t + p : fma(sb[k], p, t);
      }
      r = fma(sc[d], t, r);
    }
#pragma unroll
    for (int k = 0; k < D; ++k) r = fma(-sb[k], __shfl_xor_sync(0xffffffffu, r, 1 << k), r);
    return r;
  }
};

struct LaneArgs {
  int n_el, EB;                 // elements, elements staged at a time
  const double* Ji;             // [n_el][2^D][D*D]  2^-d (J0^{-1})_dk at the full rule's points
  const double* W;              // [n_el][2^D]
  const int* elems;
  const int* node_ptr;          // [nn + 1] into node_src
  const int* node_src;          // element * 2^D + local node of every element at the node, ascending
};

// sum of the staged element forces of elements [e0, e1) into the cell's column of f_cells
template <int D>
__device__ __forceinline__ void gather_forces(const LaneArgs& g, int nn, int n_cells, int s, int e0, int e1,
                                              const double* fes, double* __restrict__ f_cells) {
  constexpr int NEN = 1 << D;
  for (int k = threadIdx.x; k < nn * D; k += blockDim.x) {
    const int a = k / D, i = k - a * D;
    double v = 0.0;
    for (int c = g.node_ptr[a]; c < g.node_ptr[a + 1]; ++c) {
      const int src = g.node_src[c], e = src / NEN;
      if (e >= e0 && e < e1) v += fes[(size_t)(src - e0 * NEN) * D + i];
    }
    double* dst = f_cells + (size_t)k * n_cells + s;
    *dst = e0 == 0 ? v : *dst + v;
  }
}

// ---------------------------------------------------------------------------------------------
// residual: f^{int,s} for every cell, cell-stacked output [n_loc][n_cells].  Bound by the FP64
// pipe: about 220 operations per point.  1287 strut cells (3.5 M points): 1.43 ms (1.24 ms at two
// FP64 lanes per clock) against 4.93 ms for a thread per element working colour by colour (43 of 256 threads busy, 307
// operations per point).
// ---------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(kCellThreads)
    k_residual(int n_cells, int nn, LaneArgs g, const int* __restrict__ cell_nodes,
               const double* __restrict__ mu_cell, double mu_override, double lam,
               const double* __restrict__ u_glob, double* __restrict__ f_cells,
               double* __restrict__ minJ_cell) {
  constexpr int NEN = 1 << D;
  extern __shared__ double sm[];
  double* u_loc = sm;
  double* fes = sm + nn * D;    // [EB][NEN][D]
  __shared__ double red[32];
  const int s = blockIdx.x, lane = threadIdx.x & 31;
  load_cell_u(u_glob, cell_nodes + (size_t)s * nn, nn, D, u_loc);
  __syncthreads();
  const double mu = mu_override >= 0 ? mu_override : mu_cell[s];
  const LaneQ1<D> L(lane & (NEN - 1));
  const int node = L.node(), q = lane & (NEN - 1);
  double minJ = DBL_MAX;
  for (int e0 = 0; e0 < g.n_el; e0 += g.EB) {
    const int ne = min(g.EB, g.n_el - e0);
    for (int t0 = threadIdx.x - lane; t0 < ne * NEN; t0 += blockDim.x) {
      const int el = (t0 + lane) / NEN;
      const bool live = el < ne;
      const int e = e0 + min(el, ne - 1);
      const int nd = g.elems[e * NEN + node];
      double Ji[D][D], du[D][D], F[D][D], C[D][D];
#pragma unroll
      for (int d = 0; d < D; ++d)
#pragma unroll
        for (int k = 0; k < D; ++k) Ji[d][k] = g.Ji[((size_t)e * NEN + q) * D * D + d * D + k];
      const double w = g.W[e * NEN + q];
#pragma unroll
      for (int i = 0; i < D; ++i) L.gradient(u_loc[nd * D + i], lane, du[i]);
#pragma unroll
      for (int i = 0; i < D; ++i)
#pragma unroll
        for (int k = 0; k < D; ++k) {
          double v = (i == k) ? 1.0 : 0.0;
#pragma unroll
          for (int d = 0; d < D; ++d) v = fma(du[i][d], Ji[d][k], v);
          F[i][k] = v;
        }
      const double J = det_cof<D>(F, C);
      if (live) minJ = fmin(minJ, J);
      const double lnJ = J > 0 ? log(J) : 0.0;
      // P = w (mu F + (lam ln J - mu) F^{-T}),  F^{-T} = cof F / J
      const double cm = w * mu, cf = fma(w * lam, lnJ, -cm) / J;
      double fe[D];
#pragma unroll
      for (int i = 0; i < D; ++i) {
        double P[D], Q[D];
#pragma unroll
        for (int k = 0; k < D; ++k) P[k] = fma(cm, F[i][k], cf * C[i][k]);
#pragma unroll
        for (int d = 0; d < D; ++d) {
          double v = 0.0;
#pragma unroll
          for (int k = 0; k < D; ++k) v = fma(P[k], Ji[d][k], v);
          Q[d] = v;
        }
        fe[i] = L.force(Q);
      }
      if (live)
#pragma unroll
        for (int i = 0; i < D; ++i) fes[(size_t)(el * NEN + node) * D + i] = fe[i];
    }
    __syncthreads();
    gather_forces<D>(g, nn, n_cells, s, e0, e0 + ne, fes, f_cells);
    __syncthreads();
  }
  minJ = -block_max(-minJ, red);
  if (threadIdx.x == 0 && minJ_cell) minJ_cell[s] = minJ;
}

// ---------------------------------------------------------------------------------------------
// tangent: K^s on the shared pattern for a list of cells, [n_sel][nnz].  Per batch of a colour's
// elements (EB at most), a thread per quadrature point leaves h_a = F^{-T} grad phi_a of all its
// nodes in shared memory, once as it is and once times each of its two weights; then a thread per
// (element, node pair a <= b) sums its block over the points and writes K_ab and K_ba = K_ab^T.  The
// mu term's sum_q W g_a.g_b does not depend on the state: one table entry per pair (gram).  The first element to touch a block
// (in colour order; kFirst in elem_blk) stores it, later ones add, so K is not cleared first.  A
// cell is worked on by a cluster of CL CTAs that share each colour's batches and meet at a cluster
// barrier between colours: with few cells (the principals) one CTA each would leave the GPU idle
// (3 strut cells took 3.4 ms).
//
// Bound by the FP64 pipe (18 operations per pair and point in 3D, 8 in 2D).  1024 ring cells: 0.45 ms,
// 0.51 with the weights and g_a.g_b applied per pair and point, 1.35 when a thread per element row
// also repeated the kinematics; one strut principal: 0.3 ms, before 3.4.
// ---------------------------------------------------------------------------------------------
constexpr int kFirst = 1 << 30;

// smem of one element of a batch: [nq] rows of h, lam w h, (mu - lam ln J) w h (an odd length: a
// thread's row, conflict-free stores)
template <int D>
__host__ __device__ constexpr int tangent_row() { return 3 * (1 << D) * D + 1; }

template <int D>
__global__ void __launch_bounds__(kCellThreads)
    k_tangent(int nn, GeomArgs g, ColorTable ct, const int* __restrict__ cell_nodes,
              const int* __restrict__ cells, const int* __restrict__ elem_blk,
              const double* __restrict__ mu_cell, double lam, const double* __restrict__ u_glob,
              int64_t nnz, double* __restrict__ K_out, double* __restrict__ minJ_out, int geo, int EB, int CL,
              int staged) {
  constexpr int NEN = 1 << D, NP = NEN * (NEN + 1) / 2, ND = NEN * D, HS = tangent_row<D>();
  extern __shared__ double sm[];
  const int nq = g.nq;
  double* hs = sm;                          // [EB][nq][HS]
  double* u_loc = hs + (size_t)EB * nq * HS; // [nn * D] when staged
  __shared__ double red[32];
  __shared__ unsigned char pa[NP], pb[NP];
  const int si = blockIdx.x / CL, rank = blockIdx.x % CL;
  const int s = cells ? cells[si] : si;
  const int* cn = cell_nodes + (size_t)s * nn;
  if (threadIdx.x < NEN)
    for (int b = threadIdx.x, at = 0; b < NEN; ++b) {   // pair (a, b): a-major
      at = threadIdx.x * NEN - threadIdx.x * (threadIdx.x - 1) / 2 + b - threadIdx.x;
      pa[at] = (unsigned char)threadIdx.x;
      pb[at] = (unsigned char)b;
    }
  if (staged) load_cell_u(u_glob, cn, nn, D, u_loc);
  __syncthreads();
  const double mu = mu_cell[s];
  double* K = K_out + (size_t)si * nnz;
  double minJ = DBL_MAX;
  for (int c = 0; c < ct.n; ++c) {
    for (int b0 = ct.start[c] + rank * EB; b0 < ct.start[c + 1]; b0 += CL * EB) {
      const int ne = min(EB, ct.start[c + 1] - b0);
      for (int t = threadIdx.x; t < ne * nq; t += blockDim.x) {
        const int el = t / nq, q = t - el * nq;
        const int e = g.color_elems[b0 + el];
        const double* gq = g.gradX + ((size_t)(e * nq + q) * NEN) * D;
        double F[D][D], Fi[D][D];
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
          for (int k = 0; k < D; ++k) F[i][k] = (i == k) ? 1.0 : 0.0;
#pragma unroll
        for (int b = 0; b < NEN; ++b) {
          const int nd = g.elems[e * NEN + b];
          const double* ub = staged ? u_loc + nd * D : u_glob + (int64_t)cn[nd] * D;
#pragma unroll
          for (int i = 0; i < D; ++i)
#pragma unroll
            for (int k = 0; k < D; ++k) F[i][k] = fma(ub[i], gq[b * D + k], F[i][k]);
        }
        const double J = det_inv<D>(F, Fi);
        minJ = fmin(minJ, J);
        const double lnJ = J > 0 ? log(J) : 0.0;
        const double w = g.W[e * nq + q];
        const double cl = w * lam, cg = w * (mu - lam * lnJ);
        double* ht = hs + (size_t)t * HS;
#pragma unroll
        for (int a = 0; a < NEN; ++a)
#pragma unroll
          for (int i = 0; i < D; ++i) {
            double v = 0;
#pragma unroll
            for (int k = 0; k < D; ++k) v = fma(Fi[k][i], gq[a * D + k], v);
            ht[a * D + i] = v;
            ht[ND + a * D + i] = cl * v;
            ht[2 * ND + a * D + i] = cg * v;
          }
      }
      __syncthreads();
      for (int t = threadIdx.x; t < ne * NP; t += blockDim.x) {
        const int el = t / NP, pr = t - el * NP;
        const int a = pa[pr], b = pb[pr];
        const int e = g.color_elems[b0 + el];
        double acc[D][D];
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
          for (int j = 0; j < D; ++j) acc[i][j] = 0.0;
        double dg = 0.0;
        for (int q = 0; q < nq; ++q) {
          const double* ht = hs + (size_t)(el * nq + q) * HS;
          double la[D], ga[D], hb[D];
#pragma unroll
          for (int i = 0; i < D; ++i) {
            la[i] = ht[ND + a * D + i];
            ga[i] = ht[2 * ND + a * D + i];
            hb[i] = ht[b * D + i];
          }
#pragma unroll
          for (int i = 0; i < D; ++i)
#pragma unroll
            for (int j = 0; j < D; ++j) acc[i][j] = fma(la[i], hb[j], fma(hb[i], ga[j], acc[i][j]));
          if (!geo)
#pragma unroll
            for (int k = 0; k < D; ++k) dg = fma(ga[k], hb[k], dg);
        }
        // diagonal term: mu g_a.g_b holds the geometric part delta_ij J h_a^T sigma h_b =
        // mu (g_a.g_b - h_a.h_b) + lam ln J h_a.h_b; without it (geo = 0) what remains is the
        // material part, the contraction of C_ikjl alone: (mu - lam ln J) h_a.h_b
        if (geo) dg = mu * g.gram[(size_t)e * NP + pr];
#pragma unroll
        for (int i = 0; i < D; ++i) acc[i][i] += dg;
        const int ab = elem_blk[(e * NEN + a) * NEN + b], ba = elem_blk[(e * NEN + b) * NEN + a];
        double* Kab = K + (size_t)(ab & (kFirst - 1)) * D * D;
        double* Kba = K + (size_t)(ba & (kFirst - 1)) * D * D;
        const bool first = ab & kFirst;
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
          for (int j = 0; j < D; ++j) {
            Kab[i * D + j] = first ? acc[i][j] : Kab[i * D + j] + acc[i][j];
            if (a != b) Kba[j * D + i] = first ? acc[i][j] : Kba[j * D + i] + acc[i][j];
          }
      }
      __syncthreads();
    }
    if (CL > 1) {
      // the next colour's elements add to blocks that other CTAs of the cluster wrote
      __syncwarp();
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
  }
  if (minJ_out) {
    minJ = -block_max(-minJ, red);
    if (threadIdx.x == 0) minJ_out[blockIdx.x] = minJ;
  }
}

// ---------------------------------------------------------------------------------------------
// D^ref snapshots (the Remark after Eq. snapshots): the pulled-back tangent tensor of Eq.
// (tensorfunctionPulledback) at the one-point rule of every element,
//   D^ref_ijmn = |det J| sum_kl D_ijkl G_mk G_nl,   G = J^{-1}, J = dx/dxi = F J0,
//   D_ijkl = C_ikjl + delta_ij sigma_kl  (Eq. const_eq, Section 3.1.4), which expands to
//   D^ref_ijmn = |det J| [lam/J G_mi G_nj + c (delta_ij (G G^T)_mn + G_mj G_ni)
//                         + delta_ij (G sigma G^T)_mn],   c = (mu - lam ln J) / J.
// J0^{-1} follows from the reference gradients at the centre: the Q1 corner signs xi_a satisfy
// sum_a xi_a,m xi_a,m' = 2^d delta, so (J0^{-1})_mk = sum_a xi_a,m dphi_a/dX_k.  A thread per
// (cell, element); output [n_cells][n_el * d^4], entries (element, i, j, m, n) last fastest.
// ---------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(128)
    k_dref(int n_cells, int n_el, int nn, GeomArgs g, const int* __restrict__ cell_nodes,
           const double* __restrict__ mu_cell, double lam, const double* __restrict__ u_glob,
           double* __restrict__ T, double* __restrict__ minJ_cell) {
  constexpr int NEN = 1 << D;
  constexpr int D4 = D * D * D * D;
  const int s = blockIdx.y;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  __shared__ double red[32];
  double myJ = DBL_MAX;
  if (e < n_el) {
    const int* cn = cell_nodes + (size_t)s * nn;
    const double* gq = g.gradX + (size_t)e * NEN * D;   // one point per element
    double F[D][D], Fi[D][D], Ji0[D][D];
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int k = 0; k < D; ++k) {
        F[i][k] = (i == k) ? 1.0 : 0.0;
        Ji0[i][k] = 0.0;
      }
#pragma unroll
    for (int a = 0; a < NEN; ++a) {
      const int node = g.elems[e * NEN + a];
      const int64_t gn = cn[node];
      // Q1 corner a in the counter-clockwise / bottom-then-top order: signs of xi_a
      const double sx = ((a & 3) == 1 || (a & 3) == 2) ? 1.0 : -1.0;
      const double sy = ((a & 3) >= 2) ? 1.0 : -1.0;
      const double sz = a >= 4 ? 1.0 : -1.0;
      const double sg[3] = {sx, sy, sz};
#pragma unroll
      for (int i = 0; i < D; ++i) {
        const double ui = u_glob[gn * D + i];
#pragma unroll
        for (int k = 0; k < D; ++k) F[i][k] += ui * gq[a * D + k];
      }
#pragma unroll
      for (int m = 0; m < D; ++m)
#pragma unroll
        for (int k = 0; k < D; ++k) Ji0[m][k] += sg[m] * gq[a * D + k];
    }
    const double J = det_inv<D>(F, Fi);
    myJ = J;
    const double lnJ = J > 0 ? log(J) : 0.0;
    const double mu = mu_cell[s];
    const double detJ0 = g.W[e] / (double)(1 << D);         // one-point weight 2^d |det J0|
    const double dJ = fabs(J) * detJ0;
    double G[D][D];                                         // J^{-1} = J0^{-1} F^{-1}
#pragma unroll
    for (int m = 0; m < D; ++m)
#pragma unroll
      for (int k = 0; k < D; ++k) {
        double v = 0;
#pragma unroll
        for (int p = 0; p < D; ++p) v += Ji0[m][p] * Fi[p][k];
        G[m][k] = v;
      }
    double sig[D][D];                                       // Eq. (sig_eq)
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
      for (int l = 0; l < D; ++l) {
        double b = 0;
#pragma unroll
        for (int p = 0; p < D; ++p) b += F[k][p] * F[l][p];
        sig[k][l] = mu / J * (b - (k == l ? 1.0 : 0.0)) + (k == l ? lam * lnJ / J : 0.0);
      }
    double A[D][D], Sg[D][D];
#pragma unroll
    for (int m = 0; m < D; ++m)
#pragma unroll
      for (int n = 0; n < D; ++n) {
        double a1 = 0, a2 = 0;
#pragma unroll
        for (int k = 0; k < D; ++k) {
          a1 += G[m][k] * G[n][k];
          double t = 0;
#pragma unroll
          for (int l = 0; l < D; ++l) t += sig[k][l] * G[n][l];
          a2 += G[m][k] * t;
        }
        A[m][n] = a1;
        Sg[m][n] = a2;
      }
    const double cl = lam / J, cc = (mu - lam * lnJ) / J;
    double* out = T + (size_t)s * n_el * D4 + (size_t)e * D4;
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int j = 0; j < D; ++j)
#pragma unroll
        for (int m = 0; m < D; ++m)
#pragma unroll
          for (int n = 0; n < D; ++n) {
            double v = cl * G[m][i] * G[n][j] + cc * G[m][j] * G[n][i];
            if (i == j) v += cc * A[m][n] + Sg[m][n];
            out[((i * D + j) * D + m) * D + n] = dJ * v;
          }
  }
  const double mj = -block_max(-myJ, red);
  if (threadIdx.x == 0 && minJ_cell) {
    // the CTAs of a cell combine through an atomic-free per-(cell, CTA) slot
    minJ_cell[(size_t)s * gridDim.x + blockIdx.x] = mj;
  }
}

// ---------------------------------------------------------------------------------------------
// exact tangent action y = K(u) v without storing K (matrix free, full rule):
//   dP_iK = mu dF_iK + lam tr(F^{-1} dF) F^{-1}_Ki + (mu - lam ln J) (F^{-1} dF F^{-1})_Ki
// output cell-stacked local forces [n_loc][n_cells]
// ---------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(kCellThreads)
    k_tangent_apply(int n_cells, int nn, LaneArgs g, const int* __restrict__ cell_nodes,
                    const double* __restrict__ mu_cell, double lam, const double* __restrict__ u_glob,
                    const double* __restrict__ v_glob, double* __restrict__ y_cells) {
  constexpr int NEN = 1 << D;
  extern __shared__ double sm[];
  double* u_loc = sm;
  double* v_loc = sm + nn * D;
  double* fes = sm + 2 * nn * D;   // [EB][NEN][D]
  const int s = blockIdx.x, lane = threadIdx.x & 31;
  load_cell_u(u_glob, cell_nodes + (size_t)s * nn, nn, D, u_loc);
  load_cell_u(v_glob, cell_nodes + (size_t)s * nn, nn, D, v_loc);
  __syncthreads();
  const double mu = mu_cell[s];
  const LaneQ1<D> L(lane & (NEN - 1));
  const int node = L.node(), q = lane & (NEN - 1);
  for (int e0 = 0; e0 < g.n_el; e0 += g.EB) {
    const int ne = min(g.EB, g.n_el - e0);
    for (int t0 = threadIdx.x - lane; t0 < ne * NEN; t0 += blockDim.x) {
      const int el = (t0 + lane) / NEN;
      const int e = e0 + min(el, ne - 1);
      const int nd = g.elems[e * NEN + node];
      double Ji[D][D], F[D][D], dF[D][D], Fi[D][D];
#pragma unroll
      for (int d = 0; d < D; ++d)
#pragma unroll
        for (int k = 0; k < D; ++k) Ji[d][k] = g.Ji[((size_t)e * NEN + q) * D * D + d * D + k];
      const double w = g.W[e * NEN + q];
#pragma unroll
      for (int i = 0; i < D; ++i) {
        double du[D], dv[D];
        L.gradient(u_loc[nd * D + i], lane, du);
        L.gradient(v_loc[nd * D + i], lane, dv);
#pragma unroll
        for (int k = 0; k < D; ++k) {
          double f = (i == k) ? 1.0 : 0.0, df = 0.0;
#pragma unroll
          for (int d = 0; d < D; ++d) {
            f = fma(du[d], Ji[d][k], f);
            df = fma(dv[d], Ji[d][k], df);
          }
          F[i][k] = f;
          dF[i][k] = df;
        }
      }
      const double J = det_inv<D>(F, Fi);
      const double lnJ = J > 0 ? log(J) : 0.0;
      double tr = 0, FdF[D][D];
#pragma unroll
      for (int K = 0; K < D; ++K)
#pragma unroll
        for (int M = 0; M < D; ++M) {
          double v = 0;
#pragma unroll
          for (int j = 0; j < D; ++j) v = fma(Fi[K][j], dF[j][M], v);
          FdF[K][M] = v;   // (F^{-1} dF)_KM
        }
#pragma unroll
      for (int K = 0; K < D; ++K) tr += FdF[K][K];
#pragma unroll
      for (int i = 0; i < D; ++i) {
        double dP[D], Q[D];
#pragma unroll
        for (int K = 0; K < D; ++K) {
          double m = 0;
#pragma unroll
          for (int M = 0; M < D; ++M) m = fma(FdF[K][M], Fi[M][i], m);
          dP[K] = w * (mu * dF[i][K] + lam * tr * Fi[K][i] + (mu - lam * lnJ) * m);
        }
#pragma unroll
        for (int d = 0; d < D; ++d) {
          double v = 0;
#pragma unroll
          for (int K = 0; K < D; ++K) v = fma(dP[K], Ji[d][K], v);
          Q[d] = v;
        }
        const double fe = L.force(Q);
        if (el < ne) fes[(size_t)(el * NEN + node) * D + i] = fe;
      }
    }
    __syncthreads();
    gather_forces<D>(g, nn, n_cells, s, e0, e0 + ne, fes, y_cells);
    __syncthreads();
  }
}

// r[g] = sum over the copies of global node g of the cell-stacked local values
__global__ void k_scatter(int64_t n_nodes, int dim, int nn, int n_cells, const int* __restrict__ cptr,
                          const int* __restrict__ cidx, const double* __restrict__ f_cells,
                          double* __restrict__ r) {
  int64_t gnode = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (gnode >= n_nodes) return;
  for (int i = 0; i < dim; ++i) {
    double v = 0;
    for (int c = cptr[gnode]; c < cptr[gnode + 1]; ++c) {
      int sa = cidx[c];
      int s = sa / nn, a = sa - s * nn;
      v += f_cells[(size_t)(a * dim + i) * n_cells + s];
    }
    r[gnode * dim + i] = v;
  }
}

// grad[s] = sum_k w_loc[k,s] * f_mu[k,s] (cell-stacked inputs)
__global__ void k_cell_dot(int n_cells, int n_loc, const double* __restrict__ w_glob,
                           const int* __restrict__ cell_nodes, int nn, int dim,
                           const double* __restrict__ f_cells, double* __restrict__ out) {
  __shared__ double red[32];
  const int s = blockIdx.x;
  double v = 0;
  for (int k = threadIdx.x; k < n_loc; k += blockDim.x) {
    int a = k / dim, i = k - a * dim;
    v += w_glob[(int64_t)cell_nodes[(size_t)s * nn + a] * dim + i] * f_cells[(size_t)k * n_cells + s];
  }
  v = block_sum(v, red);
  if (threadIdx.x == 0) out[s] = v;
}

// deterministic two-stage reductions over global vectors
constexpr int kRedBlocks = 512;

__global__ void k_sumsq_masked(int64_t n, const double* __restrict__ x, const uint8_t* __restrict__ fixed,
                               int want_fixed, double* __restrict__ part) {
  __shared__ double red[32];
  double v = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if ((fixed[i] != 0) == (want_fixed != 0)) v += x[i] * x[i];
  v = block_sum(v, red);
  if (threadIdx.x == 0) part[blockIdx.x] = v;
}

__global__ void k_dot_masked(int64_t n, const double* __restrict__ a, const double* __restrict__ b,
                             const uint8_t* __restrict__ fixed, double* __restrict__ part) {
  __shared__ double red[32];
  double v = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (fixed[i]) v += a[i] * b[i];
  v = block_sum(v, red);
  if (threadIdx.x == 0) part[blockIdx.x] = v;
}

__global__ void k_final_sum(int n, const double* __restrict__ part, double* __restrict__ out) {
  __shared__ double red[32];
  double v = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) v += part[i];
  v = block_sum(v, red);
  if (threadIdx.x == 0) out[0] = v;
}

__global__ void k_min_reduce(int n, const double* __restrict__ x, double* __restrict__ out) {
  __shared__ double red[32];
  double v = DBL_MAX;
  for (int i = threadIdx.x; i < n; i += blockDim.x) v = fmin(v, x[i]);
  v = -block_max(-v, red);
  if (threadIdx.x == 0) out[0] = v;
}

ColorTable colors(lat_ctx* h) {
  ColorTable ct;
  ct.n = (int)h->color_start.size() - 1;
  LAT_REQUIRE(ct.n <= 32, LAT_EINVAL, "too many element colours");
  for (int c = 0; c <= ct.n; ++c) ct.start[c] = h->color_start[c];
  return ct;
}

GeomArgs geom(lat_ctx* h, int quad) {
  return GeomArgs{h->gradX[quad].p, h->W[quad].p, h->elems.p, h->color_elems.p, h->nq[quad], h->gram[quad].p};
}

// Shared memory of the lane kernels: `vecs` cell vectors and the staged element forces.  All
// elements at once where two CTAs per SM still fit (344 strut elements: 66 KB), else as many as do,
// else (cell vectors beyond that) what one CTA per SM leaves.
LaneArgs lane_args(lat_ctx* h, int vecs, size_t* shm) {
  const size_t per = (size_t)h->nen * h->dim * sizeof(double), base = (size_t)vecs * h->n_loc * sizeof(double);
  const size_t two = 108 * 1024, one = 225 * 1024;
  const size_t room = base + 64 * per <= two ? two - base : base < one ? one - base : 0;
  const int EB = (int)std::max<size_t>(1, std::min<size_t>(h->n_el, room / per));
  *shm = base + EB * per;
  return LaneArgs{h->n_el, EB, h->Jinv.p, h->W[0].p, h->elems.p, h->node_el_ptr.p, h->node_el.p};
}

template <typename K, typename... A>
void launch_cells(lat_ctx* h, K kern, size_t shm, A... args) {
  LAT_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
  LAT_LAUNCH(h, kern<<<h->n_cells, kCellThreads, shm, h->stream>>>(h->n_cells, h->n_nodes_cell, args...));
  LAT_CHECK_LAUNCH();
}

void launch_residual(lat_ctx* h, double mu_override, double lam, const double* u_glob, double* f_cells) {
  size_t shm = 0;
  const LaneArgs g = lane_args(h, 1, &shm);
  const int* cn = h->cell_nodes.p;
  const double* mu = h->mu_cell.p;
  if (h->dim == 2) launch_cells(h, k_residual<2>, shm, g, cn, mu, mu_override, lam, u_glob, f_cells, h->minJ_cell.p);
  else launch_cells(h, k_residual<3>, shm, g, cn, mu, mu_override, lam, u_glob, f_cells, h->minJ_cell.p);
}

double* scratch_scalars(lat_ctx* h) {
  h->red_part.ensure(4096);
  return h->red_part.p;
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------------------
void run_residual(lat_ctx* h, const double* u_glob, double* f_cells, double* r_glob,
                  double* min_detF_host, bool* negJ) {
  h->minJ_cell.ensure(h->n_cells);
  KernelTimer kt(h, "residual");
  launch_residual(h, -1.0, h->lam, u_glob, f_cells);
  if (r_glob) {
    LAT_LAUNCH(h, k_scatter<<<div_up(h->n_glob_nodes, 256), 256, 0, h->stream>>>(h->n_glob_nodes, h->dim,
        h->n_nodes_cell, h->n_cells, h->copy_ptr.p, h->copy_idx.p, f_cells, r_glob));
    LAT_CHECK_LAUNCH();
  }
  double* sc = scratch_scalars(h);
  LAT_LAUNCH(h, k_min_reduce<<<1, 1024, 0, h->stream>>>(h->n_cells, h->minJ_cell.p, sc));
  LAT_CHECK_LAUNCH();
  LAT_CUDA(cudaMemcpyAsync(h->h_pinned, sc, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  LAT_CUDA(cudaStreamSynchronize(h->stream));
  if (min_detF_host) *min_detF_host = h->h_pinned[0];
  if (negJ) *negJ = !(h->h_pinned[0] > 0.0);
}

void run_tangent(lat_ctx* h, const double* u_glob, int quad, const int* cells, int n_sel,
                 double* K_out, bool* negJ, bool geometric) {
  if (n_sel <= 0) return;
  auto g = geom(h, quad);
  auto ct = colors(h);
  // CTAs per cell: 8 while the cells alone would leave most SMs without a CTA
  const int CL = (int64_t)n_sel * 8 <= 2 * h->n_sm ? 8 : 1;
  h->minJ_cell.ensure(std::max((size_t)h->n_cells, (size_t)n_sel * CL));
  // elements of a batch: about one quadrature point per thread, no more than a colour's share
  int widest = 1;
  for (int c = 0; c < ct.n; ++c) widest = std::max(widest, ct.start[c + 1] - ct.start[c]);
  const size_t per = sizeof(double) * g.nq * (h->dim == 2 ? tangent_row<2>() : tangent_row<3>());
  const size_t ub = (size_t)h->n_loc * sizeof(double);
  const size_t room = ub < 64 * 1024 ? 104 * 1024 - ub : 80 * 1024;   // two CTAs per SM where u allows
  const int EB = (int)std::max<size_t>(1, std::min<size_t>({(size_t)(kCellThreads / g.nq), (size_t)div_up(widest, CL), room / per}));
  const int staged = EB * per + ub <= 200 * 1024;
  const size_t shm = EB * per + (staged ? ub : 0);
  KernelTimer kt(h, quad ? "tangent_reduced" : (geometric ? "tangent_full" : "tangent_material"));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(n_sel * CL);
  cfg.blockDim = dim3(kCellThreads);
  cfg.dynamicSmemBytes = shm;
  cfg.stream = h->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  auto go = [&](auto kern) {
    LAT_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    LAT_LAUNCH(h, LAT_CUDA(cudaLaunchKernelEx(&cfg, kern, h->n_nodes_cell, g, ct, (const int*)h->cell_nodes.p, cells,
                                              (const int*)h->elem_blk.p, (const double*)h->mu_cell.p, h->lam, u_glob,
                                              h->nnz, K_out, h->minJ_cell.p, geometric ? 1 : 0, EB, CL, staged)));
  };
  if (h->dim == 2) go(k_tangent<2>);
  else go(k_tangent<3>);
  LAT_CHECK_LAUNCH();
  if (negJ) {
    double* sc = scratch_scalars(h);
    LAT_LAUNCH(h, k_min_reduce<<<1, 1024, 0, h->stream>>>(n_sel * CL, h->minJ_cell.p, sc));
    LAT_CHECK_LAUNCH();
    LAT_CUDA(cudaMemcpyAsync(h->h_pinned, sc, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    LAT_CUDA(cudaStreamSynchronize(h->stream));
    *negJ = !(h->h_pinned[0] > 0.0);
  }
}

// D^ref snapshots of every cell: T [n_cells][n_el * d^4]
void run_dref_snapshots(lat_ctx* h, const double* u_glob, double* T, bool* negJ) {
  const int nb = div_up(h->n_el, 128);
  h->minJ_cell.ensure((size_t)h->n_cells * nb);
  auto g = geom(h, 1);
  const dim3 grid(nb, h->n_cells);
  KernelTimer kt(h, "dref_snapshots");
  if (h->dim == 2)
    LAT_LAUNCH(h, k_dref<2><<<grid, 128, 0, h->stream>>>(h->n_cells, h->n_el, h->n_nodes_cell, g, h->cell_nodes.p,
                                                          h->mu_cell.p, h->lam, u_glob, T, h->minJ_cell.p));
  else
    LAT_LAUNCH(h, k_dref<3><<<grid, 128, 0, h->stream>>>(h->n_cells, h->n_el, h->n_nodes_cell, g, h->cell_nodes.p,
                                                          h->mu_cell.p, h->lam, u_glob, T, h->minJ_cell.p));
  LAT_CHECK_LAUNCH();
  if (negJ) {
    double* sc = scratch_scalars(h);
    LAT_LAUNCH(h, k_min_reduce<<<1, 1024, 0, h->stream>>>((int)((int64_t)h->n_cells * nb), h->minJ_cell.p, sc));
    LAT_CHECK_LAUNCH();
    LAT_CUDA(cudaMemcpyAsync(h->h_pinned, sc, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    LAT_CUDA(cudaStreamSynchronize(h->stream));
    *negJ = !(h->h_pinned[0] > 0.0);
  }
}

void run_tangent_apply_exact(lat_ctx* h, const double* u_glob, const double* v_glob, double* y_glob) {
  h->f_cells.ensure((size_t)h->n_loc * h->n_cells);
  size_t shm = 0;
  const LaneArgs g = lane_args(h, 2, &shm);
  const int* cn = h->cell_nodes.p;
  const double* mu = h->mu_cell.p;
  if (h->dim == 2) launch_cells(h, k_tangent_apply<2>, shm, g, cn, mu, h->lam, u_glob, v_glob, h->f_cells.p);
  else launch_cells(h, k_tangent_apply<3>, shm, g, cn, mu, h->lam, u_glob, v_glob, h->f_cells.p);
  LAT_LAUNCH(h, k_scatter<<<div_up(h->n_glob_nodes, 256), 256, 0, h->stream>>>(h->n_glob_nodes, h->dim,
      h->n_nodes_cell, h->n_cells, h->copy_ptr.p, h->copy_idx.p, h->f_cells.p, y_glob));
  LAT_CHECK_LAUNCH();
}

// grad[s] = w^{sT} f_mu^s(u^s): internal force with mu -> base mu, lam -> 0 (d f / d theta_s)
void run_grad_mu(lat_ctx* h, const double* u_glob, const double* w_glob, double* grad) {
  h->f_cells.ensure((size_t)h->n_loc * h->n_cells);
  h->minJ_cell.ensure(h->n_cells);
  launch_residual(h, h->mu, 0.0, u_glob, h->f_cells.p);
  LAT_LAUNCH(h, k_cell_dot<<<h->n_cells, 256, 0, h->stream>>>(h->n_cells, h->n_loc, w_glob, h->cell_nodes.p,
      h->n_nodes_cell, h->dim, h->f_cells.p, grad));
  LAT_CHECK_LAUNCH();
}

double run_norm_free(lat_ctx* h, const double* r) {
  double* sc = scratch_scalars(h);
  LAT_LAUNCH(h, k_sumsq_masked<<<kRedBlocks, 256, 0, h->stream>>>(h->n_dof, r, h->dof_fixed.p, 0, sc + 16));
  LAT_LAUNCH(h, k_final_sum<<<1, 512, 0, h->stream>>>(kRedBlocks, sc + 16, sc));
  LAT_CHECK_LAUNCH();
  LAT_CUDA(cudaMemcpyAsync(h->h_pinned, sc, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  LAT_CUDA(cudaStreamSynchronize(h->stream));
  return std::sqrt(h->h_pinned[0]);
}

double run_norm_all(lat_ctx* h, const double* r) {
  double* sc = scratch_scalars(h);
  LAT_LAUNCH(h, k_sumsq_masked<<<kRedBlocks, 256, 0, h->stream>>>(h->n_dof, r, h->dof_fixed.p, 0, sc + 16));
  LAT_LAUNCH(h, k_sumsq_masked<<<kRedBlocks, 256, 0, h->stream>>>(h->n_dof, r, h->dof_fixed.p, 1, sc + 16 + kRedBlocks));
  LAT_LAUNCH(h, k_final_sum<<<1, 512, 0, h->stream>>>(2 * kRedBlocks, sc + 16, sc));
  LAT_CHECK_LAUNCH();
  LAT_CUDA(cudaMemcpyAsync(h->h_pinned, sc, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  LAT_CUDA(cudaStreamSynchronize(h->stream));
  return std::sqrt(h->h_pinned[0]);
}

double run_dot_fixed(lat_ctx* h, const double* a, const double* b) {
  double* sc = scratch_scalars(h);
  LAT_LAUNCH(h, k_dot_masked<<<kRedBlocks, 256, 0, h->stream>>>(h->n_dof, a, b, h->dof_fixed.p, sc + 16));
  LAT_LAUNCH(h, k_final_sum<<<1, 512, 0, h->stream>>>(kRedBlocks, sc + 16, sc));
  LAT_CHECK_LAUNCH();
  LAT_CUDA(cudaMemcpyAsync(h->h_pinned, sc, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  LAT_CUDA(cudaStreamSynchronize(h->stream));
  return h->h_pinned[0];
}

// ---------------------------------------------------------------------------------------------
// entry point
// ---------------------------------------------------------------------------------------------
extern "C" lat_status assemble_residual_tangent(lat_handle h, const double* u_glob, int32_t quad,
                                                const int32_t* cells, int32_t n_sel, double* r_glob,
                                                double* f_cells, double* K_vals, double* min_detF) {
  if (!h || !u_glob) return LAT_EINVAL;
  return guard(h, [&] {
    LAT_REQUIRE(quad == 0 || quad == 1, LAT_EINVAL, "quad must be 0 (full) or 1 (reduced)");
    LAT_REQUIRE(n_sel >= 0, LAT_EINVAL, "negative cell count");
    LAT_REQUIRE(cells != nullptr || n_sel == h->n_cells, LAT_EINVAL, "n_sel must equal n_cells when cells is NULL");
    LAT_REQUIRE(!(cells && (r_glob || f_cells)), LAT_EINVAL, "residual outputs need all cells");
    if (cells && n_sel > 0) {
      std::vector<int> hc(n_sel);
      LAT_CUDA(cudaMemcpy(hc.data(), cells, n_sel * sizeof(int), cudaMemcpyDeviceToHost));
      for (int c : hc) LAT_REQUIRE(c >= 0 && c < h->n_cells, LAT_EINVAL, "cell index out of range");
    }
    bool neg = false;
    double mdf = DBL_MAX;
    if (r_glob || f_cells) {
      double* fc = f_cells;
      if (!fc) {
        h->f_cells.ensure((size_t)h->n_loc * h->n_cells);
        fc = h->f_cells.p;
      }
      run_residual(h, u_glob, fc, r_glob, &mdf, &neg);
    }
    if (K_vals && n_sel > 0) {
      bool n2 = false;
      run_tangent(h, u_glob, quad, cells, n_sel, K_vals, &n2);
      neg = neg || n2;
      mdf = std::min(mdf, h->h_pinned[0]);
    }
    LAT_CUDA(cudaStreamSynchronize(h->stream));
    if (min_detF) *min_detF = mdf;
    if (neg) throw LatError{LAT_ENEG_JACOBIAN, "det F <= 0 at some quadrature point"};
  });
}
