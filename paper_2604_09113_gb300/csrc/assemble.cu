// Online assembly of the cell stiffness matrices (Sec. 4.1, Algorithms 4-5).
//
//  theta kernel (CTAs of a few cells of one model):
//    I_r(mu)  = sum_g A[g] prod_d l_{g_d}(mu_d)       (tensor GLL interpolation, Sec. 4.2.3)
//    theta    = (rho, (1 - rho) I_r)                  (Algorithm 4: I + rho (I_Pi - I))
//    Chat_k   = det J J^-1 C J^-T at the (q+1)^2 GLL interpolation nodes
//               (Eq. ELA constitutive, Eq. FAST interpolation)
//  contraction (FP64 form): I_c = theta_c U' per (k1 <= k2) pair, then
//    K[(k1 i1),(k2 i2)] = sum_{j1 j2 k3} I_c[k1 k2 k3 j1 j2] Chat_c[k3][i1 j1 i2 j2]
//  (Eq. SPEED L int), written as the packed upper triangle of each cell matrix.
#include <stdio.h>

#include <algorithm>
#include <vector>

#include "device.cuh"
#include "fx56.cuh"
#include "tables.cuh"

struct RomDev {
  const int2* At;        // [ngrid][n_r] interpolation samples, fixed point (fx56.cuh): A_t 2^-at_exp[t]
  const int* at_exp;     // [n_r] exponents with |A_t| <= 2^(at_exp - 1)
  int n_r, r;
  double lo4[4], hi4[4]; // the cluster's box per threshold
  double g01[12];        // degree-r GLL nodes of [0, 1]; node i of threshold d is lo4 + (hi4 - lo4) g01[i]
};

// the models in use, by slot, with the cells of each
struct ThetaFams {
  RomDev rom[ROMB_MAX_MODELS];
  const int* list[ROMB_MAX_MODELS];
  int count[ROMB_MAX_MODELS];
};

// FindCluster (Algorithm 5, Sec. 4.2.1): the model slot of each cell, from its
// family's cluster table: k_d = floor((mu_d - lo) / h) capped at n_k - 1
// (an interior subinterval boundary belongs to the upper cluster).  Cells
// outside their family's box are flagged and kept in the nearest cluster;
// cells of a family without models get slot -1.
struct FamTab {
  int n_k[ROMB_MAX_FAMILIES], slot0[ROMB_MAX_FAMILIES];
  double lo[ROMB_MAX_FAMILIES], hi[ROMB_MAX_FAMILIES];
};
__global__ void cell_model_kernel(FamTab T, const int32_t* __restrict__ family, const double* __restrict__ mu,
                                  int ncells, int32_t* __restrict__ slot, int32_t* __restrict__ flags) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= ncells) return;
  const int f = family[c];
  int nk = 0, s0 = -1;
  double lo = 0.0, hi = 0.0;
#pragma unroll
  for (int k = 0; k < ROMB_MAX_FAMILIES; ++k)
    if (k == f) {
      nk = T.n_k[k];
      s0 = T.slot0[k];
      lo = T.lo[k];
      hi = T.hi[k];
    }
  if (nk == 0) {
    slot[c] = -1;
    return;
  }
  const double h = (hi - lo) / nk;
  int k = 0, stride = 1;
  for (int d = 0; d < 4; ++d) {
    const double m = mu[4 * c + d];
    if (!(m >= lo && m <= hi)) atomicOr(&flags[c], ROMB_FLAG_OUT_OF_BOX);
    int kd = (int)floor((m - lo) / h);
    kd = kd < 0 ? 0 : kd > nk - 1 ? nk - 1 : kd;
    k += kd * stride;
    stride *= nk;
  }
  slot[c] = s0 + k;
}

void fill_cell_params(const romb_ctx* c, CellParams* P) {
  memset(P, 0, sizeof(*P));
  P->p = c->p;
  P->m = c->m;
  P->basis = c->basis;
  P->nB = c->nB;
  P->nI = c->nI;
  P->nU = c->nU;
  P->nx = c->nx;
  P->ny = c->ny;
  P->ncells = c->ncells;
  if (c->layout) {
    P->cell_grid = c->d_cell_grid;
    P->grid_cell = c->d_grid_cell;
    P->node_fixed = c->d_node_fixed;
  }
  P->q = c->q;
  P->nL = c->nL;
  P->dmask = c->dmask;
  P->E = c->E;
  P->nu = c->nu;
  P->rho = c->rho;
  P->lam = c->E * c->nu / (1.0 - c->nu * c->nu);
  P->mu = c->E / (2.0 * (1.0 + c->nu));
  gll_nodes01(c->p, P->gll);
  for (int i = 0; i <= c->p; ++i) {
    double den = 1.0;
    for (int j = 0; j <= c->p; ++j)
      if (j != i) den *= P->gll[i] - P->gll[j];
    P->bw[i] = 1.0 / den;
  }
  for (int i = 0; i <= c->m; ++i) {
    double den = 1.0;
    for (int j = 0; j <= c->m; ++j)
      if (j != i) den *= (double)i / c->m - (double)j / c->m;
    P->mw[i] = 1.0 / den;
  }
  gauss01(ROMB_NQ, P->gq_x, P->gq_w);
  for (int i = 0; i < ROMB_NQ; ++i) cell_basis1d(*P, P->gq_x[i], P->bq[i], nullptr);
  for (int i = 0; i <= ROMB_NQ; ++i) map_basis1d(c->m, i < ROMB_NQ ? P->gq_x[i] : 0.5, P->mq[i], P->dmq[i]);
  LocalTables T = make_local_tables(c->p);
  memcpy(P->uslot, T.uslot, sizeof(P->uslot));
  memcpy(P->islot, T.islot, sizeof(P->islot));
  memcpy(P->uslot_of_node, T.uslot_of_node, sizeof(P->uslot_of_node));
}

// ---------------------------------------------------------------------------
// family lists: cells grouped by family, in increasing cell index (one CTA)
// ---------------------------------------------------------------------------
__global__ void family_list_kernel(const int32_t* __restrict__ family, int ncells, int nfam, int* __restrict__ list,
                                   int* __restrict__ counts, int32_t* __restrict__ flags) {
  __shared__ int warp_tot[32];
  __shared__ int base;
  const int tid = threadIdx.x, nt = blockDim.x;
  int out = 0;
  for (int f = 0; f < nfam; ++f) {
    if (tid == 0) base = out;
    __syncthreads();
    for (int c0 = 0; c0 < ncells; c0 += nt) {
      const int c = c0 + tid;
      const int fam = c < ncells ? family[c] : -1;
      const int mine = fam == f;
      // block exclusive scan of `mine`
      const unsigned bal = __ballot_sync(0xffffffffu, mine);
      const int lane = tid & 31, w = tid >> 5;
      const int pre = __popc(bal & ((1u << lane) - 1u));
      if (lane == 0) warp_tot[w] = __popc(bal);
      __syncthreads();
      int wpre = 0, tot = 0;
      for (int i = 0; i < nt / 32; ++i) {
        if (i < w) wpre += warp_tot[i];
        tot += warp_tot[i];
      }
      if (mine) list[base + wpre + pre] = c;
      __syncthreads();
      if (tid == 0) base += tot;
      __syncthreads();
    }
    if (tid == 0) counts[f] = base - out;
    out = base;
    __syncthreads();
  }
  // cells whose family has no loaded model
  for (int c = tid; c < ncells; c += nt)
    if (family[c] < 0 || family[c] >= nfam) flags[c] |= ROMB_FLAG_OUT_OF_BOX;
}

// ---------------------------------------------------------------------------
// theta kernel
// ---------------------------------------------------------------------------
// Per cell: the 1D interpolation weights of its four thresholds (as
// fixed-point digits) and Chat at the 9 interpolation nodes, one thread per
// (cell, threshold) and (cell, node).  Apart from the contraction below, whose
// CTAs would wait for these serial FP64 chains.
__global__ void __launch_bounds__(128) cell_prep_kernel(CellParams P, const ThetaFams* __restrict__ F,
                                                        const int32_t* __restrict__ slot,
                                                        const double* __restrict__ ctrl,
                                                        const double* __restrict__ mu, int2* __restrict__ wts,
                                                        double* __restrict__ chat, float* __restrict__ chat32,
                                                        int32_t* __restrict__ flags) {
  const long long task = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long n4 = 4LL * P.ncells;
  if (task < n4) {
    const long long c = task >> 2;
    const int d = (int)(task & 3);
    const RomDev& R = F->rom[slot[c]];
    const int n1 = R.r + 1;
    const double m = mu[task];
    if (!(m >= R.lo4[d] && m <= R.hi4[d])) atomicOr(&flags[c], ROMB_FLAG_OUT_OF_BOX);
    double nodes[12], v[12];
    for (int i = 0; i < n1; ++i) nodes[i] = R.lo4[d] + (R.hi4[d] - R.lo4[d]) * R.g01[i];
    lagrange1d(R.r, nodes, m, v, nullptr);
    // |l| <= 1 inside the box (GLL nodes); outside it the cell is flagged
    for (int i = 0; i < n1; ++i) wts[task * 12 + i] = fx_from_double<FX_THETA>(fmin(fmax(v[i], -1.0), 1.0), 0);
    return;
  }
  if (task >= n4 + 9LL * P.ncells) return;
  const long long c = (task - n4) / 9;
  const int k3 = (int)((task - n4) % 9);
  int cx, cy;
  cell_xy(P, c, &cx, &cy);
  const double qn[3] = {0.0, 0.5, 1.0};
  double x[2], J[2][2];
  map_eval(ctrl, P.nx, P.m, cx, cy, qn[k3 % 3], qn[k3 / 3], x, J);
  const double det = J[0][0] * J[1][1] - J[0][1] * J[1][0];
  if (!(det > 0.0)) atomicOr(&flags[c], ROMB_FLAG_BAD_MAP);
  // G = J^-1, G[j][m] = dxi_j / dx_m
  const double G[2][2] = {{J[1][1] / det, -J[0][1] / det}, {-J[1][0] / det, J[0][0] / det}};
  double* out = chat + c * 144 + 16 * k3;
  for (int i = 0; i < 2; ++i)
    for (int jj = 0; jj < 2; ++jj)
      for (int k = 0; k < 2; ++k)
        for (int l = 0; l < 2; ++l) {
          // Chat_ijkl = det [lam G_ji G_lk + mu (d_ik (G G^T)_jl + G_jk G_li)]
          const double GGt = G[jj][0] * G[l][0] + G[jj][1] * G[l][1];
          // products grouped so that Chat_ijkl and Chat_klij round identically
          const double v = P.lam * (G[jj][i] * G[l][k]) + P.mu * ((i == k ? GGt : 0.0) + G[jj][k] * G[l][i]);
          out[((i * 2 + jj) * 2 + k) * 2 + l] = det * v;
          chat32[c * 144 + 16 * k3 + ((i * 2 + jj) * 2 + k) * 2 + l] = (float)(det * v);
        }
}

// The interpolation theta = A w, n_r (r+1)^4 FMA per cell (144 k at n_r = 60,
// r = 6).  A CTA takes CG groups of CT cells of one model; lanes run over the
// coefficients t, the (g3, g4) planes of the sample grid are divided among
// the warps of each group (the groups read the same samples close together,
// from L1), and the partial sums are added in warp order.  The sums run in
// 59-bit fixed point on the integer pipe: the samples are scaled per t to
// |A_t| <= 1/2 and the 1D weights satisfy |l| <= 1 (Lagrange polynomials on GLL
// nodes) with 1-norms of at most 1.98 (Lebesgue constants, r <= 7), so the sums
// over a plane stay below 1.95 (their high digit below 2^31) and those over the
// planes below 7.6 of the 8 that hi hi holds; for r = 8..10 (2.19) the samples
// take half of that.  The cross sums of r = 6 stay below 49 2^57 + 3.6 2^58 <
// 2^62.9, those of a warp's planes below 2^62.6; the general form carries
// after each line.  Bound: the integer
// multiply-adds.  Measured, the whole phase with the edge functionals, FP64
// form: 16 cells, n_r = 20: 1.30 -> 0.13 ms (one warp walked the grid
// alone); 4,096 cells, n_r = 40: 2.60 -> 0.76; 17,424 cells, n_r = 60: 7.7 ->
// 3.0 (this kernel 1.9; a double-float form on the FP32 pipe took as long
// and kept 48 bits).  Error against extended precision over max |A_t|, trained
// models of p = 3 to 8: rms 0.15 to 0.97 of the FP64 sums' (1e-16 to 3.4e-16);
// with 56 bits and samples of 1/4 it was up to 1.3 of theirs (p = 7, 8), and
// coefficients far below their largest sample lost up to 12 times as much.
#define TH_WARPS 7   // r = 6: 49 planes
__device__ inline float tf32_round_dev(float f) {
  uint32_t u = __float_as_uint(f);
  if ((u & 0x7f800000u) == 0x7f800000u) return f;
  u = (u + 0x1000u) & 0xffffe000u;
  return __uint_as_float(u);
}
__device__ __forceinline__ int2 fx_mul(int2 a, int2 b) {   // |a|, |b| <= 1
  long long hh = 0, x = 0;
  fx_mad(hh, x, a, b);
  return fx_digits<FX_THETA>(fx_sum<FX_THETA>(hh, x));
}

// the models of one launch: slot[k] owns CTAs from cta[k] to cta[k + 1]
struct ThetaCtas {
  int slot[ROMB_MAX_MODELS], cta[ROMB_MAX_MODELS + 1];
};

// NS = ceil(n_r / 32) lane slots per coefficient; N1 = r + 1 when known at
// compile time (0: from the model), so that the loads of a line (g2, g3, g4)
// are issued together.
template <int NS, int CT, int CG, int N1>
__global__ void __launch_bounds__(32 * TH_WARPS * CG) theta_kernel(
    CellParams P, const ThetaFams* __restrict__ Fams, const __grid_constant__ ThetaCtas models,
    const int2* __restrict__ wts, double* __restrict__ theta, float* __restrict__ th_hi,
    float* __restrict__ th_lo) {
  constexpr int NC = CT * CG;
  extern __shared__ __align__(16) unsigned char th_smem[];   // w12 and w34, then the warps' partial sums
  __shared__ int2 w1[NC][4][12];
  int2* w12 = reinterpret_cast<int2*>(th_smem);              // [NC][n1^2], g2 n1 + g1; then w34 [NC][n1^2]
  long long* part = reinterpret_cast<long long*>(th_smem);   // [TH_WARPS][NC][32 NS]
  const int tid = threadIdx.x, lane = tid & 31, warp = (tid >> 5) % TH_WARPS, cg = (tid >> 5) / TH_WARPS;
  const int nt = blockDim.x;
  int k = 0;   // the model of this CTA
  while ((int)blockIdx.x >= models.cta[k + 1]) ++k;
  const int fi = models.slot[k];
  const RomDev& R = Fams->rom[fi];
  const int* __restrict__ list = Fams->list[fi];
  const int count = Fams->count[fi];
  const int first = ((int)blockIdx.x - models.cta[k]) * NC;
  const int n1 = N1 > 0 ? N1 : R.r + 1, nr = R.n_r;
  for (int i = tid; i < NC * 48; i += nt) {
    const int j = i / 48;
    w1[j][(i % 48) / 12][i % 12] = first + j < count ? wts[(long long)list[first + j] * 48 + i % 48] : make_int2(0, 0);
  }
  __syncthreads();
  const int n2 = n1 * n1;
  int2* w34 = w12 + NC * n2;
  for (int i = tid; i < 2 * NC * n2; i += nt) {
    const int d = i < NC * n2 ? 0 : 2, ii = d ? i - NC * n2 : i, j = ii / n2, g = ii % n2;
    w12[i] = fx_mul(w1[j][d][g % n1], w1[j][d + 1][g / n1]);
  }
  __syncthreads();
  // lambda_t = sum_{g3 g4} w34 (sum_{g1 g2} w12 At[g][t])
  long long oh[NS][CT], ox[NS][CT];
#pragma unroll
  for (int s = 0; s < NS; ++s)
#pragma unroll
    for (int j = 0; j < CT; ++j) oh[s][j] = ox[s][j] = 0;
  const int2* wc = w12 + cg * CT * n2;
#pragma unroll 1
  for (int g34 = warp; g34 < n2; g34 += TH_WARPS) {
    long long ih[NS][CT], ix[NS][CT];
#pragma unroll
    for (int s = 0; s < NS; ++s)
#pragma unroll
      for (int j = 0; j < CT; ++j) ih[s][j] = ix[s][j] = 0;
    const int2* Ag = R.At + (long long)g34 * n2 * nr + lane;
#pragma unroll 1
    for (int g2 = 0; g2 < n1; ++g2, Ag += n1 * nr) {
      if constexpr (N1 > 0) {
        int2 av[N1][NS];
#pragma unroll
        for (int g1 = 0; g1 < N1; ++g1)
#pragma unroll
          for (int s = 0; s < NS; ++s)
            av[g1][s] = lane + 32 * s < nr ? __ldg(Ag + g1 * nr + 32 * s) : make_int2(0, 0);
#pragma unroll
        for (int g1 = 0; g1 < N1; ++g1)
#pragma unroll
          for (int j = 0; j < CT; ++j) {
            const int2 w = wc[j * n2 + g2 * N1 + g1];
#pragma unroll
            for (int s = 0; s < NS; ++s) fx_mad(ih[s][j], ix[s][j], av[g1][s], w);
          }
      } else {
        for (int g1 = 0; g1 < n1; ++g1) {
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            const int2 a = lane + 32 * s < nr ? __ldg(Ag + g1 * nr + 32 * s) : make_int2(0, 0);
#pragma unroll
            for (int j = 0; j < CT; ++j) fx_mad(ih[s][j], ix[s][j], a, wc[j * n2 + g2 * n1 + g1]);
          }
        }
#pragma unroll
        for (int s = 0; s < NS; ++s)   // carry: 64 terms and more could pass 2^63
#pragma unroll
          for (int j = 0; j < CT; ++j) {
            ih[s][j] += ix[s][j] >> (FX_THETA - 30);
            ix[s][j] &= (1LL << (FX_THETA - 30)) - 1;
          }
      }
    }
#pragma unroll
    for (int j = 0; j < CT; ++j) {
      const int2 w = w34[(cg * CT + j) * n2 + g34];
#pragma unroll
      for (int s = 0; s < NS; ++s) 
        fx_mad(oh[s][j], ox[s][j], fx_digits<FX_THETA>(fx_sum<FX_THETA>(ih[s][j], ix[s][j])), w);
    }
  }
  __syncthreads();   // the weights are read no more: their memory takes the partial sums
#pragma unroll
  for (int s = 0; s < NS; ++s)
#pragma unroll
    for (int j = 0; j < CT; ++j)
      part[(warp * NC + cg * CT + j) * (32 * NS) + lane + 32 * s] =
          fx_sum<FX_THETA>(oh[s][j], ox[s][j]);
  __syncthreads();
  for (int i = tid; i < NC * 128; i += nt) {
    const int j = i >> 7, t = i & 127;   // slot t of theta: 0 rho, 1.. the coefficients
    if (first + j >= count) break;
    const long long c = list[first + j];
    double v = 0.0;
    if (t == 0) {
      v = P.rho;
    } else if (t <= nr) {
      long long sum = 0;
#pragma unroll
      for (int w = 0; w < TH_WARPS; ++w) sum += part[(w * NC + j) * (32 * NS) + t - 1];
      const int e = R.at_exp[t - 1];
      v = (1.0 - P.rho) * (e == FX_NAN ? nan("") : ldexp((double)sum, e - FX_THETA));
    }
    if (t <= nr) theta[128 * c + t] = v;
    // TF32 hi / lo split of the tensor-core slots of theta (0 and 2..; slot 1
    // is applied in the epilogue), zero padded to 128 slots
    if (t == 1) v = 0.0;
    const float h = tf32_round_dev((float)v);
    th_hi[128 * c + t] = h;
    th_lo[128 * c + t] = tf32_round_dev((float)(v - (double)h));
  }
}

// ---------------------------------------------------------------------------
// FP64 contraction: 32 cells x 4 pairs per CTA
// ---------------------------------------------------------------------------
#define A64_CELLS 32
#define A64_PAIRS 4
__global__ void __launch_bounds__(128) assemble_fp64_kernel(const double* __restrict__ U, long long n_half, int K,
                                                             const int* __restrict__ list, int count,
                                                             const int2* __restrict__ pairs, int npairs, int ndof,
                                                             const double* __restrict__ theta,
                                                             const double* __restrict__ chat,
                                                             double* __restrict__ Kout) {
  extern __shared__ double sm[];
  const int KS = K | 1;                      // odd stride: no bank conflicts across cells
  double* sU = sm;                           // [K][A64_PAIRS*36]
  double* sT = sU + (size_t)K * A64_PAIRS * 36;   // [32][KS]
  double* sC = sT + A64_CELLS * KS;          // [32][145]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int pair0 = blockIdx.y * A64_PAIRS;
  const int c0 = blockIdx.x * A64_CELLS;
  const int npl = min(A64_PAIRS, npairs - pair0);
  for (int i = tid; i < K * A64_PAIRS * 36; i += blockDim.x) {
    const int t = i / (A64_PAIRS * 36), e = i % (A64_PAIRS * 36);
    sU[i] = (e < npl * 36) ? U[(long long)t * n_half + (long long)pair0 * 36 + e] : 0.0;
  }
  for (int i = tid; i < A64_CELLS * K; i += blockDim.x) {
    const int j = i / K, t = i % K;
    const int c = c0 + j < count ? list[c0 + j] : -1;
    sT[j * KS + t] = c >= 0 ? theta[128 * (long long)c + t] : 0.0;
  }
  for (int i = tid; i < A64_CELLS * 144; i += blockDim.x) {
    const int j = i / 144, e = i % 144;
    const int c = c0 + j < count ? list[c0 + j] : -1;
    sC[j * 145 + e] = c >= 0 ? chat[144 * (long long)c + e] : 0.0;
  }
  __syncthreads();
  const int pl = warp;
  if (pl >= npl) return;
  const int cl = lane;
  const int cell = c0 + cl < count ? list[c0 + cl] : -1;
  double acc[36];
#pragma unroll
  for (int e = 0; e < 36; ++e) acc[e] = 0.0;
  const double* u = sU + pl * 36;
  const double* th = sT + cl * KS;
  for (int t = 0; t < K; ++t) {
    const double a = th[t];
    const double* ut = u + t * A64_PAIRS * 36;
#pragma unroll
    for (int e = 0; e < 36; ++e) acc[e] = fma(a, ut[e], acc[e]);
  }
  if (cell < 0) return;
  const int2 kk = pairs[pair0 + pl];
  const double* C = sC + cl * 145;
  double* Kc = Kout + (long long)cell * ((long long)ndof * (ndof + 1) / 2);
#pragma unroll
  for (int i1 = 0; i1 < 2; ++i1)
#pragma unroll
    for (int i2 = 0; i2 < 2; ++i2) {
      if (kk.x == kk.y && i1 > i2) continue;
      double v = 0.0;
#pragma unroll
      for (int k3 = 0; k3 < 9; ++k3)
#pragma unroll
        for (int j1 = 0; j1 < 2; ++j1)
#pragma unroll
          for (int j2 = 0; j2 < 2; ++j2)
            v = fma(acc[k3 * 4 + 2 * j1 + j2], C[16 * k3 + ((i1 * 2 + j1) * 2 + i2) * 2 + j2], v);
      const long long r = 2 * kk.x + i1, q = 2 * kk.y + i2;
      Kc[r * ndof - r * (r - 1) / 2 + (q - r)] = v;
    }
}

// dense [cells][ndof][ndof] -> packed upper triangle
__global__ void pack_dense_kernel(const double* __restrict__ dense, int ndof, long long cells,
                                  double* __restrict__ Kout) {
  const long long kp = (long long)ndof * (ndof + 1) / 2;
  const long long total = cells * kp;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long c = i / kp;
    long long t = i % kp;
    // row r: entries t in [r*ndof - r(r-1)/2, ...)
    int r = 0;
    long long rowlen = ndof;
    while (t >= rowlen) {
      t -= rowlen;
      ++r;
      --rowlen;
    }
    const int q = r + (int)t;
    Kout[i] = dense[(c * ndof + r) * ndof + q];
  }
}

__global__ void flag_or_kernel(const int32_t* __restrict__ flags, long long n, int* __restrict__ out) {
  int v = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    v |= flags[i];
  for (int o = 16; o > 0; o >>= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v) atomicOr(out, v);
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static romb_status ensure_pairs(romb_ctx* c) {
  if (c->d_pairs) return ROMB_OK;
  const int nB = c->nB;
  std::vector<int2> pr;
  for (int k1 = 0; k1 < nB; ++k1)
    for (int k2 = k1; k2 < nB; ++k2) pr.push_back(make_int2(k1, k2));
  romb_status s = romb_alloc_t(c, &c->d_pairs, pr.size());
  if (s != ROMB_OK) return s;
  ROMB_CUDA(cudaMemcpy(c->d_pairs, pr.data(), sizeof(int2) * pr.size(), cudaMemcpyHostToDevice));
  return ROMB_OK;
}

romb_status launch_theta(romb_ctx* c) {
  romb_status s;
  if ((s = ensure_pairs(c)) != ROMB_OK) return s;
  // the model slot of every cell, then the cells grouped by slot
  {
    FamTab T;
    for (int f = 0; f < ROMB_MAX_FAMILIES; ++f) {
      T.n_k[f] = c->fams[f].n_k;
      T.slot0[f] = c->fams[f].slot0;
      T.lo[f] = c->fams[f].lo;
      T.hi[f] = c->fams[f].hi;
    }
    cell_model_kernel<<<(c->ncells + 255) / 256, 256, 0, c->stream>>>(T, c->d_family, c->d_mu, c->ncells, c->d_slot,
                                                                      c->d_flags); ++c->launches;
    ROMB_CUDA(cudaGetLastError());
  }
  int* d_counts = (int*)(c->d_red + 64);
  family_list_kernel<<<1, 1024, 0, c->stream>>>(c->d_slot, c->ncells, c->nslots, c->d_famlist, d_counts,
                                                c->d_flags); ++c->launches;
  ROMB_CUDA(cudaGetLastError());
  int counts[ROMB_MAX_MODELS] = {0};
  if (c->nslots > 0)
    ROMB_CUDA(cudaMemcpyAsync(counts, d_counts, sizeof(int) * c->nslots, cudaMemcpyDeviceToHost, c->stream));
  ROMB_CUDA(cudaStreamSynchronize(c->stream));
  CellParams P;
  fill_cell_params(c, &P);
  int start = 0;
  for (int f = 0; f < ROMB_MAX_MODELS; ++f) {
    c->famstart[f] = start;
    c->famcount[f] = counts[f];
    start += counts[f];
  }
  // cells of a family without models (slot -1) fall in no group
  if (start != c->ncells) return ROMB_E_ARG;
  // the table of the models in use, by slot
  c->h_fams.resize(sizeof(ThetaFams));
  ThetaFams& F = *reinterpret_cast<ThetaFams*>(c->h_fams.data());
  memset(&F, 0, sizeof(F));
  for (int f = 0; f < ROMB_MAX_MODELS; ++f) {
    if (counts[f] == 0) continue;
    const RombRom& Rr = c->roms[f];
    RomDev& R = F.rom[f];
    R.At = Rr.Atfx;
    R.at_exp = Rr.at_exp;
    R.n_r = Rr.n_r;
    R.r = Rr.r;
    for (int d = 0; d < 4; ++d) {
      R.lo4[d] = Rr.lo4[d];
      R.hi4[d] = Rr.hi4[d];
    }
    gll_nodes01(Rr.r, R.g01);
    F.list[f] = c->d_famlist + c->famstart[f];
    F.count[f] = counts[f];
  }
  ThetaFams* d_fams = reinterpret_cast<ThetaFams*>(c->d_fams);
  // the table of the context: the copy is done before the next call writes it
  // again (the wait for the counts above)
  ROMB_CUDA(cudaMemcpyAsync(d_fams, &F, sizeof(F), cudaMemcpyHostToDevice, c->stream));
  cell_prep_kernel<<<(int)((13LL * c->ncells + 127) / 128), 128, 0, c->stream>>>(
      P, d_fams, c->d_slot, c->d_ctrl, c->d_mu, c->d_wts, c->d_chat, c->d_chat32, c->d_flags);
  ++c->launches;
  ROMB_CUDA(cudaGetLastError());
  if (c->plain64 && c->prec == ROMB_FP64) return launch_theta_fp64(c);
  // one launch per group of models that share the kernel's template arguments
  bool done[ROMB_MAX_MODELS] = {false};
  for (int f0 = 0; f0 < ROMB_MAX_MODELS; ++f0) {
    if (done[f0] || counts[f0] == 0) continue;
    const int ns = (c->roms[f0].n_r + 31) / 32;
    const bool r6 = c->roms[f0].r == 6;
    // Cells per CTA: every sample read serves the CT cells of a group from
    // registers and the groups' from L1; wide models keep CT = 2 for
    // registers.  A lattice of few cells takes one group of 2, so that its
    // CTAs spread over the SMs.
    const bool few = c->ncells < 8 * c->sms;
    const int ct = few || ns > 2 ? 2 : 4, cg = few ? 1 : 2, nc = ct * cg;
    ThetaCtas models;
    int grid = 0, n1max = 0, nm = 0;
    for (int f = f0; f < ROMB_MAX_MODELS; ++f) {
      const RombRom& Rr = c->roms[f];
      if (done[f] || counts[f] == 0 || (Rr.n_r + 31) / 32 != ns || (Rr.r == 6) != r6) continue;
      done[f] = true;
      models.slot[nm] = f;
      models.cta[nm++] = grid;
      n1max = std::max(n1max, Rr.r + 1);
      grid += (counts[f] + nc - 1) / nc;
    }
    models.cta[nm] = grid;
#define TH_(NS_) (few ? (r6 ? theta_kernel<NS_, 2, 1, 7> : theta_kernel<NS_, 2, 1, 0>) \
                      : (r6 ? theta_kernel<NS_, NS_ <= 2 ? 4 : 2, 2, 7> : theta_kernel<NS_, NS_ <= 2 ? 4 : 2, 2, 0>))
    auto k = ns <= 1 ? TH_(1) : ns == 2 ? TH_(2) : ns == 3 ? TH_(3) : TH_(4);
#undef TH_
    const size_t smem = 8 * std::max((size_t)2 * nc * n1max * n1max, (size_t)TH_WARPS * nc * 32 * ns);
    ROMB_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k<<<grid, 32 * TH_WARPS * cg, smem, c->stream>>>(P, d_fams, models, c->d_wts, c->d_theta, c->d_theta_hi,
                                                     c->d_theta_lo);
    ++c->launches;
    ROMB_CUDA(cudaGetLastError());
  }
  return ROMB_OK;
}

// bytes of the device table of launch_theta
size_t theta_table_bytes() { return sizeof(ThetaFams); }

romb_status launch_assemble_fp64(romb_ctx* c) {
  if (!c->plain64) {
    bool done = false;
    const romb_status sd = launch_assemble_digits(c, &done);
    if (sd != ROMB_OK || done) return sd;
  }
  // the FP64 pipe: asked for, or no device memory for the digit tiles
  const int npairs = c->nB * (c->nB + 1) / 2;
  for (int f = 0; f < ROMB_MAX_MODELS; ++f) {
    if (c->famcount[f] == 0) continue;
    const RombRom& R = c->roms[f];
    const int K = R.n_r + 1;
    const size_t smem = 8 * ((size_t)K * A64_PAIRS * 36 + A64_CELLS * (K | 1) + A64_CELLS * 145);
    static bool attr_done = false;
    if (!attr_done) {
      ROMB_CUDA(cudaFuncSetAttribute(assemble_fp64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
      attr_done = true;
    }
    dim3 grid((c->famcount[f] + A64_CELLS - 1) / A64_CELLS, (npairs + A64_PAIRS - 1) / A64_PAIRS);
    assemble_fp64_kernel<<<grid, 128, smem, c->stream>>>(R.U64, R.n_half, K, c->d_famlist + c->famstart[f],
                                                         c->famcount[f], c->d_pairs, npairs, c->ndof, c->d_theta,
                                                         c->d_chat, c->d_K); ++c->launches;
    ROMB_CUDA(cudaGetLastError());
  }
  return ROMB_OK;
}

// The FP64 contraction for a list of cells against a given U' (K rows, half
// layout) and the cells' own theta rows.
romb_status launch_assemble_cells_fp64(romb_ctx* c, const double* U, long long n_half, int K, const int* d_list,
                                       int count) {
  const int npairs = c->nB * (c->nB + 1) / 2;
  const size_t smem = 8 * ((size_t)K * A64_PAIRS * 36 + A64_CELLS * (K | 1) + A64_CELLS * 145);
  ROMB_CUDA(cudaFuncSetAttribute(assemble_fp64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  dim3 grid((count + A64_CELLS - 1) / A64_CELLS, (npairs + A64_PAIRS - 1) / A64_PAIRS);
  assemble_fp64_kernel<<<grid, 128, smem, c->stream>>>(U, n_half, K, d_list, count, c->d_pairs, npairs, c->ndof,
                                                       c->d_theta, c->d_chat, c->d_K);
  ++c->launches;
  ROMB_CUDA(cudaGetLastError());
  return ROMB_OK;
}

romb_status launch_pack_dense(romb_ctx* c, const double* d_dense) {
  pack_dense_kernel<<<4 * c->sms, 256, 0, c->stream>>>(d_dense, c->ndof, c->ncells, c->d_K); ++c->launches;
  ROMB_CUDA(cudaGetLastError());
  return ROMB_OK;
}

romb_status launch_flag_or(romb_ctx* c, int* d_any) {
  flag_or_kernel<<<c->sms, 256, 0, c->stream>>>(c->d_flags, c->ncells, d_any); ++c->launches;
  ROMB_CUDA(cudaGetLastError());
  return ROMB_OK;
}
