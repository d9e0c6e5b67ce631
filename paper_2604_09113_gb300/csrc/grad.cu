// Compliance and its gradient (discrete adjoint of the assembled model).
//
// c = f^T u with K u = f; K symmetric, so dc = 2 u^T df - sum_i u_i^T dK_i u_i.
// Cell matrices of Algorithm 4: K_i = sum_e I'_i[e] Chat_i[e] with
// I'_i = U'^T theta_i, theta_i = (rho, (1 - rho) I_r(mu_i)), so
//   u_i^T (dK_i/dx) u_i  = sum_e W_i[e] . dChat_i[e]/dx,
//   W_i[k3][i1 j1 i2 j2] = sum_{k1 k2} u[k1 i1] I'_i[k1 k2 k3 j1 j2] u[k2 i2],
//   u_i^T (dK_i/dtheta_t) u_i = Q_i[t] = sum_{k1 k2 e} U'_t[k1 k2 e] (u u Chat)[k1 k2 e],
//   dc/dmu_d = -(1 - rho) sum_t dI_r,t/dmu_d Q_i[t+1].
// W and Q are formed by one pass over U' (grad_wq_kernel); dChat/dJ is
// analytic; the traction term uses dj/dx of the loaded edges.  Control-point gradients are gathered over the sharing cells in a
// fixed order.
#include <math.h>
#include <stdio.h>

#include <algorithm>

#include "bulk.cuh"
#include "device.cuh"
#include "tables.cuh"

struct GradNodes {
  double nd[4][12];   // the GLL nodes of each threshold's interval of the model's box
  double lo4[4], hi4[4], g01[12];   // the box and the nodes on [0, 1]
};

// theta = (rho, (1 - rho) I_r(mu)) on the FP64 pipe (romb_set_fp64_arithmetic),
// one thread per (cell, coefficient), the sums in one fixed order.  0.8 ms at
// 4,096 cells, n_r = 40, r = 6 (FP64-bound).
#define GT_CELLS 32
__global__ void __launch_bounds__(256) theta_fp64_kernel(CellParams P, const double* __restrict__ At, int n_r, int r,
                                                         GradNodes N, const int* __restrict__ list, int count,
                                                         const double* __restrict__ mu,
                                                         double* __restrict__ theta) {
  __shared__ double wts[GT_CELLS][4][12];
  const int per = min(GT_CELLS, 256 / n_r), c0 = blockIdx.x * per, n1 = r + 1, tid = threadIdx.x;
  for (int i = tid; i < 4 * per; i += blockDim.x) {
    if (c0 + i / 4 >= count) break;
    double nodes[12], v[12];
    for (int k = 0; k < n1; ++k) nodes[k] = N.lo4[i % 4] + (N.hi4[i % 4] - N.lo4[i % 4]) * N.g01[k];
    lagrange1d(r, nodes, mu[4 * (long long)list[c0 + i / 4] + i % 4], v, nullptr);
    for (int k = 0; k < n1; ++k) wts[i / 4][i % 4][k] = v[k];
  }
  __syncthreads();
  const int j = tid / n_r, t = tid % n_r;
  if (j >= per || c0 + j >= count) return;
  const long long cell = list[c0 + j];
  double* th = theta + 128 * cell;
  const double* w1 = wts[j][0];
  double acc = 0.0;
  const double* a = At + t;
  for (int g4 = 0; g4 < n1; ++g4)
    for (int g3 = 0; g3 < n1; ++g3) {
      const double w34 = wts[j][2][g3] * wts[j][3][g4];
      for (int g2 = 0; g2 < n1; ++g2) {
        double inner = 0.0;
#pragma unroll 7
        for (int g1 = 0; g1 < n1; ++g1, a += n_r) inner = fma(__ldg(a), w1[g1], inner);
        acc = fma(wts[j][1][g2] * w34, inner, acc);
      }
    }
  if (t == 0) th[0] = P.rho;
  th[1 + t] = (1.0 - P.rho) * acc;
}

// W and Q of CPC cells by one CTA, thread (cell, e = (k3, j1, j2)), the pairs
// k1 <= k2 in order with U' of the next pair copied meanwhile (cp.async):
//   I'_e = sum_t theta_t U'_t[e],  W += (u u) I',  Y_e = (u u) Chat,
//   Q_t += sum_e U'_t[e] Y_e,
// all in FP64: W and Q cancel from |u|^2 to the strain energy and lose about six
// digits, so 56-bit fixed point (tried: 1.6e-9 in dc/dmu against 3e-10) does
// not serve.  CPC = 8 fills nine warps, several CTAs an SM; lattices of few
// cells take fewer cells per CTA, so that the sequence of pairs is walked on
// all SMs.  Bound: FP64 issue (2 K 36 + 600 FMA per cell and pair).  Before, 36
// of 64 lanes worked, in CTAs one to an SM: 4,096 cells, n_r = 40: 61.5 -> 36.8 ms
// (17.8 G FMA: 34 ms at the measured FP64 rate); 35 cells: 9.3 -> 7.2.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
template <int CPC>
__global__ void __launch_bounds__(CPC == 1 ? 64 : CPC == 2 ? 96 : CPC == 4 ? 160 : 288) grad_wq_kernel(
    CellParams P, const double* __restrict__ U, long long n_half, int K, const int* __restrict__ list, int count,
    const int2* __restrict__ pairs, int npairs, const double* __restrict__ theta, const double* __restrict__ chat,
    const double* __restrict__ unodal, double* __restrict__ Wout, double* __restrict__ Qout) {
  extern __shared__ __align__(16) unsigned char gsm[];
  const int ND = 2 * P.nB, LD = 38;                    // row stride of U' (a multiple of 16 bytes)
  double* Ut = reinterpret_cast<double*>(gsm);         // [2][K][LD]
  double* Y = Ut + 2 * K * LD;                         // [CPC][36]
  double* uu = Y + CPC * 36;                           // [2][CPC][8] products of u of a pair
  double* su = uu + 2 * CPC * 8;                       // [CPC][2 nB]
  double* sth = su + CPC * ND;                         // [CPC][K]
  const int tid = threadIdx.x, nt = blockDim.x;
  const int j = tid / 36, e = tid % 36;
  const int ci = blockIdx.x * CPC + j;
  const bool valid = j < CPC && ci < count;
  const int p = P.p;
  const long long gnx = (long long)p * P.nx + 1;
  auto cell_of = [&](int jj) { return blockIdx.x * CPC + jj < count ? (long long)list[blockIdx.x * CPC + jj] : -1LL; };
  auto stage = [&](int pr) {   // U' of pair pr: K rows of 288 bytes
    double* dst = Ut + (size_t)(pr & 1) * K * LD;
    for (int i = tid; i < K * 18; i += nt)
      cp_async16(dst + (i / 18) * LD + (i % 18) * 2, U + (long long)(i / 18) * n_half + (long long)pr * 36 + (i % 18) * 2);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  stage(0);
  for (int i = tid; i < CPC * ND; i += nt) {
    const long long c = cell_of(i / ND);
    const int d = i % ND, k = d >> 1, a = k % (p + 1), b = k / (p + 1);
    const int cx = c < 0 ? 0 : (int)(c % P.nx), cy = c < 0 ? 0 : (int)(c / P.nx);
    su[i] = c >= 0 ? unodal[2 * ((long long)(p * cy + b) * gnx + (p * cx + a)) + (d & 1)] : 0.0;
  }
  for (int i = tid; i < CPC * K; i += nt) {
    const long long c = cell_of(i / K);
    sth[i] = c >= 0 ? theta[c * 128 + i % K] : 0.0;
  }
  // Chat of the thread's (k3, j1, j2) and of (k3, j2, j1), by 2 i1 + i2
  const long long cell = valid ? list[ci] : 0;
  const int k3 = e >> 2, j1 = (e >> 1) & 1, j2 = e & 1;
  const int swp = (j1 != j2) ? 3 : 0;   // lane of (k3, j2, j1): groups of four do not cross warps
  double C[4], Cs[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int o = 16 * k3 + 8 * (i >> 1) + 2 * (i & 1);
    C[i] = valid ? chat[cell * 144 + o + 4 * j1 + j2] : 0.0;
    Cs[i] = valid ? chat[cell * 144 + o + 4 * j2 + j1] : 0.0;
  }
  // products u[2 k1 + i1] u[2 k2 + i2] (0..3) and u[2 k2 + i1] u[2 k1 + i2]
  // (4..7, zero on the diagonal) of pair pr
  auto products = [&](int pr) {
    const int2 kk = pairs[pr];
    for (int i = tid; i < CPC * 8; i += nt) {
      const double* u = su + (i >> 3) * ND;
      const int i1 = (i >> 1) & 1, i2 = i & 1, sw = (i >> 2) & 1;
      uu[((pr & 1) * CPC) * 8 + i] =
          sw && kk.x == kk.y ? 0.0 : u[2 * (sw ? kk.y : kk.x) + i1] * u[2 * (sw ? kk.x : kk.y) + i2];
    }
  };
  __syncthreads();
  products(0);
  double w[4] = {0.0, 0.0, 0.0, 0.0};   // W by 2 i1 + i2
  double q[4] = {0.0, 0.0, 0.0, 0.0};   // Q of the items (cell, t) = tid, tid + nt, ..
  const double* th = sth + (j < CPC ? j : 0) * K;
  for (int pr = 0; pr < npairs; ++pr) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const double* Uc = Ut + (size_t)(pr & 1) * K * LD;
    if (pr + 1 < npairs) stage(pr + 1);
    double Ie = 0.0;
#pragma unroll 4
    for (int t = 0; t < K; ++t) Ie = fma(th[t], Uc[t * LD + e], Ie);
    const double Is = __shfl_xor_sync(0xffffffffu, Ie, swp);
    const double* ab = uu + ((pr & 1) * CPC + (j < CPC ? j : 0)) * 8;
    double y = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double a = ab[i], b = ab[4 + i];
      w[i] = fma(a, Ie, fma(b, Is, w[i]));
      y = fma(a, C[i], fma(b, Cs[i], y));
    }
    if (j < CPC) Y[j * 36 + e] = y;
    __syncthreads();
    if (pr + 1 < npairs) products(pr + 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int item = tid + k * nt;
      if (item >= CPC * K) break;
      const double2* Yc = reinterpret_cast<const double2*>(Y + (item / K) * 36);
      const double2* Ur = reinterpret_cast<const double2*>(Uc + (item % K) * LD);
      double s = 0.0;
#pragma unroll 6
      for (int ee = 0; ee < 18; ++ee) {
        const double2 a = Ur[ee], b = Yc[ee];
        s = fma(a.x, b.x, s);
        s = fma(a.y, b.y, s);
      }
      q[k] += s;
    }
  }
  if (valid) {
    double* Wc = Wout + cell * 144;
#pragma unroll
    for (int i = 0; i < 4; ++i) Wc[16 * k3 + 8 * (i >> 1) + 4 * j1 + 2 * (i & 1) + j2] = w[i];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int item = tid + k * nt;
    if (item >= CPC * K) break;
    const long long c = cell_of(item / K);
    if (c >= 0) Qout[c * 128 + item % K] = q[k];
  }
}

// Per cell: -sum_e W[e] dChat[e]/dx for each local control point.  A CTA takes
// 32 cells (lanes), its nine warps the nodes k3, whose terms are then added in
// order; one thread per cell ran the FP64 chains of all nodes alone
// (4,096 cells: 2.6 -> 0.5 ms).
__global__ void __launch_bounds__(288) grad_chain_kernel(CellParams P, const double* __restrict__ ctrl,
                                                         const double* __restrict__ W, double* __restrict__ gloc) {
  extern __shared__ double gc_smem[];   // [9][2 (m+1)^2][32]
  const int lane = threadIdx.x & 31, k3 = threadIdx.x >> 5;
  const int m = P.m, nx = P.nx;
  const int ncp = (m + 1) * (m + 1);
  const long long cell = (long long)blockIdx.x * 32 + lane;
  auto sacc = [&](int k, int i) -> double& { return gc_smem[(k * 2 * ncp + i) * 32 + lane]; };
  if (cell < P.ncells) {
    const int cx = (int)(cell % nx), cy = (int)(cell / nx);
    const double qn[3] = {0.0, 0.5, 1.0};
    const double* Wc = W + cell * 144;
    const double x1 = qn[k3 % 3], x2 = qn[k3 / 3];
    double x[2], J[2][2];
    map_eval(ctrl, nx, m, cx, cy, x1, x2, x, J);
    const double det = J[0][0] * J[1][1] - J[0][1] * J[1][0];
    const double G[2][2] = {{J[1][1] / det, -J[0][1] / det}, {-J[1][0] / det, J[0][0] / det}};
    double v1[5], d1[5], v2[5], d2[5];
    map_basis1d(m, x1, v1, d1);
    map_basis1d(m, x2, v2, d2);
    // Chat at this node (needed for the det J term)
    double Ch[16];
    for (int i = 0; i < 2; ++i)
      for (int j = 0; j < 2; ++j)
        for (int k = 0; k < 2; ++k)
          for (int l = 0; l < 2; ++l) {
            const double GGt = G[j][0] * G[l][0] + G[j][1] * G[l][1];
            const double v = P.lam * (G[j][i] * G[l][k]) + P.mu * ((i == k ? GGt : 0.0) + G[j][k] * G[l][i]);
            Ch[((i * 2 + j) * 2 + k) * 2 + l] = det * v;
          }
    for (int b = 0; b <= m; ++b)
      for (int a = 0; a <= m; ++a) {
        const double dN[2] = {d1[a] * v2[b], v1[a] * d2[b]};
        for (int comp = 0; comp < 2; ++comp) {
          // dJ[r][s] = delta(r, comp) dN[s];  H = G dJ G, tr(G dJ) = sum_s G[s][comp] dN[s]
          const double tr = G[0][comp] * dN[0] + G[1][comp] * dN[1];
          double H[2][2];
          for (int r = 0; r < 2; ++r)
            for (int s = 0; s < 2; ++s) H[r][s] = G[r][comp] * (dN[0] * G[0][s] + dN[1] * G[1][s]);
          double acc = 0.0;
          for (int i = 0; i < 2; ++i)
            for (int j = 0; j < 2; ++j)
              for (int k = 0; k < 2; ++k)
                for (int l = 0; l < 2; ++l) {
                  // d(G_jm C_imkn G_ln) with dG = -H
                  const double dGGt = H[j][0] * G[l][0] + H[j][1] * G[l][1] + G[j][0] * H[l][0] + G[j][1] * H[l][1];
                  const double dv = P.lam * (H[j][i] * G[l][k] + G[j][i] * H[l][k]) +
                                    P.mu * ((i == k ? dGGt : 0.0) + H[j][k] * G[l][i] + G[j][k] * H[l][i]);
                  const int idx = ((i * 2 + j) * 2 + k) * 2 + l;
                  acc += Wc[16 * k3 + idx] * (tr * Ch[idx] - det * dv);
                }
          sacc(k3, 2 * (b * (m + 1) + a) + comp) = acc;
        }
      }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 32 * 2 * ncp; i += blockDim.x) {
    const int c = i / (2 * ncp), o = i % (2 * ncp);
    if ((long long)blockIdx.x * 32 + c >= P.ncells) break;
    double s = 0.0;
    for (int k = 0; k < 9; ++k) s -= gc_smem[(k * 2 * ncp + o) * 32 + c];
    gloc[((long long)blockIdx.x * 32 + c) * 2 * ncp + o] = s;
  }
}

// The traction term 2 u . df/dx of the cells on loaded lattice edges, added to
// their control-point gradients; one thread per boundary cell.
__global__ void grad_traction_kernel(CellParams P, const double* __restrict__ ctrl,
                                     const double* __restrict__ eiv, const double* __restrict__ unodal,
                                     const double* __restrict__ trac, double* __restrict__ gloc) {
  const int nx = P.nx, ny = P.ny, m = P.m, p = P.p;
  int i = blockIdx.x * blockDim.x + threadIdx.x;   // bottom row, top row, then the sides between
  int cx, cy;
  if (i < nx) {
    cx = i;
    cy = 0;
  } else if (i < nx + (ny > 1 ? nx : 0)) {
    cx = i - nx;
    cy = ny - 1;
  } else {
    i -= nx + (ny > 1 ? nx : 0);
    const int sides = nx > 1 ? 2 : 1;
    if (i >= sides * (ny - 2)) return;
    cx = (i % sides) ? nx - 1 : 0;
    cy = 1 + i / sides;
  }
  const long long cell = cx + (long long)nx * cy;
  double* out = gloc + cell * (m + 1) * (m + 1) * 2;
  // traction term: f[2k+i] = int b_k(t) t_i j(t) dt over the solid part of loaded edges
  const long long gnx = (long long)p * nx + 1;
  for (int e = 0; e < 4; ++e) {
    const bool on = (e == 0 && cx == 0) || (e == 1 && cx == nx - 1) || (e == 2 && cy == 0) || (e == 3 && cy == P.ny - 1);
    const double t0 = trac[2 * e], t1 = trac[2 * e + 1];
    if (!on || (t0 == 0.0 && t1 == 0.0)) continue;
    const double* o = eiv + (cell * 4 + e) * ROMB_EIV;   // the edge's solid intervals
    const int nint = (int)o[0];
    for (int iv = 0; iv < nint; ++iv) {
      const double lo = o[1 + 2 * iv], len = o[2 + 2 * iv] - lo;
      for (int qq = 0; qq < ROMB_NQ; ++qq) {
        const double t = lo + len * P.gq_x[qq];
        // the edge tangent dx/dt: on the edge one factor of the tensor map basis
        // is a Kronecker delta, so only the edge's m+1 control points vary
        double vs[5], ds[5];
        map_basis1d(m, t, vs, ds);
        double tg[2] = {0.0, 0.0};
        for (int s2 = 0; s2 <= m; ++s2) {
          const int ea = e == 0 ? 0 : e == 1 ? m : s2, eb = e == 2 ? 0 : e == 3 ? m : s2;
          const double* X = ctrl_pt(ctrl, nx, m, cx, cy, ea, eb);
          tg[0] = fma(ds[s2], X[0], tg[0]);
          tg[1] = fma(ds[s2], X[1], tg[1]);
        }
        const double jj = hypot(tg[0], tg[1]);
        double bv[ROMB_MAX_P + 1];
        cell_basis1d(P, t, bv, nullptr);
        // u . (b t) along the edge
        double ub = 0.0;
        for (int s = 0; s <= p; ++s) {
          const int k = e == 0 ? (p + 1) * s : e == 1 ? p + (p + 1) * s : e == 2 ? s : s + (p + 1) * p;
          const int a = k % (p + 1), bb = k / (p + 1);
          const long long node = (long long)(p * cy + bb) * gnx + (p * cx + a);
          ub += bv[s] * (unodal[2 * node] * t0 + unodal[2 * node + 1] * t1);
        }
        const double wq = len * P.gq_w[qq];
        for (int s2 = 0; s2 <= m; ++s2) {   // d N / dt along the edge: ds for the edge's control points
          const int ea = e == 0 ? 0 : e == 1 ? m : s2, eb = e == 2 ? 0 : e == 3 ? m : s2;
          for (int comp = 0; comp < 2; ++comp)
            out[2 * (eb * (m + 1) + ea) + comp] += 2.0 * wq * ub * tg[comp] * ds[s2] / jj;
        }
      }
    }
  }
}

// dc/dmu_d = -(1 - rho) sum_t dI_r,t/dmu_d Q[t+1]: one warp per GM_CELLS cells,
// lanes over the grid (a sample read serves all of them).
#define GM_CELLS 4
__global__ void __launch_bounds__(128) grad_mu_kernel(CellParams P, const double* __restrict__ A, int n_r, int r,
                                                      GradNodes N, const int* __restrict__ list, int count,
                                                      const double* __restrict__ mu, const double* __restrict__ Q,
                                                      double* __restrict__ dmu) {
  __shared__ double sv[4][GM_CELLS][4][12], sd[4][GM_CELLS][4][12], sq[4][GM_CELLS][128];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c0 = (blockIdx.x * 4 + warp) * GM_CELLS;
  if (c0 >= count) return;
  const int n1 = r + 1;
  if (lane < 4 * GM_CELLS) {   // lane = (cell, threshold)
    const int j = lane >> 2, k = lane & 3;
    double nodes[12], v[12], d[12];
    for (int i = 0; i < n1; ++i) nodes[i] = N.nd[k][i];
    const long long c = list[min(c0 + j, count - 1)];
    lagrange1d(r, nodes, mu[4 * c + k], v, d);
    for (int i = 0; i < n1; ++i) {
      sv[warp][j][k][i] = v[i];
      sd[warp][j][k][i] = d[i];
    }
  }
  for (int j = 0; j < GM_CELLS; ++j) {
    const long long c = list[min(c0 + j, count - 1)];
    for (int t = lane; t < n_r; t += 32) sq[warp][j][t] = Q[c * 128 + 1 + t];
  }
  __syncwarp();
  double s[GM_CELLS][4];
#pragma unroll
  for (int j = 0; j < GM_CELLS; ++j)
#pragma unroll
    for (int k = 0; k < 4; ++k) s[j][k] = 0.0;
  const int ng = n1 * n1 * n1 * n1;
  for (int gg = lane; gg < ng; gg += 32) {
    double z[GM_CELLS];
#pragma unroll
    for (int j = 0; j < GM_CELLS; ++j) z[j] = 0.0;
#pragma unroll 4
    for (int t = 0; t < n_r; ++t) {
      const double a = __ldg(A + (long long)t * ng + gg);
#pragma unroll
      for (int j = 0; j < GM_CELLS; ++j) z[j] = fma(a, sq[warp][j][t], z[j]);
    }
    const int g1 = gg % n1, g2 = (gg / n1) % n1, g3 = (gg / (n1 * n1)) % n1, g4 = gg / (n1 * n1 * n1);
#pragma unroll
    for (int j = 0; j < GM_CELLS; ++j) {
      const double (*v)[12] = sv[warp][j], (*d)[12] = sd[warp][j];
      s[j][0] = fma(z[j], d[0][g1] * v[1][g2] * v[2][g3] * v[3][g4], s[j][0]);
      s[j][1] = fma(z[j], v[0][g1] * d[1][g2] * v[2][g3] * v[3][g4], s[j][1]);
      s[j][2] = fma(z[j], v[0][g1] * v[1][g2] * d[2][g3] * v[3][g4], s[j][2]);
      s[j][3] = fma(z[j], v[0][g1] * v[1][g2] * v[2][g3] * d[3][g4], s[j][3]);
    }
  }
#pragma unroll
  for (int j = 0; j < GM_CELLS; ++j)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double t = warp_sum(s[j][k]);
      if (lane == 0 && c0 + j < count) dmu[4 * (long long)list[c0 + j] + k] = -(1.0 - P.rho) * t;
    }
}

// global control point gradient: sum over the cells sharing the point
__global__ void grad_gather_kernel(CellParams P, const double* __restrict__ gloc, double* __restrict__ out) {
  const int m = P.m, nx = P.nx, ny = P.ny;
  const long long gnx = (long long)m * nx + 1, n = gnx * ((long long)m * ny + 1);
  const int ncp = (m + 1) * (m + 1);
  for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < n; id += (long long)gridDim.x * blockDim.x) {
    const int gx = (int)(id % gnx), gy = (int)(id / gnx);
    double s0 = 0.0, s1 = 0.0;
    for (int dy = (gy % m == 0) ? -1 : 0; dy <= 0; ++dy)
      for (int dx = (gx % m == 0) ? -1 : 0; dx <= 0; ++dx) {
        const int cx = gx / m + dx, cy = gy / m + dy;
        if (cx < 0 || cy < 0 || cx >= nx || cy >= ny) continue;
        const int a = gx - m * cx, b = gy - m * cy;
        const double* l = gloc + ((long long)cy * nx + cx) * ncp * 2 + 2 * (b * (m + 1) + a);
        s0 += l[0];
        s1 += l[1];
      }
    out[2 * id] = s0;
    out[2 * id + 1] = s1;
  }
}

// The per-threshold GLL nodes of a model's box (as the theta kernel forms them).
static GradNodes grad_nodes(const RombRom& R) {
  GradNodes N;
  memset(&N, 0, sizeof(N));
  double* g1 = N.g01;
  gll_nodes01(R.r, g1);
  for (int k = 0; k < 4; ++k) {
    N.lo4[k] = R.lo4[k];
    N.hi4[k] = R.hi4[k];
    for (int i = 0; i <= R.r; ++i) N.nd[k][i] = R.lo4[k] + (R.hi4[k] - R.lo4[k]) * g1[i];
  }
  return N;
}

// The gradient's kernels with the given intermediate arrays: W [cells][144],
// Q [cells][128], gloc [cells][2 (m+1)^2].
static romb_status grad_kernels(romb_ctx* c, double* W, double* Q, double* gloc, double* d_dctrl, double* d_dmu) {
  CellParams P;
  fill_cell_params(c, &P);
  const int npairs = c->nB * (c->nB + 1) / 2;
  for (int f = 0; f < ROMB_MAX_MODELS; ++f) {
    const int count = c->famcount[f];
    if (count == 0) continue;
    const RombRom& R = c->roms[f];
    const int K = R.n_r + 1;
    const int* list = c->d_famlist + c->famstart[f];
    const int cpc = count <= 2 * c->sms ? 1 : count <= 4 * c->sms ? 2 : count <= 8 * c->sms ? 4 : 8;
    const size_t smem = 8 * ((size_t)2 * K * 38 + cpc * (36 + 16 + 2 * c->nB + K));
    auto k = cpc == 1 ? grad_wq_kernel<1> : cpc == 2 ? grad_wq_kernel<2> : cpc == 4 ? grad_wq_kernel<4>
                                                                           : grad_wq_kernel<8>;
    ROMB_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k<<<(count + cpc - 1) / cpc, (36 * cpc + 31) / 32 * 32, smem, c->stream>>>(
        P, R.U64, R.n_half, K, list, count, c->d_pairs, npairs, c->d_theta, c->d_chat,
        c->lane[0].d_u, W, Q);
    ++c->launches;
    ROMB_CUDA(cudaGetLastError());
    if (d_dmu) {
      grad_mu_kernel<<<(count + 4 * GM_CELLS - 1) / (4 * GM_CELLS), 128, 0, c->stream>>>(
          P, R.A, R.n_r, R.r, grad_nodes(R), list, count, c->d_mu, Q, d_dmu);
      ++c->launches;
      ROMB_CUDA(cudaGetLastError());
    }
  }
  const size_t csm = 8 * (size_t)9 * 2 * (c->m + 1) * (c->m + 1) * 32;
  ROMB_CUDA(cudaFuncSetAttribute(grad_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)csm));
  grad_chain_kernel<<<(c->ncells + 31) / 32, 288, csm, c->stream>>>(P, c->d_ctrl, W, gloc);
  const int nb = 2 * (c->nx + c->ny);
  grad_traction_kernel<<<(nb + 31) / 32, 32, 0, c->stream>>>(P, c->d_ctrl, c->d_eiv, c->lane[0].d_u,
                                                             c->lane[0].d_traction, gloc);
  grad_gather_kernel<<<4 * c->sms, 256, 0, c->stream>>>(P, gloc, d_dctrl);
  c->launches += 3;
  ROMB_CUDA(cudaGetLastError());
  return ROMB_OK;
}

romb_status launch_grad(romb_ctx* c, double* d_dctrl, double* d_dmu) {
  romb_status s;
  if (!c->d_gW) {
    if ((s = romb_alloc_t(c, &c->d_gW, (size_t)c->ncells * 144)) != ROMB_OK) return s;
    if ((s = romb_alloc_t(c, &c->d_gQ, (size_t)c->ncells * 128)) != ROMB_OK) return s;
    const int ncp = (c->m + 1) * (c->m + 1);
    if ((s = romb_alloc_t(c, &c->d_gloc, (size_t)c->ncells * ncp * 2)) != ROMB_OK) return s;
  }
  return grad_kernels(c, c->d_gW, c->d_gQ, c->d_gloc, d_dctrl, d_dmu);
}

// launch_grad with caller-supplied intermediate arrays (the no-allocation
// gradient).
romb_status launch_grad_scratch(romb_ctx* c, double* W, double* Q, double* gloc, double* d_dctrl, double* d_dmu) {
  return grad_kernels(c, W, Q, gloc, d_dctrl, d_dmu);
}

// theta of every cell on the FP64 pipe (romb_set_fp64_arithmetic).
romb_status launch_theta_fp64(romb_ctx* c) {
  CellParams P;
  fill_cell_params(c, &P);
  for (int f = 0; f < ROMB_MAX_MODELS; ++f) {
    const int count = c->famcount[f];
    if (count == 0) continue;
    const RombRom& R = c->roms[f];
    const int per = std::min(GT_CELLS, 256 / R.n_r);
    theta_fp64_kernel<<<(count + per - 1) / per, 256, 0, c->stream>>>(
        P, R.At, R.n_r, R.r, grad_nodes(R), c->d_famlist + c->famstart[f], count, c->d_mu, c->d_theta);
    ++c->launches;
    ROMB_CUDA(cudaGetLastError());
  }
  return ROMB_OK;
}
