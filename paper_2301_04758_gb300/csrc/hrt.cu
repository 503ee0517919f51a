// Hybridized Raviart-Thomas (HRT) VEF solve: element-local elimination, the reduced
// system for the Lagrange multiplier, and the recovery of the scalar flux and current
// (paper Sec. "Hybridization": "Extension to VEF" and "Implementation Details").
//
// Per element K the local mixed system couples the broken RT_p current J and the Y_p
// scalar flux phi:
//     [ A  G ] [J  ]   [g - C2 lambda]        A  = int sigma_t v.J + int_Gb (1/E_b)(v.E n)(J.n)
//     [ D  Ma] [phi] = [f            ]        G  = -int grad v : E phi   (Piola gradient)
//                                             D  = int u div J,  Ma = int sigma_a u phi
//                                             g  = int v.Q1 + 2 int_Gb (1/E_b)(v.E n) J_in
//                                             f  = int u Q0
// with C2 lambda = int_G0 (v.{E} n) lambda (the face multipliers) and the constraint
// C1 J = int_G0 mu [[J.n]] = 0.  hrt_local_kernel assembles these blocks for one element per
// CTA in shared memory (the map's derivatives and the Eddington tensor evaluated once per
// Gauss point; D and C1 are the same on every element and come from host tables);
// hrt_invert_kernel, at a higher occupancy, inverts [[A, G], [D, Ma]] by Gauss-Jordan
// elimination with partial pivoting in registers, and forms the element's share of the reduced
// system (the two kernels and the recovery: 3.0 ms at 128^2 Q2, 7.5 when divergent lanes, zero
// components and shared-memory traffic took most of the issue),
//     H_e = C1 W C2,   r_e = C1 (W g + X f),   [[W, X], [Y, Z]] = [[A, G], [D, Ma]]^{-1}.
// The multiplier system H lambda = r (H = sum_e H_e over the interior faces, not symmetric
// for a general Eddington tensor) is solved by BiCGStab with a two-level additive Schwarz
// preconditioner (element patches plus a coarse bilinear space), the matrix applied face by
// face from the two sides' rows of H_e (no atomics) and the Krylov scalars kept on the
// device.  hrt_recover_kernel then forms J and phi element by element.
//
// Spaces (identical to the CPU reference of this discretisation): RT_p on the reference
// square with the x component in Q_{p+1} x Q_p and the y component in Q_p x Q_{p+1}, nodal
// at the p+2 Gauss-Lobatto points across (normal flux on the end nodes) and the p+1
// Gauss-Legendre points along; contravariant Piola transform v = F v_hat / J, whose
// gradient (d v / d xi) F^{-1} uses the map's second derivatives; the transport's DG basis
// for phi; degree-p Lagrange multipliers at the p+1 Gauss-Legendre points of each interior
// face; the transport's Gauss-Legendre rules, so the Eddington tensor is P / phi from the
// closure pass's nodal moments.  Interior faces: vertical first (j (nx-1) + i), then
// horizontal ((nx-1) ny + j nx + i).
#include <algorithm>
#include <cmath>
#include <memory>

#include "device.cuh"

namespace vef {
namespace {

// 1D tables of one order p and mesh order m (host): index k < nq is the Gauss point s_k, nq is
// the point 0 and nq + 1 the point 1.
struct HrtTab {
  int p, m, nq;
  double w[kMaxNq];                               // Gauss weights
  double cl[kMaxP + 2][kMaxNq + 2], dcl[kMaxP + 2][kMaxNq + 2];   // p+2 Gauss-Lobatto nodes
  double op[kMaxP + 1][kMaxNq + 2], dop[kMaxP + 1][kMaxNq + 2];   // p+1 Gauss-Legendre nodes
  double dg[kMaxP + 1][kMaxNq + 2];               // DG basis (p+1 Gauss-Lobatto nodes)
  double mv[kMaxM + 1][kMaxNq + 2], md[kMaxM + 1][kMaxNq + 2], mdd[kMaxM + 1][kMaxNq + 2];
};

HrtTab make_hrt_tab(int p, int m) {
  HrtTab t{};
  t.p = p;
  t.m = m;
  t.nq = p + 2;
  double s[kMaxNq], gw[kMaxNq];
  gauss_legendre(t.nq, s, gw);
  for (int k = 0; k < t.nq; ++k) t.w[k] = gw[k];
  double cl[kMaxP + 2], op[kMaxP + 1], dg[kMaxP + 1], mn[kMaxM + 1], dummy[kMaxNq];
  gll_nodes(p + 1, cl);
  gauss_legendre(p + 1, op, dummy);
  gll_nodes(p, dg);
  gll_nodes(m, mn);
  for (int k = 0; k < t.nq + 2; ++k) {
    const double x = k < t.nq ? s[k] : (k == t.nq ? 0.0 : 1.0);
    double v[kMaxP + 2], d[kMaxP + 2];
    lagrange_eval(p + 2, cl, x, v, d);
    for (int a = 0; a < p + 2; ++a) { t.cl[a][k] = v[a]; t.dcl[a][k] = d[a]; }
    lagrange_eval(p + 1, op, x, v, d);
    for (int a = 0; a < p + 1; ++a) { t.op[a][k] = v[a]; t.dop[a][k] = d[a]; }
    lagrange_eval(p + 1, dg, x, v, d);
    for (int a = 0; a < p + 1; ++a) t.dg[a][k] = v[a];
    // control-point basis: values, first and second derivatives (second by differencing the
    // exact first derivatives would lose digits; use the product-rule sum instead)
    lagrange_eval(m + 1, mn, x, v, d);
    for (int a = 0; a <= m; ++a) {
      t.mv[a][k] = v[a];
      t.md[a][k] = d[a];
      double s2 = 0.0;
      for (int i = 0; i <= m; ++i) {
        if (i == a) continue;
        for (int j = 0; j <= m; ++j) {
          if (j == a || j == i) continue;
          double term = 1.0 / ((mn[a] - mn[i]) * (mn[a] - mn[j]));
          for (int c = 0; c <= m; ++c)
            if (c != a && c != i && c != j) term *= (x - mn[c]) / (mn[a] - mn[c]);
          s2 += term;
        }
      }
      t.mdd[a][k] = s2;
    }
  }
  return t;
}

template <int P>
struct HrtShape {
  static constexpr int Q = P + 1, N = Q * Q, NQ = P + 2, NQ2 = NQ * NQ;
  static constexpr int NX = (P + 2) * (P + 1);   // dofs of one component
  static constexpr int NJ = 2 * NX;
  static constexpr int MM = NJ + N;               // local system size
  static constexpr int LD = MM + 1;
  static constexpr int NL = P + 1, NL4 = 4 * NL;
};

// the nonzero component of reference RT basis function a (component a / NX) at table points
// (kx, ky): value, d/dxi, d/deta
template <int P>
void rt_ref(const HrtTab& t, int a, int kx, int ky, double& v, double& dxi, double& deta) {
  using S = HrtShape<P>;
  if (a < S::NX) {
    const int ax = a % (P + 2), bx = a / (P + 2);
    v = t.cl[ax][kx] * t.op[bx][ky];
    dxi = t.dcl[ax][kx] * t.op[bx][ky];
    deta = t.cl[ax][kx] * t.dop[bx][ky];
  } else {
    const int b = a - S::NX, ay = b % (P + 1), by = b / (P + 1);
    v = t.op[ay][kx] * t.cl[by][ky];
    dxi = t.dop[ay][kx] * t.cl[by][ky];
    deta = t.op[ay][kx] * t.dcl[by][ky];
  }
}

// face-point table indices of face f, point k
__host__ __device__ __forceinline__ void face_pt(int f, int k, int nq, int& kx, int& ky) {
  kx = f == 0 ? k : (f == 1 ? nq + 1 : (f == 2 ? k : nq));
  ky = f == 0 ? nq : (f == 1 ? k : (f == 2 ? nq + 1 : k));
}

struct HrtIn {
  const double* ctrl;   // [E][(m+1)^2][2]
  const double* Mm;     // [E][n][n] mass matrices
  const double* nds;    // [E][4][nq][2]
  const double* sigma_t;
  const double* sigma_s;
  const double* phi;    // [E][n] transport scalar flux (nodal)
  const double* P;      // [3][E][n] second moment (nodal)
  const double* Eb;     // [nbf][nq]
  const double* Jin;    // [nbf][nq]
  const double* Q0;     // [E][n] nodal
  const double* Q1;     // [2][E][n] nodal or null
};

struct HrtOut {
  double* Li;   // [E][MM][MM] inverse of the local system (row-major)
  double* C2;   // [E][NJ][NL4]
  double* g;    // [E][NJ]
  double* f;    // [E][N]
  double* He;   // [E][NL4][NL4]
  double* re;   // [E][NL4]
};

// What the elimination needs that depends on no element, formed once per mesh on the host from
// the 1D tables and kept on the device with the handle.  Points: NQ2 volume points (k1 + NQ k2),
// then NQ per face.
template <int P>
struct HrtRef {
  using S = HrtShape<P>;
  static constexpr int NPT = S::NQ2 + 4 * S::NQ, NT = S::NJ * (S::NJ + 1) / 2;
  double D[S::N * S::NJ];           // int u div_hat v_hat (the Piola transform makes int u div J dx this)
  double C1[S::NL4 * S::NJ];        // int_f mu (v_hat . n_hat) (rows of boundary faces are dropped per element)
  double rs[S::NQ2][S::NJ];         // the RT functions' nonzero component at the volume points: value,
  double r0[S::NQ2][S::NJ], r1[S::NQ2][S::NJ];   // d/dxi, d/deta
  double fv[4 * S::NQ][S::NJ];      // its value at the face points
  double c2[S::NL4][S::NQ][S::NJ];  // times the multiplier basis: op_t(s_k) fv
  double bt[NPT][S::N];             // DG basis at the points
  double w[NPT];                    // w_k1 w_k2, and w_k at the face points
  double gt[5][(kMaxM + 1) * (kMaxM + 1)][NPT];  // control-point basis: d/dxi, d/deta, second derivatives xx, xy, yy
  int tri[NT];                      // (r << 8) | c, c >= r: the upper triangle of A
};

template <int P>
static void make_hrt_ref(const HrtTab& t, HrtRef<P>& o) {
  using S = HrtShape<P>;
  using R = HrtRef<P>;
  constexpr int Q = P + 1, N = S::N, NQ = S::NQ, NQ2 = S::NQ2, NJ = S::NJ, NL = S::NL;
  for (int pt = 0; pt < R::NPT; ++pt) {
    const int f = pt < NQ2 ? -1 : (pt - NQ2) / NQ, k = pt < NQ2 ? 0 : (pt - NQ2) % NQ;
    int kx = pt % NQ, ky = pt / NQ;
    if (f >= 0) face_pt(f, k, NQ, kx, ky);
    o.w[pt] = f < 0 ? t.w[kx] * t.w[ky] : t.w[k];
    for (int j = 0; j < N; ++j) o.bt[pt][j] = t.dg[j % Q][kx] * t.dg[j / Q][ky];
    const int q = t.m + 1;
    for (int c = 0; c < q * q; ++c) {
      const int a = c % q, b = c / q;
      o.gt[0][c][pt] = t.md[a][kx] * t.mv[b][ky];
      o.gt[1][c][pt] = t.mv[a][kx] * t.md[b][ky];
      o.gt[2][c][pt] = t.mdd[a][kx] * t.mv[b][ky];
      o.gt[3][c][pt] = t.md[a][kx] * t.md[b][ky];
      o.gt[4][c][pt] = t.mv[a][kx] * t.mdd[b][ky];
    }
    for (int a = 0; a < NJ; ++a) {
      double v, dx, dy;
      rt_ref<P>(t, a, kx, ky, v, dx, dy);
      if (f < 0) {
        o.rs[pt][a] = v;
        o.r0[pt][a] = dx;
        o.r1[pt][a] = dy;
      } else {
        o.fv[pt - NQ2][a] = v;
        for (int tt = 0; tt < NL; ++tt) o.c2[f * NL + tt][k][a] = t.op[tt][k] * v;
      }
    }
  }
  // D and C1 round the same way on every element, and phi collects what breaks the balance of
  // D's columns with C1's: the order of these products is kept (another one tripled phi's error
  // at p = 1 in thin media)
  for (int r = 0; r < N; ++r)
    for (int c = 0; c < NJ; ++c) {
      double s = 0.0;
      for (int k2 = 0; k2 < NQ; ++k2)
        for (int k1 = 0; k1 < NQ; ++k1) {
          double v, dx, dy;
          rt_ref<P>(t, c, k1, k2, v, dx, dy);
          s += t.w[k1] * t.w[k2] * t.dg[r % Q][k1] * t.dg[r / Q][k2] * (c < S::NX ? dx : dy);
        }
      o.D[r * NJ + c] = s;
    }
  for (int f = 0; f < 4; ++f) {
    const double n0 = f == 1 ? 1.0 : (f == 3 ? -1.0 : 0.0), n1 = f == 2 ? 1.0 : (f == 0 ? -1.0 : 0.0);
    for (int tt = 0; tt < NL; ++tt)
      for (int a = 0; a < NJ; ++a) {
        double s = 0.0;
        for (int k = 0; k < NQ; ++k) s += t.w[k] * t.op[tt][k] * (o.fv[f * NQ + k][a] * (a < S::NX ? n0 : n1));
        o.C1[(f * NL + tt) * NJ + a] = s;
      }
  }
  for (int r = 0, i = 0; r < NJ; ++r)
    for (int c = r; c < NJ; ++c) o.tri[i++] = (r << 8) | c;
}

template <int P>
struct HrtSmem {
  using S = HrtShape<P>;
  using R = HrtRef<P>;
  double rs[S::NQ2][S::NJ];          // HrtRef::rs, read by every product below
  double L[S::MM * S::LD];
  double ms[2][S::NQ2][S::NJ];       // sigma_t w J (F^T F / J^2)_{c, comp(a)} times the reference value
  double sg[S::NQ2][S::NJ];          // -w J (grad v : E) at the volume points
  double C2[S::NJ][S::NL4];
  double gv[S::NJ];
  double ctrl[(kMaxM + 1) * (kMaxM + 1) * 2];
  double mom[5][4][S::N];            // nodal phi, P of the element and its face neighbours
  double geo[R::NPT][10];            // map derivatives: (xi, eta[, xi xi, xi eta, eta eta]) of x and y
  double ed[S::NQ2 + 8 * S::NQ][4];  // phi and P at the points, then at the face points from outside
  // per volume point: m00, m01, m11 (sigma_t w J F^T F / J^2), then per component c the weights
  // of (value, d/dxi, d/deta) in -w J (grad v : E); (w F^T Q1) (2)
  double pv[S::NQ2][11];
  // per face point: interior faces w (F^T {E} n ds) / J (2); boundary faces (F^T E n^) / J (2),
  // (F^T n^) / J (2), w |n ds| / E_b and 2 w |n ds| J_in / E_b
  double pf[4 * S::NQ][6];
};

// Assembly of one element per CTA at a time.  The work is cut into items that fill warps: the
// map's derivatives and the moments at the points as small matrix products with the reference
// tables; then, per point, everything that multiplies a reference basis value, so that A is
//   A_ab = sum_q [sigma_t w J (F^T F / J^2)_{comp a, comp b} v_a] v_b   (upper triangle),
// and -w J (grad v_a : E) = K0 v_a + K1 dv_a/dxi + K2 dv_a/deta with three numbers per point
// and component: an RT function has one nonzero reference component, so its Piola image and
// gradient need no more.  FP64 issue bounds it: ~35 k lane operations per element at p = 2.
template <int P>
__global__ void __launch_bounds__(256, P <= 2 ? 4 : P == 3 ? 3 : 2)
hrt_local_kernel(long long E, int nx, int ny, int qc, const HrtRef<P>* __restrict__ ref, HrtIn in, HrtOut out) {
  using S = HrtShape<P>;
  using R = HrtRef<P>;
  constexpr int N = S::N, NQ = S::NQ, NQ2 = S::NQ2, NJ = S::NJ, MM = S::MM, LD = S::LD, NL = S::NL, NL4 = S::NL4;
  constexpr int NF = 4 * NQ;
  extern __shared__ __align__(16) unsigned char hrt_smem[];
  HrtSmem<P>& sm = *reinterpret_cast<HrtSmem<P>*>(hrt_smem);
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int i = tid; i < NQ2 * NJ; i += nth) (&sm.rs[0][0])[i] = (&ref->rs[0][0])[i];
  const long long En = E * N;
  for (long long e = blockIdx.x; e < E; e += gridDim.x) {
    __syncthreads();
    int nb[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) nb[f] = nb_elem(nx, ny, (int)e, f);
    const bool inner = nb[0] >= 0 && nb[1] >= 0 && nb[2] >= 0 && nb[3] >= 0;
    for (int i = tid; i < 2 * qc; i += nth) sm.ctrl[i] = in.ctrl[(size_t)e * 2 * qc + i];
    for (int i = tid; i < 20 * N; i += nth) {
      const int who = i / (4 * N), c = (i / N) & 3, j = i % N;
      const long long ee = who == 0 ? e : nb[who - 1];
      if (ee >= 0) sm.mom[who][c][j] = c == 0 ? in.phi[(size_t)ee * N + j] : in.P[(size_t)(c - 1) * En + ee * N + j];
    }
    const double st = in.sigma_t[e], sa = in.sigma_t[e] - in.sigma_s[e];
    __syncthreads();
    // (1) the map's derivatives (second ones at the volume points only) and the moments at
    // the points: lanes along the points
    for (int i = tid; i < NQ2 * 10 + NF * 4; i += nth) {
      const bool vol = i < NQ2 * 10;
      const int d = vol ? i / NQ2 : (i - NQ2 * 10) / NF, pt = vol ? i % NQ2 : NQ2 + (i - NQ2 * 10) % NF;
      const int type = d >> 1, comp = d & 1;
      double s = 0.0;
      for (int c = 0; c < qc; ++c) s = fma(ref->gt[type][c][pt], sm.ctrl[2 * c + comp], s);
      sm.geo[pt][d] = s;
    }
    for (int i = tid; i < (NQ2 + 2 * NF) * 4; i += nth) {
      const int c = i / (NQ2 + 2 * NF), q = i % (NQ2 + 2 * NF);
      // q: volume points, face points from inside, face points from the neighbour (its own
      // table points are those of the opposite face)
      int pt = q, who = 0;
      if (q >= NQ2 + NF) {
        const int f = (q - NQ2 - NF) / NQ;
        who = 1 + f;
        pt = NQ2 + ((f + 2) & 3) * NQ + (q - NQ2 - NF) % NQ;
        if (nb[f] < 0) continue;
      }
      const double* m = sm.mom[who][c];
      double s = 0.0;
#pragma unroll
      for (int j = 0; j < N; ++j) s = fma(ref->bt[pt][j], m[j], s);
      sm.ed[q][c] = s;
    }
    for (int idx = tid; idx < NL4 * NJ; idx += nth) (&sm.C2[0][0])[idx] = 0.0;
    __syncthreads();
    // (2) per point: the numbers that multiply reference basis values
    for (int pt = tid; pt < NQ2 + NF; pt += nth) {
      const double* g = sm.geo[pt];
      // F = [x_xi x_eta; y_xi y_eta]
      const double F[4] = {g[0], g[2], g[1], g[3]};
      const double rJ = 1.0 / (F[0] * F[3] - F[1] * F[2]);
      const double* o = sm.ed[pt];
      const double rf = 1.0 / o[0];
      const double E0 = o[1] * rf, E1 = o[2] * rf, E2 = o[3] * rf;
      if (pt < NQ2) {
        double* v = sm.pv[pt];
        const double w = ref->w[pt], wr = st * w * rJ;   // w J / J^2 = w / J
        v[0] = wr * (F[0] * F[0] + F[2] * F[2]);
        v[1] = wr * (F[0] * F[1] + F[2] * F[3]);
        v[2] = wr * (F[1] * F[1] + F[3] * F[3]);
        // second derivatives H[i][k][l] = d^2 x_i / dxi_k dxi_l and Jacobi's formula
        // dJ / dxi_l = tr(adj F dF / dxi_l)
        const double H[2][2][2] = {{{g[4], g[6]}, {g[6], g[8]}}, {{g[5], g[7]}, {g[7], g[9]}}};
        // grad v : E = sum_il dv_i / dxi_l B_il / J, B = E adj(F)^T / J; with
        // dv_i / dxi_l = (H_icl v + F_ic dv_l - dJ_l F_ic v / J) / J and the weight -w J
        const double adj[2][2] = {{F[3], -F[1]}, {-F[2], F[0]}};
        double dJ[2], B[2][2];
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          dJ[l] = adj[0][0] * H[0][0][l] + adj[0][1] * H[1][0][l] + adj[1][0] * H[0][1][l] + adj[1][1] * H[1][1][l];
          B[0][l] = -w * rJ * (adj[l][0] * E0 + adj[l][1] * E1);
          B[1][l] = -w * rJ * (adj[l][0] * E1 + adj[l][1] * E2);
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const double f0 = F[c], f1 = F[2 + c];
          double k0 = 0.0;
#pragma unroll
          for (int l = 0; l < 2; ++l) {
            const double t = dJ[l] * rJ;
            k0 += B[0][l] * (H[0][c][l] - t * f0) + B[1][l] * (H[1][c][l] - t * f1);
            v[4 + 3 * c + l] = B[0][l] * f0 + B[1][l] * f1;
          }
          v[3 + 3 * c] = k0;
        }
        if (in.Q1) {   // int v . Q1: w J (F v / J) . Q1
          double q1x = 0.0, q1y = 0.0;
          for (int j = 0; j < N; ++j) {
            q1x += ref->bt[pt][j] * in.Q1[(size_t)e * N + j];
            q1y += ref->bt[pt][j] * in.Q1[En + (size_t)e * N + j];
          }
          v[9] = w * (F[0] * q1x + F[2] * q1y);
          v[10] = w * (F[1] * q1x + F[3] * q1y);
        }
      } else {
        const int fp = pt - NQ2, f = fp / NQ, k = fp % NQ;
        double* r = sm.pf[fp];
        const double* nd = in.nds + (((size_t)e * 4 + f) * NQ + k) * 2;
        const double w = ref->w[pt];
        if (nb[f] >= 0) {
          const double* on = sm.ed[pt + NF];
          const double rn = 1.0 / on[0];
          const double a00 = 0.5 * (E0 + on[1] * rn), a01 = 0.5 * (E1 + on[2] * rn), a11 = 0.5 * (E2 + on[3] * rn);
          const double En0 = a00 * nd[0] + a01 * nd[1], En1 = a01 * nd[0] + a11 * nd[1];
          // v_a . {E} n ds = v_hat_a . F^T ({E} n ds) / J
          r[0] = w * (F[0] * En0 + F[2] * En1) * rJ;
          r[1] = w * (F[1] * En0 + F[3] * En1) * rJ;
        } else {
          const long long bf = bface(nx, ny, (int)e, f);
          const double ln = sqrt(nd[0] * nd[0] + nd[1] * nd[1]);
          const double un0 = nd[0] / ln, un1 = nd[1] / ln;
          const double En0 = E0 * un0 + E1 * un1, En1 = E1 * un0 + E2 * un1;
          const double eb = in.Eb[bf * NQ + k];
          r[0] = (F[0] * En0 + F[2] * En1) * rJ;
          r[1] = (F[1] * En0 + F[3] * En1) * rJ;
          r[2] = (F[0] * un0 + F[2] * un1) * rJ;
          r[3] = (F[1] * un0 + F[3] * un1) * rJ;
          r[4] = w * ln / eb;
          r[5] = 2.0 * w * ln * in.Jin[bf * NQ + k] / eb;
        }
      }
    }
    __syncthreads();
    // (3) per (volume point, basis function); the multiplier couplings of the interior faces
    for (int idx = tid; idx < NQ2 * NJ; idx += nth) {
      const int q = idx / NJ, a = idx % NJ, c = a < S::NX ? 0 : 1;
      const double* v = sm.pv[q];
      const double s = sm.rs[q][a];
      sm.ms[0][q][a] = v[c] * s;
      sm.ms[1][q][a] = v[1 + c] * s;
      sm.sg[q][a] = fma(v[3 + 3 * c], s, fma(v[4 + 3 * c], ref->r0[q][a], v[5 + 3 * c] * ref->r1[q][a]));
    }
    for (int idx = tid; idx < NL4 * NJ; idx += nth) {
      const int ft = idx / NJ, a = idx % NJ, f = ft / NL, c = a < S::NX ? 0 : 1;
      if (nb[f] < 0) continue;
      double s = 0.0;
#pragma unroll
      for (int k = 0; k < NQ; ++k) s = fma(ref->c2[ft][k][a], sm.pf[f * NQ + k][c], s);
      sm.C2[a][ft] = s;
    }
    __syncthreads();
    // (4) A (upper triangle, mirrored), G, D (reference), sigma_a M, f, g
    for (int idx = tid; idx < R::NT; idx += nth) {
      const int rc = ref->tri[idx], r = rc >> 8, c = rc & 0xff, cc = c < S::NX ? 0 : 1;
      double s = 0.0;
#pragma unroll 4
      for (int q = 0; q < NQ2; ++q) s = fma(sm.ms[cc][q][r], sm.rs[q][c], s);
      sm.L[r * LD + c] = s;
      sm.L[c * LD + r] = s;
    }
    for (int idx = tid; idx < NJ * N; idx += nth) {
      const int c = idx / NJ, a = idx % NJ;
      double s = 0.0;
#pragma unroll 4
      for (int q = 0; q < NQ2; ++q) s = fma(sm.sg[q][a], ref->bt[q][c], s);
      sm.L[a * LD + NJ + c] = s;
      sm.L[(NJ + c) * LD + a] = ref->D[idx];
    }
    for (int idx = tid; idx < N * N; idx += nth)
      sm.L[(NJ + idx / N) * LD + NJ + idx % N] = sa * in.Mm[(size_t)e * N * N + idx];
    for (int c = tid; c < N + NJ; c += nth) {
      double s = 0.0;
      if (c < N) {
        for (int j = 0; j < N; ++j) s += in.Mm[((size_t)e * N + c) * N + j] * in.Q0[(size_t)e * N + j];
        out.f[(size_t)e * N + c] = s;
      } else {
        const int a = c - N, k = a < S::NX ? 9 : 10;
        if (in.Q1)
          for (int q = 0; q < NQ2; ++q) s += sm.rs[q][a] * sm.pv[q][k];
        sm.gv[a] = s;
      }
    }
    __syncthreads();
    // (5) Miften-Larsen terms of the boundary faces
    for (int f = 0; f < 4 && !inner; ++f) {
      if (nb[f] >= 0) continue;
      const double (*o)[6] = sm.pf + f * NQ;
      for (int idx = tid; idx < NJ * NJ + NJ; idx += nth) {
        const int a = idx < NJ * NJ ? idx / NJ : idx - NJ * NJ, b = idx < NJ * NJ ? idx % NJ : -1;
        const int ca = a < S::NX ? 0 : 1, cb = b < S::NX ? 0 : 1;
        double s = 0.0;
        if (b >= 0) {
          for (int k = 0; k < NQ; ++k)
            s += o[k][4] * (ref->fv[f * NQ + k][a] * o[k][ca]) * (ref->fv[f * NQ + k][b] * o[k][2 + cb]);
          sm.L[a * LD + b] += s;
        } else {
          for (int k = 0; k < NQ; ++k) s += o[k][5] * (ref->fv[f * NQ + k][a] * o[k][ca]);
          sm.gv[a] += s;
        }
      }
      __syncthreads();
    }
    // the assembled local system (inverted by hrt_invert_kernel) and the couplings
    for (int idx = tid; idx < MM * MM; idx += nth)
      out.Li[(size_t)e * MM * MM + idx] = sm.L[(idx / MM) * LD + idx % MM];
    for (int idx = tid; idx < NJ * NL4; idx += nth) out.C2[(size_t)e * NJ * NL4 + idx] = (&sm.C2[0][0])[idx];
    for (int a = tid; a < NJ; a += nth) out.g[(size_t)e * NJ + a] = sm.gv[a];
  }
}

// Inversion of the assembled local systems and the element's share of the reduced system,
// apart from the assembly so that it runs many CTAs per SM.  Gauss-Jordan with partial
// pivoting and the matrix in registers, rows tr + TR u and columns tc + TC v on thread
// (tr, tc): per step the pivot's column is already in shared memory, every warp picks the pivot
// row from it, the row's owners publish R = row / pivot and every entry takes one FMA,
// a = R_j (-c_i) + a, where the pivot's own row and column start from zero (R_k = 1 / pivot,
// -c_k = 1), so no lane of a warp takes another path; the owners of the next column publish it
// as they update it.  The grids of threads leave few idle: 11 x 11 with 3 x 3 entries each for
// 33 unknowns (p = 2), 28 x 8 with 2 x 7 for 56, 15 x 17 with 6 x 5 for 85.  Rows stay
// where they are: step k's pivot row perm[k] ends as row k of the inverse, and column j belongs
// to the right-hand side of equation perm[j].  The pivoting is needed: on optically thin
// elements A's entries are small against G's, and diagonal pivots left phi an error of 2e-10 to
// 4e-9 at sigma_t = 1e-7 (1e-16 with pivoting; one element, p = 1..4).  It costs 0.5 of the
// 3.0 ms at 128^2 Q2, 1.9 of 32.5 at Q4.
template <int P>
struct HrtInvSmem {
  using S = HrtShape<P>;
  double L[S::MM * S::LD];
  double C2[S::NJ][S::NL4];
  double gf[S::MM];                  // g, f
  double T1[S::NL4][S::NL4];         // rows of W C2 at the face unknowns
  double u[S::NL4];                  // W g + X f there
  double col[2][S::MM];              // the pivot's column, this step's and the next one's
  double R[S::MM];                   // row / pivot
  int perm[S::MM], step[S::MM];      // pivot row of each step, and its inverse
};
template <int P> struct HrtInvShape {
  static constexpr int MM = HrtShape<P>::MM;
  static constexpr int TR = P == 1 ? 8 : P == 2 ? 11 : P == 3 ? 28 : 15, TC = P == 1 ? 16 : P == 2 ? 11 : P == 3 ? 8 : 17;
  static constexpr int NU = (MM + TR - 1) / TR, NV = (MM + TC - 1) / TC, T = (TR * TC + 31) / 32 * 32;
  static_assert(NV * TC == MM, "whole columns");
};

template <int P>
__global__ void __launch_bounds__(HrtInvShape<P>::T)
hrt_invert_kernel(long long E, int nx, int ny, const HrtRef<P>* __restrict__ ref, HrtOut out, unsigned int* status) {
  using S = HrtShape<P>;
  constexpr int N = S::N, NJ = S::NJ, MM = S::MM, LD = S::LD, NL = S::NL, NL4 = S::NL4, NX = S::NX;
  using I = HrtInvShape<P>;
  constexpr int T = I::T, TR = I::TR, TC = I::TC, NU = I::NU, NV = I::NV, RPW = (MM + 31) / 32;
  constexpr unsigned FULL = 0xffffffffu;
  extern __shared__ __align__(16) unsigned char hrt_inv_smem[];
  HrtInvSmem<P>& sm = *reinterpret_cast<HrtInvSmem<P>*>(hrt_inv_smem);
  const int tid = threadIdx.x, lane = tid & 31, nth = T;
  // this thread's rows and columns (a thread past the grid holds row MM and up: none)
  const int tr = tid < TR * TC ? tid / TC : MM, tc = tid < TR * TC ? tid % TC : 0;
  // the RT unknown with a normal flux on face f at tangential node b (C1's columns)
  auto face_unknown = [](int f, int b) {
    return f == 3 ? (P + 2) * b : f == 1 ? P + 1 + (P + 2) * b : f == 0 ? NX + b : NX + b + (P + 1) * (P + 1);
  };
  for (long long e = blockIdx.x; e < E; e += gridDim.x) {
    __syncthreads();
    for (int idx = tid; idx < NL4 * NJ; idx += nth) (&sm.C2[0][0])[idx] = out.C2[(size_t)e * NJ * NL4 + idx];
    for (int a = tid; a < MM; a += nth) sm.gf[a] = a < NJ ? out.g[(size_t)e * NJ + a] : out.f[(size_t)e * N + a - NJ];
    double* Lg = out.Li + (size_t)e * MM * MM;
    double a[NU][NV];
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      const int i = tr + TR * u;
#pragma unroll
      for (int v = 0; v < NV; ++v) a[u][v] = i < MM ? Lg[i * MM + tc + TC * v] : 0.0;
      if (i < MM && tc == 0) sm.col[0][i] = a[u][0];
    }
    unsigned used = 0;   // which of rows lane, lane + 32, ... have been pivots
    for (int k = 0; k < MM; ++k) {
      __syncthreads();
      const double* col = sm.col[k & 1];
      // the largest magnitude of the rows left (not a NaN; the lowest such row): high words,
      // then low words, then the index; -1 where a row takes no part
      int hi[RPW], best = -1;
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        const int i = lane + 32 * q;
        hi[q] = i < MM && !((used >> q) & 1) ? __double2hiint(col[i]) & 0x7fffffff : -1;
        if (hi[q] > 0x7ff00000) hi[q] = -2;
        best = max(best, hi[q]);
      }
      best = __reduce_max_sync(FULL, best);
      unsigned lo[RPW], blo = 0;
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        const int i = lane + 32 * q;
        lo[q] = i < MM ? (unsigned)__double2loint(col[i]) : 0;
        if (hi[q] == best) blo = max(blo, lo[q]);
      }
      blo = __reduce_max_sync(FULL, blo);
      int pr = MM;
#pragma unroll
      for (int q = RPW - 1; q >= 0; --q) {
        if (best >= 0 ? hi[q] == best && lo[q] == blo : hi[q] == -2) pr = lane + 32 * q;
      }
      pr = __reduce_min_sync(FULL, pr);
      if ((pr & 31) == lane) used |= 1u << (pr >> 5);
      const double piv = col[pr];
      if (tid == 0) {
        sm.perm[k] = pr;
        sm.step[pr] = k;
        if (best < 0 || !(fabs(piv) > 1e-300)) atomicOr(status, kDevSingular);
      }
      const int ur = pr / TR, vk = k / TC, vn = (k + 1) / TC;
      const bool own_row = tr == pr - ur * TR, own_col = tc == k - vk * TC, own_next = tc == k + 1 - vn * TC;
      if (own_row) {
        const double inv = 1.0 / piv;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          double x = a[0][v];
#pragma unroll
          for (int u = 1; u < NU; ++u) x = u == ur ? a[u][v] : x;
          sm.R[tc + TC * v] = own_col && v == vk ? inv : x * inv;
        }
      }
      __syncthreads();
      double R[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) R[v] = sm.R[tc + TC * v];
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        const int i = tr + TR * u;
        const bool prow = own_row && u == ur;
        const double c = i < MM ? (prow ? 1.0 : -col[i]) : 0.0;
        double next = 0.0;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          a[u][v] = fma(c, R[v], prow || (own_col && v == vk) ? 0.0 : a[u][v]);
          next = v == vn ? a[u][v] : next;
        }
        if (own_next && i < MM) sm.col[(k + 1) & 1][i] = next;
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      const int i = tr + TR * u;
      if (i < MM) {
#pragma unroll
        for (int v = 0; v < NV; ++v) sm.L[sm.step[i] * LD + sm.perm[tc + TC * v]] = a[u][v];
      }
    }
    __syncthreads();
    for (int idx = tid; idx < MM * MM; idx += nth) Lg[idx] = sm.L[(idx / MM) * LD + idx % MM];
    // W C2 and W g + X f at the unknowns with a normal flux on a face (the others have zero
    // columns in C1), then H_e = C1 (W C2) and r_e = C1 (W g + X f)
    for (int idx = tid; idx < NL4 * NL4 + NL4; idx += nth) {
      const int r = idx < NL4 * NL4 ? idx / NL4 : idx - NL4 * NL4;
      const double* Lr = sm.L + face_unknown(r / NL, r % NL) * LD;
      double s = 0.0;
      if (idx < NL4 * NL4) {
        const int c = idx % NL4;
        for (int b = 0; b < NJ; ++b) s = fma(Lr[b], sm.C2[b][c], s);
        sm.T1[r][c] = s;
      } else {
        for (int b = 0; b < MM; ++b) s = fma(Lr[b], sm.gf[b], s);
        sm.u[r] = s;
      }
    }
    __syncthreads();
    for (int idx = tid; idx < NL4 * NL4 + NL4; idx += nth) {
      const int r = idx < NL4 * NL4 ? idx / NL4 : idx - NL4 * NL4, f = r / NL;
      double s = 0.0;
      if (nb_elem(nx, ny, (int)e, f) >= 0) {
#pragma unroll
        for (int b = 0; b < NL; ++b) {
          const double c1 = ref->C1[r * NJ + face_unknown(f, b)];
          s = fma(c1, idx < NL4 * NL4 ? sm.T1[f * NL + b][idx % NL4] : sm.u[f * NL + b], s);
        }
      }
      if (idx < NL4 * NL4) out.He[(size_t)e * NL4 * NL4 + idx] = s;
      else out.re[(size_t)e * NL4 + r] = s;
    }
  }
}

// global multiplier index of face f of element e, or -1 on the boundary
__device__ __forceinline__ long long face_index(int nx, int ny, int e, int f) {
  const int i = e % nx, j = e / nx;
  const long long nv = (long long)(nx - 1) * ny;
  if (f == 1) return i < nx - 1 ? (long long)j * (nx - 1) + i : -1;
  if (f == 3) return i > 0 ? (long long)j * (nx - 1) + i - 1 : -1;
  if (f == 2) return j < ny - 1 ? nv + (long long)j * nx + i : -1;
  return j > 0 ? nv + (long long)(j - 1) * nx + i : -1;
}

// the two elements and local faces on either side of interior face fid
__device__ __forceinline__ void face_sides(int nx, int ny, long long fid, long long& e1, int& f1, long long& e2,
                                           int& f2) {
  const long long nv = (long long)(nx - 1) * ny;
  if (fid < nv) {
    const long long j = fid / (nx - 1), i = fid % (nx - 1);
    e1 = j * nx + i; f1 = 1; e2 = e1 + 1; f2 = 3;
  } else {
    const long long h = fid - nv, j = h / nx, i = h % nx;
    e1 = j * nx + i; f1 = 2; e2 = e1 + nx; f2 = 0;
  }
}

// r[face dof] = the two sides' rows of r_e (the reduced right-hand side)
template <int P>
__global__ void hrt_gather_kernel(int nx, int ny, long long nfaces, const double* __restrict__ z,
                                  double* __restrict__ y) {
  constexpr int NL = P + 1, NL4 = 4 * NL;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= nfaces * NL) return;
  long long e1, e2;
  int f1, f2;
  face_sides(nx, ny, t / NL, e1, f1, e2, f2);
  const int tt = (int)(t % NL);
  y[t] = z[e1 * NL4 + f1 * NL + tt] + z[e2 * NL4 + f2 * NL + tt];
}

// Element-patch additive Schwarz preconditioner: for each element the restriction of H to
// the multipliers of its interior faces, H_e plus, on each such face, the neighbour's
// diagonal block of that face (its only contribution there), inverted; the preconditioner
// applies every element's inverse to its faces' values and sums the two elements' results on
// each face.  One warp per element with the matrix in shared memory, Gauss-Jordan with
// partial pivoting; the rows and columns of boundary faces are the identity, so they stay
// decoupled and carry zeros.
template <int P>
__global__ void __launch_bounds__(128)
hrt_asm_setup_kernel(long long E, int nx, int ny, const double* __restrict__ He, double* __restrict__ Pinv,
                     unsigned int* status) {
  constexpr int NL = P + 1, NL4 = 4 * NL, LDP = NL4 + 1;
  __shared__ double sm[4][NL4 * LDP];
  __shared__ double scol[4][NL4];     // column k before the step
  __shared__ int sperm[4][NL4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long e = blockIdx.x * 4LL + w;
  if (e >= E) return;   // whole warps leave together; the kernel has no block barrier
  double* A = sm[w];
  int nbe[4], nbf[4];
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    nbe[f] = nb_elem(nx, ny, (int)e, f);
    nbf[f] = (f + 2) & 3;
  }
  for (int idx = lane; idx < NL4 * NL4; idx += 32) {
    const int r = idx / NL4, c = idx % NL4, fr = r / NL, fc = c / NL;
    double v;
    if (nbe[fr] < 0 || nbe[fc] < 0) {
      v = r == c ? 1.0 : 0.0;
    } else {
      v = He[(size_t)e * NL4 * NL4 + idx];
      if (fr == fc) {
        const int on = nbf[fr] * NL;
        v += He[(size_t)nbe[fr] * NL4 * NL4 + (size_t)(on + r % NL) * NL4 + on + c % NL];
      }
    }
    A[r * LDP + c] = v;
  }
  __syncwarp();
  bool singular = false;
  for (int k = 0; k < NL4; ++k) {
    double best = -1.0;
    int bi = k;
    for (int i = k + lane; i < NL4; i += 32) {
      const double v = fabs(A[i * LDP + k]);
      if (v > best) { best = v; bi = i; }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, off);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    singular = singular || !(best > 1e-300);
    if (lane == 0) sperm[w][k] = bi;
    if (bi != k)
      for (int j = lane; j < NL4; j += 32) {
        const double t = A[k * LDP + j];
        A[k * LDP + j] = A[bi * LDP + j];
        A[bi * LDP + j] = t;
      }
    __syncwarp();
    const double inv = 1.0 / A[k * LDP + k];
    for (int i = lane; i < NL4; i += 32) scol[w][i] = A[i * LDP + k];
    __syncwarp();
    for (int j = lane; j < NL4; j += 32)
      if (j != k) A[k * LDP + j] *= inv;
    __syncwarp();
    for (int idx = lane; idx < NL4 * NL4; idx += 32) {
      const int i = idx / NL4, j = idx % NL4;
      if (i == k) continue;
      const double cik = scol[w][i];
      if (j == k) A[i * LDP + k] = -cik * inv;
      else A[i * LDP + j] -= cik * A[k * LDP + j];
    }
    __syncwarp();
    if (lane == 0) A[k * LDP + k] = inv;
    __syncwarp();
  }
  for (int k = NL4 - 1; k >= 0; --k) {   // undo the row interchanges as column interchanges
    const int pr = sperm[w][k];
    if (pr != k)
      for (int i = lane; i < NL4; i += 32) {
        const double t = A[i * LDP + k];
        A[i * LDP + k] = A[i * LDP + pr];
        A[i * LDP + pr] = t;
      }
    __syncwarp();
  }
  for (int idx = lane; idx < NL4 * NL4; idx += 32) Pinv[(size_t)e * NL4 * NL4 + idx] = A[(idx / NL4) * LDP + idx % NL4];
  if (lane == 0 && singular) atomicOr(status, kDevSingular);
}

// [J; phi] = Li [g - C2 lambda_e; f]
template <int P>
__global__ void hrt_recover_kernel(long long E, int nx, int ny, const double* __restrict__ Li,
                                   const double* __restrict__ C2, const double* __restrict__ g,
                                   const double* __restrict__ f, const double* __restrict__ lam,
                                   double* __restrict__ Jout, double* __restrict__ phi_out) {
  using S = HrtShape<P>;
  constexpr int N = S::N, NJ = S::NJ, MM = S::MM, NL = S::NL, NL4 = S::NL4;
  __shared__ double rhs[MM];
  __shared__ double le[NL4];
  for (long long e = blockIdx.x; e < E; e += gridDim.x) {
    __syncthreads();
    for (int r = threadIdx.x; r < NL4; r += blockDim.x) {
      const long long fi = face_index(nx, ny, (int)e, r / NL);
      le[r] = fi < 0 ? 0.0 : lam[fi * NL + r % NL];
    }
    __syncthreads();
    for (int a = threadIdx.x; a < MM; a += blockDim.x) {
      if (a < NJ) {
        double s = g[(size_t)e * NJ + a];
        for (int c = 0; c < NL4; ++c) s -= C2[(size_t)e * NJ * NL4 + (size_t)a * NL4 + c] * le[c];
        rhs[a] = s;
      } else {
        rhs[a] = f[(size_t)e * N + a - NJ];
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < MM; i += blockDim.x) {
      const double* row = Li + (size_t)e * MM * MM + (size_t)i * MM;
      double s = 0.0;
      for (int j = 0; j < MM; ++j) s += row[j] * rhs[j];
      if (i < NJ) Jout[(size_t)e * NJ + i] = s;
      else phi_out[(size_t)e * N + i - NJ] = s;
    }
  }
}

// ---- the multiplier system's Krylov solve: BiCGStab (van der Vorst) with the two-level
// Schwarz preconditioner (the element patches above and the coarse space below) as one
// cooperative kernel, kry_solve_kernel.  The mesh is cut into tiles of whole elements, each
// inside one coarse cell (kry_cut); a CTA takes a tile (or several) and owns the multipliers of the
// left and bottom faces of its elements.  Vectors that other tiles read live in global
// memory and are read past L1; a phase's own intermediate (the vector the element patches or
// the matrix act on, with its halo) sits in shared memory.  One iteration is four phases,
// each closed by a grid barrier:
//   A  omega, rho and beta from the last phase's dots; lambda, r and p of the owned
//      multipliers; z_e = Pinv_e p|e per element; the cell's restriction of p; r.r
//   B  p_hat = the two sides' z + the coarse correction, on the tile and
//      its halo; v = H p_hat; r_hat.v
//   C  convergence test on r.r; alpha; s = r - alpha v; z_e = Pinv_e s|e; restriction of s; r_hat.s
//   D  s_hat as in B; t = H s_hat; t.s, t.t, r_hat.t
// (rho of the next iteration is r_hat.s - omega r_hat.t, so it needs no barrier of its own).
// Every dot product is summed in a fixed order (per tile, then over the tiles), so the
// iteration is deterministic.  The waits at the barriers are bounded.  66 us per iteration at
// 128^2 Q2, where the FP64 pipe of the 121 SMs with a tile is busy 65 % of the time and shared
// memory's latency and the block and grid barriers take the rest; about 30 at 24 x 20 Q3, mostly
// barriers.  11 launches replayed from a graph took 78 and 62.
constexpr int kKT = 512, kCheck = 256;   // threads per CTA; iterations per launch
enum { kDotRR = 0, kDotRV = 1, kDotRS = 2, kDotTS = 3, kDotTT = 4, kDotRT = 5, kNumDots = 6 };
constexpr size_t kTileSmemMax = 160 * 1024;
constexpr int kTileMin = 16;   // elements
constexpr unsigned kGridPolls = 1u << 22;   // a poll takes 0.23 us (vef_grid_wait_selftest), so about a second

struct KState {
  int done;      // 1: converged, 2: breakdown
  int iters;     // iterations completed when done was set
  int base;      // iterations completed by earlier launches
  unsigned bar;  // arrivals at the grid barrier of the running launch
  double bb;     // ||r0||^2
  double rr;     // ||r||^2 at the last check
  double tol2;   // squared relative tolerance
  double rho, alpha;   // of the last completed iteration
};
static_assert(sizeof(KState) % sizeof(double) == 0, "KState is carved from a double buffer");

struct Kry {
  int nx, ny;
  long long nl;
  const double* He;
  const double* Pinv;   // [E][4 (p+1)][4 (p+1)] element-patch inverses of the preconditioner
  double* z;            // [E][4 (p+1)] the preconditioner's element results
  // coarse space of the preconditioner: bilinear functions on a grid of (ncx+1) x (ncy+1)
  // vertices whose cells hold cx x cy elements (the last ones fewer)
  int ncx, ncy, cx, cy, nc;
  // tiles: each cell cut into sx x sy sub-blocks of tw x th elements (the last ones fewer)
  int sx, sy, tw, th, ntiles;
  double gl[kMaxP + 1];   // the multiplier nodes on [0, 1]
  double2* cw;            // [nl] each multiplier's local coordinates (xi, eta) in its coarse cell
  double* A0;             // [nc][nc] the coarse operator R0 H R0^T, then its inverse
  double* pc;             // [ntiles][4] per tile: its multipliers' restriction to its cell's vertices
  double *x, *r, *rh, *p[2], *v, *s, *t, *ph, *sh;
  double* part;   // [kNumDots][ntiles]
  KState* st;
};

// ---- coarse space of the preconditioner (two-level additive Schwarz): the coarse
// functions are bilinear on a grid of at most 12 x 12 vertices laid over the elements, taken
// at the multiplier nodes of every interior face; the coarse operator A0 = R0 H R0^T is
// assembled from the elements' H_e and inverted once per solve, and each application adds
// R0^T A0^{-1} R0 x to the element-patch part.
// (144 vertices: the coarse operator is inverted in one CTA's shared memory)
constexpr int kCoarseMaxCells = 11, kCoarseMax = (kCoarseMaxCells + 1) * (kCoarseMaxCells + 1);

// the coarse cell holding multiplier node tt of interior face fid (its lower-left vertex v0)
// and the node's local coordinates in it.  A node on a cell's left or lower line belongs to
// that cell, one on the domain's right or upper coarse line to the last cell: so vertical
// faces on lines x = i0 .. i1 - 1 and horizontal faces on lines y = j0 .. j1 - 1 of the
// cell's element range [i0, i1) x [j0, j1) are its own.
__device__ __forceinline__ void coarse_coords(const Kry& k, long long fid, int tt, int& v0, double& xi,
                                              double& eta) {
  const long long nv = (long long)(k.nx - 1) * k.ny;
  double X, Y;   // in element widths from the lower-left corner
  if (fid < nv) {
    const long long j = fid / (k.nx - 1), i = fid % (k.nx - 1);
    X = (double)(i + 1);
    Y = (double)j + k.gl[tt];
  } else {
    const long long h = fid - nv, j = h / k.nx, i = h % k.nx;
    X = (double)i + k.gl[tt];
    Y = (double)(j + 1);
  }
  const int kx = min((int)(X / k.cx), k.ncx - 1), ky = min((int)(Y / k.cy), k.ncy - 1);
  const double x0 = (double)(kx * k.cx), x1 = (double)min((kx + 1) * k.cx, k.nx);
  const double y0 = (double)(ky * k.cy), y1 = (double)min((ky + 1) * k.cy, k.ny);
  xi = (X - x0) / (x1 - x0);
  eta = (Y - y0) / (y1 - y0);
  v0 = ky * (k.ncx + 1) + kx;
}

// the four bilinear weights, vertices in the order v0, v0 + 1, v0 + W, v0 + W + 1
__device__ __forceinline__ void bilinear(double xi, double eta, double w[4]) {
  w[0] = (1.0 - xi) * (1.0 - eta);
  w[1] = xi * (1.0 - eta);
  w[2] = (1.0 - xi) * eta;
  w[3] = xi * eta;
}

// coarse vertices and bilinear weights of multiplier node tt of interior face fid
__device__ __forceinline__ void coarse_weights(const Kry& k, long long fid, int tt, int v[4], double w[4]) {
  double xi, eta;
  coarse_coords(k, fid, tt, v[0], xi, eta);
  const int W = k.ncx + 1;
  v[1] = v[0] + 1;
  v[2] = v[0] + W;
  v[3] = v[2] + 1;
  bilinear(xi, eta, w);
}

// the node table of the coarse space, once per solve
template <int P>
__global__ void hrt_coarse_nodes_kernel(Kry k) {
  constexpr int NL = P + 1;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= k.nl) return;
  int v0;
  double xi, eta;
  coarse_coords(k, t / NL, (int)(t % NL), v0, xi, eta);
  k.cw[t] = make_double2(xi, eta);
}

// per coarse cell (one CTA): the sum over its elements of P_e^T H_e P_e, P_e the element's
// multipliers' weights on the cell's four vertices (every face of an element inside the
// cell lies in the cell's closure); threads take elements in a fixed stride and the block
// sums in a fixed order
template <int P>
__global__ void __launch_bounds__(128) hrt_coarse_cell_kernel(Kry k, double* __restrict__ Acell) {
  constexpr int NL = P + 1, NL4 = 4 * NL;
  const int cell = blockIdx.x, kx = cell % k.ncx, ky = cell / k.ncx;
  const int i0 = kx * k.cx, i1 = min(i0 + k.cx, k.nx), j0 = ky * k.cy, j1 = min(j0 + k.cy, k.ny);
  const int ni = i1 - i0, nel = ni * (j1 - j0);
  const int W = k.ncx + 1;
  double acc[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) acc[q] = 0.0;
  for (int t = threadIdx.x; t < nel; t += blockDim.x) {
    const long long e = (long long)(j0 + t / ni) * k.nx + i0 + t % ni;
    double Pw[NL4][4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const long long fi = face_index(k.nx, k.ny, (int)e, g);
#pragma unroll
      for (int tt = 0; tt < NL; ++tt) {
#pragma unroll
        for (int c = 0; c < 4; ++c) Pw[g * NL + tt][c] = 0.0;
        if (fi < 0) continue;
        int v[4];
        double w[4];
        coarse_weights(k, fi, tt, v, w);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          // a face on the cell's upper or right line may be assigned to the next cell, whose
          // far vertices then carry weight zero: keep the cell's own four
          const int lx = v[c] % W - kx, ly = v[c] / W - ky;
          if (lx < 0 || lx > 1 || ly < 0 || ly > 1) continue;
          Pw[g * NL + tt][ly * 2 + lx] += w[c];
        }
      }
    }
    const double* He = k.He + (size_t)e * NL4 * NL4;
    for (int i = 0; i < NL4; ++i) {
      double T[4] = {0.0, 0.0, 0.0, 0.0};   // (H_e P_e)[i][:]
      for (int j = 0; j < NL4; ++j) {
        const double h = He[i * NL4 + j];
#pragma unroll
        for (int b = 0; b < 4; ++b) T[b] = fma(h, Pw[j][b], T[b]);
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a * 4 + b] = fma(Pw[i][a], T[b], acc[a * 4 + b]);
    }
  }
  __shared__ double red[4][16];   // blockDim 128: four warps
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    double x = acc[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][q] = x;
  }
  __syncthreads();
  if (threadIdx.x < 16)
    Acell[(size_t)cell * 16 + threadIdx.x] =
        ((red[0][threadIdx.x] + red[1][threadIdx.x]) + red[2][threadIdx.x]) + red[3][threadIdx.x];
}

// the dense coarse operator, one row per thread from the cells around its vertex
__global__ void hrt_coarse_assemble_kernel(Kry k, const double* __restrict__ Acell) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= k.nc) return;
  const int W = k.ncx + 1, ax = a % W, ay = a / W;
  double* row = k.A0 + (size_t)a * k.nc;
  for (int b = 0; b < k.nc; ++b) row[b] = 0.0;
  for (int cy = ay - 1; cy <= ay; ++cy)
    for (int cx = ax - 1; cx <= ax; ++cx) {
      if (cx < 0 || cy < 0 || cx >= k.ncx || cy >= k.ncy) continue;
      const int cell = cy * k.ncx + cx, la = (ay - cy) * 2 + (ax - cx);
      for (int lb = 0; lb < 4; ++lb) {
        const int b = (cy + lb / 2) * W + cx + lb % 2;
        row[b] += Acell[(size_t)cell * 16 + la * 4 + lb];
      }
    }
  // a coarse function that vanishes on every interior face (a domain corner's when its cell
  // is one element wide) has an empty row and column: put 1 on the diagonal, its restriction
  // being zero, so it contributes nothing and A0 stays invertible
  double mx = 0.0;
  for (int b = 0; b < k.nc; ++b) mx = fmax(mx, fabs(row[b]));
  if (mx == 0.0) row[a] = 1.0;
}

// Gauss-Jordan inverse of the coarse operator, in FP32 in one CTA, of A0 scaled by its
// largest entry; written back in FP64 over A0.  The coarse solve is part of the
// preconditioner only: its accuracy changes the iteration count, not the FP64 Krylov
// iteration's answer.  (FP64 here is held to one SM's two FP64 FMA per clock: n^3 = 3 M FMA
// is 0.75 ms, FP32 runs at 64 times that rate.)  A0 is close to symmetric positive definite
// (it is for E = I/3), so the elimination takes the diagonal pivots in order: 1024 threads
// hold the matrix in registers, entry (i, j) on warp i mod 32, lane j mod 32, and a step
// publishes the pivot row and column through a double buffer in shared memory, one barrier
// and at most 25 FMA per thread.  A pivot below 2^-14 of its row's largest entry, or not
// finite, leaves A0 as it is and raises *fallback, and hrt_coarse_pivot_kernel inverts it with
// partial pivoting instead.
constexpr int kCoarseTile = (kCoarseMax + 31) / 32;
__global__ void __launch_bounds__(1024) hrt_coarse_invert_kernel(Kry k, int* __restrict__ fallback) {
  const int n = k.nc, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ float srow[2][32 * kCoarseTile], scol[2][32 * kCoarseTile];
  __shared__ double wmax[32];
  float a[kCoarseTile][kCoarseTile], scale[kCoarseTile];
  double m = 0.0;
  for (int idx = threadIdx.x; idx < n * n; idx += 1024) m = fmax(m, fabs(k.A0[idx]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) wmax[warp] = m;
  __syncthreads();
  m = wmax[lane];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  const double rs = m > 0.0 ? 1.0 / m : 1.0;
#pragma unroll
  for (int u = 0; u < kCoarseTile; ++u) {
    float mx = 0.0f;
#pragma unroll
    for (int v = 0; v < kCoarseTile; ++v) {
      const int i = warp + 32 * u, j = lane + 32 * v;
      a[u][v] = i < n && j < n ? (float)(k.A0[i * n + j] * rs) : 0.0f;
      mx = fmaxf(mx, fabsf(a[u][v]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    scale[u] = mx;
  }
  bool bad = false;
#pragma unroll
  for (int u0 = 0; u0 < kCoarseTile; ++u0) {
    for (int kk = 0; kk < 32; ++kk) {
      const int step = 32 * u0 + kk, b = step & 1;
      if (step >= n) break;
      if (warp == kk) {
#pragma unroll
        for (int v = 0; v < kCoarseTile; ++v) srow[b][lane + 32 * v] = a[u0][v];
      }
      if (lane == kk) {
#pragma unroll
        for (int u = 0; u < kCoarseTile; ++u) scol[b][warp + 32 * u] = a[u][u0];
      }
      __syncthreads();
      const float piv = srow[b][step], inv = 1.0f / piv;
      if (warp == kk) bad = bad || !(fabsf(piv) > scale[u0] * 6.103515625e-05f) || !isfinite(inv);
      float r[kCoarseTile];
#pragma unroll
      for (int v = 0; v < kCoarseTile; ++v) r[v] = srow[b][lane + 32 * v] * inv;
#pragma unroll
      for (int u = 0; u < kCoarseTile; ++u) {
        const float c = scol[b][warp + 32 * u];
#pragma unroll
        for (int v = 0; v < kCoarseTile; ++v) a[u][v] = fmaf(-c, r[v], a[u][v]);
        if (lane == kk) a[u][u0] = -c * inv;
      }
      if (warp == kk) {
#pragma unroll
        for (int v = 0; v < kCoarseTile; ++v) a[u0][v] = r[v];
        if (lane == kk) a[u0][u0] = inv;
      }
    }
  }
  const bool any = __syncthreads_or(bad) != 0;
  if (threadIdx.x == 0) *fallback = any;
  if (any) return;
#pragma unroll
  for (int u = 0; u < kCoarseTile; ++u)
#pragma unroll
    for (int v = 0; v < kCoarseTile; ++v) {
      const int i = warp + 32 * u, j = lane + 32 * v;
      if (i < n && j < n) k.A0[i * n + j] = (double)a[u][v] * rs;
    }
}

// The same inverse with partial pivoting, for an A0 whose diagonal pivots were too small (the
// kernel leaves at once otherwise).
// Per pivot step two barriers: every warp finds the pivot row itself (same order, same
// result), the pivot row, the row it changes places with and the pivot column go to
// buffers, and each thread then updates only its own entries, reading the row that moves
// to row pr from the buffer.  A pivot below 1e-30 of the largest entry (A0 singular in
// FP32) drops the coarse part: the inverse is written as zero and the preconditioner is the
// element patches alone.
constexpr int kCoarseInvThreads = 512, kCoarsePerLane = (kCoarseMax + 31) / 32;
__global__ void __launch_bounds__(kCoarseInvThreads)
hrt_coarse_pivot_kernel(Kry k, const int* __restrict__ fallback) {
  if (*fallback == 0) return;
  const int n = k.nc, ld = n | 1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int nwarp = kCoarseInvThreads / 32;
  extern __shared__ float A[];   // [n][ld]
  __shared__ float R[kCoarseMax], krow[kCoarseMax], colk[kCoarseMax];
  __shared__ int perm[kCoarseMax], src[kCoarseMax];
  __shared__ double wmax[nwarp];
  __shared__ int singular;
  if (tid == 0) singular = 0;
  double m = 0.0;
  for (int idx = tid; idx < n * n; idx += kCoarseInvThreads) m = fmax(m, fabs(k.A0[idx]));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) wmax[warp] = m;
  __syncthreads();
  m = 0.0;
  for (int w = 0; w < nwarp; ++w) m = fmax(m, wmax[w]);
  const double rs = m > 0.0 ? 1.0 / m : 1.0;
  for (int idx = tid; idx < n * n; idx += kCoarseInvThreads) A[(idx / n) * ld + idx % n] = (float)(k.A0[idx] * rs);
  __syncthreads();
  for (int kk = 0; kk < n; ++kk) {
    float best = -1.0f;
    int pr = kk;
#pragma unroll
    for (int q = 0; q < kCoarsePerLane; ++q) {
      const int i = kk + lane + 32 * q;
      const float v = i < n ? fabsf(A[i * ld + kk]) : -1.0f;
      if (v > best) { best = v; pr = i; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const float ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, pr, o);
      if (ob > best || (ob == best && oi < pr)) { best = ob; pr = oi; }
    }
    if (tid == 0) {
      perm[kk] = pr;
      if (!(best > 1e-30f)) singular = 1;
    }
    const float iv = 1.0f / A[pr * ld + kk];
    for (int j = tid; j < n; j += kCoarseInvThreads) {
      R[j] = j == kk ? iv : A[pr * ld + j] * iv;
      krow[j] = A[kk * ld + j];
      colk[j] = j == kk ? A[pr * ld + kk] : (j == pr ? A[kk * ld + kk] : A[j * ld + kk]);
    }
    __syncthreads();
    float r[kCoarsePerLane];   // this lane's columns of the new pivot row
#pragma unroll
    for (int q = 0; q < kCoarsePerLane; ++q) r[q] = lane + 32 * q < n ? R[lane + 32 * q] : 0.0f;
    for (int i = warp; i < n; i += nwarp) {
      float* Ai = A + i * ld;
      const float c = colk[i];
      const bool moved = i == pr;   // row pr now holds the old row kk
      float a[kCoarsePerLane];      // all loads of the row before its stores
#pragma unroll
      for (int q = 0; q < kCoarsePerLane; ++q) {
        const int j = lane + 32 * q;
        a[q] = j < n ? (moved ? krow[j] : Ai[j]) : 0.0f;
      }
#pragma unroll
      for (int q = 0; q < kCoarsePerLane; ++q) {
        const int j = lane + 32 * q;
        if (j < n) Ai[j] = i == kk ? r[q] : (j == kk ? -c * iv : fmaf(-c, r[q], a[q]));
      }
    }
    __syncthreads();
  }
  // the row interchanges, undone as column interchanges in reverse order, as one gather
  if (tid == 0) {
    for (int j = 0; j < n; ++j) src[j] = j;
    for (int kk = n - 1; kk >= 0; --kk) {
      const int t = src[kk];
      src[kk] = src[perm[kk]];
      src[perm[kk]] = t;
    }
  }
  __syncthreads();
  for (int idx = tid; idx < n * n; idx += kCoarseInvThreads) {
    const int i = idx / n, j = idx % n;
    k.A0[idx] = singular ? 0.0 : (double)A[i * ld + src[j]] * rs;
  }
}

// element ranges of tile q: its cell (kx, ky) and [i0, i1) x [j0, j1) (empty for a sub-block
// past a short cell's end); r1, r2: multipliers for division by the width + 1, + 2
struct KTile { int kx, ky, i0, i1, j0, j1; unsigned r0, r1, r2; };
__device__ __forceinline__ KTile kry_tile(const Kry& k, int q) {
  const int ns = k.sx * k.sy, cell = q / ns, sub = q - cell * ns;
  KTile t;
  t.kx = cell % k.ncx;
  t.ky = cell / k.ncx;
  const int ie = min((t.kx + 1) * k.cx, k.nx), je = min((t.ky + 1) * k.cy, k.ny);
  t.i0 = min(t.kx * k.cx + (sub % k.sx) * k.tw, ie);
  t.j0 = min(t.ky * k.cy + (sub / k.sx) * k.th, je);
  t.i1 = min(t.i0 + k.tw, ie);
  t.j1 = min(t.j0 + k.th, je);
  const unsigned w = (unsigned)(t.i1 - t.i0);
  t.r0 = w > 1 ? 0xffffffffu / w + 1 : 0;
  t.r1 = w > 0 ? 0xffffffffu / (w + 1) + 1 : 0;
  t.r2 = 0xffffffffu / (w + 2) + 1;
  return t;
}
// a / d by the multiplier r = 2^32 / d rounded up (0 stands for d = 1): exact for the element
// counts of a tile (a d < 2^32)
__device__ __forceinline__ int kry_div(int a, unsigned r) { return r ? (int)__umulhi((unsigned)a, r) : a; }
// multiplier of node tt on the left (side 0) or bottom face of element (i, j)
template <int P>
__device__ __forceinline__ int kry_dof(const Kry& k, int side, int i, int j, int tt) {
  return (side == 0 ? j * (k.nx - 1) + i - 1 : (k.nx - 1) * k.ny + (j - 1) * k.nx + i) * (P + 1) + tt;
}

__device__ __forceinline__ bool kry_barrier(KState* st, unsigned& epoch, unsigned int* status) {
  return grid_barrier(&st->bar, epoch, gridDim.x, kGridPolls, status);
}

// The scalars of the iteration, kept by thread 0 of every CTA (the same values in the same
// order everywhere) and read by the others from shared memory: an FP64 division or comparison
// costs its warp's sub-partition as much as a multiply-add, and 16 warps repeating it cost 16
// times that.
struct KryScal {
  double dot[4];
  double rho, rho_new, alpha, omega, beta, bb, rr, tol2;
  int done, iters, brk;
};

// a / b to within two ulp: the approximate reciprocal refined by two Newton-Raphson steps
// (pivot_rcp), at a third of a division's dependent FP64 operations; a b of magnitude 2^1021 and
// up, whose reciprocal is below the normal range and would come out as zero, and results that
// are not finite divide
__device__ __forceinline__ double kry_quot(double a, double b) {
  const double q = a * pivot_rcp(b);
  return isfinite(q) && (__double2hiint(b) & 0x7fffffff) < ((1021 + 1023) << 20) ? q : a / b;
}

// the sums over the tiles of nq <= 4 dots q, warp w summing dot q[w] in a fixed order, into
// sc.dot; ends with a block barrier
__device__ __forceinline__ void kry_sums(const Kry& k, KryScal& sc, int q0, int q1, int q2, int q3, int nq) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w < nq) {
    const double* p = k.part + (size_t)(w == 0 ? q0 : w == 1 ? q1 : w == 2 ? q2 : q3) * k.ntiles;
    double a = 0.0;
    for (int i = lane; i < k.ntiles; i += 32) a += __ldcg(p + i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) sc.dot[w] = a;
  }
  __syncthreads();
}

// K values per lane (a power of two) summed over the warp in log2(K) halving exchanges and a
// butterfly of one value: K - 1 + 5 - log2(K) additions instead of 5 K.  Lane l ends with the
// total of value kry_which<K>(l) in v[0].
template <int K>
__device__ __forceinline__ void kry_warp_sums(double (&v)[K]) {
  const int lane = threadIdx.x & 31;
  int off = 16;
#pragma unroll
  for (int h = K / 2; h >= 1; h >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
    off >>= 1;
  }
#pragma unroll
  for (; off > 0; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
}
template <int K>
__device__ __forceinline__ int kry_which(int lane) {
  int idx = 0;
  for (int h = K / 2, bit = 4; h >= 1; h >>= 1, --bit) idx += ((lane >> bit) & 1) * h;
  return idx;
}

// block sums of NV <= K values per thread in a fixed order; store(i, total) is called once per
// value.  Only the warps that had one of the `items` work items add (16 idle warps' shuffled
// additions would cost a microsecond).  Ends with a block barrier.
template <int NV, int K, typename F>
__device__ __forceinline__ void kry_block_sums(double (&val)[K], int items, F store) {
  __shared__ double red[K][kKT / 32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = min(kKT / 32, max(1, (items + 31) / 32));
  if (w < nw) {
    kry_warp_sums<K>(val);
    if ((lane & (32 / K - 1)) == 0) red[kry_which<K>(lane)][w] = val[0];
  }
  __syncthreads();
  if (w < NV) {
    double a = lane < nw ? red[w][lane] : 0.0;
    for (int o = nw > 4 ? kKT / 64 : nw > 1 ? 2 : 0; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) store(w, a);
  }
  __syncthreads();
}

// one row of an element matrix (H_e or Pinv_e) times the element's multipliers, staged at x0 of a buffer W elements
// wide (faces in order bottom, right = the next element's left, top = the upper one's bottom,
// left)
template <int P>
__device__ __forceinline__ double kry_row(const double* __restrict__ M, int e, int row,
                                          const double* __restrict__ x0, int W) {
  constexpr int NL = P + 1, NL4 = 4 * NL;
  const double2* A = reinterpret_cast<const double2*>(M + (size_t)(e * NL4 + row) * NL4);
  const double* xf[4] = {x0 + NL, x0 + 2 * NL, x0 + (size_t)W * 2 * NL + NL, x0};
  double s = 0.0;
#pragma unroll
  for (int h = 0; h < NL4 / 2; ++h) {
    const double2 a = __ldg(A + h);
    s = fma(a.x, xf[(2 * h) / NL][(2 * h) % NL], s);
    s = fma(a.y, xf[(2 * h + 1) / NL][(2 * h + 1) % NL], s);
  }
  return s;
}

// z_e = Pinv_e x|e for the tile's elements, x staged in sx as [element of the tile widened by
// one column and row][left, bottom][node]
template <int P>
__device__ __forceinline__ void kry_patches(const Kry& k, const KTile& t, const double* __restrict__ sx) {
  constexpr int NL = P + 1, NL4 = 4 * NL;
  const int w = t.i1 - t.i0, nel = w * (t.j1 - t.j0), W = w + 1;
  for (int q = threadIdx.x; q < nel * NL4; q += kKT) {
    const int le = q / NL4, row = q - le * NL4, lj = kry_div(le, t.r0), li = le - lj * w;
    const int e = (t.j0 + lj) * k.nx + t.i0 + li;
    k.z[e * NL4 + row] = kry_row<P>(k.Pinv, e, row, sx + (size_t)(lj * W + li) * 2 * NL, W);
  }
}

// The coarse correction around the tile's cell: every CTA sums the restriction per vertex
// from the cells around it (fixed order), multiplies the rows of A0^{-1} it needs and forms
// each of the 3 x 3 cells' bilinear coefficients: correction = c0 + c1 xi + (c2 + c3 xi) eta.
// The matrix needs the correction on the tile, on the faces of the elements to its left and
// below, and on the left / bottom faces of the next column / row, which lie on that cell's
// line (xi = 0 / eta = 0): vertices (kx - 1 .. kx + 1) x (ky - 1 .. ky + 1); the vertices
// beyond are taken as zero.  A tile's restriction comes as
// the sums of x, xi x, eta x and xi eta x over its multipliers.
__device__ __forceinline__ void kry_coarse(const Kry& k, const double (*a0)[kCoarseMax], double* vc, double* zc,
                                           double (*cc)[4]) {
  const int W = k.ncx + 1, ns = k.sx * k.sy;
  for (int a = threadIdx.x; a < k.nc; a += kKT) {
    const int ay = a / W, ax = a - ay * W;
    // the vertex is cell c's upper right (c = 0), upper left, lower right, lower left corner
    double q[4];
    if (ns == 1) {   // the cells' values read together
      double2 s01[4], s23[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int cx = ax - 1 + (c & 1), cy = ay - 1 + (c >> 1);
        const bool in = cx >= 0 && cy >= 0 && cx < k.ncx && cy < k.ncy;
        const double2* p = reinterpret_cast<const double2*>(k.pc) + (in ? cy * k.ncx + cx : 0) * 2;
        s01[c] = in ? __ldcg(p) : make_double2(0.0, 0.0);
        s23[c] = in ? __ldcg(p + 1) : make_double2(0.0, 0.0);
      }
      q[0] = s23[0].y;
      q[1] = s23[1].x - s23[1].y;
      q[2] = s01[2].y - s23[2].y;
      q[3] = (s01[3].x - s01[3].y) - (s23[3].x - s23[3].y);
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int cx = ax - 1 + (c & 1), cy = ay - 1 + (c >> 1);
        double v = 0.0;
        if (cx >= 0 && cy >= 0 && cx < k.ncx && cy < k.ncy) {
          const double2* p = reinterpret_cast<const double2*>(k.pc) + (size_t)(cy * k.ncx + cx) * ns * 2;
          for (int u = 0; u < ns; ++u) {
            const double2 s01 = __ldcg(p + 2 * u), s23 = __ldcg(p + 2 * u + 1);
            v += c == 0 ? s23.y : c == 1 ? s23.x - s23.y : c == 2 ? s01.y - s23.y : (s01.x - s01.y) - (s23.x - s23.y);
          }
        }
        q[c] = v;
      }
    }
    vc[a] = (q[0] + q[1]) + (q[2] + q[3]);
  }
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w < 4) {   // warp w: the three vertices of row ky - 1 + w
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    if (w < 3) {
      for (int b = lane; b < k.nc; b += 32) {
        const double vb = vc[b];
#pragma unroll
        for (int i = 0; i < 3; ++i) s[i] = fma(a0[3 * w + i][b], vb, s[i]);
      }
      kry_warp_sums<4>(s);
    }
    if ((lane & 7) == 0) zc[4 * w + kry_which<4>(lane)] = s[0];
  }
  __syncthreads();
  if (threadIdx.x < 9) {
    const double* z = zc + (threadIdx.x / 3) * 4 + threadIdx.x % 3;
    double* c = cc[threadIdx.x];
    c[0] = z[0];
    c[1] = z[1] - z[0];
    c[2] = z[4] - z[0];
    c[3] = (z[5] - z[4]) - (z[1] - z[0]);
  }
  __syncthreads();
}
// the rows of A0^{-1} of the vertices (kx - 1 .. kx + 1) x (ky - 1 .. ky + 1) into shared memory
__device__ __forceinline__ void kry_load_rows(const Kry& k, const KTile& t, double (*a0)[kCoarseMax]) {
  for (int i = threadIdx.x; i < 9 * k.nc; i += kKT) {
    const int r = i / k.nc, b = i - r * k.nc, ax = t.kx - 1 + r % 3, ay = t.ky - 1 + r / 3;
    a0[r][b] = ax >= 0 && ay >= 0 ? k.A0[(size_t)(ay * (k.ncx + 1) + ax) * k.nc + b] : 0.0;
  }
  __syncthreads();
}

// y = M^{-1} x on the tile and one element around it: the two sides' element-patch results
// plus the coarse correction, into sy as [element of the widened tile][left, bottom][node]
// (zero on boundary faces); the owned values also to out
template <int P>
__device__ __forceinline__ void kry_gather(const Kry& k, const KTile& t, const double (*cc)[4], double* sy,
                                           double* __restrict__ out) {
  constexpr int NL = P + 1, NL4 = 4 * NL;
  const int W = t.i1 - t.i0 + 2, nel = W * (t.j1 - t.j0 + 2);
  // the coarse cells' lines around the tile's cell
  const int xl = t.kx * k.cx, xr = xl + k.cx, yl = t.ky * k.cy, yr = yl + k.cy;
  for (int q = threadIdx.x; q < nel * 2 * NL; q += kKT) {
    const int le = q / (2 * NL), c = q - le * 2 * NL, side = c / NL, tt = c - side * NL;
    const int lj = kry_div(le, t.r2), i = t.i0 - 1 + le - lj * W, j = t.j0 - 1 + lj;
    double y = 0.0;
    if (i >= 0 && j >= 0 && i < k.nx && j < k.ny && (side == 0 ? i > 0 : j > 0)) {
      const int e = j * k.nx + i, m = kry_dof<P>(k, side, i, j, tt);
      const double z1 = __ldcg(k.z + (side == 0 ? (e - 1) * NL4 + NL : (e - k.nx) * NL4 + 2 * NL) + tt);
      const double z2 = __ldcg(k.z + e * NL4 + (side == 0 ? 3 * NL : 0) + tt);
      const double2 cw = k.cw[m];
      // the face's cell is its element's
      const double* d = cc[(j < yl ? 0 : j < yr ? 3 : 6) + (i < xl ? 0 : i < xr ? 1 : 2)];
      y = fma(cw.y, fma(cw.x, d[3], d[2]), fma(cw.x, d[1], d[0] + (z1 + z2)));
      if (i >= t.i0 && i < t.i1 && j >= t.j0 && j < t.j1) out[m] = y;
    }
    sy[q] = y;
  }
  __syncthreads();
}

// y = H x on the tile's owned multipliers (x staged by kry_gather); use(index, y) for each.
// Large tiles: a lane per multiplier sums both sides' rows of H_e.  Small ones (at most kKT
// items): two lanes per multiplier, one for each side's row, which keeps more sub-partitions at
// work; the row, which does not depend on x, is fetched before x is formed (kry_fetch), so
// that its latency overlaps the coarse solve and the gather.
template <int P>
__device__ __forceinline__ int kry_apply_items(const KTile& t) {
  const int own = (t.i1 - t.i0) * (t.j1 - t.j0) * 2 * (P + 1);
  return 2 * own <= kKT ? 2 * own : own;
}
template <int P>
struct KFetch {
  double2 a[2 * (P + 1)];
  const double* x0;   // the row's element in the staged buffer
  int m;              // the multiplier, or -1
};
template <int P>
__device__ __forceinline__ void kry_fetch(const Kry& k, const KTile& t, const double* sy, KFetch<P>& r) {
  constexpr int NL = P + 1, NL4 = 4 * NL;
  const int w = t.i1 - t.i0, own = w * (t.j1 - t.j0) * 2 * NL, W = w + 2;
  r.m = -1;
  if (2 * own > kKT || (int)threadIdx.x >= 2 * own) return;
  const int d = threadIdx.x >> 1, which = threadIdx.x & 1;
  const int le = d / (2 * NL), c = d - le * 2 * NL, side = c / NL, tt = c - side * NL;
  const int lj = kry_div(le, t.r0), li = le - lj * w, i = t.i0 + li, j = t.j0 + lj;
  if (side == 0 ? i == 0 : j == 0) return;
  // the element on the left / below (its right / top face), or the owner
  const int di = which == 0 && side == 0, dj = which == 0 && side == 1;
  const int e = (j - dj) * k.nx + i - di, row = (which == 0 ? (side == 0 ? NL : 2 * NL) : (side == 0 ? 3 * NL : 0)) + tt;
  r.m = kry_dof<P>(k, side, i, j, tt);
  r.x0 = sy + ((lj + 1 - dj) * W + li + 1 - di) * 2 * NL;
  const double2* A = reinterpret_cast<const double2*>(k.He + (size_t)(e * NL4 + row) * NL4);
#pragma unroll
  for (int h = 0; h < NL4 / 2; ++h) r.a[h] = __ldg(A + h);
}
template <int P, typename F>
__device__ __forceinline__ void kry_apply(const Kry& k, const KTile& t, const double* __restrict__ sy,
                                          const KFetch<P>& r, F use) {
  constexpr int NL = P + 1, NL4 = 4 * NL;
  const int w = t.i1 - t.i0, own = w * (t.j1 - t.j0) * 2 * NL, W = w + 2;
  if (2 * own <= kKT) {
    double s = 0.0;
    if (r.m >= 0) {
      const double* x0 = r.x0;
      const double* xf[4] = {x0 + NL, x0 + 2 * NL, x0 + W * 2 * NL + NL, x0};
#pragma unroll
      for (int h = 0; h < NL4 / 2; ++h) {
        s = fma(r.a[h].x, xf[(2 * h) / NL][(2 * h) % NL], s);
        s = fma(r.a[h].y, xf[(2 * h + 1) / NL][(2 * h + 1) % NL], s);
      }
    }
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (r.m >= 0 && (threadIdx.x & 1)) use(r.m, s);
    return;
  }
  for (int q = threadIdx.x; q < own; q += kKT) {
    const int le = q / (2 * NL), c = q - le * 2 * NL, side = c / NL, tt = c - side * NL;
    const int lj = kry_div(le, t.r0), li = le - lj * w, i = t.i0 + li, j = t.j0 + lj;
    if (side == 0 ? i == 0 : j == 0) continue;
    const int e = j * k.nx + i;
    const double* x0 = sy + ((lj + 1) * W + li + 1) * 2 * NL;
    use(kry_dof<P>(k, side, i, j, tt),
        side == 0 ? kry_row<P>(k.He, e - 1, NL + tt, x0 - 2 * NL, W) + kry_row<P>(k.He, e, 3 * NL + tt, x0, W)
                  : kry_row<P>(k.He, e - k.nx, 2 * NL + tt, x0 - W * 2 * NL, W) + kry_row<P>(k.He, e, tt, x0, W));
  }
}

template <int P>
__device__ __forceinline__ int kry_stage_items(const KTile& t) {
  return (t.i1 - t.i0 + 1) * (t.j1 - t.j0 + 1) * 2 * (P + 1);
}
// Stages x on the tile and one column and row to its right and top for kry_patches: value(m)
// gives x at multiplier m, own(m, x, (xi, eta)) is called for the owned ones with their
// local coordinates in the coarse cell.  Zero on boundary faces.
template <int P, typename V, typename O>
__device__ __forceinline__ void kry_stage(const Kry& k, const KTile& t, double* sx, V value, O own) {
  constexpr int NL = P + 1;
  const int W = t.i1 - t.i0 + 1, nel = W * (t.j1 - t.j0 + 1);
  for (int q = threadIdx.x; q < nel * 2 * NL; q += kKT) {
    const int le = q / (2 * NL), c = q - le * 2 * NL, side = c / NL, tt = c - side * NL;
    const int lj = kry_div(le, t.r1), i = t.i0 + le - lj * W, j = t.j0 + lj;
    double x = 0.0;
    if (i < k.nx && j < k.ny && (side == 0 ? i > 0 : j > 0)) {
      const int m = kry_dof<P>(k, side, i, j, tt);
      x = value(m);
      if (i < t.i1 && j < t.j1) own(m, x, k.cw[m]);
    }
    sx[q] = x;
  }
  __syncthreads();
}

// sums of x, xi x, eta x and xi eta x: a tile's restriction to its coarse cell
__device__ __forceinline__ void kry_restrict(double (&acc)[8], double x, double2 c) {
  const double tx = c.x * x;
  acc[0] += x;
  acc[1] += tx;
  acc[2] = fma(c.y, x, acc[2]);
  acc[3] = fma(c.y, tx, acc[3]);
}

// n iterations from the state left by the last launch (st->base of them done); check: then
// the convergence test on the residual they leave.  Dynamic shared memory: the staged vector
// of one tile with its halo.
template <int P>
__global__ void __launch_bounds__(kKT, 1) kry_solve_kernel(Kry k, int n, int check, unsigned int* status) {
  extern __shared__ double sv[];
  __shared__ double vc[kCoarseMax], zc[16], cc[9][4], a0[9][kCoarseMax];
  __shared__ KryScal sc;
  KState* st = k.st;
  const bool lead = threadIdx.x == 0;
  unsigned epoch = 0;
  int it = st->base;
  if (lead) {
    sc.rho = st->rho;
    sc.alpha = st->alpha;
    sc.bb = st->bb;
    sc.rr = st->rr;
    sc.tol2 = st->tol2;
    sc.done = st->done;
    sc.iters = st->iters;
  }
  __syncthreads();
  auto part = [&](int q, int tile) -> double& { return k.part[(size_t)q * k.ntiles + tile]; };
  // usually one tile per CTA: its ranges and rows of A0^{-1} are kept
  const KTile t0 = kry_tile(k, min((int)blockIdx.x, k.ntiles - 1));
  const bool one = k.ntiles <= (int)gridDim.x;
  kry_load_rows(k, t0, a0);
  for (int j = 0; !sc.done; ++j) {
    if (j == n && !check) break;
    // ---- A
    if (it > 0) {
      kry_sums(k, sc, kDotTS, kDotTT, kDotRS, kDotRT, 4);
      if (threadIdx.x < 32) {
        // beta = (rho' / rho) (alpha / omega): its three divisions on three lanes at once
        const int l = threadIdx.x;
        const double q = kry_quot(l == 0 ? sc.dot[0] : l == 1 ? sc.dot[1] : sc.alpha,
                                  l == 0 ? sc.dot[1] : l == 1 ? sc.dot[0] : sc.rho);
        const double ti = __shfl_sync(0xffffffffu, q, 1), ar = __shfl_sync(0xffffffffu, q, 2);
        if (lead) {
          const double omega = sc.dot[1] > 0.0 ? q : 0.0;
          const double rho = sc.dot[2] - omega * sc.dot[3];
          const bool brk = rho == 0.0 || !isfinite(rho) || omega == 0.0;
          sc.omega = omega;
          sc.rho_new = rho;
          sc.brk = brk;
          sc.beta = brk ? 0.0 : rho * ar * ti;
        }
      }
      __syncthreads();
    }
    const double omega = sc.omega, beta = sc.beta, alpha = sc.alpha;
    const double* po = k.p[it & 1];
    double* pn = k.p[(it & 1) ^ 1];
    for (int tile = blockIdx.x; tile < k.ntiles; tile += gridDim.x) {
      const KTile t = one ? t0 : kry_tile(k, tile);
      double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
      double ri = 0.0;   // r at the value just formed
      kry_stage<P>(
          k, t, sv,
          [&](int m) {
            if (it == 0) return ri = __ldcg(k.r + m);
            ri = fma(-omega, __ldcg(k.t + m), __ldcg(k.s + m));
            return fma(beta, fma(-omega, __ldcg(k.v + m), __ldcg(po + m)), ri);
          },
          [&](int m, double pm, double2 cw) {
            if (it == 0) {
              k.rh[m] = ri;
              k.x[m] = 0.0;
            } else {
              k.x[m] += fma(omega, k.sh[m], alpha * k.ph[m]);   // one rounding at the size of x
              k.r[m] = ri;
            }
            pn[m] = pm;
            kry_restrict(acc, pm, cw);
            acc[4] = fma(ri, ri, acc[4]);
          });
      if (j < n) kry_patches<P>(k, t, sv);
      kry_block_sums<5, 8>(acc, kry_stage_items<P>(t), [&](int i, double a) {
        if (i < 4) k.pc[4 * tile + i] = a;
        else part(kDotRR, tile) = a;
      });
    }
    if (!kry_barrier(st, epoch, status)) return;
    // the convergence test waits for the next phase's dots (its sum would cost a round trip of
    // its own), except at the end
    auto test = [&](double rr, bool last) {
      sc.rr = rr;
      if (it == 0) {
        sc.bb = rr;
        sc.rho_new = rr;
        sc.brk = rr == 0.0 || !isfinite(rr);
      }
      const bool conv = rr <= sc.tol2 * sc.bb;
      if (conv || (sc.brk && !last)) {
        sc.done = conv ? 1 : 2;
        sc.iters = it;
      }
      sc.rho = sc.rho_new;
    };
    if (j == n) {
      kry_sums(k, sc, kDotRR, 0, 0, 0, 1);
      if (lead) test(sc.dot[0], true);
      __syncthreads();
      break;
    }
    // ---- B
    for (int tile = blockIdx.x; tile < k.ntiles; tile += gridDim.x) {
      const KTile t = one ? t0 : kry_tile(k, tile);
      KFetch<P> row;
      kry_fetch<P>(k, t, sv, row);
      if (!one) kry_load_rows(k, t, a0);
      kry_coarse(k, a0, vc, zc, cc);
      kry_gather<P>(k, t, cc, sv, k.ph);
      double acc[1] = {0.0};
      kry_apply<P>(k, t, sv, row, [&](int m, double y) {
        k.v[m] = y;
        acc[0] = fma(k.rh[m], y, acc[0]);
      });
      kry_block_sums<1, 1>(acc, kry_apply_items<P>(t), [&](int, double a) { part(kDotRV, tile) = a; });
    }
    if (!kry_barrier(st, epoch, status)) return;
    // ---- C
    kry_sums(k, sc, kDotRV, kDotRR, 0, 0, 2);
    if (lead) {
      test(sc.dot[1], false);
      sc.alpha = kry_quot(sc.rho, sc.dot[0]);
      if (!sc.done && !isfinite(sc.alpha)) {
        sc.done = 2;
        sc.iters = it;
      }
    }
    __syncthreads();
    if (sc.done) break;
    const double a1 = sc.alpha;
    for (int tile = blockIdx.x; tile < k.ntiles; tile += gridDim.x) {
      const KTile t = one ? t0 : kry_tile(k, tile);
      double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
      kry_stage<P>(
          k, t, sv, [&](int m) { return fma(-a1, __ldcg(k.v + m), __ldcg(k.r + m)); },
          [&](int m, double sm, double2 cw) {
            k.s[m] = sm;
            kry_restrict(acc, sm, cw);
            acc[4] = fma(k.rh[m], sm, acc[4]);
          });
      kry_patches<P>(k, t, sv);
      kry_block_sums<5, 8>(acc, kry_stage_items<P>(t), [&](int i, double a) {
        if (i < 4) k.pc[4 * tile + i] = a;
        else part(kDotRS, tile) = a;
      });
    }
    if (!kry_barrier(st, epoch, status)) return;
    // ---- D
    for (int tile = blockIdx.x; tile < k.ntiles; tile += gridDim.x) {
      const KTile t = one ? t0 : kry_tile(k, tile);
      KFetch<P> row;
      kry_fetch<P>(k, t, sv, row);
      if (!one) kry_load_rows(k, t, a0);
      kry_coarse(k, a0, vc, zc, cc);
      kry_gather<P>(k, t, cc, sv, k.sh);
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      kry_apply<P>(k, t, sv, row, [&](int m, double y) {
        k.t[m] = y;
        acc[0] = fma(k.s[m], y, acc[0]);
        acc[1] = fma(y, y, acc[1]);
        acc[2] = fma(k.rh[m], y, acc[2]);
      });
      kry_block_sums<3, 4>(acc, kry_apply_items<P>(t), [&](int i, double a) { part(i == 0 ? kDotTS : i == 1 ? kDotTT : kDotRT, tile) = a; });
    }
    ++it;
    if (!kry_barrier(st, epoch, status)) return;
  }
  if (blockIdx.x == 0 && lead) {
    st->done = sc.done;
    st->iters = sc.iters;
    st->base = it;
    st->bb = sc.bb;
    st->rr = sc.rr;
    st->rho = sc.rho;
    st->alpha = sc.alpha;
  }
}

static inline unsigned nblk(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// The tiles of the Krylov kernel: a coarse cell each, cut along its longer side while its staged
// vector with its halo does not fit a CTA's shared memory, and on while every tile still has an
// SM of its own and more than kTileMin elements.  The second rule serves strips, whose coarse grid
// has few cells: whole solves 10000 x 1 Q2 12.7 -> 5.4 ms, 1000 x 4 3.6 -> 2.7, 500 x 5 2.5 -> 2.2;
// with a limit of 8 elements 100 x 3 Q3 takes 1.29 ms instead of 1.22 (shorter tiles, the same
// barriers), with 64 1000 x 4 takes 3.1.  A mesh of 11 x 11 cells is cut for shared memory only.
template <typename Fits>
static void kry_cut(Kry& k, int sms, Fits fits) {
  k.sx = k.sy = 1;
  k.tw = k.cx;
  k.th = k.cy;
  for (;;) {
    const bool wide = k.tw >= k.th;
    // the fewest parts shorter than now, of even length: none is empty in a whole cell
    const int sx = wide && k.tw > 1 ? (k.cx + k.tw - 2) / (k.tw - 1) : k.sx;
    const int sy = !wide && k.th > 1 ? (k.cy + k.th - 2) / (k.th - 1) : k.sy;
    const int w = (k.cx + sx - 1) / sx, h = (k.cy + sy - 1) / sy;
    if (fits() && ((long long)k.ncx * k.ncy * sx * sy > sms || k.tw * k.th <= kTileMin)) return;
    k.tw = w;
    k.th = h;
    k.sx = sx;
    k.sy = sy;
  }
}

template <int P>
static vef_status hrt_run(Mesh& M, const HrtIn& in, double tol, int max_iter, double* phi, double* J,
                          double* lambda, vef_hrt_info* info, cudaStream_t s, bool& launched) {
  using S = HrtShape<P>;
  const long long E = M.E;
  const long long nfaces = (long long)(M.nx - 1) * M.ny + (long long)M.nx * (M.ny - 1);
  const long long nl = nfaces * S::NL;
  const size_t per_e = (size_t)S::MM * S::MM + (size_t)S::NJ * S::NL4 + S::NJ + S::N + (size_t)S::NL4 * S::NL4 +
                       S::NL4;
  const size_t vec = (size_t)std::max(1LL, nl);
  if (!M.hrt_ref) {   // the reference tables, once per mesh
    auto refh = std::make_unique<HrtRef<P>>();
    make_hrt_ref<P>(make_hrt_tab(P, M.m), *refh);
    void* dev = nullptr;
    size_t cap = 0;
    vef_status st = ensure_buffer(&dev, &cap, sizeof(HrtRef<P>));
    if (st != VEF_OK) return st;
    cudaError_t ce = cudaMemcpyAsync(dev, refh.get(), sizeof(HrtRef<P>), cudaMemcpyHostToDevice, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) {
      cudaFree(dev);
      return cuda_fail(ce, "copying the HRT reference tables");
    }
    M.hrt_ref = dev;
  }
  const HrtRef<P>* ref = (const HrtRef<P>*)M.hrt_ref;
  // the coarse grid: at most kCoarseMaxCells cells per direction
  Kry k{};
  k.cx = (M.nx + kCoarseMaxCells - 1) / kCoarseMaxCells;
  k.cy = (M.ny + kCoarseMaxCells - 1) / kCoarseMaxCells;
  k.ncx = (M.nx + k.cx - 1) / k.cx;
  k.ncy = (M.ny + k.cy - 1) / k.cy;
  const int nc = (k.ncx + 1) * (k.ncy + 1);
  k.nc = nc;
  {
    double gw[kMaxP + 1];
    gauss_legendre(P + 1, k.gl, gw);
  }
  int dev = 0, sms = 0, inv_per_sm = 0;
  VEF_CUDA_TRY(cudaGetDevice(&dev));
  VEF_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  auto tile_smem = [&] { return (size_t)(k.tw + 2) * (k.th + 2) * 2 * S::NL * sizeof(double); };
  kry_cut(k, sms, [&] { return tile_smem() <= kTileSmemMax; });
  k.ntiles = k.ncx * k.ncy * k.sx * k.sy;
  const size_t total = per_e * E + 10 * vec + (size_t)(S::NL4 * S::NL4 + S::NL4) * E +
                       (size_t)nc * nc + 16 * (size_t)k.ncx * k.ncy + 4 * (size_t)k.ntiles + 2 * vec +
                       (size_t)kNumDots * k.ntiles + sizeof(KState) / sizeof(double) +
                       32;   // each of the takes below rounded up to two doubles
  vef_status st = ensure_buffer((void**)&M.work, &M.work_cap, total * sizeof(double));
  if (st != VEF_OK) return st;
  double* base = M.work;
  // 16-byte aligned pieces (cw is read as double2)
  auto take = [&](size_t n) { double* q = base; base += (n + 1) & ~(size_t)1; return q; };
  double* Li = take((size_t)S::MM * S::MM * E);
  double* C2 = take((size_t)S::NJ * S::NL4 * E);
  double* g = take((size_t)S::NJ * E);
  double* f = take((size_t)S::N * E);
  double* He = take((size_t)S::NL4 * S::NL4 * E);
  double* re = take((size_t)S::NL4 * E);
  k.nx = M.nx; k.ny = M.ny; k.nl = nl; k.He = He;
  k.x = lambda && nl > 0 ? lambda : take(vec);
  k.r = take(vec); k.rh = take(vec); k.p[0] = take(vec); k.p[1] = take(vec); k.v = take(vec); k.s = take(vec);
  k.t = take(vec); k.ph = take(vec); k.sh = take(vec);
  double* Pinv = take((size_t)S::NL4 * S::NL4 * E);
  k.Pinv = Pinv;
  k.z = take((size_t)S::NL4 * E);
  k.A0 = take((size_t)nc * nc);
  k.pc = take((size_t)4 * k.ntiles);
  double* Acell = take((size_t)16 * k.ncx * k.ncy);
  k.cw = reinterpret_cast<double2*>(take(2 * vec));
  k.part = take((size_t)kNumDots * k.ntiles);
  k.st = reinterpret_cast<KState*>(take(sizeof(KState) / sizeof(double)));
  HrtOut out{Li, C2, g, f, He, re};
  const size_t smem = sizeof(HrtSmem<P>), ismem = sizeof(HrtInvSmem<P>);
  const size_t csmem = (size_t)nc * (nc | 1) * sizeof(float);
  if ((st = allow_dynamic_smem<hrt_local_kernel<P>>()) != VEF_OK) return st;
  if ((st = allow_dynamic_smem<hrt_invert_kernel<P>>()) != VEF_OK) return st;
  if ((st = allow_dynamic_smem<hrt_coarse_pivot_kernel>()) != VEF_OK) return st;
  VEF_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&inv_per_sm, hrt_invert_kernel<P>, HrtInvShape<P>::T, ismem));
  launched = true;
  {
    KTimer kt(&M, VEF_K_HRT, s);
    hrt_local_kernel<P><<<(unsigned)std::min<long long>(E, (long long)sms * 8), 256, smem, s>>>(
        E, M.nx, M.ny, (M.m + 1) * (M.m + 1), ref, in, out);
    hrt_invert_kernel<P><<<(unsigned)std::min<long long>(E, (long long)sms * std::max(1, inv_per_sm)),
                           HrtInvShape<P>::T, ismem, s>>>(E, M.nx, M.ny, ref, out, M.dev_status);
    VEF_CUDA_TRY(cudaGetLastError());
  }
  int it = 0;
  KState hs{};
  if (nl > 0) {
    hrt_gather_kernel<P><<<nblk(nl, 256), 256, 0, s>>>(M.nx, M.ny, nfaces, re, k.r);
    hrt_asm_setup_kernel<P><<<(unsigned)((E + 3) / 4), 128, 0, s>>>(E, M.nx, M.ny, He, Pinv, M.dev_status);
    hrt_coarse_nodes_kernel<P><<<nblk(nl, 256), 256, 0, s>>>(k);
    hrt_coarse_cell_kernel<P><<<(unsigned)(k.ncx * k.ncy), 128, 0, s>>>(k, Acell);
    hrt_coarse_assemble_kernel<<<nblk(nc, 128), 128, 0, s>>>(k, Acell);
    int* fallback = (int*)&k.st->done;   // the state is set after the setup
    hrt_coarse_invert_kernel<<<1, 1024, 0, s>>>(k, fallback);
    hrt_coarse_pivot_kernel<<<1, kCoarseInvThreads, csmem, s>>>(k, fallback);
    VEF_CUDA_TRY(cudaGetLastError());
    hs.tol2 = tol * tol;
    VEF_CUDA_TRY(cudaMemcpyAsync(k.st, &hs, sizeof(KState), cudaMemcpyHostToDevice, s));
    const size_t ksmem = tile_smem();
    if ((st = allow_dynamic_smem<kry_solve_kernel<P>>()) != VEF_OK) return st;
    int per_sm = 0;
    VEF_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kry_solve_kernel<P>, kKT, ksmem));
    int grid = std::max(1, std::min(k.ntiles, sms * std::max(1, per_sm)));
    while (!hs.done && it < max_iter) {
      int n = std::min(kCheck, max_iter - it), check = it + n == max_iter;
      unsigned int* status = M.dev_status;
      void* args[] = {&k, &n, &check, &status};
      // a context limited to part of the device refuses a grid that does not fit it: halve it
      // (a CTA then takes several tiles)
      for (;; grid = (grid + 1) / 2) {
        VEF_CUDA_TRY(cudaMemsetAsync(&k.st->bar, 0, sizeof(unsigned), s));
        const cudaError_t e = cudaLaunchCooperativeKernel((const void*)kry_solve_kernel<P>, dim3((unsigned)grid),
                                                          dim3(kKT), args, ksmem, s);
        if (e == cudaSuccess) break;
        (void)cudaGetLastError();
        if (e != cudaErrorCooperativeLaunchTooLarge || grid == 1)
          return cuda_fail(e, "cudaLaunchCooperativeKernel(kry_solve_kernel)");
      }
      VEF_CUDA_TRY(cudaMemcpyAsync(&hs, k.st, sizeof(KState), cudaMemcpyDeviceToHost, s));
      VEF_CUDA_TRY(cudaStreamSynchronize(s));
      it += n;
      if (!hs.done && hs.base != it) {   // a grid barrier's wait ran out: the launch left early
        st = collect_status(M, s, nullptr);
        if (st != VEF_OK && st != VEF_ERR_TIMEOUT) return st;
        set_last_error("a grid barrier of the HRT multiplier solve gave up (a bounded device-side wait ran out)");
        return VEF_ERR_TIMEOUT;
      }
    }
    if (hs.done) it = hs.iters;
  }
  {
    KTimer kt(&M, VEF_K_HRT, s);
    hrt_recover_kernel<P><<<(unsigned)std::min<long long>(E, (long long)sms * 8), 128, 0, s>>>(
        E, M.nx, M.ny, Li, C2, g, f, k.x, J, phi);
    VEF_CUDA_TRY(cudaGetLastError());
  }
  const bool conv = nl == 0 || hs.done == 1;
  const double rel = nl == 0 || hs.bb <= 0.0 ? 0.0 : std::sqrt(hs.rr / hs.bb);
  if (info) {
    info->iterations = it;
    info->rel_residual = rel;
    info->multipliers = nl;
  }
  if (!conv) {
    set_last_error(hs.done == 2 ? "HRT multiplier solve broke down (BiCGStab)"
                                : "HRT multiplier solve did not reach its tolerance");
    return VEF_ERR_NOT_CONVERGED;
  }
  return VEF_OK;
}

}  // namespace
}  // namespace vef

using namespace vef;

extern "C" vef_status vef_hrt_solve(vef_mesh mesh, const double* sigma_t, const double* sigma_s,
                                    const double* phi_tr, const double* P_tr, const double* Eb,
                                    const double* Jin, const double* Q0, const double* Q1, double tol,
                                    int max_iter, double* phi, double* J, double* lambda,
                                    vef_hrt_info* info, void* stream) {
  if (!mesh || !sigma_t || !sigma_s || !phi_tr || !P_tr || !Eb || !Jin || !Q0 || !phi || !J) {
    set_last_error("mesh, sigma_t, sigma_s, phi_tr, P_tr, Eb, Jin, Q0, phi and J are required");
    return VEF_ERR_INVALID_ARG;
  }
  if (!(tol > 0.0) || max_iter < 1) {
    set_last_error("tol must be positive and max_iter >= 1");
    return VEF_ERR_INVALID_ARG;
  }
  Mesh& M = mesh->impl;
  int dev = 0;
  VEF_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != M.device) { set_last_error("mesh belongs to another device"); return VEF_ERR_INVALID_ARG; }
  HrtIn in{M.ctrl_dev, M.Mmat, M.nds, sigma_t, sigma_s, phi_tr, P_tr, Eb, Jin, Q0, Q1};
  cudaStream_t s = (cudaStream_t)stream;
  vef_status st;
  bool launched = false;
  switch (M.p) {
    case 1: st = hrt_run<1>(M, in, tol, max_iter, phi, J, lambda, info, s, launched); break;
    case 2: st = hrt_run<2>(M, in, tol, max_iter, phi, J, lambda, info, s, launched); break;
    case 3: st = hrt_run<3>(M, in, tol, max_iter, phi, J, lambda, info, s, launched); break;
    default: st = hrt_run<4>(M, in, tol, max_iter, phi, J, lambda, info, s, launched); break;
  }
  if (st == VEF_OK) return collect_status(M, s, nullptr);
  return launched ? collect_status_failed(M, s, st) : st;
}
