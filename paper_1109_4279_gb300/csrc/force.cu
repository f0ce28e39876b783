// Fermion force (Sec. 1: the inversions feed the HMC force): for
// L = Re(phi^+ x), x = D^-1 phi, y = D^-+ phi and the link deformation
// U_mu(x) -> exp(i theta_a lambda_a / 2) U_mu(x),
//   F_a(x, mu) = dL/dtheta_a = -Re(y^+ (dD/dtheta_a) x).
//
// Hopping part (the link appears in D at x and at x + mu):
//   F_a = -(eta/4) Im tr[lambda_a (U P1 - P2 U^+)] = -(eta/4) Im tr[lambda_a U (P1 + P2^+)],
//   P1 = sum_s h_s k_s^+,  h = proj_(1-g)(x(x+mu)), k = proj_(1-g)(y(x)),
//   P2 = sum_s h'_s k'_s^+, h' = proj_(1+g)(x(x)),  k' = proj_(1+g)(y(x+mu)),
// where proj keeps the two upper spin components of (1 -+ g_mu) psi (the
// lower two are fixed by them, which folds the spin trace to two terms).
//
// Clover part: with both orientations summed, the clover term equals
// (i c_sw / 16) sum_{rho != sigma} sigma_{rho sigma} (x) Q_{rho sigma}, so
//   F_a = (c_sw / 32) Re tr[lambda_a sum U S]   (sum over the 24 leaf
// occurrences of the link; a daggered occurrence contributes -S U^+), where S
// is the rest of the leaf read cyclically from the link, with
// W_{rho sigma}(z) = X + X^+, X = sum_{s,t} sigma_{rho sigma}[s][t] x_t(z) y_s(z)^+,
// inserted at the leaf's corner z.
//
// GB300's FP64 units (2 per SM and clock) bound all of this, so the work is
// arranged by the number of 3x3 products: one thread takes one plaquette and
// forms the contributions to its four links together, which shares the corner
// products and the products with W -- 25 matrix products per plaquette where
// link by link it takes 4 x 13.  Each contribution is 8 reals in a slot of the
// link's site; a second kernel adds a link's slots in a fixed order, so nothing
// is accumulated atomically.  24^3 x 48: 86.3 -> 20.6 ms per qcd_force (the version with
// one thread per link also kept its matrices in local memory).
#include "internal.h"

namespace qcd {

typedef cpx<double> cd;

struct C3 {
  cd m[3][3];
};

// Hermitian 3x3: the diagonal, then (0,1), (0,2), (1,2)
struct H3 {
  double d[3];
  cd o[3];
  __device__ __forceinline__ cd at(int i, int j) const {  // i != j
    return i < j ? o[i + j - 1] : conjg(o[i + j - 1]);
  }
};

// r += a b
__device__ __forceinline__ void c3mac(C3& r, const C3& a, const C3& b) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int k = 0; k < 3; ++k) r.m[i][j] = cmadd(a.m[i][k], b.m[k][j], r.m[i][j]);
}

__device__ __forceinline__ C3 c3mul(const C3& a, const C3& b) {
  C3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cd v = cmul(a.m[i][0], b.m[0][j]);
      v = cmadd(a.m[i][1], b.m[1][j], v);
      r.m[i][j] = cmadd(a.m[i][2], b.m[2][j], v);
    }
  return r;
}

// r += a h (h Hermitian: its diagonal is real)
__device__ __forceinline__ void c3mac(C3& r, const C3& a, const H3& h) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (k == j)
          fadd(r.m[i][j], h.d[k], a.m[i][k]);
        else
          r.m[i][j] = cmadd(a.m[i][k], h.at(k, j), r.m[i][j]);
      }
}

// r += h a
__device__ __forceinline__ void c3mac(C3& r, const H3& h, const C3& a) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (k == i)
          fadd(r.m[i][j], h.d[k], a.m[k][j]);
        else
          r.m[i][j] = cmadd(h.at(i, k), a.m[k][j], r.m[i][j]);
      }
}

__device__ __forceinline__ C3 c3zero() {
  C3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) r.m[i][j] = {0, 0};
  return r;
}

__device__ __forceinline__ C3 c3dag(const C3& a) {
  C3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) r.m[i][j] = conjg(a.m[j][i]);
  return r;
}

// Re tr(lambda_a M), a = 1..8
__device__ __forceinline__ void re_trace_lambda(const C3& M, double t[8]) {
  const double r3 = 0.57735026918962576451;  // 1 / sqrt(3)
  t[0] = M.m[1][0].re + M.m[0][1].re;
  t[1] = M.m[1][0].im - M.m[0][1].im;
  t[2] = M.m[0][0].re - M.m[1][1].re;
  t[3] = M.m[2][0].re + M.m[0][2].re;
  t[4] = M.m[2][0].im - M.m[0][2].im;
  t[5] = M.m[2][1].re + M.m[1][2].re;
  t[6] = M.m[2][1].im - M.m[1][2].im;
  t[7] = r3 * (M.m[0][0].re + M.m[1][1].re - 2.0 * M.m[2][2].re);
}

// Im tr(lambda_a M)
__device__ __forceinline__ void im_trace_lambda(const C3& M, double t[8]) {
  const double r3 = 0.57735026918962576451;
  t[0] = M.m[1][0].im + M.m[0][1].im;
  t[1] = M.m[0][1].re - M.m[1][0].re;
  t[2] = M.m[0][0].im - M.m[1][1].im;
  t[3] = M.m[2][0].im + M.m[0][2].im;
  t[4] = M.m[0][2].re - M.m[2][0].re;
  t[5] = M.m[2][1].im + M.m[1][2].im;
  t[6] = M.m[1][2].re - M.m[2][1].re;
  t[7] = r3 * (M.m[0][0].im + M.m[1][1].im - 2.0 * M.m[2][2].im);
}

__device__ __forceinline__ C3 link64(const Geom& g, const double2* U, long long s, int mu) {
  const int blk = (int)(s / g.Vb), r = (int)(s - (long long)blk * g.Vb);
  SU3<double> u = load_link<P64, double>(U, g.Vb, blk, r, mu);
  C3 o;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) o.m[i][j] = u.m[i][j];
  return o;
}

// internal index of x + s_mu mu-hat + s_nu nu-hat (periodic).  Written with
// selects only: no dynamically indexed local arrays, whose copies the
// compiler is free to place in overlapping stack slots.
__device__ __forceinline__ long long shifted(const Geom& g, const int x[4], int mu, int smu, int nu, int snu) {
  int y[4];
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    const int o = (d == mu ? smu : 0) + (d == nu ? snu : 0);
    y[d] = (x[d] + o + g.L[d]) % g.L[d];
  }
  return internal_index(g, y);
}

// the two directions mu < nu of plane 0 .. 5: 01 02 03 12 13 23
__device__ __forceinline__ void plane_dirs(int p, int& mu, int& nu) {
  mu = p < 3 ? 0 : (p < 5 ? 1 : 2);
  nu = p < 3 ? p + 1 : (p < 5 ? p - 1 : 3);
}

// W_{rho sigma}(z) = X + X^+ for np planes from p0 on; X = sum_st sigma[s][t] x_t y_s^+.
// sigma_0k = diag(s_k, -s_k), sigma_jk = -eps_jkl diag(s_l, s_l) in the chiral basis.
// W is Hermitian: 9 reals per site and plane, [plane][9][site] (the earlier
// [site][plane][18] made every store and load of a warp touch 32 lines).
__global__ void __launch_bounds__(128) force_w_kernel(Geom g, FieldPtr xf, FieldPtr yf, double* __restrict__ W, int p0,
                                                      int np) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  const int blk = (int)(s / g.Vb), r = (int)(s - (long long)blk * g.Vb);
  const Spinor<double> x = load_spinor<P64, double>(xf, g.Vb, blk, r);
  const Spinor<double> y = load_spinor<P64, double>(yf, g.Vb, blk, r);
#pragma unroll 1
  for (int q = 0; q < np; ++q) {
    // the Pauli index l and signs of sigma in the upper / lower chiral block:
    // 01: s1, 02: s2, 03: s3 (opposite in the lower block); 12: -s3, 13: s2, 23: -s1
    const int p = p0 + q;
    const int l = p < 3 ? p : 5 - p;
    const double su = p == 3 || p == 5 ? -1.0 : 1.0, sl = p < 3 ? -1.0 : su;
    C3 X = c3zero();
#pragma unroll
    for (int ch = 0; ch < 2; ++ch) {
      // sum_t sigma[s][t] x_t for s = 0, 1 (times the sign), then the outer products with y_s
      cd z[2][3];
      const double sg = ch == 0 ? su : sl;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const cd x0 = x.c[2 * ch][a], x1 = x.c[2 * ch + 1][a];
        const cd z0 = l == 0 ? x1 : (l == 1 ? mti(x1) : x0), z1 = l == 0 ? x0 : (l == 1 ? ti(x0) : -x1);
        z[0][a] = {sg * z0.re, sg * z0.im};
        z[1][a] = {sg * z1.re, sg * z1.im};
      }
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = 0; b < 3; ++b) X.m[a][b] = cjmadd(y.c[2 * ch + k][b], z[k][a], X.m[a][b]);
    }
    double* w = W + (long long)q * 9 * g.V + s;
#pragma unroll
    for (int a = 0; a < 3; ++a) w[(long long)a * g.V] = 2.0 * X.m[a][a].re;
    int k = 3;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = a + 1; b < 3; ++b) {
        w[(long long)k * g.V] = X.m[a][b].re + X.m[b][a].re;
        w[(long long)(k + 1) * g.V] = X.m[a][b].im - X.m[b][a].im;
        k += 2;
      }
  }
}

__device__ __forceinline__ H3 load_w(const double* __restrict__ W, long long V, long long s) {
  H3 h;
#pragma unroll
  for (int a = 0; a < 3; ++a) h.d[a] = __ldg(W + (long long)a * V + s);
#pragma unroll
  for (int k = 0; k < 3; ++k) h.o[k] = {__ldg(W + (long long)(3 + 2 * k) * V + s), __ldg(W + (long long)(4 + 2 * k) * V + s)};
  return h;
}

__device__ __forceinline__ void store_slot(double* __restrict__ S, long long V, long long s, const C3& M, double f) {
  double t[8];
  re_trace_lambda(M, t);
#pragma unroll
  for (int a = 0; a < 8; ++a) S[(long long)a * V + s] = f * t[a];
}

// One thread per plaquette (x; mu < nu) of plane p0 + blockIdx.y: links
// C0 = U_mu(x), C1 = U_nu(x+mu), C2 = U_mu(x+nu)^+, C3 = U_nu(x)^+ between the
// corners 0 = x, 1 = x+mu, 2 = x+mu+nu, 3 = x+nu with their W0 .. W3.  Reading
// the loop from the corner where a link starts (its own site), with W inserted
// once at every corner, the link's matrices are
//   U_nu(x+mu): M1 = (G2 + d W3) e + d K
//   U_mu(x+nu): M2 = -((W3 e + K) d + e G2)
//   U_mu(x):    M0 = T + L W0
//   U_nu(x):    M3 = -(T + W0 L),  T = (G1 + a W2) b + a G3, L = a b
// with the corner products a = C0 C1, b = C2 C3, d = C1 C2, e = C3 C0, the
// corners' insertions G1 = C0 W1 C1, G3 = C2 W3 C3, G2 = C1 W2 C2, G0 = C3 W0 C0
// and K = G0 + e W1.  Slots [plane][4][8][site]: M0 and M3 at x, M1 at x+mu, M2
// at x+nu.  Links and W are loaded again where they are used again (from L1 or
// L2): the FP64 pipe is the bound, and the registers hold the products.
__global__ void __launch_bounds__(128) force_plaquette_kernel(Geom g, const double2* __restrict__ U,
                                                              const double* __restrict__ W, double* __restrict__ S,
                                                              double f, int p0) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int mu, nu;
  plane_dirs(p0 + blockIdx.y, mu, nu);
  W += (long long)blockIdx.y * 9 * g.V;
  S += (long long)blockIdx.y * 32 * g.V;
  int x[4];
  global_coords(g, (int)(s / g.Vb), (int)(s % g.Vb), x);
  const long long s1 = shifted(g, x, mu, 1, -1, 0), s2 = shifted(g, x, mu, 1, nu, 1), s3 = shifted(g, x, nu, 1, -1, 0);
  {
    C3 G2, d;  // G2 = C1 W2 C2, d = C1 C2
    {
      const C3 C1 = link64(g, U, s1, nu), C2 = c3dag(link64(g, U, s3, mu));
      C3 t = c3zero();
      c3mac(t, C1, load_w(W, g.V, s2));
      G2 = c3mul(t, C2);
      d = c3mul(C1, C2);
    }
    C3 K, e;  // K = C3 W0 C0 + e W1, e = C3 C0
    {
      const C3 C3_ = c3dag(link64(g, U, s, nu)), C0 = link64(g, U, s, mu);
      C3 t = c3zero();
      c3mac(t, C3_, load_w(W, g.V, s));
      K = c3mul(t, C0);
      e = c3mul(C3_, C0);
    }
    c3mac(K, e, load_w(W, g.V, s1));
    const H3 W3 = load_w(W, g.V, s3);
    C3 t = G2;
    c3mac(t, d, W3);
    C3 M = c3mul(t, e);
    c3mac(M, d, K);
    store_slot(S + 16 * g.V, g.V, s1, M, f);
    c3mac(K, W3, e);
    M = c3mul(K, d);
    c3mac(M, e, G2);
    store_slot(S + 24 * g.V, g.V, s3, M, -f);
  }
  {
    C3 T, a;  // T = C0 W1 C1 + a W2, a = C0 C1
    {
      const C3 C0 = link64(g, U, s, mu), C1 = link64(g, U, s1, nu);
      C3 t = c3zero();
      c3mac(t, C0, load_w(W, g.V, s1));
      T = c3mul(t, C1);
      a = c3mul(C0, C1);
    }
    c3mac(T, a, load_w(W, g.V, s2));
    C3 L;
    {
      const C3 C2 = c3dag(link64(g, U, s3, mu)), C3_ = c3dag(link64(g, U, s, nu));
      const C3 b = c3mul(C2, C3_);
      T = c3mul(T, b);
      L = c3mul(a, b);
      C3 t = c3zero();
      c3mac(t, C2, load_w(W, g.V, s3));
      const C3 G3 = c3mul(t, C3_);
      c3mac(T, a, G3);
    }
    const H3 W0 = load_w(W, g.V, s);
    C3 M = T;
    c3mac(M, L, W0);
    store_slot(S, g.V, s, M, f);
    c3mac(T, W0, L);
    store_slot(S + 8 * g.V, g.V, s, T, -f);
  }
}

template <int S>
__device__ __forceinline__ void project_both(int mu, const Spinor<double>& p, const Spinor<double>& q, Half<double>& h,
                                             Half<double>& k) {
  switch (mu) {
    case 0: h = project<0, S>(p); k = project<0, S>(q); break;
    case 1: h = project<1, S>(p); k = project<1, S>(q); break;
    case 2: h = project<2, S>(p); k = project<2, S>(q); break;
    default: h = project<3, S>(p); k = project<3, S>(q); break;
  }
}

// One thread per link (site, mu = blockIdx.y): the hopping part (first group
// of planes) plus the slots of the planes p0 .. p0 + np - 1 that contain mu.
__global__ void __launch_bounds__(128) force_kernel(Geom g, const double2* __restrict__ U, FieldPtr xf, FieldPtr yf,
                                                    const double* __restrict__ S, int p0, int np, int first,
                                                    double* __restrict__ F) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  const int mu = blockIdx.y;
  const int blk = (int)(s / g.Vb), r = (int)(s - (long long)blk * g.Vb);
  int x[4];
  global_coords(g, blk, r, x);
  // F is a caller's array, aligned to 8 bytes only: one double at a time
  double* o = F + (lex_index(g, x) * 4 + mu) * 8;
  double out[8];
  if (first) {
    const long long sp = shifted(g, x, mu, 1, -1, 0);
    const int bp = (int)(sp / g.Vb), rp = (int)(sp - (long long)bp * g.Vb);
    const int xmu = mu == 0 ? x[0] : (mu == 1 ? x[1] : (mu == 2 ? x[2] : x[3]));
    const int Lmu = mu == 0 ? g.L[0] : (mu == 1 ? g.L[1] : (mu == 2 ? g.L[2] : g.L[3]));
    const double bcmu = mu == 0 ? g.bc[0] : (mu == 1 ? g.bc[1] : (mu == 2 ? g.bc[2] : g.bc[3]));
    const double eta = (xmu == Lmu - 1) ? bcmu : 1.0;
    C3 P = c3zero();  // P1 + P2^+ = sum_s h_s k_s^+ + k'_s h'_s^+
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      // half 0: h from x(x+mu), k from y(x), projector 1 - g; half 1: k' from y(x+mu), h' from x(x), 1 + g
      const Spinor<double> up = load_spinor<P64, double>(half ? yf : xf, g.Vb, bp, rp);
      const Spinor<double> here = load_spinor<P64, double>(half ? xf : yf, g.Vb, blk, r);
      Half<double> h, k;
      if (half == 0)
        project_both<-1>(mu, up, here, h, k);
      else
        project_both<+1>(mu, up, here, h, k);
#pragma unroll
      for (int sp_ = 0; sp_ < 2; ++sp_)
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = 0; b < 3; ++b) P.m[a][b] = cjmadd(k.c[sp_][b], h.c[sp_][a], P.m[a][b]);
    }
    im_trace_lambda(c3mul(link64(g, U, s, mu), P), out);
#pragma unroll
    for (int a = 0; a < 8; ++a) out[a] *= -0.25 * eta;
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) out[k] = o[k];
  }
#pragma unroll 1
  for (int q = 0; q < np; ++q) {
    int m, n;
    plane_dirs(p0 + q, m, n);
    if (m != mu && n != mu) continue;
    // the lower direction of the plane: slots 0 (own plaquette) and 3 (the one at x - nu);
    // the upper one: slots 1 and 2 (the one at x - mu)
    const double* a = S + ((long long)q * 4 + (m == mu ? 0 : 1)) * 8 * g.V + s;
    const double* b = S + ((long long)q * 4 + (m == mu ? 3 : 2)) * 8 * g.V + s;
#pragma unroll
    for (int k = 0; k < 8; ++k) out[k] += __ldg(a + (long long)k * g.V) + __ldg(b + (long long)k * g.V);
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) o[k] = out[k];
}

int force_apply(qcd_ctx* c, const Rec& x, const Rec& y, double* F, cudaStream_t s) {
  if (x.prec != P64 || y.prec != P64) return QCD_ERR_ARG;
  QCD_TRY(ensure_gauge(c, P64, s));
  // W (9 reals) and the four slots (32 reals) of a plane are 328 bytes per site: all
  // six planes in one launch up to 4 GiB of them and where the device has room, else
  // plane by plane (less memory than W alone used to take, the same sums in the same
  // order, and a large lattice fills the GPU with one plane)
  const size_t per_plane = (size_t)c->V * 41 * sizeof(double);
  int group = 6 * per_plane <= ((size_t)4 << 30) ? 6 : 1;
  const bool clover = c->p.csw != 0.0;
  Scratch mem;
  if (clover) {
    int st = mem.get(c, kScratchForce, per_plane * group);
    if (st == QCD_ERR_NOMEM && group > 1) st = mem.get(c, kScratchForce, per_plane * (group = 1));
    QCD_TRY(st);
  }
  double* W = (double*)mem.p;
  double* S = W + (size_t)c->V * 9 * group;
  const unsigned grid = (unsigned)((c->V + 127) / 128);
  const double2* U = (const double2*)c->U[P64];
  int st = QCD_OK;
  auto launched = [&st](const char* what) {
    const cudaError_t e = cudaGetLastError();
    g_launches.fetch_add(1);
    if (e != cudaSuccess) st = cuda_fail(e, what);
  };
  for (int p0 = 0; p0 < 6 && st == QCD_OK; p0 += group) {
    if (clover) {
      force_w_kernel<<<grid, 128, 0, s>>>(c->g, x.ptr(), y.ptr(), W, p0, group);
      launched("force_w_kernel");
      if (st == QCD_OK) {
        force_plaquette_kernel<<<dim3(grid, group), 128, 0, s>>>(c->g, U, W, S, c->p.csw / 32.0, p0);
        launched("force_plaquette_kernel");
      }
    }
    if (st == QCD_OK) {
      force_kernel<<<dim3(grid, 4), 128, 0, s>>>(c->g, U, x.ptr(), y.ptr(), S, p0, clover ? group : 0, p0 == 0, F);
      launched("force_kernel");
    }
    if (!clover) break;
  }
  cudaStreamSynchronize(s);
  return st;
}

}  // namespace qcd
