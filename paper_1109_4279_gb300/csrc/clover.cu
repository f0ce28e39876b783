// Clover term (abstract / Sec. 1: "Wilson-Dirac solver with Clover term"):
// A(x) = (4 + m0) + c_sw (i/4) sum_{mu != nu} sigma_{mu nu} Fhat_{mu nu}(x),
// built once per gauge field in FP64, plus the inverse of its two 6x6 chiral
// blocks on odd sites for the even/odd block solver (Sec. 5, Table 1).
#include "internal.h"

namespace qcd {

typedef cpx<double> cd;

struct M3 {
  cd m[3][3];
};

__device__ __forceinline__ M3 m3mul(const M3& a, const M3& b) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cd v = cmul(a.m[i][0], b.m[0][j]);
      v = cmadd(a.m[i][1], b.m[1][j], v);
      v = cmadd(a.m[i][2], b.m[2][j], v);
      r.m[i][j] = v;
    }
  return r;
}

__device__ __forceinline__ M3 m3dag(const M3& a) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) r.m[i][j] = conjg(a.m[j][i]);
  return r;
}

// q - q^+ of the product q = a b in 9 reals: twice the imaginary diagonal,
// then (re, im) of the elements (0,1), (0,2), (1,2).  The real diagonal is never
// formed, which leaves 90 of a product's 108 FP64 operations.
__device__ __forceinline__ void antiherm_product(const M3& a, const M3& b, double t[9]) {
  const M3 q = m3mul(a, b);
#pragma unroll
  for (int i = 0; i < 3; ++i) t[i] = 2.0 * q.m[i][i].im;
  int k = 3;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i + 1; j < 3; ++j) {
      t[k++] = q.m[i][j].re - q.m[j][i].re;
      t[k++] = q.m[i][j].im + q.m[j][i].im;
    }
}

__device__ __forceinline__ M3 link_of(const Geom& g, const double2* U64, long long s, int mu) {
  const int blk = (int)(s / g.Vb), r = (int)(s - (long long)blk * g.Vb);
  const SU3<double> u = load_link<P64, double>(U64, g.Vb, blk, r, mu);
  M3 o;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) o.m[i][j] = u.m[i][j];
  return o;
}

// internal index of x + s_mu mu-hat + s_nu nu-hat (periodic; selects only, no
// dynamically indexed writes)
__device__ __forceinline__ long long site_at(const Geom& g, const int x[4], int mu, int smu, int nu, int snu) {
  int y[4];
#pragma unroll
  for (int d = 0; d < 4; ++d) y[d] = (x[d] + (d == mu ? smu : 0) + (d == nu ? snu : 0) + g.L[d]) % g.L[d];
  return internal_index(g, y);
}

// the j-th of a site's 72 reals in a clover record's memory ([blk][36 double2][Vb]),
// which the build uses as scratch: a site's reals are its own, so the last pass can
// turn them into the record in place
__device__ __forceinline__ double* rec_real(double* rec, const Geom& g, long long s, int j) {
  const long long blk = s / g.Vb, r = s - blk * g.Vb;
  return rec + 2 * ((blk * 36 + (j >> 1)) * g.Vb + r) + (j & 1);
}

// planes 0 .. 5 in the order 01, 23, 02, 13, 03, 12: a launch takes two of them
__device__ __forceinline__ void plane_dirs(int q, int& mu, int& nu) {
  mu = (q & 1) == 0 ? 0 : (q == 5 ? 1 : (q == 3 ? 1 : 2));
  nu = q == 0 ? 1 : (q == 1 ? 3 : (q == 2 ? 2 : (q == 3 ? 3 : (q == 4 ? 3 : 2))));
}

// The four leaves of one plaquette (x; mu < nu), one thread each, for the plane
// q0 + blockIdx.y.  A leaf is the plaquette read from one of its corners, so
//   x:        U_mu(x) (D U_nu(x)^+)            x+mu:  D E
//   x+mu+nu:  U_mu(x+nu)^+ (E U_nu(x+mu))      x+nu:  E D
// with D = U_nu(x+mu) U_mu(x+nu)^+ and E = U_nu(x)^+ U_mu(x): 8 products where
// every site on its own takes 12 for its four leaves.  FP64 arithmetic is the
// bound, so the anti-Hermitian parts (9 reals) go through memory to the sites
// they belong to: slots [plane][leaf][9] in the 72 reals of Ahat's record.  With
// the packed inverse below, qcd_build_clover on 16^3 x 32 went from 3.0 ms (one
// kernel, its FP64 pipe 91 % busy, matrices in local memory) to 1.4 ms: this kernel
// 1.15 (the operations alone 1.0), the sums 0.05, the records and inverses 0.22.
__global__ void __launch_bounds__(128) clover_leaf_kernel(Geom g, const double2* __restrict__ U64, double* slots,
                                                          int q0) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int mu, nu, x[4];
  plane_dirs(q0 + blockIdx.y, mu, nu);
  global_coords(g, (int)(s / g.Vb), (int)(s % g.Vb), x);
  const long long s1 = site_at(g, x, mu, 1, -1, 0), s2 = site_at(g, x, mu, 1, nu, 1), s3 = site_at(g, x, nu, 1, -1, 0);
  const int j0 = 36 * blockIdx.y;
  double t[9];
  const M3 D = m3mul(link_of(g, U64, s1, nu), m3dag(link_of(g, U64, s3, mu)));
  {
    const M3 E = m3mul(m3dag(link_of(g, U64, s, nu)), link_of(g, U64, s, mu));
    antiherm_product(D, E, t);
#pragma unroll
    for (int k = 0; k < 9; ++k) *rec_real(slots, g, s1, j0 + 9 + k) = t[k];
    antiherm_product(E, D, t);
#pragma unroll
    for (int k = 0; k < 9; ++k) *rec_real(slots, g, s3, j0 + 27 + k) = t[k];
    antiherm_product(m3dag(link_of(g, U64, s3, mu)), m3mul(E, link_of(g, U64, s1, nu)), t);
#pragma unroll
    for (int k = 0; k < 9; ++k) *rec_real(slots, g, s2, j0 + 18 + k) = t[k];
  }
  antiherm_product(link_of(g, U64, s, mu), m3mul(D, m3dag(link_of(g, U64, s, nu))), t);
#pragma unroll
  for (int k = 0; k < 9; ++k) *rec_real(slots, g, s, j0 + k) = t[k];
}

// Fhat (9 reals, the form above) of two planes at a site: an eighth of its leaves' sum
__device__ __forceinline__ void leaf_sum(const double* slots, const Geom& g, long long s, double f[18]) {
  double2 v[36];
  const double2* p = (const double2*)rec_real(const_cast<double*>(slots), g, s, 0);
#pragma unroll
  for (int k = 0; k < 36; ++k) v[k] = p[(long long)k * g.Vb];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      double sum = 0;
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        const int j = 36 * q + 9 * l + k;
        const double w = (j & 1) ? v[j >> 1].y : v[j >> 1].x;
        sum = l == 0 ? w : sum + w;
      }
      f[9 * q + k] = 0.125 * sum;
    }
}

// Fhat of the launch's two planes into reals 18 (q0 / 2) .. + 17 of A's record memory
__global__ void __launch_bounds__(128) clover_sum_kernel(Geom g, const double* __restrict__ slots, double* F, int q0) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  double f[18];
  leaf_sum(slots, g, s, f);
  double2* o = (double2*)rec_real(F, g, s, 9 * q0);
#pragma unroll
  for (int k = 0; k < 9; ++k) o[(long long)k * g.Vb] = make_double2(f[2 * k], f[2 * k + 1]);
}

// pack the Hermitian 6x6 M into 36 reals: 6 diagonal, then (i < j) pairs row-major
__device__ __forceinline__ void pack_herm(const cd M[6][6], double* out) {
  for (int i = 0; i < 6; ++i) out[i] = M[i][i].re;
  int k = 6;
  for (int i = 0; i < 6; ++i)
    for (int j = i + 1; j < 6; ++j) {
      out[k++] = M[i][j].re;
      out[k++] = M[i][j].im;
    }
}

// Gauss-Jordan inverse with partial pivoting; returns false if singular
__device__ bool invert6(cd M[6][6], cd Inv[6][6]) {
  double scale = 0;
  for (int i = 0; i < 6; ++i)
    for (int j = 0; j < 6; ++j) {
      Inv[i][j] = {i == j ? 1.0 : 0.0, 0.0};
      scale = fmax(scale, fabs(M[i][j].re) + fabs(M[i][j].im));
    }
  for (int col = 0; col < 6; ++col) {
    int piv = col;
    double best = 0;
    for (int r = col; r < 6; ++r) {
      double a = fabs(M[r][col].re) + fabs(M[r][col].im);
      if (a > best) {
        best = a;
        piv = r;
      }
    }
    if (!(best > 1e-14 * scale)) return false;
    if (piv != col)
      for (int j = 0; j < 6; ++j) {
        cd t = M[col][j]; M[col][j] = M[piv][j]; M[piv][j] = t;
        t = Inv[col][j]; Inv[col][j] = Inv[piv][j]; Inv[piv][j] = t;
      }
    cd d = M[col][col];
    double den = d.re * d.re + d.im * d.im;
    cd dinv = {d.re / den, -d.im / den};
    for (int j = 0; j < 6; ++j) {
      M[col][j] = cmul(M[col][j], dinv);
      Inv[col][j] = cmul(Inv[col][j], dinv);
    }
    for (int r = 0; r < 6; ++r) {
      if (r == col) continue;
      cd f = M[r][col];
      for (int j = 0; j < 6; ++j) {
        M[r][j] = M[r][j] - cmul(f, M[col][j]);
        Inv[r][j] = Inv[r][j] - cmul(f, Inv[col][j]);
      }
    }
  }
  return true;
}

// i times element (a, b) of an anti-Hermitian matrix in 9 reals (Hermitian result)
__device__ __forceinline__ cd times_i_at(const double f[9], int a, int b) {
  if (a == b) return {-f[a], 0.0};
  const int k = 3 + 2 * (a + b - 1);
  return a < b ? cd{-f[k + 1], f[k]} : cd{-f[k + 1], -f[k]};
}

// Inverse of a Hermitian 6x6 in packed form by six sweeps: for each pivot k,
//   B_ij = A_ij - A_ik A_kj / A_kk,  B_ik = A_ik / A_kk,  B_kk = -1 / A_kk,
// which keeps the matrix Hermitian (60 FP64 operations per pivot where the
// elimination of M beside a unit matrix takes 288) and leaves minus the
// inverse.  Takes the pivots on the diagonal in order, as the elimination with
// column pivoting does whenever each is the largest of its column; returns
// false otherwise (m is then spoilt and the caller eliminates with pivoting).
__device__ __forceinline__ int herm_at(int i, int j) {  // packed index of (i < j)'s real part
  return 6 + 2 * (i * (11 - i) / 2 + (j - i - 1));
}
__device__ __forceinline__ bool invert6_sweep(double m[36]) {
  double scale = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) scale = fmax(scale, fabs(m[i]));
#pragma unroll
  for (int k = 6; k < 36; k += 2) scale = fmax(scale, fabs(m[k]) + fabs(m[k + 1]));
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double piv = fabs(m[k]);
    ok &= piv > 1e-14 * scale;
#pragma unroll
    for (int i = k + 1; i < 6; ++i) ok &= !(fabs(m[herm_at(k, i)]) + fabs(m[herm_at(k, i) + 1]) > piv);
    const double d = 1.0 / m[k];
    cd col[6], sc[6];  // A_ik and A_ik / A_kk
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      if (i == k) continue;
      const int p = i < k ? herm_at(i, k) : herm_at(k, i);
      col[i] = {m[p], i < k ? m[p + 1] : -m[p + 1]};
      sc[i] = d * col[i];
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      if (i == k) continue;
      m[i] = fma(-sc[i].re, col[i].re, fma(-sc[i].im, col[i].im, m[i]));
#pragma unroll
      for (int j = i + 1; j < 6; ++j) {  // A_ij -= (A_ik / A_kk) conj(A_jk)
        if (j == k) continue;
        const int p = herm_at(i, j);
        m[p] = fma(-sc[i].re, col[j].re, fma(-sc[i].im, col[j].im, m[p]));
        m[p + 1] = fma(-sc[i].im, col[j].re, fma(sc[i].re, col[j].im, m[p + 1]));
      }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      if (i == k) continue;
      const int p = i < k ? herm_at(i, k) : herm_at(k, i);
      m[p] = sc[i].re;
      m[p + 1] = i < k ? sc[i].im : -sc[i].im;
    }
    m[k] = -d;
  }
#pragma unroll
  for (int k = 0; k < 36; ++k) m[k] = -m[k];
  return ok;
}

// the general inverse of a packed Hermitian block (pivoting, matrices in local memory)
__device__ __noinline__ bool invert6_packed(double* m) {
  cd M[6][6], Inv[6][6];
  int k = 6;
  for (int i = 0; i < 6; ++i) {
    M[i][i] = {m[i], 0.0};
    for (int j = i + 1; j < 6; ++j) {
      M[i][j] = {m[k], m[k + 1]};
      M[j][i] = conjg(M[i][j]);
      k += 2;
    }
  }
  const bool ok = invert6(M, Inv);
  // symmetrise the inverse (Hermitian up to rounding)
  for (int i = 0; i < 6; ++i)
    for (int j = i; j < 6; ++j) {
      const cd a = Inv[i][j], b = conjg(Inv[j][i]);
      Inv[i][j] = 0.5 * (a + b);
      Inv[j][i] = conjg(Inv[i][j]);
    }
  pack_herm(Inv, m);
  return ok;
}

// A and Ahat of a site from Fhat: planes 01, 23, 02, 13 from A's record memory,
// 03 and 12 from the last leaves in Ahat's; both are then overwritten by the
// records (a thread reads and writes its own site's reals only)
__global__ void __launch_bounds__(128) clover_build_kernel(Geom g, double m0, double csw, FieldPtr A, FieldPtr Ahat,
                                                           int* bad) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  const int blk = (int)(s / g.Vb), r = (int)(s - (long long)blk * g.Vb);
  double f[54];  // [01, 23, 02, 13, 03, 12][9]
  {
    const double2* p = (const double2*)rec_real((double*)A.data, g, s, 0);
#pragma unroll
    for (int k = 0; k < 18; ++k) {
      const double2 v = p[(long long)k * g.Vb];
      f[2 * k] = v.x;
      f[2 * k + 1] = v.y;
    }
    leaf_sum((const double*)Ahat.data, g, s, f + 36);
  }
  // sigma_0k = diag(s_k, -s_k); sigma_jk = -eps_jkl diag(s_l, s_l).  Hence
  // upper block: (i c/2) sum_k s_k (x) E_k, E = (F01 - F23, F02 + F13, F03 - F12);
  // lower block: -(i c/2) sum_k s_k (x) B_k, B = (F01 + F23, F02 - F13, F03 + F12).
  double2* out = (double2*)A.data + (long long)blk * 36 * g.Vb + r;
  double2* hat = (double2*)Ahat.data + (long long)blk * 36 * g.Vb + r;
  const bool odd = r >= g.Vbh;
#pragma unroll 1
  for (int chir = 0; chir < 2; ++chir) {
    const double sg = chir == 0 ? 1.0 : -1.0, c = 0.5 * csw * sg;
    double e[3][9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      e[0][k] = f[k] - sg * f[9 + k];
      e[1][k] = f[18 + k] + sg * f[27 + k];
      e[2][k] = f[36 + k] - sg * f[45 + k];
    }
    // s1 E1 + s2 E2 + s3 E3 = [[E3, E1 - i E2], [E1 + i E2, -E3]], times i c
    double m[36];
#pragma unroll
    for (int i = 0; i < 6; ++i) m[i] = 4.0 + m0 + (i < 3 ? c : -c) * times_i_at(e[2], i % 3, i % 3).re;
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
      for (int j = i + 1; j < 6; ++j) {
        cd v;
        if ((i < 3) == (j < 3)) {
          const cd h = times_i_at(e[2], i % 3, j % 3);
          v = i < 3 ? h : -h;
        } else {
          v = times_i_at(e[0], i, j - 3) + mti(times_i_at(e[1], i, j - 3));
        }
        m[herm_at(i, j)] = c * v.re;
        m[herm_at(i, j) + 1] = c * v.im;
      }
#pragma unroll
    for (int k = 0; k < 18; ++k) out[(long long)(18 * chir + k) * g.Vb] = make_double2(m[2 * k], m[2 * k + 1]);
    if (odd) {
      double w[36];
#pragma unroll
      for (int k = 0; k < 36; ++k) w[k] = m[k];
      if (!invert6_sweep(w)) {
        double t[36];
#pragma unroll
        for (int k = 0; k < 36; ++k) t[k] = m[k];
        if (!invert6_packed(t)) atomicExch(bad, 1);
#pragma unroll
        for (int k = 0; k < 36; ++k) w[k] = t[k];
      }
#pragma unroll
      for (int k = 0; k < 36; ++k) m[k] = w[k];
    }
#pragma unroll
    for (int k = 0; k < 18; ++k) hat[(long long)(18 * chir + k) * g.Vb] = make_double2(m[2 * k], m[2 * k + 1]);
  }
}

int build_clover(qcd_ctx* c, cudaStream_t s) {
  if (!c->gauge_loaded) return QCD_ERR_STATE;
  ++c->gen;  // captured graphs hold the records of the last build
  // After qcd_load_gauge the FP64 records are written again in place: nothing can still
  // be reading them, or it would be reading links that the load replaced.  A term built
  // a second time on the same links may have readers queued on any stream, so all its
  // records are freed, which waits for them, and allocated anew.  (Not
  // cudaDeviceSynchronize: that fails while another thread captures a stream, and
  // contexts are independent.)
  const bool keep = !c->clover_built;
  c->clover_built = false;  // A's memory is scratch until the last pass
  for (int p = 0; p < 5; ++p) {
    if (keep && p == P64 && c->A[p].data && c->Ahat[p].data) continue;
    rec_free(c->A[p]);
    rec_free(c->Ahat[p]);
  }
  if (!c->A[P64].data) QCD_TRY(rec_alloc(c->A[P64], P64, 72, c->V));
  if (!c->Ahat[P64].data) QCD_TRY(rec_alloc(c->Ahat[P64], P64, 72, c->V));
  int* d_bad = (int*)c->d_scalars;
  QCD_CUDA(cudaMemsetAsync(d_bad, 0, sizeof(int), s));
  const unsigned grid = (unsigned)((c->V + 127) / 128);
  double* slots = (double*)c->Ahat[P64].data;
  for (int q = 0; q < 6; q += 2) {
    clover_leaf_kernel<<<dim3(grid, 2), 128, 0, s>>>(c->g, (const double2*)c->U[P64], slots, q);
    QCD_LAUNCHED();
    if (q == 4) break;  // the last two planes' leaves are summed by the pass that uses them
    clover_sum_kernel<<<grid, 128, 0, s>>>(c->g, slots, (double*)c->A[P64].data, q);
    QCD_LAUNCHED();
  }
  clover_build_kernel<<<grid, 128, 0, s>>>(c->g, c->p.m0, c->p.csw, c->A[P64].ptr(), c->Ahat[P64].ptr(), d_bad);
  QCD_LAUNCHED();
  int h = 0;
  QCD_CUDA(cudaMemcpyAsync(&h, d_bad, sizeof(int), cudaMemcpyDeviceToHost, s));
  QCD_CUDA(cudaStreamSynchronize(s));
  if (h) return QCD_ERR_SINGULAR_CLOVER;
  c->clover_built = true;
  return QCD_OK;
}

int ensure_clover(qcd_ctx* c, int prec, cudaStream_t s) {
  if (!c->clover_built) return QCD_ERR_STATE;
  if (c->A[prec].data) return QCD_OK;
  ++c->gen;
  QCD_TRY(rec_alloc(c->A[prec], prec, 72, c->V));
  QCD_TRY(rec_alloc(c->Ahat[prec], prec, 72, c->V));
  QCD_TRY(convert_rec(c, c->A[P64], c->A[prec], s));
  QCD_TRY(convert_rec(c, c->Ahat[P64], c->Ahat[prec], s));
  return QCD_OK;
}

}  // namespace qcd
