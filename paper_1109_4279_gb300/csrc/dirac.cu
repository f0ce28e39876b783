// Full-lattice clover Wilson-Dirac operator (Sec. 4: the matrix-vector product
// applied to a spinor field; Sec. 6: the double precision operator of the
// outer solver).  One thread per site; the 8 neighbour spinors are gathered
// through L1/L2 (the Schwarz blocks are contiguous and CTAs follow the block
// order, so block faces are re-read from cache, not HBM); links come from the
// site itself (forward hops) and from the backward neighbour.
#include "internal.h"

namespace qcd {

template <int P>
struct Arith {
  typedef float T;
};
template <>
struct Arith<P64> {
  typedef double T;
};

// a neighbour's spinor with its 16-bit scale left out (returned in `scale`,
// 1 for FP32/FP64), so the scale joins the hop coefficient
template <int P, typename T>
__device__ __forceinline__ Spinor<T> load_spinor_unscaled(const FieldPtr& f, int Vb, int blk, int r, T& scale) {
  if constexpr (P == P16 || P == PB16) {
    float v[24];
    scale = load_record_raw<P, 24>(f, Vb, blk, r, v);
    Spinor<T> s;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) s.c[a][b] = {v[6 * a + 2 * b], v[6 * a + 2 * b + 1]};
    return s;
  } else {
    scale = T(1);
    return load_spinor<P, T>(f, Vb, blk, r);
  }
}

// acc += -1/2 [eta U (1 -/+ g) psi(x + mu) + eta U^+ (1 +/- g) psi(x - mu)]; the
// factor -1/2, the boundary sign and the neighbour's 16-bit scale are one
// coefficient per hop (U h is linear in h)
template <int MU, int P, int DAG, typename T>
__device__ __forceinline__ void hop_pair(const Geom& g, const void* U, const FieldPtr& in, int blk, int r,
                                         const int y[4], const int n[4], Spinor<T>& acc) {
  constexpr int SF = DAG ? +1 : -1;  // D: (1 - g) psi(x + mu); D^+: (1 + g) psi(x + mu)
  {
    Nbr f = neighbour(g, blk, y, n, MU, +1);
    T sc;
    Spinor<T> p = load_spinor_unscaled<P, T>(in, g.Vb, f.blk, f.r, sc);
    Half<T> h = project<MU, SF>(p);
    SU3<T> u = load_link<P, T>(U, g.Vb, blk, r, MU);
    Half<T> w = umul(u, h);
    expand_add<MU, SF>(acc, w, (f.wrap ? T(-0.5) * bc_of<T>(g, MU) : T(-0.5)) * sc);
  }
  {
    Nbr b = neighbour(g, blk, y, n, MU, -1);
    T sc;
    Spinor<T> p = load_spinor_unscaled<P, T>(in, g.Vb, b.blk, b.r, sc);
    Half<T> h = project<MU, -SF>(p);
    SU3<T> u = load_link<P, T>(U, g.Vb, b.blk, b.r, MU);
    Half<T> w = udmul(u, h);
    expand_add<MU, -SF>(acc, w, (b.wrap ? T(-0.5) * bc_of<T>(g, MU) : T(-0.5)) * sc);
  }
}

// two FP32 numbers in one 64-bit register, for the packed instructions
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ uint64_t mul2p(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2p(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// (D psi)(site) or (D^+ psi)(site); A is Hermitian so D^+ only swaps projectors
template <int P, int DAG, typename T, bool PACK = false>
__device__ __forceinline__ Spinor<T> dirac_site(const Geom& g, const void* U, const FieldPtr& A, const FieldPtr& in,
                                               int blk, int r) {
  int n[4], y[4];
  block_coords(g, blk, n);
  const int packed = __ldg(g.r2y + r);
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) y[mu] = ycoord(packed, mu);
  Spinor<T> acc;
  zero(acc);
  hop_pair<0, P, DAG, T>(g, U, in, blk, r, y, n, acc);
  hop_pair<1, P, DAG, T>(g, U, in, blk, r, y, n, acc);
  hop_pair<2, P, DAG, T>(g, U, in, blk, r, y, n, acc);
  hop_pair<3, P, DAG, T>(g, U, in, blk, r, y, n, acc);
  T sp;
  Spinor<T> psi = load_spinor_unscaled<P, T>(in, g.Vb, blk, r, sp);
  if constexpr (P == P16 || P == PB16) {
    // one chiral 6x6 block at a time: chunks 4 hb .. 4 hb + 4 hold its 18
    // packed pairs from pair 2 hb on
    const uint4* d = (const uint4*)A.data + (long long)blk * 9 * g.Vb + r;
    const T s = (A.norm ? __ldg(A.norm + (long long)blk * g.Vb + r) : 1.0f) * sp;
#pragma unroll
    for (int hb = 0; hb < 2; ++hb) {
      uint32_t w[20];
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const uint4 v = __ldg(d + (long long)(4 * hb + k) * g.Vb);
        w[4 * k] = v.x;
        w[4 * k + 1] = v.y;
        w[4 * k + 2] = v.z;
        w[4 * k + 3] = v.w;
      }
      T c[36];
#pragma unroll
      for (int k = 0; k < 18; ++k) {
        const float2 x = to_f2<P>(w[2 * hb + k]);
        c[2 * k] = x.x;
        c[2 * k + 1] = x.y;
      }
      // PACK: packed FP32x2 instructions, one for the two parts of a number (x[i] the
      // input, ix[i] = i x[i]).  The compiler's register allocation decides: in the
      // 4^4 instantiation they take bf16 on 32^3 x 64 from 0.221 to 0.1785 ms and 12
      // FP16 right-hand sides on 24^3 x 48 from 0.670 to 0.620 ms, with 8 x 4^3
      // blocks they change nothing (0.176 and 0.61 ms), with general shapes they cost
      // 7 % (two right-hand sides on 24^3 x 48 0.129 against 0.139 ms).
      if constexpr (PACK) {
        uint64_t x[6], ix[6], o[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          const cpx<T> v = psi.c[2 * hb + i / 3][i % 3];
          x[i] = pack2(v.re, v.im);
          ix[i] = pack2(-v.im, v.re);
          o[i] = mul2p(pack2(c[i], c[i]), x[i]);
        }
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
          for (int j = i + 1; j < 6; ++j) {
            const int k = 6 + 2 * (5 * i - i * (i - 1) / 2 + j - i - 1);
            const uint64_t re = pack2(c[k], c[k]);
            o[i] = fma2p(re, x[j], fma2p(pack2(c[k + 1], c[k + 1]), ix[j], o[i]));
            o[j] = fma2p(re, x[i], fma2p(pack2(-c[k + 1], -c[k + 1]), ix[i], o[j]));
          }
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          cpx<T>& a = acc.c[2 * hb + i / 3][i % 3];
          float re, im;
          unpack2(o[i], re, im);
          a = {fma(s, re, a.re), fma(s, im, a.im)};
        }
      } else {
        cpx<T> i6[6], o6[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) i6[i] = psi.c[2 * hb + i / 3][i % 3];
        clover_block_apply(c, i6, o6);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          cpx<T>& a = acc.c[2 * hb + i / 3][i % 3];
          a = {fma(s, o6[i].re, a.re), fma(s, o6[i].im, a.im)};
        }
      }
    }
  } else {
    T c[72];
    load_record<P, 72, T>(A, g.Vb, blk, r, c);
    const Spinor<T> o = clover_apply(c, psi);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) acc.c[a][b] = acc.c[a][b] + o.c[a][b];
  }
  return acc;
}

// Schwarz block shapes with their own instantiation: BS = 1 for 4^4 and 2 for
// 8 x 4^3 (time extent 8); the in-block extents, strides and volume are then
// compile-time constants, which shortens the neighbour and address arithmetic
static int block_shape_id(const Geom& g) {
  if (g.b[1] == 4 && g.b[2] == 4 && g.b[3] == 4) {
    if (g.b[0] == 4) return 1;
    if (g.b[0] == 8) return 2;
  }
  return 0;
}

template <int BS>
__device__ __forceinline__ void fix_block_shape(Geom& g) {
  if constexpr (BS != 0) {
    constexpr int b0 = BS == 1 ? 4 : 8;
    g.b[0] = b0;
    g.b[1] = g.b[2] = g.b[3] = 4;
    g.ystr[0] = 64;
    g.ystr[1] = 16;
    g.ystr[2] = 4;
    g.ystr[3] = 1;
    g.Vb = 64 * b0;
    g.Vbh = 32 * b0;
  }
}

// one thread per site; with nrhs > 1 the thread applies the operator to every
// right-hand side in turn (fields nrhs apart by `stride` sites), so the
// site's links and clover block come from HBM once and from L1 afterwards.
// The FP32 instantiation is told it runs one 512-thread CTA per SM (the full
// 128 registers, used to issue more gathers ahead); the others keep the
// compiler's default
template <int P, int DAG, int BS>
__global__ void __launch_bounds__(512, P == P32 ? 1 : 0) dirac_kernel(Geom g0, const void* __restrict__ U, FieldPtr A, FieldPtr in,
                                                    FieldPtr out, int nrhs, const int* __restrict__ mask,
                                                    int out_df) {
  typedef typename Arith<P>::T T;
  Geom g = g0;
  fix_block_shape<BS>(g);
  long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int blk = (int)(s / g.Vb), r = (int)(s - (long long)blk * g.Vb);
  constexpr int NC = P == P64 ? 12 : (P == P32 ? 6 : 3);
#pragma unroll 1
  for (int k = 0; k < nrhs; ++k) {
    if (mask && !mask[k]) continue;  // a right-hand side of a batch that is not being iterated
    FieldPtr fi = in, fo = out;
    fi.data = (char*)in.data + (size_t)k * g.V * NC * 16;
    fo.data = (char*)out.data + (size_t)k * g.V * NC * 16;
    if (in.norm) fi.norm = in.norm + (size_t)k * g.V;
    if (out.norm) fo.norm = out.norm + (size_t)k * g.V;
    Spinor<T> o = dirac_site<P, DAG, T, BS == 1>(g, U, A, fi, blk, r);
    if constexpr (P == P64) {
      if (out_df) {  // the FP64 result split into double-float pairs for a df64 recursion
        store_spinor<PDF, T>(fo, g.Vb, blk, r, o);
        continue;
      }
    }
    store_spinor<P, T>(fo, g.Vb, blk, r, o);
  }
}

// ------------------------------------------------------------------------
// Two threads per site (16-bit storage).  The one-thread form above needs all
// 128 registers for a site's eight hops, which leaves 16 warps per SM to hide
// the gathers.  Here thread half hf of a CTA (warp-uniform: threads
// hf * 128 .. hf * 128 + 127) computes the hops in directions 2 hf and
// 2 hf + 1 of 128 sites and owns spin components 2 hf, 2 hf + 1 of their
// results: the partial hop sums of the other two components go to the partner
// through shared memory (a named barrier of the two warps that hold the same
// 32 sites), the clover term acts on the owned chiral half alone (it is block
// diagonal in chirality), and the per-site 16-bit scale of the result is the
// larger of the two halves' maxima.
// ------------------------------------------------------------------------
static constexpr int kPairSites = 128;  // sites per CTA of the two-thread form (256 threads)
// resident CTAs per SM the two-thread form is compiled for (its register budget)
#ifndef QCD_PAIR_MIN_CTAS
#define QCD_PAIR_MIN_CTAS 2
#endif

// owned half (spins 2 hf, 2 hf + 1) of a 16-bit spinor record without its scale
// (16-bit words 6 hf .. 6 hf + 5: chunk 2 hf and the hf-th 8-byte half of chunk 1)
template <int P>
__device__ __forceinline__ Half<float> load_half16_unscaled(const FieldPtr& f, int Vb, int blk, int r, int hf) {
  const uint4* d = (const uint4*)f.data + (long long)blk * 3 * Vb + r;
  const uint4 a = __ldg(d + (long long)(2 * hf) * Vb);
  const uint2 b = __ldg((const uint2*)(d + Vb) + hf);
  const uint32_t w[6] = {hf ? b.x : a.x, hf ? b.y : a.y, hf ? a.x : a.z, hf ? a.y : a.w, hf ? a.z : b.x, hf ? a.w : b.y};
  Half<float> h;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float2 x = to_f2<P>(w[k]);
    h.c[k / 3][k % 3] = {x.x, x.y};
  }
  return h;
}

// store the owned half with the site's scale (the maximum over both halves)
template <int P>
__device__ __forceinline__ void store_half16(const FieldPtr& f, int Vb, int blk, int r, int hf, const Half<float>& h,
                                             float scale) {
  typedef typename Storage<P>::real hr;
  const float inv = scale > 0.f ? 1.0f / scale : 0.f;
  uint32_t w[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    hr* q = reinterpret_cast<hr*>(&w[k]);
    q[0] = from_f<P>(h.c[k / 3][k % 3].re * inv);
    q[1] = from_f<P>(h.c[k / 3][k % 3].im * inv);
  }
  uint4* d = (uint4*)f.data + (long long)blk * 3 * Vb + r;
  if (hf == 0) {
    d[0] = make_uint4(w[0], w[1], w[2], w[3]);
    *((uint2*)(d + Vb)) = make_uint2(w[4], w[5]);
    f.norm[(long long)blk * Vb + r] = scale;
  } else {
    *((uint2*)(d + Vb) + 1) = make_uint2(w[0], w[1]);
    d[2 * (long long)Vb] = make_uint4(w[2], w[3], w[4], w[5]);
  }
}

template <int P, int DAG, int BS>
__global__ void __launch_bounds__(2 * kPairSites, QCD_PAIR_MIN_CTAS) dirac_pair_kernel(Geom g0, const void* __restrict__ U, FieldPtr A,
                                                                  FieldPtr in, FieldPtr out, int nrhs,
                                                                  const int* __restrict__ mask) {
  static_assert(P == P16 || P == PB16, "16-bit storage only");
  __shared__ float xch[2][12][kPairSites];  // [receiving half][real][site]
  __shared__ float mx[2][kPairSites];
  Geom g = g0;
  fix_block_shape<BS>(g);
  const int hf = threadIdx.x / kPairSites, li = threadIdx.x - hf * kPairSites;
  const long long s = (long long)blockIdx.x * kPairSites + li;
  const bool act = s < g.V;
  const long long sc = act ? s : 0;
  const int blk = (int)(sc / g.Vb), r = (int)(sc - (long long)blk * g.Vb);
  int n[4], y[4];
  block_coords(g, blk, n);
  {
    const int packed = __ldg(g.r2y + r);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) y[mu] = ycoord(packed, mu);
  }
  const int pair_bar = 1 + (li >> 5);  // named barrier of warps li / 32 and li / 32 + 4
#pragma unroll 1
  for (int k = 0; k < nrhs; ++k) {
    if (mask && !mask[k]) continue;
    FieldPtr fi = in, fo = out;
    fi.data = (char*)in.data + (size_t)k * g.V * 3 * 16;
    fo.data = (char*)out.data + (size_t)k * g.V * 3 * 16;
    fi.norm = in.norm + (size_t)k * g.V;
    fo.norm = out.norm + (size_t)k * g.V;
    Spinor<float> acc;
    zero(acc);
    if (hf) {
      hop_pair<2, P, DAG, float>(g, U, fi, blk, r, y, n, acc);
      hop_pair<3, P, DAG, float>(g, U, fi, blk, r, y, n, acc);
    } else {
      hop_pair<0, P, DAG, float>(g, U, fi, blk, r, y, n, acc);
      hop_pair<1, P, DAG, float>(g, U, fi, blk, r, y, n, acc);
    }
    // hand the partner its components
#pragma unroll
    for (int sp = 0; sp < 2; ++sp)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const cpx<float> v = acc.c[2 * (1 - hf) + sp][c];
        xch[1 - hf][6 * sp + 2 * c][li] = v.re;
        xch[1 - hf][6 * sp + 2 * c + 1][li] = v.im;
      }
    asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
    Half<float> o;
#pragma unroll
    for (int sp = 0; sp < 2; ++sp)
#pragma unroll
      for (int c = 0; c < 3; ++c)
        o.c[sp][c] = {acc.c[2 * hf + sp][c].re + xch[hf][6 * sp + 2 * c][li],
                      acc.c[2 * hf + sp][c].im + xch[hf][6 * sp + 2 * c + 1][li]};
    // clover: chiral block hf on the site's own half
    {
      const Half<float> psi = load_half16_unscaled<P>(fi, g.Vb, blk, r, hf);
      const float ps = __ldg(fi.norm + (long long)blk * g.Vb + r);
      const uint4* d = (const uint4*)A.data + (long long)blk * 9 * g.Vb + r;
      const float scl = (A.norm ? __ldg(A.norm + (long long)blk * g.Vb + r) : 1.0f) * ps;
      uint32_t w[20];
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const uint4 v = __ldg(d + (long long)(4 * hf + q) * g.Vb);
        w[4 * q] = v.x;
        w[4 * q + 1] = v.y;
        w[4 * q + 2] = v.z;
        w[4 * q + 3] = v.w;
      }
      float cb[36];
#pragma unroll
      for (int q = 0; q < 18; ++q) {
        const float2 x = to_f2<P>(hf ? w[q + 2] : w[q]);
        cb[2 * q] = x.x;
        cb[2 * q + 1] = x.y;
      }
      cpx<float> i6[6], o6[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) i6[q] = psi.c[q / 3][q % 3];
      clover_block_apply(cb, i6, o6);
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        cpx<float>& a = o.c[q / 3][q % 3];
        a = {fmaf(scl, o6[q].re, a.re), fmaf(scl, o6[q].im, a.im)};
      }
    }
    float m = 0.f;
#pragma unroll
    for (int sp = 0; sp < 2; ++sp)
#pragma unroll
      for (int c = 0; c < 3; ++c) m = fmaxf(m, fmaxf(fabsf(o.c[sp][c].re), fabsf(o.c[sp][c].im)));
    mx[hf][li] = m;
    asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
    m = fmaxf(m, mx[1 - hf][li]);
    if (act) store_half16<P>(fo, g.Vb, blk, r, hf, o, m);
  }
}

// ------------------------------------------------------------------------
// The operator in double-float arithmetic: spinors, links (all 18 reals) and
// clover as (hi, lo) pairs of FP32 values (the FP64 layouts with float4 =
// (re hi, re lo, im hi, im lo) per complex number), computed on the FP32
// units with error-free transformations.  Every output real is a double-float
// running sum; a hop's projection adds pairs by TwoSum, its SU(3)
// product accumulates exact FP32 products and their cross terms, its
// expansion and the -1/2 (a power of two) are exact.  About 12 FP32 operations
// per real multiply-add in place of one FP64 fused multiply-add, on units 64
// times faster on GB300; the result agrees with the FP64 operator to about
// 2^-46 relative.
// ------------------------------------------------------------------------
//
// The arithmetic is written on packed FP32x2 instructions, two independent
// values per instruction: the FP32 lanes are the same, but half the issue slots
// go by, and issue was what the scalar form ran out of (59 % of the slots, the
// FMA pipe at 46 %).  In a hop the two lanes are the two rows of the projected
// spinor (upper spins 0, 1, then lower spins 2, 3), so a link entry serves both;
// in the clover term they are the real and imaginary part of one component.
// The order of the operations on every value is that of the scalar form, and
// so are the results to the last rounding.  32^3 x 64 with an FP32 input: 1.41 ->
// 1.09 ms, and 0.96 ms with the hops' data asked for ahead in registers (below);
// on 8^3 x 16 34 -> 17 us.  The FMA pipe alone needs 0.69 ms.
// the 24 output reals of a site: [spin pair][colour], lanes = the pair's spins
struct SpinAcc {
  acc2 re[2][3], im[2][3];
};
// real (part 0) or imaginary part of component (spin, colour) as a double-float
__device__ __forceinline__ df acc_real(const SpinAcc& a, int sp, int c, int part) {
  const acc2& v = part ? a.im[sp >> 1][c] : a.re[sp >> 1][c];
  return (sp & 1) ? two_sum(v.s.y, v.c.y) : two_sum(v.s.x, v.c.x);
}

// what a double-float hop needs to find its neighbour: the site's in-block
// lexicographic index, its packed local coordinates (8 bits each), its block
// coordinates (16 bits each) and its parity; kept in five registers (a table
// of the eight neighbours would take 24 and make the kernel spill), the
// neighbours are computed per hop
struct DfSite {
  int j, py, pn01, pn23, par;
};

__device__ __forceinline__ DfSite df_site_info(const Geom& g, int blk, int r) {
  int n[4];
  block_coords(g, blk, n);
  DfSite d;
  d.py = __ldg(g.r2y + r);
  d.pn01 = n[0] | (n[1] << 16);
  d.pn23 = n[2] | (n[3] << 16);
  d.j = 0;
  d.par = 0;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    d.j += ycoord(d.py, mu) * g.ystr[mu];
    d.par += ycoord(d.py, mu);
  }
  d.par &= 1;
  return d;
}

// neighbour of hop h (mu = h / 2, forward for even h): block, site and the
// hop's coefficient -1/2 (times the boundary sign where it wraps around)
__device__ __forceinline__ void df_hop_nbr(const Geom& g, int blk, const DfSite& d, int h, int& hb, int& hr,
                                           float& cf) {
  const int mu = h >> 1;
  const int ymu = ycoord(d.py, mu), nmu = ((mu < 2 ? d.pn01 : d.pn23) >> (16 * (mu & 1))) & 0xffff;
  const int b = g.b[mu], ys = g.ystr[mu], nb = g.nb[mu], bs = g.bstr[mu];
  int j = d.j;
  bool wrap = false;
  hb = blk;
  if ((h & 1) == 0) {
    if (ymu + 1 < b) {
      j += ys;
    } else {
      j -= (b - 1) * ys;
      wrap = nmu + 1 == nb;
      hb += wrap ? -(nb - 1) * bs : bs;
    }
  } else {
    if (ymu > 0) {
      j -= ys;
    } else {
      j += (b - 1) * ys;
      wrap = nmu == 0;
      hb += wrap ? (nb - 1) * bs : -bs;
    }
  }
  hr = (d.par ^ 1) * g.Vbh + (j >> 1);  // even block extents: rank among the parity is j >> 1
  cf = wrap ? -0.5f * g.bcf[mu] : -0.5f;
}

__device__ __forceinline__ float2 lane_swap(float2 v) { return make_float2(v.y, v.x); }
__device__ __forceinline__ void lane_swap(acc2& a) {
  a.s = lane_swap(a.s);
  a.c = lane_swap(a.c);
}

// What a hop reads, in registers: the neighbour's spinor record (double-float:
// (re hi, re lo, im hi, im lo) per complex number 3 spin + colour; IN32: two
// complex numbers per chunk, the low parts being 0) and the link's rows (of the
// transposed link for a backward hop).  A hop's data are asked for while the
// hop before it computes, each piece as soon as its registers are free: waiting
// for them was the largest stall (4.9 of 9.2 cycles per issue), also with the
// next hop's lines prefetched to L1.
template <bool IN32>
struct DfHopData {
  static constexpr int NQ = IN32 ? 6 : 12;
  float4 p[NQ], u[9];
  const float4 *fp, *up;
  int sa, sb;
  float cf;  // -1/2, times the boundary sign where the hop wraps around
  __device__ __forceinline__ void locate(const Geom& g, const float4* __restrict__ U, const float4* __restrict__ fin,
                                         int blk, int r, const DfSite& ds, int h) {
    int hb, hr;
    df_hop_nbr(g, blk, ds, h, hb, hr, cf);
    const int mu = h >> 1, bwd = h & 1;
    fp = fin + (long long)hb * NQ * g.Vb + hr;
    up = U + ((long long)((bwd ? hb : blk) * 4 + mu) * 9) * g.Vb + (bwd ? hr : r);
    sa = bwd ? g.Vb : 3 * g.Vb;
    sb = bwd ? 3 * g.Vb : g.Vb;
  }
  __device__ __forceinline__ void load_spinor(int Vb) {
#pragma unroll
    for (int k = 0; k < NQ; ++k) p[k] = __ldg(fp + (long long)k * Vb);
  }
  __device__ __forceinline__ void load_row(int a) {
#pragma unroll
    for (int b = 0; b < 3; ++b) u[3 * a + b] = __ldg(up + a * sa + b * sb);
  }
  // real (part 0) or imaginary part of the components (spin s0, colour a), (spin s1, colour a)
  __device__ __forceinline__ df2 pair(int s0, int s1, int a, int part) const {
    const int c0 = 3 * s0 + a, c1 = 3 * s1 + a;
    if constexpr (IN32) {
      const float4 x = p[c0 >> 1], y = p[c1 >> 1];
      const float vx = (c0 & 1) ? (part ? x.w : x.z) : (part ? x.y : x.x);
      const float vy = (c1 & 1) ? (part ? y.w : y.z) : (part ? y.y : y.x);
      return {make_float2(vx, vy), bc2(0.f)};
    } else {
      const float4 x = p[c0], y = p[c1];
      return part ? df2{make_float2(x.z, y.z), make_float2(x.w, y.w)}
                  : df2{make_float2(x.x, y.x), make_float2(x.y, y.y)};
    }
  }
};

// one hop in direction MU: forward (bwd = 0) or backward, S = -1 for the
// projector 1 - g, +1 for 1 + g; d holds its data and is refilled for the next
// hop (located by `next`) on the way.  In directions 1 and 2 the upper rows 0, 1
// pair with spins 3, 2: there the lower lanes of acc are (3, 2), swapped by the
// caller.  U^+ h = conj(U^T conj(h)): a backward hop conjugates h and the result.
template <int MU, bool IN32, typename Next>
__device__ __forceinline__ void df_hop(DfHopData<IN32>& d, int Vb, int bwd, float S, bool more, Next next,
                                       SpinAcc& acc) {
  constexpr bool kSwap = MU == 1 || MU == 2, kImag = MU == 1 || MU == 3;
  const float cj = bwd ? -1.f : 1.f, cf = d.cf;
  df2 hre[3], him[3];
  {
    // q = S (phase) p_lower: phases (-1, -1), (-i, -i), (-1, +1), (-i, +i) for MU = 0 .. 3
    const float s1 = MU >= 2 ? -S : S;  // lane 1 has the opposite sign in directions 2, 3
    const float2 qr = kImag ? make_float2(S, s1) : make_float2(-S, -s1), qi = make_float2(-S, -s1);
    constexpr int l0 = kSwap ? 3 : 2, l1 = kSwap ? 2 : 3;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const df2 ur = d.pair(0, 1, a, 0), ui = d.pair(0, 1, a, 1);
      const df2 lr = d.pair(l0, l1, a, kImag ? 1 : 0), li = d.pair(l0, l1, a, kImag ? 0 : 1);
      two_sum2(ur.hi, __fmul2_rn(qr, lr.hi), hre[a].hi, hre[a].lo);
      two_sum2(ui.hi, __fmul2_rn(qi, li.hi), him[a].hi, him[a].lo);
      if (!IN32) {
        hre[a].lo = add2(hre[a].lo, add2(ur.lo, __fmul2_rn(qr, lr.lo)));
        him[a].lo = add2(him[a].lo, add2(ui.lo, __fmul2_rn(qi, li.lo)));
      }
      him[a].hi = __fmul2_rn(bc2(cj), him[a].hi);
      him[a].lo = __fmul2_rn(bc2(cj), him[a].lo);
    }
  }
  if (more) {
    next();
    d.load_spinor(Vb);
  }
  const float2 fu = bc2(cf), fui = bc2(cj * cf);
  // the lower rows get conj(phase) S w: factors of their real and imaginary part
  const float fl0 = MU == 0 || MU == 2 ? -S * cf : S * cf, fl1 = MU >= 2 ? -fl0 : fl0;
  const float2 fl = make_float2(fl0, fl1), flj = make_float2(cj * fl0, cj * fl1);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    acc2 wr, wi;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const float4 u = d.u[3 * a + b];
      if (b == 0)
        acc2_set<true>(wr, bc2(u.x), bc2(u.y), hre[b].hi, hre[b].lo);
      else
        acc2_prod<true>(wr, bc2(u.x), bc2(u.y), hre[b].hi, hre[b].lo);
      acc2_prod<true>(wr, bc2(-u.z), bc2(-u.w), him[b].hi, him[b].lo);
      if (b == 0)
        acc2_set<true>(wi, bc2(u.x), bc2(u.y), him[b].hi, him[b].lo);
      else
        acc2_prod<true>(wi, bc2(u.x), bc2(u.y), him[b].hi, him[b].lo);
      acc2_prod<true>(wi, bc2(u.z), bc2(u.w), hre[b].hi, hre[b].lo);
    }
    if (more) d.load_row(a);
    acc2_add(acc.re[0][a], fu, wr);
    acc2_add(acc.im[0][a], fui, wi);
    if (kImag) {  // times i
      acc2_add(acc.re[1][a], neg2(flj), wi);
      acc2_add(acc.im[1][a], fl, wr);
    } else {
      acc2_add(acc.re[1][a], fl, wr);
      acc2_add(acc.im[1][a], flj, wi);
    }
  }
}

template <int MU, int DAG, bool IN32>
__device__ __forceinline__ void df_hop_pair(const Geom& g, const float4* __restrict__ U,
                                            const float4* __restrict__ fin, int blk, int r, const DfSite& ds,
                                            DfHopData<IN32>& d, SpinAcc& acc) {
  constexpr float SF = DAG ? 1.f : -1.f;  // D: (1 - g) psi(x + mu); D^+: (1 + g) psi(x + mu)
  // the two hops of a direction share their code (its four copies fit the
  // instruction cache; eight of the scalar form did not: no_instruction stalls
  // of 8.6 per issue)
#pragma unroll 1
  for (int bwd = 0; bwd < 2; ++bwd) {
    const int h = 2 * MU + bwd;
    df_hop<MU, IN32>(d, g.Vb, bwd, bwd ? -SF : SF, h < 7, [&] { d.locate(g, U, fin, blk, r, ds, h + 1); }, acc);
  }
}

// (D psi)(x) (D^+ with DAG) at site (blk, r) of the field fin (double-float,
// or FP32 with IN32), into the double-float accumulators acc
template <int DAG, bool IN32 = false>
__device__ __forceinline__ void df_site(const Geom& g, const float4* __restrict__ U, const FieldPtr& A,
                                        const float4* __restrict__ fin, int blk, int r, const DfSite& ds,
                                        SpinAcc& acc) {
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < 3; ++c) acc.re[h][c] = acc.im[h][c] = acc2{bc2(0.f), bc2(0.f)};
  DfHopData<IN32> d;
  d.locate(g, U, fin, blk, r, ds, 0);
  d.load_spinor(g.Vb);
#pragma unroll
  for (int a = 0; a < 3; ++a) d.load_row(a);
  df_hop_pair<0, DAG, IN32>(g, U, fin, blk, r, ds, d, acc);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    lane_swap(acc.re[1][c]);
    lane_swap(acc.im[1][c]);
  }
  df_hop_pair<1, DAG, IN32>(g, U, fin, blk, r, ds, d, acc);
  df_hop_pair<2, DAG, IN32>(g, U, fin, blk, r, ds, d, acc);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    lane_swap(acc.re[1][c]);
    lane_swap(acc.im[1][c]);
  }
  df_hop_pair<3, DAG, IN32>(g, U, fin, blk, r, ds, d, acc);
  // clover: two Hermitian 6x6 chiral blocks (6 diagonal reals, then the 15
  // upper off-diagonal elements), record chunk 18 hb + j = reals 36 hb + 2 j, + 1;
  // lanes (re, im)
  const float4* ca = (const float4*)A.data + (long long)blk * 36 * g.Vb + r;
#pragma unroll 1
  for (int hb = 0; hb < 2; ++hb) {
    df2 psi[6], rot[6];  // psi and i psi
    if constexpr (IN32) {
      const float4* p = fin + ((long long)blk * 6 + 3 * hb) * g.Vb + r;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float4 v = __ldg(p + (long long)k * g.Vb);
        psi[2 * k].hi = make_float2(v.x, v.y);
        psi[2 * k + 1].hi = make_float2(v.z, v.w);
      }
    } else {
      const float4* p = fin + ((long long)blk * 12 + 6 * hb) * g.Vb + r;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const float4 v = __ldg(p + (long long)k * g.Vb);
        psi[k] = {make_float2(v.x, v.z), make_float2(v.y, v.w)};
      }
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      rot[k].hi = make_float2(-psi[k].hi.y, psi[k].hi.x);
      if (!IN32) rot[k].lo = make_float2(-psi[k].lo.y, psi[k].lo.x);
    }
    acc2 t[6];
#pragma unroll
    for (int i = 0; i < 6; i += 2) {  // diagonal reals i, i + 1
      const float4 dv = __ldg(ca + (long long)(18 * hb + i / 2) * g.Vb);
      acc2_set<!IN32>(t[i], bc2(dv.x), bc2(dv.y), psi[i].hi, psi[i].lo);
      acc2_set<!IN32>(t[i + 1], bc2(dv.z), bc2(dv.w), psi[i + 1].hi, psi[i + 1].lo);
    }
    int kk = 3;
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
      for (int j = i + 1; j < 6; ++j) {
        const float4 a = __ldg(ca + (long long)(18 * hb + kk) * g.Vb);
        ++kk;
        acc2_prod<!IN32>(t[i], bc2(a.x), bc2(a.y), psi[j].hi, psi[j].lo);
        acc2_prod<!IN32>(t[i], bc2(a.z), bc2(a.w), rot[j].hi, rot[j].lo);
        acc2_prod<!IN32>(t[j], bc2(a.x), bc2(a.y), psi[i].hi, psi[i].lo);
        acc2_prod<!IN32>(t[j], bc2(-a.z), bc2(-a.w), rot[i].hi, rot[i].lo);
      }
    // into spins 2 hb (components 0 .. 2) and 2 hb + 1 (3 .. 5)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const acc2 zr = {make_float2(t[c].s.x, t[c + 3].s.x), make_float2(t[c].c.x, t[c + 3].c.x)};
      const acc2 zi = {make_float2(t[c].s.y, t[c + 3].s.y), make_float2(t[c].c.y, t[c + 3].c.y)};
      if (hb == 0) {
        acc2_add(acc.re[0][c], bc2(1.f), zr);
        acc2_add(acc.im[0][c], bc2(1.f), zi);
      } else {
        acc2_add(acc.re[1][c], bc2(1.f), zr);
        acc2_add(acc.im[1][c], bc2(1.f), zi);
      }
    }
  }
}

//
// IN32: the input is an FP32 field (an FP32-exact operand, e.g. a preconditioner
// output), read at half the bytes; the arithmetic is the same
template <int DAG, bool IN32>
__global__ void __launch_bounds__(256, 1) dirac_df_kernel(Geom g, const float4* __restrict__ U, FieldPtr A,
                                                          FieldPtr in, FieldPtr out, int nrhs,
                                                          const int* __restrict__ mask) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  const int blk = (int)(s / g.Vb), r = (int)(s - (long long)blk * g.Vb);
  const DfSite ds = df_site_info(g, blk, r);
#pragma unroll 1
  for (int k = 0; k < nrhs; ++k) {
    if (mask && !mask[k]) continue;
    const float4* fin = (const float4*)in.data + (size_t)k * g.V * (IN32 ? 6 : 12);
    float4* fout = (float4*)out.data + (size_t)k * g.V * 12;
    SpinAcc acc;
    df_site<DAG, IN32>(g, U, A, fin, blk, r, ds, acc);
    float4* o = fout + (long long)blk * 12 * g.Vb + r;
#pragma unroll
    for (int q = 0; q < 12; ++q) {
      const df re = acc_real(acc, q / 3, q % 3, 0), im = acc_real(acc, q / 3, q % 3, 1);
      o[(long long)q * g.Vb] = make_float4(re.hi, re.lo, im.hi, im.lo);
    }
  }
}

// deterministic block sum of a double: warp shuffles, then warps in order
__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double t = 0;
  if (threadIdx.x == 0)
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += sh[k];
  return t;
}

// r = b - D x with x given as its double-float split: D x in double-float
// arithmetic (as dirac_df_kernel), the difference and |r|^2 in FP64;
// partial[blockIdx.x] = sum |r|^2 over the CTA, blockIdx.y a right-hand side
// of a batch (fields V sites apart, partial sums ps doubles apart)
__global__ void __launch_bounds__(kDfThreads, 2) residual_df_kernel(Geom g, const float4* __restrict__ U, FieldPtr A,
                                                             FieldPtr b, FieldPtr x, FieldPtr r_out, double* partial,
                                                             long long ps, const int* __restrict__ mask) {
  __shared__ double sh[32];
  if (mask && !mask[blockIdx.y]) return;
  const long long o = (long long)blockIdx.y * g.V * 12;  // double2 / float4 elements per field
  const double2* bb = (const double2*)b.data + o;
  const float4* xx = (const float4*)x.data + o;
  double2* rr = (double2*)r_out.data + o;
  partial += blockIdx.y * ps;
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double nrm = 0;
  if (s < g.V) {
    const int blk = (int)(s / g.Vb), r = (int)(s - (long long)blk * g.Vb);
    SpinAcc acc;
    df_site<0>(g, U, A, xx, blk, r, df_site_info(g, blk, r), acc);
    const long long e = (long long)blk * 12 * g.Vb + r;
#pragma unroll
    for (int q = 0; q < 12; ++q) {
      const double2 bv = __ldg(bb + e + (long long)q * g.Vb);
      const double2 v = make_double2(bv.x - df_to_f64(acc_real(acc, q / 3, q % 3, 0)),
                                     bv.y - df_to_f64(acc_real(acc, q / 3, q % 3, 1)));
      rr[e + (long long)q * g.Vb] = v;
      nrm = fma(v.x, v.x, fma(v.y, v.y, nrm));
    }
  }
  const double t = block_sum(nrm, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

// r = b - D x (FP64), partial[blockIdx.x] = sum |r|^2 over the CTA; blockIdx.y
// selects a right-hand side of a batch (fields V sites apart, partial sums ps
// doubles apart), skipped when masked out
__global__ void __launch_bounds__(kF64Threads) residual64_kernel(Geom g, const void* __restrict__ U, FieldPtr A, FieldPtr b,
                                                         FieldPtr x, FieldPtr r_out, double* partial, long long ps,
                                                         const int* __restrict__ mask) {
  __shared__ double sh[32];
  if (mask && !mask[blockIdx.y]) return;
  {
    const long long o = (long long)blockIdx.y * g.V * 12;  // double2 elements per FP64 field
    b.data = (double2*)b.data + o;
    x.data = (double2*)x.data + o;
    r_out.data = (double2*)r_out.data + o;
    partial += blockIdx.y * ps;
  }
  long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double nrm = 0;
  if (s < g.V) {
    int blk = (int)(s / g.Vb), r = (int)(s - (long long)blk * g.Vb);
    Spinor<double> o = dirac_site<P64, 0, double>(g, U, A, x, blk, r);
    Spinor<double> bb = load_spinor<P64, double>(b, g.Vb, blk, r);
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        o.c[sp][a] = bb.c[sp][a] - o.c[sp][a];
        nrm += o.c[sp][a].re * o.c[sp][a].re + o.c[sp][a].im * o.c[sp][a].im;
      }
    store_spinor<P64, double>(r_out, g.Vb, blk, r, o);
  }
  double t = block_sum(nrm, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

// ------------------------------------------------------------------------
// The FP64 operator with a site's work split over the four warps of a CTA of 32
// sites, for lattices whose sites alone do not keep the FP64 units busy: a warp's
// FP64 operation holds a quarter of an SM for 64 cycles, so one thread's 1150 of
// them last 36 us however few warps there are.  Warp w computes the two hops of
// direction w; the partial sums meet in shared memory, and warp w finishes spin w
// (its three rows of the chiral clover block).  RES: out = b - D x and the sum of
// its squares per CTA instead of out = D x.
// ------------------------------------------------------------------------
static constexpr int kSplitSites = 32;

// rows R0 .. R0 + 2 of a packed Hermitian 6x6 block (chunks of record a) times in
template <int R0>
__device__ __forceinline__ void clover_rows(const double2* __restrict__ a, int Vb, const cpx<double>* in,
                                            cpx<double>* out) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int i = R0 + c;
    const double2 dv = __ldg(a + (long long)(i >> 1) * Vb);
    out[c] = ((i & 1) ? dv.y : dv.x) * in[i];
  }
  int k = 3;
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = i + 1; j < 6; ++j, ++k) {
      const bool row_i = i >= R0 && i < R0 + 3, row_j = j >= R0 && j < R0 + 3;
      if (!row_i && !row_j) continue;
      const double2 v = __ldg(a + (long long)k * Vb);
      const cpx<double> e = {v.x, v.y};
      if (row_i) out[i - R0] = cmadd(e, in[j], out[i - R0]);
      if (row_j) out[j - R0] = cjmadd(e, in[i], out[j - R0]);
    }
}

template <int DAG, bool RES>
__global__ void __launch_bounds__(4 * kSplitSites, 4) dirac_split_kernel(Geom g, const void* __restrict__ U, FieldPtr A,
                                                                         FieldPtr in, FieldPtr out, FieldPtr b,
                                                                         const int* __restrict__ mask, int out_df,
                                                                         double* partial, long long ps) {
  __shared__ double part[4][24][kSplitSites];
  __shared__ double sh[4];
  if (mask && !mask[blockIdx.y]) return;
  const long long fo = (long long)blockIdx.y * g.V * 12;  // 16-byte chunks per field
  in.data = (double2*)in.data + fo;
  out.data = (double2*)out.data + fo;
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const long long s0 = (long long)blockIdx.x * kSplitSites + l;
  const bool on = s0 < g.V;
  const long long s = on ? s0 : 0;
  const int blk = (int)(s / g.Vb), r = (int)(s - (long long)blk * g.Vb);
  {
    int n[4], y[4];
    block_coords(g, blk, n);
    const int packed = __ldg(g.r2y + r);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) y[mu] = ycoord(packed, mu);
    Spinor<double> acc;
    zero(acc);
    switch (w) {
      case 0: hop_pair<0, P64, DAG, double>(g, U, in, blk, r, y, n, acc); break;
      case 1: hop_pair<1, P64, DAG, double>(g, U, in, blk, r, y, n, acc); break;
      case 2: hop_pair<2, P64, DAG, double>(g, U, in, blk, r, y, n, acc); break;
      default: hop_pair<3, P64, DAG, double>(g, U, in, blk, r, y, n, acc); break;
    }
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        part[w][6 * sp + 2 * c][l] = acc.c[sp][c].re;
        part[w][6 * sp + 2 * c + 1][l] = acc.c[sp][c].im;
      }
  }
  // spin w: its clover rows while the other warps arrive
  const int hb = w >> 1;
  cpx<double> psi[6], o[3];
  const double2* f = (const double2*)in.data + ((long long)blk * 12 + 6 * hb) * g.Vb + r;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double2 v = __ldg(f + (long long)k * g.Vb);
    psi[k] = {v.x, v.y};
  }
  const double2* a = (const double2*)A.data + ((long long)blk * 36 + 18 * hb) * g.Vb + r;
  if (w & 1)
    clover_rows<3>(a, g.Vb, psi, o);
  else
    clover_rows<0>(a, g.Vb, psi, o);
  __syncthreads();
  double nrm = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int e = 6 * w + 2 * c;
    cpx<double> h = {part[0][e][l], part[0][e + 1][l]};
#pragma unroll
    for (int q = 1; q < 4; ++q) h = h + cpx<double>{part[q][e][l], part[q][e + 1][l]};
    h = h + o[c];
    const long long at = ((long long)blk * 12 + 3 * w + c) * g.Vb + r;
    if (RES) {
      const double2 bv = __ldg((const double2*)b.data + fo + at);
      h = cpx<double>{bv.x, bv.y} - h;
      if (on) nrm += h.re * h.re + h.im * h.im;
    }
    if (!on) continue;
    if (out_df) {
      const df x = df_from_f64(h.re), y = df_from_f64(h.im);
      ((float4*)out.data)[at] = make_float4(x.hi, x.lo, y.hi, y.lo);
    } else {
      ((double2*)out.data)[at] = make_double2(h.re, h.im);
    }
  }
  if (RES) {
    const double t = block_sum(nrm, sh);
    if (threadIdx.x == 0) partial[blockIdx.y * ps + blockIdx.x] = t;
  }
}

// The split form where its warps fill the SM quarters better (and no CTA size was set
// for the operator, which applies to the other form): FP64 operations that
// one quarter runs through, per warp 1150 (one thread per site, right-hand sides in
// turn) or 306 (split, right-hand sides side by side), times the warps it gets.
// One right-hand side, one thread per site / split: 256 sites 41 / 15 us, 8192 43 / 25,
// 16384 43 / 45, 32768 80 / 74, 41472 107 / 94, 65536 147 / 146, 131072 271 / 275.
bool use_split(const qcd_ctx* c, int nrhs) {
  if (nrhs > 65535) return false;  // (a grid dimension)
  const long long q = 4LL * c->sms;
  const long long whole = (c->V + 32 * q - 1) / (32 * q) * nrhs, split = (c->V * nrhs + 8 * q - 1) / (8 * q);
  return split * 306 < whole * 1150;
}

static double bytes_per_site(int prec) {
  if (prec == P64) return 2 * 24 * 8 + 4 * 18 * 8 + 72 * 8;
  if (prec == P32) return 2 * 24 * 4 + 4 * 12 * 4 + 72 * 4;
  return 2 * (24 * 2 + 4) + 4 * 12 * 2 + (72 * 2 + 4);
}

int dirac_apply(qcd_ctx* c, const Rec& in, const Rec& out, int dagger, cudaStream_t s, int nrhs, const int* mask) {
  const int prec = in.prec;
  if (prec == PDF || (prec == P32 && out.prec == PDF)) {
    // the double-float operator: double-float in and out, or an FP32 input
    // (FP32-exact operand) with a double-float result
    if (out.prec != PDF || in.nreal != 24 || out.nreal != 24 || nrhs < 1) return QCD_ERR_ARG;
    QCD_TRY(ensure_gauge(c, PDF, s));
    QCD_TRY(ensure_clover(c, PDF, s));
    const bool in32 = prec == P32;
    const int threads = c->dirac_threads[PDF];
    const unsigned grid = (unsigned)((c->V + threads - 1) / threads);
    // algorithmic bytes: links and clover as pairs (576 + 576), spinor out 192, in 192 or 96
    ProfScope ps(c, QCD_KERNEL_DIRAC, s, (1344.0 + (in32 ? 96.0 : 192.0)) * (double)c->V * nrhs,
                 1824.0 * (double)c->V * nrhs);
    const float4* U = (const float4*)c->U[PDF];
    const FieldPtr A = c->A[PDF].ptr();
    if (in32) {
      if (dagger)
        dirac_df_kernel<1, true><<<grid, threads, 0, s>>>(c->g, U, A, in.ptr(), out.ptr(), nrhs, mask);
      else
        dirac_df_kernel<0, true><<<grid, threads, 0, s>>>(c->g, U, A, in.ptr(), out.ptr(), nrhs, mask);
    } else if (dagger) {
      dirac_df_kernel<1, false><<<grid, threads, 0, s>>>(c->g, U, A, in.ptr(), out.ptr(), nrhs, mask);
    } else {
      dirac_df_kernel<0, false><<<grid, threads, 0, s>>>(c->g, U, A, in.ptr(), out.ptr(), nrhs, mask);
    }
    QCD_LAUNCHED();
    return QCD_OK;
  }
  // FP64 in and double-float out: the FP64 operator with its result split
  const int out_df = prec == P64 && out.prec == PDF;
  if ((out.prec != prec && !out_df) || in.nreal != 24 || out.nreal != 24 || nrhs < 1) return QCD_ERR_ARG;
  QCD_TRY(ensure_gauge(c, prec, s));
  QCD_TRY(ensure_clover(c, prec, s));
  const int threads = c->dirac_threads[prec];
  const unsigned grid = (unsigned)((c->V + threads - 1) / threads);
  const void* U = c->U[prec];
  FieldPtr A = c->A[prec].ptr();
  // algorithmic bytes: links and clover once, spinors per right-hand side
  const double spin = prec == P64 ? 384 : (prec == P32 ? 192 : 104);
  const double bytes = ((bytes_per_site(prec) - spin) + spin * nrhs) * (double)c->V;
  ProfScope ps(c, QCD_KERNEL_DIRAC, s, bytes, 1824.0 * (double)c->V * nrhs);
#define LAUNCH(PP, BS)                                                                                 \
  if (dagger)                                                                                          \
    dirac_kernel<PP, 1, BS><<<grid, threads, 0, s>>>(c->g, U, A, in.ptr(), out.ptr(), nrhs, mask, out_df); \
  else                                                                                                     \
    dirac_kernel<PP, 0, BS><<<grid, threads, 0, s>>>(c->g, U, A, in.ptr(), out.ptr(), nrhs, mask, out_df);
  // 16-bit storage (FP16, BF16) is issue-bound, so it gets the fixed-shape
  // instantiations, and the two-threads-per-site form when the context asks for it
  const int bs = block_shape_id(c->g);
  if ((prec == P16 || prec == PB16) && c->dirac_tps[prec] == 2) {
    const unsigned g2 = (unsigned)((c->V + kPairSites - 1) / kPairSites);
#define LAUNCH2(PP, DD, BB) \
  dirac_pair_kernel<PP, DD, BB><<<g2, 2 * kPairSites, 0, s>>>(c->g, U, A, in.ptr(), out.ptr(), nrhs, mask)
#define LAUNCH2_BS(PP, DD) \
  if (bs == 1) LAUNCH2(PP, DD, 1); else if (bs == 2) LAUNCH2(PP, DD, 2); else LAUNCH2(PP, DD, 0);
    if (prec == P16) {
      if (dagger) { LAUNCH2_BS(P16, 1) } else { LAUNCH2_BS(P16, 0) }
    } else {
      if (dagger) { LAUNCH2_BS(PB16, 1) } else { LAUNCH2_BS(PB16, 0) }
    }
#undef LAUNCH2_BS
#undef LAUNCH2
    QCD_LAUNCHED();
    return QCD_OK;
  }
  if (prec == P64 && !c->f64_threads_set && use_split(c, nrhs)) {
    const dim3 g2((unsigned)((c->V + kSplitSites - 1) / kSplitSites), nrhs);
    if (dagger)
      dirac_split_kernel<1, false><<<g2, 4 * kSplitSites, 0, s>>>(c->g, U, A, in.ptr(), out.ptr(), FieldPtr{}, mask,
                                                                  out_df, nullptr, 0);
    else
      dirac_split_kernel<0, false><<<g2, 4 * kSplitSites, 0, s>>>(c->g, U, A, in.ptr(), out.ptr(), FieldPtr{}, mask,
                                                                  out_df, nullptr, 0);
    QCD_LAUNCHED();
    return QCD_OK;
  }
  switch (prec) {
    case P64: LAUNCH(P64, 0); break;
    case P32: LAUNCH(P32, 0); break;
    case P16:
      if (bs == 1) {
        LAUNCH(P16, 1);
      } else if (bs == 2) {
        LAUNCH(P16, 2);
      } else {
        LAUNCH(P16, 0);
      }
      break;
    case PB16:
      if (bs == 1) {
        LAUNCH(PB16, 1);
      } else if (bs == 2) {
        LAUNCH(PB16, 2);
      } else {
        LAUNCH(PB16, 0);
      }
      break;
    default: return QCD_ERR_ARG;
  }
#undef LAUNCH
  QCD_LAUNCHED();
  return QCD_OK;
}

int residual64(qcd_ctx* c, double* part, const Rec& b, const Rec& x, const Rec& r, double* d_norm2, cudaStream_t s,
               const Batch& B) {
  NvtxRange nv("residual64");
  if (b.prec != P64 || x.prec != P64 || r.prec != P64) return QCD_ERR_ARG;
  QCD_TRY(ensure_gauge(c, P64, s));
  QCD_TRY(ensure_clover(c, P64, s));
  const bool split = use_split(c, B.n);
  const int sites = split ? kSplitSites : kF64Threads;  // per CTA
  const unsigned grid = (unsigned)((c->V + sites - 1) / sites);
  {
    ProfScope ps(c, QCD_KERNEL_RESIDUAL, s, (bytes_per_site(P64) + 192) * (double)c->V * B.n,
                 1848.0 * (double)c->V * B.n);
    if (split)
      dirac_split_kernel<0, true><<<dim3(grid, B.n), 4 * kSplitSites, 0, s>>>(
          c->g, c->U[P64], c->A[P64].ptr(), x.ptr(), r.ptr(), b.ptr(), B.mask, 0, part + kPartHead, B.ps);
    else
      residual64_kernel<<<dim3(grid, B.n), kF64Threads, 0, s>>>(c->g, c->U[P64], c->A[P64].ptr(), b.ptr(), x.ptr(), r.ptr(),
                                                       part + kPartHead, B.ps, B.mask);
    QCD_LAUNCHED();
  }
  return reduce_partials(part + kPartHead, (int)grid, 1, 1, d_norm2, s, B);
}

int residual_df(qcd_ctx* c, double* part, const Rec& b, const Rec& x, const Rec& r, const Rec& tmp, double* d_norm2,
                cudaStream_t s, const Batch& B, bool presplit) {
  NvtxRange nv("residual_df");
  if (b.prec != P64 || x.prec != P64 || r.prec != P64 || tmp.prec != PDF || tmp.bytes < (size_t)c->V * 192 * B.n)
    return QCD_ERR_ARG;
  QCD_TRY(ensure_gauge(c, PDF, s));
  QCD_TRY(ensure_clover(c, PDF, s));
  if (!presplit) QCD_TRY(blas_df_split(c, (const double*)x.data, (float*)tmp.data, s, B));
  const unsigned grid = (unsigned)((c->V + kDfThreads - 1) / kDfThreads);
  {
    ProfScope ps(c, QCD_KERNEL_RESIDUAL, s, (bytes_per_site(P64) + 192) * (double)c->V * B.n,
                 1848.0 * (double)c->V * B.n);
    residual_df_kernel<<<dim3(grid, B.n), kDfThreads, 0, s>>>(c->g, (const float4*)c->U[PDF], c->A[PDF].ptr(), b.ptr(),
                                                        tmp.ptr(), r.ptr(), part + kPartHead, B.ps, B.mask);
    QCD_LAUNCHED();
  }
  return reduce_partials(part + kPartHead, (int)grid, 1, 1, d_norm2, s, B);
}

// ------------------------------------------------------------------------
// Even/odd split of D over the whole lattice (the global parity of a site is
// its block-local parity, block extents being even).  For the sites of
// parity `par` (r = par * Vbh + rr):
//   PRE = 1:  out = c1 * M x + c2 * H y
//   PRE = 0:  out = M (c1 x + c2 H y)
// with H y = -1/2 sum of the hops from the opposite parity (D's hopping term,
// its adjoint's with DAG), M = Ahat on these sites (A_ee on even, A_oo^-1 on
// odd) if USE_M, else 1.  x and out are read / written on parity par only, y
// on the other parity only, so out may be y.  c2 = 0 skips the hops, c1 = 0
// the load of x.  FP64 throughout.
// ------------------------------------------------------------------------
template <int DAG, int PRE, int USE_M>
__global__ void __launch_bounds__(kF64Threads, 8) eo_kernel(Geom g, const void* __restrict__ U, FieldPtr Ahat, FieldPtr x,
                                                 FieldPtr y, FieldPtr out, int par, double c1, double c2) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= g.V / 2) return;
  const int blk = (int)(t / g.Vbh), r = (int)(t - (long long)blk * g.Vbh) + par * g.Vbh;
  Spinor<double> h;
  zero(h);
  if (c2 != 0.0) {
    int n[4], yc[4];
    block_coords(g, blk, n);
    const int packed = __ldg(g.r2y + r);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) yc[mu] = ycoord(packed, mu);
    hop_pair<0, P64, DAG, double>(g, U, y, blk, r, yc, n, h);
    hop_pair<1, P64, DAG, double>(g, U, y, blk, r, yc, n, h);
    hop_pair<2, P64, DAG, double>(g, U, y, blk, r, yc, n, h);
    hop_pair<3, P64, DAG, double>(g, U, y, blk, r, yc, n, h);
  }
  Spinor<double> v;
  zero(v);
  if (c1 != 0.0) v = load_spinor<P64, double>(x, g.Vb, blk, r);
  double cm[72];
  if (USE_M) load_record<P64, 72, double>(Ahat, g.Vb, blk, r, cm);
  if (PRE && USE_M) v = clover_apply(cm, v);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b)
      v.c[a][b] = {fma(c2, h.c[a][b].re, c1 * v.c[a][b].re), fma(c2, h.c[a][b].im, c1 * v.c[a][b].im)};
  if (!PRE && USE_M) v = clover_apply(cm, v);
  store_spinor<P64, double>(out, g.Vb, blk, r, v);
}

int eo_apply(qcd_ctx* c, const Rec& x, const Rec& y, const Rec& out, int par, int dagger, int pre, int use_m,
             double c1, double c2, cudaStream_t s) {
  if (x.prec != P64 || y.prec != P64 || out.prec != P64 || (par != 0 && par != 1)) return QCD_ERR_ARG;
  QCD_TRY(ensure_gauge(c, P64, s));
  QCD_TRY(ensure_clover(c, P64, s));
  const unsigned grid = (unsigned)((c->V / 2 + kF64Threads - 1) / kF64Threads);
  // algorithmic bytes: per site of parity par, 8 neighbour spinors and 8 links
  // (hops), x and the clover record (if used) and the result
  const double sites = (double)c->V / 2;
  const double bytes = sites * ((c2 != 0.0 ? 8 * 192 + 8 * 144 : 0) + (c1 != 0.0 ? 192 : 0) + (use_m ? 576 : 0) + 192);
  ProfScope ps(c, QCD_KERNEL_DIRAC, s, bytes, sites * ((c2 != 0.0 ? 1320.0 : 0.0) + (use_m ? 504.0 : 0.0)));
  const void* U = c->U[P64];
  const FieldPtr A = c->Ahat[P64].ptr();
#define EO(D, P, M) eo_kernel<D, P, M><<<grid, kF64Threads, 0, s>>>(c->g, U, A, x.ptr(), y.ptr(), out.ptr(), par, c1, c2)
  if (dagger) {
    if (pre) { if (use_m) EO(1, 1, 1); else EO(1, 1, 0); }
    else { if (use_m) EO(1, 0, 1); else EO(1, 0, 0); }
  } else {
    if (pre) { if (use_m) EO(0, 1, 1); else EO(0, 1, 0); }
    else { if (use_m) EO(0, 0, 1); else EO(0, 0, 0); }
  }
#undef EO
  QCD_LAUNCHED();
  return QCD_OK;
}

// out_e = Dhat x_e = A_ee x_e - H_eo A_oo^-1 H_oe x_e (dagger: Dhat^+, the same
// with the adjoint's hops); tmp receives A_oo^-1 H_oe x_e on the odd sites.
// Only the even sites of x and out are read / written.
int schur_apply(qcd_ctx* c, const Rec& x, const Rec& tmp, const Rec& out, int dagger, cudaStream_t s) {
  QCD_TRY(eo_apply(c, x, x, tmp, 1, dagger, 0, 1, 0.0, 1.0, s));
  return eo_apply(c, x, tmp, out, 0, dagger, 1, 1, 1.0, -1.0, s);
}

}  // namespace qcd
