// Layout transforms (canonical lexicographic <-> domain-major) and the clover build.
//
// Canonical layouts (the library's public formats):
//   spinor: [t][z][y][x][spin 4][colour 3][re, im]   (FP64 or FP32)
//   gauge:  [t][z][y][x][mu 4][row 3][col 3][re, im] (FP64), forward links U_mu(x).
// The antiperiodic time boundary of the fermion field is folded into the internal copy
// of the links: U_t(x) at t = L_t - 1 is stored negated.  Every plaquette that crosses
// the boundary holds two such links, so the clover term is unaffected; it is built here
// from the canonical (unsigned) links.
#include "dd_kernels.hpp"

namespace dd {

__device__ inline void site_global(const Geom& g, const Site& st, int x[4]) {
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) x[mu] = st.n[mu] * g.b[mu] + st.l[mu];
}

__device__ inline long long canon_index(const Geom& g, const int x[4]) {
  return x[0] + (long long)g.L[0] * (x[1] + (long long)g.L[1] * (x[2] + (long long)g.L[2] * x[3]));
}

// One site of a canonical field, 24 reals in a row, in 16-byte accesses where the field's
// address allows them (VEC): 24 scalar accesses a site, each of a warp in 32 lines, bound
// the layout passes (whole calls, FP32 24^3x48: unpacking 91 -> 35 us, packing 40 -> 31 us).
template <bool VEC> __device__ __forceinline__ void canon_load(const double* q, double v[24]) {
#pragma unroll
  for (int k = 0; k < 24; k += 2) {
    if constexpr (VEC) {
      const double2 w = *reinterpret_cast<const double2*>(q + k);
      v[k] = w.x; v[k + 1] = w.y;
    } else {
      v[k] = q[k]; v[k + 1] = q[k + 1];
    }
  }
}
template <bool VEC> __device__ __forceinline__ void canon_load(const float* q, float v[24]) {
#pragma unroll
  for (int k = 0; k < 24; k += 4) {
    if constexpr (VEC) {
      const float4 w = *reinterpret_cast<const float4*>(q + k);
      v[k] = w.x; v[k + 1] = w.y; v[k + 2] = w.z; v[k + 3] = w.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[k + e] = q[k + e];
    }
  }
}
template <bool VEC> __device__ __forceinline__ void canon_store(double* q, const double v[24]) {
#pragma unroll
  for (int k = 0; k < 24; k += 2) {
    if constexpr (VEC) {
      *reinterpret_cast<double2*>(q + k) = make_double2(v[k], v[k + 1]);
    } else {
      q[k] = v[k]; q[k + 1] = v[k + 1];
    }
  }
}
template <bool VEC> __device__ __forceinline__ void canon_store(float* q, const float v[24]) {
#pragma unroll
  for (int k = 0; k < 24; k += 4) {
    if constexpr (VEC) {
      *reinterpret_cast<float4*>(q + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) q[k + e] = v[k + e];
    }
  }
}

template <typename C, typename T, bool VEC>
__global__ void pack_spinor_kernel(Geom g, const C* canon, SpinorPtr<T> out) {
  long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  Site st = decode(g, s);
  int x[4];
  site_global(g, st, x);
  C q[24];
  canon_load<VEC>(canon + 24 * canon_index(g, x), q);
  Spinor<typename Arith<T>::type> v;
#pragma unroll
  for (int k = 0; k < 12; ++k) v.c[k / 3][k % 3] = mk<typename Arith<T>::type>(q[2 * k], q[2 * k + 1]);
  out.store(g, s, v);
}

template <typename T, typename C, bool VEC>
__global__ void unpack_spinor_kernel(Geom g, SpinorPtr<T> in, C* canon) {
  long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  Site st = decode(g, s);
  int x[4];
  site_global(g, st, x);
  Spinor<typename Arith<T>::type> v;
  in.load(g, s, v);
  C q[24];
#pragma unroll
  for (int k = 0; k < 12; ++k) { q[2 * k] = (C)v.c[k / 3][k % 3].re; q[2 * k + 1] = (C)v.c[k / 3][k % 3].im; }
  canon_store<VEC>(canon + 24 * canon_index(g, x), q);
}

static inline unsigned nblk(long long n, int t) { return (unsigned)((n + t - 1) / t); }

template <typename C, bool VEC>
static void pack_dispatch(const Geom& g, const C* canon, FieldView out, cudaStream_t st) {
  unsigned nb = nblk(g.V, 256);
  if (out.prec == P64) pack_spinor_kernel<C, double, VEC><<<nb, 256, 0, st>>>(g, canon, SpinorPtr<double>{(double2*)out.data});
  else if (out.prec == P32) pack_spinor_kernel<C, float, VEC><<<nb, 256, 0, st>>>(g, canon, SpinorPtr<float>{(float4*)out.data});
  else pack_spinor_kernel<C, __half, VEC><<<nb, 256, 0, st>>>(g, canon, SpinorPtr<__half>{(uint4*)out.data, out.norm});
}

static bool vec_aligned(const void* p) { return (uintptr_t)p % 16 == 0; }

void launch_pack_spinor(const Geom& g, const void* canon, int canon_prec, FieldView out, cudaStream_t st) {
  const bool vec = vec_aligned(canon);
  if (canon_prec == P64)
    vec ? pack_dispatch<double, true>(g, (const double*)canon, out, st) : pack_dispatch<double, false>(g, (const double*)canon, out, st);
  else
    vec ? pack_dispatch<float, true>(g, (const float*)canon, out, st) : pack_dispatch<float, false>(g, (const float*)canon, out, st);
}

template <typename C, bool VEC>
static void unpack_dispatch(const Geom& g, FieldView in, C* canon, cudaStream_t st) {
  unsigned nb = nblk(g.V, 256);
  if (in.prec == P64) unpack_spinor_kernel<double, C, VEC><<<nb, 256, 0, st>>>(g, SpinorPtr<double>{(double2*)in.data}, canon);
  else if (in.prec == P32) unpack_spinor_kernel<float, C, VEC><<<nb, 256, 0, st>>>(g, SpinorPtr<float>{(float4*)in.data}, canon);
  else unpack_spinor_kernel<__half, C, VEC><<<nb, 256, 0, st>>>(g, SpinorPtr<__half>{(uint4*)in.data, in.norm}, canon);
}

void launch_unpack_spinor(const Geom& g, FieldView in, void* canon, int canon_prec, cudaStream_t st) {
  const bool vec = vec_aligned(canon);
  if (canon_prec == P64)
    vec ? unpack_dispatch<double, true>(g, in, (double*)canon, st) : unpack_dispatch<double, false>(g, in, (double*)canon, st);
  else
    vec ? unpack_dispatch<float, true>(g, in, (float*)canon, st) : unpack_dispatch<float, false>(g, in, (float*)canon, st);
}

__global__ void pack_gauge_kernel(Geom g, const double* canon, int anti, double2* u64, float2* u32, uint4* u16) {
  long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  Site st = decode(g, s);
  int x[4];
  site_global(g, st, x);
  const double* q = canon + 72 * canon_index(g, x);
  long long d = st.d, r = s & (g.Vd - 1);
  for (int mu = 0; mu < 4; ++mu) {
    double sg = (anti && mu == 3 && x[3] == g.L[3] - 1) ? -1.0 : 1.0;
    uint32_t w[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const int j = 3 * link_row(k) + link_col(k);
      double re = sg * q[18 * mu + 2 * j], im = sg * q[18 * mu + 2 * j + 1];
      const long long a = ((d * 4 + mu) * 9) << g.lgVd;
      u64[a + ((long long)j << g.lgVd) + r] = make_double2(re, im);
      u32[a + ((long long)k << g.lgVd) + r] = make_float2((float)re, (float)im);
      w[k] = f2h((float)re, (float)im);
    }
    uint4* b = u16 + ((d * 10) << g.lgVd);
    b[((2 * mu) << g.lgVd) + r] = make_uint4(w[3], w[4], w[5], w[0]);
    b[((2 * mu + 1) << g.lgVd) + r] = make_uint4(w[6], w[7], w[8], w[0]);
    reinterpret_cast<uint2*>(b + (8 << g.lgVd))[(mu << g.lgVd) + r] = make_uint2(w[1], w[2]);
  }
}

void launch_pack_gauge(const Geom& g, const double* canon, int anti, double2* u64, float2* u32, uint4* u16,
                       cudaStream_t st) {
  pack_gauge_kernel<<<nblk(g.V, 128), 128, 0, st>>>(g, canon, anti, u64, u32, u16);
}

// ------------------------------------------------------------------ clover build (FP64)
// Bound by GB300's FP64 rate (two lanes per SM), so the count of FP64 instructions is what
// matters: ten 3x3 products per plane instead of the twelve of four separate leaves, and
// Hermitian 6x6 blocks inverted by symmetric sweeps over their 36 real numbers.
// Set-up of a 24^3x48 configuration with its first FP64 operator and preconditioner
// application: 27.6 ms with four leaves and pivoted inverses (19.2k FP64 instructions per
// site), 19.5 ms with those as fused multiply-adds, 10.7 ms in this form; two or three blocks
// per SM measure the same.
struct M3 { cx<double> e[3][3]; };

struct CanonLinks {
  const double* U;
  __device__ __forceinline__ void get(long long site, int mu, M3& m) const {
    const double2* q = reinterpret_cast<const double2*>(U + 72 * site + 18 * mu);
#pragma unroll
    for (int j = 0; j < 9; ++j) { const double2 v = q[j]; m.e[j / 3][j % 3] = mk(v.x, v.y); }
  }
};

// c (+)= s a b with a or b replaced by its adjoint; s = -1 when NEG.
template <bool ADAG, bool BDAG, bool ACC, bool NEG>
__device__ __forceinline__ void m3_mul(M3& c, const M3& a, const M3& b) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cx<double> v = ACC ? c.e[i][j] : mk(0.0, 0.0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        cx<double> x = ADAG ? a.e[k][i] : a.e[i][k], y = BDAG ? b.e[j][k] : b.e[k][j];
        if (ADAG) x.im = -x.im;
        if (BDAG) y.im = -y.im;
        if (!ACC && k == 0) v = NEG ? cmul(mk(-x.re, -x.im), y) : cmul(x, y);
        else v = NEG ? cnmac(v, x, y) : cmac(v, x, y);
      }
      c.e[i][j] = v;
    }
}

// F = Q - Q^dag of one plane, Q the sum of the four plaquette leaves at x oriented m -> n.
// Replacing two of the leaves by minus their adjoints leaves F unchanged and lets the outer
// links be factored out:
//   l1 - l4^dag = U_m(x)   [ U_n(x+m) U_m(x+n)^dag U_n(x)^dag - (U_m(x-n) U_n(x+m-n))^dag U_n(x-n) ]
//   l2 - l3^dag = [ U_n(x) (U_n(x-m) U_m(x-m+n))^dag - U_n(x-n)^dag U_m(x-m-n)^dag U_n(x-m-n) ] U_m(x-m)
// fm, fn, bm, bn: site index steps to x + m, x + n, x - m, x - n.  F is anti-Hermitian: its nine
// reals go to f[0..2] (imaginary diagonal) and f[3..8] (entries 10, 20, 21), `ld` apart.
__device__ __forceinline__ void plane_field(const CanonLinks& L, long long x, int m, int n, long long fm, long long fn,
                                            long long bm, long long bn, double* f, int ld) {
  M3 a, b, p, t, X;
  L.get(x + fm, n, a);
  L.get(x + fn, m, b);
  m3_mul<false, true, false, false>(p, a, b);
  L.get(x, n, a);
  m3_mul<false, true, false, false>(t, p, a);
  L.get(x + bn, m, a);
  L.get(x + fm + bn, n, b);
  m3_mul<false, false, false, false>(p, a, b);
  L.get(x + bn, n, a);
  m3_mul<true, false, true, true>(t, p, a);
  L.get(x, m, b);
  m3_mul<false, false, false, false>(X, b, t);
  L.get(x + bm, n, a);
  L.get(x + bm + fn, m, b);
  m3_mul<false, false, false, false>(p, a, b);
  L.get(x, n, a);
  m3_mul<false, true, false, false>(t, a, p);
  L.get(x + bm + bn, m, a);
  L.get(x + bm + bn, n, b);
  m3_mul<true, false, false, false>(p, a, b);
  L.get(x + bn, n, a);
  m3_mul<true, false, true, true>(t, a, p);
  L.get(x + bm, m, b);
  m3_mul<false, false, true, false>(X, t, b);
#pragma unroll
  for (int i = 0; i < 3; ++i) f[i * ld] = 2.0 * X.e[i][i].im;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int i = k == 0 ? 1 : 2, j = k == 2 ? 1 : 0;
    f[(3 + 2 * k) * ld] = X.e[i][j].re - X.e[j][i].re;
    f[(4 + 2 * k) * ld] = X.e[i][j].im + X.e[j][i].im;
  }
}

// Gauss-Jordan inverse of a 6x6 complex matrix with partial pivoting.  Returns the
// smallest pivot magnitude relative to the largest entry.
__device__ double inv6(cx<double> a[6][6], cx<double> inv[6][6]) {
  double amax = 0;
  for (int i = 0; i < 6; ++i)
    for (int j = 0; j < 6; ++j) {
      inv[i][j] = mk(i == j ? 1.0 : 0.0, 0.0);
      amax = fmax(amax, hypot(a[i][j].re, a[i][j].im));
    }
  double minpiv = 1e300;
  for (int c = 0; c < 6; ++c) {
    int pr = c;
    double best = -1;
    for (int r = c; r < 6; ++r) {
      double v = hypot(a[r][c].re, a[r][c].im);
      if (v > best) { best = v; pr = r; }
    }
    minpiv = fmin(minpiv, best);
    if (best == 0.0) return 0.0;
    if (pr != c)
      for (int j = 0; j < 6; ++j) {
        cx<double> t = a[c][j]; a[c][j] = a[pr][j]; a[pr][j] = t;
        t = inv[c][j]; inv[c][j] = inv[pr][j]; inv[pr][j] = t;
      }
    cx<double> p = a[c][c];
    double pn = p.re * p.re + p.im * p.im;
    cx<double> pi = mk(p.re / pn, -p.im / pn);
    for (int j = 0; j < 6; ++j) { a[c][j] = cmul(a[c][j], pi); inv[c][j] = cmul(inv[c][j], pi); }
    for (int r = 0; r < 6; ++r) {
      if (r == c) continue;
      cx<double> f = a[r][c];
      for (int j = 0; j < 6; ++j) {
        a[r][j] = cnmac(a[r][j], f, a[c][j]);
        inv[r][j] = cnmac(inv[r][j], f, inv[c][j]);
      }
    }
  }
  return amax > 0 ? minpiv / amax : 0.0;
}

// Pack a Hermitian 6x6 block (its lower triangle and real diagonal) into 36 reals.
__device__ inline void pack_block(cx<double> a[6][6], double* out) {
  for (int i = 0; i < 6; ++i) out[i] = a[i][i].re;
  for (int i = 1; i < 6; ++i)
    for (int j = 0; j < i; ++j) {
      // Hermitian part of the pair (i, j), (j, i)
      out[6 + 2 * tri(i, j)] = 0.5 * (a[i][j].re + a[j][i].re);
      out[6 + 2 * tri(i, j) + 1] = 0.5 * (a[i][j].im - a[j][i].im);
    }
}

// Inverse of a packed Hermitian block in place by Gauss-Jordan with partial pivoting: the
// general path, for blocks whose natural pivots are too small.
__device__ __noinline__ double inv6_packed(double* m) {
  cx<double> a[6][6], b[6][6];
  for (int i = 0; i < 6; ++i) {
    a[i][i] = mk(m[i], 0.0);
    for (int j = 0; j < i; ++j) {
      const double re = m[6 + 2 * tri(i, j)], im = m[6 + 2 * tri(i, j) + 1];
      a[i][j] = mk(re, im);
      a[j][i] = mk(re, -im);
    }
  }
  const double rel = inv6(a, b);
  if (rel > 0.0) pack_block(b, m);
  return rel;
}

// Symmetric sweep of a packed Hermitian block with its natural (diagonal) pivots:
//   d = a_kk, a_ij -= a_ik conj(a_jk) / d, a_ik /= d, a_kk = -1 / d,
// which leaves -A^{-1} after all six (FULL), or only the elimination below the diagonal, for
// the pivots.  Pivots are real, so a sweep costs ten complex and five real updates.  Returns
// false when a pivot is less than half of an entry it eliminates (threshold pivoting would
// exchange rows there) or below 1e-9 of the largest entry; m is then unusable.
template <bool FULL>
__device__ __forceinline__ bool sweep6(double m[36]) {
  double amax2 = 0.0, minp = 1e300;
#pragma unroll
  for (int i = 0; i < 6; ++i) amax2 = fmax(amax2, m[i] * m[i]);
#pragma unroll
  for (int k = 0; k < 15; ++k) amax2 = fmax(amax2, fma(m[6 + 2 * k], m[6 + 2 * k], m[7 + 2 * k] * m[7 + 2 * k]));
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double d = m[k], d2 = d * d;
    minp = fmin(minp, d2);
    cx<double> b[6];   // column k
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      if (i == k || (!FULL && i < k)) continue;
      const int t = 6 + 2 * (i > k ? tri(i, k) : tri(k, i));
      b[i] = mk(m[t], i > k ? m[t + 1] : -m[t + 1]);
      if (i > k) ok = ok && 4.0 * d2 >= fma(b[i].re, b[i].re, b[i].im * b[i].im);
    }
    const double r = 1.0 / d;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      if (i == k || (!FULL && i < k)) continue;
      const cx<double> s = mk(b[i].re * r, b[i].im * r);
      m[i] = fma(-s.re, b[i].re, fma(-s.im, b[i].im, m[i]));
#pragma unroll
      for (int j = 0; j < i; ++j) {
        if (j == k || (!FULL && j < k)) continue;
        const int t = 6 + 2 * tri(i, j);   // a_ij -= s_i conj(b_j)
        m[t] = fma(-s.im, b[j].im, fma(-s.re, b[j].re, m[t]));
        m[t + 1] = fma(s.re, b[j].im, fma(-s.im, b[j].re, m[t + 1]));
      }
      if (FULL) {
        const int t = 6 + 2 * (i > k ? tri(i, k) : tri(k, i));
        m[t] = s.re;
        m[t + 1] = i > k ? s.im : -s.im;
      }
    }
    if (FULL) m[k] = -r;
  }
  if (FULL) {
#pragma unroll
    for (int k = 0; k < 36; ++k) m[k] = -m[k];
  }
  return ok && minp > 0.0 && minp >= 1e-18 * amax2;
}

constexpr int CLOVER_THREADS = 128;
__global__ void __launch_bounds__(CLOVER_THREADS, 2)
    build_clover_kernel(Geom g, const double* canon, double kappa, double csw, double2* c64, float4* c32, uint4* c16,
                        float4* s32, uint4* s16, int* status) {
  extern __shared__ double fs[];   // [6 planes][9][thread]
  const long long s = blockIdx.x * (long long)CLOVER_THREADS + threadIdx.x;
  if (s >= g.V) return;
  const Site st = decode(g, s);
  int x[4];
  site_global(g, st, x);
  const long long at = canon_index(g, x);
  const CanonLinks L{canon};
  double* const f = fs + threadIdx.x;
  // Planes (0,1) (0,2) (0,3) (1,2) (1,3) (2,3), one at a time: one copy of the code.
  long long up[4], dn[4], stride = 1;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    up[mu] = x[mu] + 1 < g.L[mu] ? stride : -(g.L[mu] - 1) * stride;
    dn[mu] = x[mu] > 0 ? -stride : (g.L[mu] - 1) * stride;
    stride *= g.L[mu];
  }
#pragma unroll 1
  for (int k = 0; k < 6; ++k) {
    const int m = k < 3 ? 0 : k < 5 ? 1 : 2, n = k < 3 ? k + 1 : k < 5 ? k - 1 : 3;
    const long long fm = m == 0 ? up[0] : m == 1 ? up[1] : up[2], bm = m == 0 ? dn[0] : m == 1 ? dn[1] : dn[2];
    const long long fn = n == 1 ? up[1] : n == 2 ? up[2] : up[3], bn = n == 1 ? dn[1] : n == 2 ? dn[2] : dn[3];
    plane_field(L, at, m, n, fm, fn, bm, bn, f + 9 * k * CLOVER_THREADS, CLOVER_THREADS);
  }
  // Chiral blocks: D_cl = -(c_sw/16) sum_{mu<nu} gamma_mu gamma_nu (x) F_mu,nu.  With
  // E = (F_yz, -F_xz, F_xy), G = (F_xt, F_yt, F_zt) and X_l = i (E_l -/+ G_l) for the
  // upper / lower chirality, each block is -(c_sw/16) [[X3, X1 - i X2], [X1 + i X2, -X3]].
  const double c = -csw / 16.0, diag = 1.0 / (2.0 * kappa);
  int singular = 0;
#pragma unroll 1
  for (int blk = 0; blk < 2; ++blk) {
    const double sg = blk == 0 ? -1.0 : 1.0;
    // v_l = c (E_l + sg G_l), anti-Hermitian: v[l][0..2] the imaginary diagonal, then 10, 20, 21
    double v[3][9];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const double* q = f + e * CLOVER_THREADS;
      v[0][e] = c * fma(sg, q[9 * 2 * CLOVER_THREADS], q[9 * 3 * CLOVER_THREADS]);
      v[1][e] = c * fma(sg, q[9 * 4 * CLOVER_THREADS], -q[9 * 1 * CLOVER_THREADS]);
      v[2][e] = c * fma(sg, q[9 * 5 * CLOVER_THREADS], q[0]);
    }
    // entry (a, b) of v_l as a complex number
    auto at_l = [&](int l, int a, int b) -> cx<double> {
      if (a == b) return mk(0.0, v[l][a]);
      const int hi = a > b ? a : b, lo = a > b ? b : a, k = hi == 1 ? 0 : lo == 0 ? 1 : 2;
      const double re = v[l][3 + 2 * k], im = v[l][4 + 2 * k];
      return a > b ? mk(re, im) : mk(-re, im);
    };
    double m[36];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      m[a] = diag - v[2][a];       // c X3 = i v3, on the diagonal i (i v) = -v
      m[3 + a] = diag + v[2][a];
#pragma unroll
      for (int b = 0; b < a; ++b) {
        const cx<double> z = ti(at_l(2, a, b));
        m[6 + 2 * tri(a, b)] = z.re;
        m[6 + 2 * tri(a, b) + 1] = z.im;
        m[6 + 2 * tri(3 + a, 3 + b)] = -z.re;
        m[6 + 2 * tri(3 + a, 3 + b) + 1] = -z.im;
      }
#pragma unroll
      for (int b = 0; b < 3; ++b) {   // c (X1 + i X2) = i v1 - v2
        const cx<double> z = ti(at_l(0, a, b)) - at_l(1, a, b);
        m[6 + 2 * tri(3 + a, b)] = z.re;
        m[6 + 2 * tri(3 + a, b) + 1] = z.im;
      }
    }
#pragma unroll
    for (int u = 0; u < 18; ++u) c64[unit_addr(g, s, 36, 18 * blk + u)] = make_double2(m[2 * u], m[2 * u + 1]);
    float w[36];
#pragma unroll
    for (int u = 0; u < 36; ++u) w[u] = (float)m[u];
#pragma unroll
    for (int u = 0; u < 9; ++u)
      c32[unit_addr(g, s, 18, 9 * blk + u)] = make_float4(w[4 * u], w[4 * u + 1], w[4 * u + 2], w[4 * u + 3]);
    // FP16 clover: words 18 blk .. 18 blk + 17 of the site's 36, as 8-byte halves of its units
    uint2* h16 = reinterpret_cast<uint2*>(c16);
#pragma unroll
    for (int u = 0; u < 9; ++u) {
      const int k = 9 * blk + u;
      h16[2 * unit_addr(g, s, 9, k >> 1) + (k & 1)] =
          make_uint2(f2h(w[4 * u], w[4 * u + 1]), f2h(w[4 * u + 2], w[4 * u + 3]));
    }
    // Schwarz matrix: the block on even sites, its inverse on odd ones (a warp holds sites of one
    // parity).  The pivots are wanted on both, to report singular blocks.
    const bool ok = st.p ? sweep6<true>(m) : sweep6<false>(m);
    if (!ok) {   // the general path, from the copy just written
      double b[36];
      for (int u = 0; u < 18; ++u) {
        const double2 q = c64[unit_addr(g, s, 36, 18 * blk + u)];
        b[2 * u] = q.x;
        b[2 * u + 1] = q.y;
      }
      if (!(inv6_packed(b) >= 1e-12)) singular = 1;
#pragma unroll
      for (int k = 0; k < 36; ++k) m[k] = b[k];
    }
    if (st.p) {
#pragma unroll
      for (int u = 0; u < 36; ++u) w[u] = (float)m[u];
    }
#pragma unroll
    for (int u = 0; u < 9; ++u)
      s32[unit_addr(g, s, 18, 9 * blk + u)] = make_float4(w[4 * u], w[4 * u + 1], w[4 * u + 2], w[4 * u + 3]);
    // FP16 form: units 4 blk .. 4 blk + 3 hold words 0..15 of the block, unit 8 the last two of
    // both, so each block is four 16-byte units and one 8-byte half unit
    uint32_t h[18];
#pragma unroll
    for (int k = 0; k < 18; ++k) h[k] = f2h(w[2 * k], w[2 * k + 1]);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      s16[unit_addr(g, s, 9, 4 * blk + u)] = make_uint4(h[4 * u], h[4 * u + 1], h[4 * u + 2], h[4 * u + 3]);
    reinterpret_cast<uint2*>(s16)[2 * unit_addr(g, s, 9, 8) + blk] = make_uint2(h[16], h[17]);
  }
  if (singular) atomicAdd(status, 1);
}

void launch_build_clover(const Geom& g, const double* canon, double kappa, double csw, double2* c64, float4* c32,
                         uint4* c16, float4* s32, uint4* s16, int* status, cudaStream_t st) {
  const size_t smem = sizeof(double) * 54 * CLOVER_THREADS;
  static SmemAllowed allowed;
  allow_smem(allowed, device_info(), (const void*)build_clover_kernel, smem);
  build_clover_kernel<<<nblk(g.V, CLOVER_THREADS), CLOVER_THREADS, smem, st>>>(g, canon, kappa, csw, c64, c32, c16, s32,
                                                                             s16, status);
}

}  // namespace dd
