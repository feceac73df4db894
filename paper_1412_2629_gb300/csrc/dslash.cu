// Full-lattice Wilson-clover operator A = 1/(2 kappa) - 1/2 D_w + D_cl (Eq. 1-3).
//
// One thread per site in the domain-major layout: consecutive threads are consecutive
// sites of one parity of one domain, so the site's own spinor, links and clover are read
// with fully coalesced 16-byte (8- or 4-byte for links) loads, and most neighbours are
// adjacent sites of the other parity (read through L1/L2).  Hops that leave the domain
// go to the neighbouring domain's block; the antiperiodic time boundary is already in
// the links.  The diagonal 1/(2 kappa) is folded into the stored clover.
// Bytes per site (algorithmic, each field read once): 4 links + clover + in + out =
// 192 reals; FP32 768 B, FP64 1536 B, FP16 384 B + 8 B of spinor norms.  The stored FP16 links
// hold one entry of each twice for the Schwarz kernel's loads, so FP16 moves 400 + 8 B; with three
// vector loads a link instead of nine words, and fused products, it is faster all the same
// (24^3x48 150 -> 107 us).
#include <type_traits>

#include "dd_kernels.hpp"

namespace dd {

template <int MU, typename T>
__device__ inline void hop_pair(const Geom& g, const Site& st, long long s, const SpinorPtr<T>& in,
                                const LinkPtr<T>& U, Spinor<typename Arith<T>::type>& acc) {
  typedef typename Arith<T>::type R;
  Spinor<R> psi;
  Half<R> h, uh;
  Link<R> L;
  // forward: (1 - gamma_mu) U_mu(x) psi(x + mu)
  long long sf = neighbour(g, st, MU, +1);
  in.load(g, sf, psi);
  project<MU, -1>(psi, h);
  U.load(g, s, MU, L);
  su3_mul(L, h, uh);
  accum_recon<MU, -1>(acc, uh);
  // backward: (1 + gamma_mu) U_mu(x - mu)^dag psi(x - mu)
  long long sb = neighbour(g, st, MU, -1);
  in.load(g, sb, psi);
  project<MU, +1>(psi, h);
  U.load(g, sb, MU, L);
  su3_dag_mul(L, h, uh);
  accum_recon<MU, +1>(acc, uh);
}

template <typename T>
__global__ void __launch_bounds__(256) apply_A_kernel(Geom g, LinkPtr<T> U, CloverPtr<T> C, SpinorPtr<T> in,
                                                       SpinorPtr<T> out, SpinorPtr<T> f, int residual,
                                                       const double2* in_norm2) {
  typedef typename Arith<T>::type R;
  long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  if (in_norm2 && in_norm2->x == 0.0) {   // f - A 0
    Spinor<R> fv;
    f.load(g, s, fv);
    out.store(g, s, fv);
    return;
  }
  Site st = decode(g, s);
  Spinor<R> hop;
  zero(hop);
  hop_pair<0, T>(g, st, s, in, U, hop);
  hop_pair<1, T>(g, st, s, in, U, hop);
  hop_pair<2, T>(g, st, s, in, U, hop);
  hop_pair<3, T>(g, st, s, in, U, hop);
  Spinor<R> x, y;
  in.load(g, s, x);
  R m[72];
  C.load(g, s, m);
  clover_mul(m, x, y);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) y.c[a][b] = y.c[a][b] - R(0.5) * hop.c[a][b];
  if (residual) {
    Spinor<R> fv;
    f.load(g, s, fv);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) y.c[a][b] = fv.c[a][b] - y.c[a][b];
  }
  out.store(g, s, y);
}

// ------------------------------------------------------------------ FP32, shape known at compile time
// The same one-thread-per-site operator for FP32 fields with the domain shape as
// compile-time constants (SHAPE 1: 8x4x4x4, 2: 4x4x4x4): the site decoding and every
// neighbour and unit address then fold into shifts and immediate offsets, which takes the
// integer work off the issue slots that the loads need.  Two CTAs of 256 per SM: the
// compiler may then use 128 registers, and spends them on keeping more of the neighbour
// and link loads in flight (measured 20 % faster than the same code at 88 registers).
template <int SHAPE>
__global__ void __launch_bounds__(256, 2) apply_A_shape_kernel(Geom g0, LinkPtr<float> U, CloverPtr<float> C,
                                                            SpinorPtr<float> in, SpinorPtr<float> out,
                                                            SpinorPtr<float> f, int residual) {
  const Geom g = fixed_shape<SHAPE>(g0);
  long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  Site st = decode(g, s);
  Spinor<float> hop;
  zero(hop);
  hop_pair<0, float>(g, st, s, in, U, hop);
  hop_pair<1, float>(g, st, s, in, U, hop);
  hop_pair<2, float>(g, st, s, in, U, hop);
  hop_pair<3, float>(g, st, s, in, U, hop);
  Spinor<float> x, y;
  in.load(g, s, x);
  float m[72];
  C.load(g, s, m);
  clover_mul(m, x, y);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) y.c[a][b] = y.c[a][b] - 0.5f * hop.c[a][b];
  if (residual) {
    Spinor<float> fv;
    f.load(g, s, fv);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) y.c[a][b] = fv.c[a][b] - y.c[a][b];
  }
  out.store(g, s, y);
}

// Threads per block: `most`, halved until the grid has two blocks per SM (or a block is one
// warp), so that a small lattice uses the whole chip.  FP64 blocks start at 64 threads: two
// FP64 lanes per SM are busy with two warps, and on 8^4 the 16 blocks of 256 threads left
// nine SMs in ten idle (107 -> 49 us cold; FP32 8.3 -> 7.7 us).  24^3x48 gains from the shorter
// tail too: 1.42 -> 1.37 ms.
static int block_threads(long long V, int most) {
  const int sms = device_info().sms;
  while (most > 32 && V / most < 2 * sms) most >>= 1;
  return most;
}

void launch_apply_A(const Geom& g, GaugeView U, CloverView C, FieldView in, FieldView out, const FieldView* f,
                    cudaStream_t st, const double2* in_norm2) {
  const int nt = block_threads(g.V, in.prec == P64 ? 64 : 256);
  const unsigned nb = (unsigned)((g.V + nt - 1) / nt);
  int res = f != nullptr;
  if (in.prec == P32 && domain_shape_id(g) != 0) {
    const LinkPtr<float> L{(const float2*)U.links};
    const CloverPtr<float> Cp{(const float4*)C.m};
    const SpinorPtr<float> vi{(float4*)in.data}, vo{(float4*)out.data}, fi{res ? (float4*)f->data : nullptr};
    if (domain_shape_id(g) == 1) apply_A_shape_kernel<1><<<nb, nt, 0, st>>>(g, L, Cp, vi, vo, fi, res);
    else apply_A_shape_kernel<2><<<nb, nt, 0, st>>>(g, L, Cp, vi, vo, fi, res);
    return;
  }
  if (in.prec == P64) {
    SpinorPtr<double> fi{res ? (double2*)f->data : nullptr};
    apply_A_kernel<double><<<nb, nt, 0, st>>>(g, LinkPtr<double>{(const double2*)U.links},
                                               CloverPtr<double>{(const double2*)C.m},
                                               SpinorPtr<double>{(double2*)in.data},
                                               SpinorPtr<double>{(double2*)out.data}, fi, res, res ? in_norm2 : nullptr);
  } else if (in.prec == P32) {
    SpinorPtr<float> fi{res ? (float4*)f->data : nullptr};
    apply_A_kernel<float><<<nb, nt, 0, st>>>(g, LinkPtr<float>{(const float2*)U.links},
                                              CloverPtr<float>{(const float4*)C.m},
                                              SpinorPtr<float>{(float4*)in.data}, SpinorPtr<float>{(float4*)out.data},
                                              fi, res, nullptr);
  } else {
    SpinorPtr<__half> fi{res ? (uint4*)f->data : nullptr, res ? f->norm : nullptr};
    apply_A_kernel<__half><<<nb, nt, 0, st>>>(g, LinkPtr<__half>{(const uint4*)U.links},
                                               CloverPtr<__half>{(const uint4*)C.m},
                                               SpinorPtr<__half>{(uint4*)in.data, in.norm},
                                               SpinorPtr<__half>{(uint4*)out.data, out.norm}, fi, res, nullptr);
  }
}

// ------------------------------------------------------------------ canonical fields
// The operator on the caller's own fields ([t][z][y][x][spin][colour]), without the two layout
// passes: a thread keeps its place in the domain-major order (links and clover are read as
// above) and finds its site and the eight neighbours in the canonical field by their index
// steps.  The strided 16-byte spinor accesses cost L1 wavefronts, which hide behind FP64
// arithmetic and cost less than the passes in FP32: FP64 24^3x48 1514 -> 1357 us (1350 us on
// internal fields), FP32 32^3x64 635 -> 413 us (270 internal), FP32 8^4 27 -> 15.6 us.
template <typename T> struct CanonField;
template <> struct CanonField<float> {
  const float4* p;
  __device__ __forceinline__ void load(long long x, Spinor<float>& v) const {
#pragma unroll
    for (int u = 0; u < 6; ++u) {
      const float4 q = p[6 * x + u];
      const int k = 2 * u;
      v.c[k / 3][k % 3] = mk(q.x, q.y);
      v.c[(k + 1) / 3][(k + 1) % 3] = mk(q.z, q.w);
    }
  }
  __device__ __forceinline__ void store(long long x, const Spinor<float>& v) const {
#pragma unroll
    for (int u = 0; u < 6; ++u) {
      const int k = 2 * u;
      const_cast<float4*>(p)[6 * x + u] = make_float4(v.c[k / 3][k % 3].re, v.c[k / 3][k % 3].im,
                                                      v.c[(k + 1) / 3][(k + 1) % 3].re, v.c[(k + 1) / 3][(k + 1) % 3].im);
    }
  }
};
template <> struct CanonField<double> {
  const double2* p;
  __device__ __forceinline__ void load(long long x, Spinor<double>& v) const {
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const double2 q = p[12 * x + k];
      v.c[k / 3][k % 3] = mk(q.x, q.y);
    }
  }
  __device__ __forceinline__ void store(long long x, const Spinor<double>& v) const {
#pragma unroll
    for (int k = 0; k < 12; ++k)
      const_cast<double2*>(p)[12 * x + k] = make_double2(v.c[k / 3][k % 3].re, v.c[k / 3][k % 3].im);
  }
};

template <int MU, typename T>
__device__ __forceinline__ void hop_pair_canon(const Geom& g, const Site& st, long long s, long long x,
                                               long long stride, const CanonField<T>& in, const LinkPtr<T>& U,
                                               Spinor<T>& acc) {
  Spinor<T> psi;
  Half<T> h, uh;
  Link<T> L;
  const int c = st.n[MU] * g.b[MU] + st.l[MU];
  in.load(c + 1 < g.L[MU] ? x + stride : x - (g.L[MU] - 1) * stride, psi);
  project<MU, -1>(psi, h);
  U.load(g, s, MU, L);
  su3_mul(L, h, uh);
  accum_recon<MU, -1>(acc, uh);
  in.load(c > 0 ? x - stride : x + (g.L[MU] - 1) * stride, psi);
  project<MU, +1>(psi, h);
  U.load(g, neighbour(g, st, MU, -1), MU, L);
  su3_dag_mul(L, h, uh);
  accum_recon<MU, +1>(acc, uh);
}

template <typename T, int SHAPE>
__global__ void __launch_bounds__(256) apply_A_canon_kernel(Geom g0, LinkPtr<T> U, CloverPtr<T> C, CanonField<T> in,
                                                            CanonField<T> out) {
  const Geom g = fixed_shape<SHAPE>(g0);
  const long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  const Site st = decode(g, s);
  long long x = 0, stride[4], n = 1;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    stride[mu] = n;
    x += (st.n[mu] * g.b[mu] + st.l[mu]) * n;
    n *= g.L[mu];
  }
  Spinor<T> hop;
  zero(hop);
  hop_pair_canon<0, T>(g, st, s, x, stride[0], in, U, hop);
  hop_pair_canon<1, T>(g, st, s, x, stride[1], in, U, hop);
  hop_pair_canon<2, T>(g, st, s, x, stride[2], in, U, hop);
  hop_pair_canon<3, T>(g, st, s, x, stride[3], in, U, hop);
  Spinor<T> v, y;
  in.load(x, v);
  T m[72];
  C.load(g, s, m);
  clover_mul(m, v, y);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) y.c[a][b] = y.c[a][b] - T(0.5) * hop.c[a][b];
  out.store(x, y);
}

void launch_apply_A_canonical(const Geom& g, GaugeView U, CloverView C, const void* in, void* out, int prec,
                              cudaStream_t st) {
  const int nt = block_threads(g.V, prec == P64 ? 64 : 256);
  const unsigned nb = (unsigned)((g.V + nt - 1) / nt);
  if (prec == P64) {
    apply_A_canon_kernel<double, 0><<<nb, nt, 0, st>>>(g, LinkPtr<double>{(const double2*)U.links},
                                                       CloverPtr<double>{(const double2*)C.m},
                                                       CanonField<double>{(const double2*)in},
                                                       CanonField<double>{(const double2*)out});
    return;
  }
  const LinkPtr<float> L{(const float2*)U.links};
  const CloverPtr<float> Cp{(const float4*)C.m};
  const CanonField<float> a{(const float4*)in}, b{(const float4*)out};
  switch (domain_shape_id(g)) {
    case 1: apply_A_canon_kernel<float, 1><<<nb, nt, 0, st>>>(g, L, Cp, a, b); break;
    case 2: apply_A_canon_kernel<float, 2><<<nb, nt, 0, st>>>(g, L, Cp, a, b); break;
    default: apply_A_canon_kernel<float, 0><<<nb, nt, 0, st>>>(g, L, Cp, a, b); break;
  }
}

}  // namespace dd

namespace dd {

// ------------------------------------------------------------------ several right-hand sides
__device__ inline void shift_norm(SpinorPtr<float>&, long long) {}
__device__ inline void shift_norm(SpinorPtr<__half>& p, long long d) { p.norm += d; }

// Thread per site, NR right-hand sides per thread: every link and the clover block are
// loaded once and applied to NR spinors, so per right-hand side the operator moves
// (4 links + clover) / NR + in + out bytes instead of all 192 reals.
template <int MU, typename T, int NR>
__device__ inline void hop_pair_multi(const Geom& g, const Site& st, long long s, const SpinorPtr<T>* in,
                                      const LinkPtr<T>& U, Spinor<typename Arith<T>::type>* acc) {
  typedef typename Arith<T>::type R;
  Spinor<R> psi;
  Half<R> h, uh;
  Link<R> L;
  long long sf = neighbour(g, st, MU, +1);
  U.load(g, s, MU, L);
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    in[r].load(g, sf, psi);
    project<MU, -1>(psi, h);
    su3_mul(L, h, uh);
    accum_recon<MU, -1>(acc[r], uh);
  }
  long long sb = neighbour(g, st, MU, -1);
  U.load(g, sb, MU, L);
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    in[r].load(g, sb, psi);
    project<MU, +1>(psi, h);
    su3_dag_mul(L, h, uh);
    accum_recon<MU, +1>(acc[r], uh);
  }
}

// The fields r0 .. r0 + NR - 1 at site s; in_list / out_list: FP32 fields anywhere in memory.
template <typename T, int NR>
__device__ __forceinline__ void apply_A_multi_site(const Geom& g, long long s, int r0, const LinkPtr<T>& U,
                                                   const CloverPtr<T>& C, const SpinorPtr<T>& in0,
                                                   const SpinorPtr<T>& out0, long long unit_stride,
                                                   long long norm_stride, const float4* const* in_list,
                                                   float4* const* out_list) {
  typedef typename Arith<T>::type R;
  SpinorPtr<T> in[NR], out[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int rr = r0 + r;
    in[r] = in0;
    out[r] = out0;
    in[r].p += rr * unit_stride;
    out[r].p += rr * unit_stride;
    shift_norm(in[r], rr * norm_stride);
    shift_norm(out[r], rr * norm_stride);
    if constexpr (std::is_same<T, float>::value) {
      if (in_list) {
        in[r].p = const_cast<float4*>(in_list[rr]);
        out[r].p = out_list[rr];
      }
    }
  }
  Site st = decode(g, s);
  Spinor<R> acc[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) zero(acc[r]);
  hop_pair_multi<0, T, NR>(g, st, s, in, U, acc);
  hop_pair_multi<1, T, NR>(g, st, s, in, U, acc);
  hop_pair_multi<2, T, NR>(g, st, s, in, U, acc);
  hop_pair_multi<3, T, NR>(g, st, s, in, U, acc);
  R m[72];
  C.load(g, s, m);
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    Spinor<R> x, y;
    in[r].load(g, s, x);
    clover_mul(m, x, y);
#pragma unroll
    for (int a2 = 0; a2 < 4; ++a2)
#pragma unroll
      for (int b2 = 0; b2 < 3; ++b2) y.c[a2][b2] = y.c[a2][b2] - R(0.5) * acc[r].c[a2][b2];
    out[r].store(g, s, y);
  }
}

// Blocks that work on the same 128 sites with other pairs of fields are neighbours in launch order,
// so the links and clover blocks come from HBM once and from L2 afterwards.  Bound by the latency
// of the neighbours' loads (L1 and L2): three blocks per SM at 168 registers, with a few spilled,
// beat two at 255 and four at 128 (six fields of 24^3x48: 355, 430 and 377 us; with 4x4x4x8
// domains, whose shape is not compiled in, three and two blocks: 434 and 541 us), and three
// fields per thread gain nothing over two.  The domain shape as compile-time constants and the
// launch order took six fields from 541 to 349 us (169 us of traffic).
//
// A field left over from the pairs runs alone, in blocks behind all pairs.  Between the pairs of
// the same sites its code and theirs, both fully unrolled, evict each other from the instruction
// caches (8.0 warps waiting for instructions per issue, against 0.7): three FP16 fields of 24^3x48
// 352 us (4x4x4x8 domains 435), behind the pairs 189 (226); FP32 226 (400) and 216 (293) us; 13
// FP32 fields of 16^3x32, which gain from the links they share, 149 and 155 us.
//
// Both forms below number blocks and fields alike.  Where the compiler knows the shape, the
// field number as an expression of each branch is 2 % faster (six FP32 fields 344 for 351 us);
// where it does not, one computed before the branch spills less (429 for 451 us).
constexpr int MULTI_THREADS = 128;
template <typename T, int SHAPE>
__global__ void __launch_bounds__(MULTI_THREADS, 3)
    apply_A_multi_kernel(Geom g0, LinkPtr<T> U, CloverPtr<T> C, SpinorPtr<T> in, SpinorPtr<T> out, long long unit_stride,
                         long long norm_stride, int nrhs, unsigned site_blocks, const float4* const* in_list,
                         float4* const* out_list) {
  const Geom g = fixed_shape<SHAPE>(g0);
  const unsigned pairs = (unsigned)nrhs >> 1, paired = site_blocks * pairs;   // pairs of fields, their blocks
  if constexpr (SHAPE != 0) {
    const bool alone = blockIdx.x >= paired;
    const unsigned b = alone ? blockIdx.x - paired : blockIdx.x / pairs;
    const long long s = b * (long long)MULTI_THREADS + threadIdx.x;
    if (s >= g.V) return;
    if (alone)
      apply_A_multi_site<T, 1>(g, s, 2 * pairs, U, C, in, out, unit_stride, norm_stride, in_list, out_list);
    else
      apply_A_multi_site<T, 2>(g, s, 2 * (blockIdx.x % pairs), U, C, in, out, unit_stride, norm_stride, in_list, out_list);
  } else {
    const bool pair = blockIdx.x < paired;
    const unsigned per = pair ? pairs : 1u, x = pair ? blockIdx.x : blockIdx.x - paired;
    const long long s = (x / per) * (long long)MULTI_THREADS + threadIdx.x;
    if (s >= g.V) return;
    const int r0 = pair ? (x % per) * 2 : nrhs - 1;
    if (r0 + 1 < nrhs)
      apply_A_multi_site<T, 2>(g, s, r0, U, C, in, out, unit_stride, norm_stride, in_list, out_list);
    else
      apply_A_multi_site<T, 1>(g, s, r0, U, C, in, out, unit_stride, norm_stride, in_list, out_list);
  }
}

template <typename T>
static void multi_launch(const Geom& g, LinkPtr<T> U, CloverPtr<T> C, SpinorPtr<T> in, SpinorPtr<T> out,
                         long long unit_stride, long long norm_stride, int nrhs, const float4* const* in_list,
                         float4* const* out_list, cudaStream_t st) {
  const unsigned nb = (unsigned)((g.V + MULTI_THREADS - 1) / MULTI_THREADS);
  auto launch = [&](auto kernel) {
    kernel<<<nb * (nrhs / 2 + nrhs % 2), MULTI_THREADS, 0, st>>>(g, U, C, in, out, unit_stride, norm_stride, nrhs, nb,
                                                                 in_list, out_list);
  };
  switch (domain_shape_id(g)) {
    case 1: launch(apply_A_multi_kernel<T, 1>); break;
    case 2: launch(apply_A_multi_kernel<T, 2>); break;
    default: launch(apply_A_multi_kernel<T, 0>); break;
  }
}

void launch_apply_A_multi(const Geom& g, GaugeView U, CloverView C, FieldView in, FieldView out, int nrhs,
                          cudaStream_t st) {
  if (in.prec == P32) {
    multi_launch<float>(g, LinkPtr<float>{(const float2*)U.links}, CloverPtr<float>{(const float4*)C.m},
                        SpinorPtr<float>{(float4*)in.data}, SpinorPtr<float>{(float4*)out.data}, g.V * 6, 0, nrhs,
                        nullptr, nullptr, st);
  } else {
    // FP16 fields are V * 52 bytes each (values, then the per-site norms) and follow each
    // other: 13 V / 4 uint4 units or 13 V floats apart (V is a multiple of 64)
    multi_launch<__half>(g, LinkPtr<__half>{(const uint4*)U.links}, CloverPtr<__half>{(const uint4*)C.m},
                         SpinorPtr<__half>{(uint4*)in.data, in.norm}, SpinorPtr<__half>{(uint4*)out.data, out.norm},
                         13 * g.V / 4, 13 * g.V, nrhs, nullptr, nullptr, st);
  }
}

void launch_apply_A_multi_list(const Geom& g, GaugeView U, CloverView C, const float4* const* in,
                               float4* const* out, int nrhs, cudaStream_t st) {
  multi_launch<float>(g, LinkPtr<float>{(const float2*)U.links}, CloverPtr<float>{(const float4*)C.m},
                      SpinorPtr<float>{nullptr}, SpinorPtr<float>{nullptr}, 0, 0, nrhs, in, out, st);
}

}  // namespace dd
