// Multiplicative Schwarz (SAP) half-sweep: every domain of one colour is solved
// approximately in one launch, one CTA per domain (Sec. II-D, Table I).
//
// Formulation.  Per site the state is u (accumulated solution) and, on even sites only,
// the residual r of the last solve of its domain (the odd residual after a solve is
// exactly zero, Eq. 5).  Between two visits of a domain its neighbours (all of the other
// colour) changed their solution by delta'; their face buffers hold the half-spinors of
// delta' that enter the coupling R.  A visit does:
//   1. r = stored r (or the input v on the first sweep); r -= R delta' from the faces.
//   2. even-odd: t_o = A_oo^{-1} r_o;  f_e = r_e - D_eo t_o.
//   3. MR on D~_ee = A_ee - D_eo A_oo^{-1} D_oe, I_domain steps from x = 0.
//   4. delta_e = x, delta_o = A_oo^{-1} (r_o - D_oe x); u += delta; store r = MR residual.
//   5. write the projected half-spinors of delta on the eight faces.
// D_eo, D_oe are the hops inside the domain with factor -1/2; A_ee is the clover block
// (diagonal 1/(2 kappa) included), A_oo^{-1} its per-site inverse.
//
// Data movement.  The domain's links and Schwarz matrices (clover on even sites, inverse on
// odd sites) form contiguous blocks in HBM, and so does each face of a neighbouring domain;
// all of them are staged into shared memory with bulk asynchronous copies (TMA engine,
// completion on mbarriers) while the threads load the residual.  The even-site and odd-site
// work vectors live in shared memory as FP32; x, rho and the odd solution stay in registers,
// so every MR step runs on chip.  The MR inner products are reduced with warp shuffles and
// one exchange through shared memory.  There are two kernels: one thread per site
// (sap_kernel) and the default with two (sap_kernel_pair).
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "dd_kernels.hpp"
#include "dd_tma.cuh"

namespace dd {

// ------------------------------------------------------------------ matrix views
// Links and Schwarz matrices of one domain, in shared or global memory.  link<...>(mu, r, h)
// is U_mu of site r for h = 0 and its adjoint for h = 1 (h may differ between lanes: see the
// diagonal grouping of the link layout); block(r, h) the packed Hermitian 6x6 block of
// chirality h.
template <typename MT> struct MatBlock;

template <> struct MatBlock<__half> {
  const uint4* l4;     // [mu][2][Vd], then
  const uint2* l2;     // [mu][Vd]
  const uint4* cm;     // [8][Vd], then 8-byte halves [Vd][2]
  int Vd;
  __device__ void set_links(const void* p) {
    l4 = reinterpret_cast<const uint4*>(p);
    l2 = reinterpret_cast<const uint2*>(l4 + 8 * Vd);
  }
  __device__ void set_mats(const void* p) { cm = reinterpret_cast<const uint4*>(p); }
  // the nine entries (re, im) in the order D0, D1, D2 of U (h = 0) or U^dag (h = 1)
  __device__ void words(int mu, int r, int h, uint32_t w[9]) const {
    const uint4 a = l4[(2 * mu + h) * Vd + r], b = l4[(2 * mu + 1 - h) * Vd + r];
    const uint2 c = l2[mu * Vd + r];
    const uint32_t conj = h ? 0x80000000u : 0u;   // the sign of the imaginary halves
    const uint32_t v[9] = {a.w, c.x, c.y, a.x, a.y, a.z, b.x, b.y, b.z};
#pragma unroll
    for (int k = 0; k < 9; ++k) w[k] = v[k] ^ conj;
  }
  __device__ void link(int mu, int r, int h, Link<float>& U) const {
    uint32_t w[9];
    words(mu, r, h, w);
#pragma unroll
    for (int k = 0; k < 9; ++k) { float2 v = h2f(w[k]); U.e[link_row(k)][link_col(k)] = mk(v.x, v.y); }
  }
  __device__ void block_words(int r, int h, uint32_t w[18]) const {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint4 v = cm[(4 * h + u) * Vd + r];
      w[4 * u] = v.x;
      w[4 * u + 1] = v.y;
      w[4 * u + 2] = v.z;
      w[4 * u + 3] = v.w;
    }
    const uint2 v = reinterpret_cast<const uint2*>(cm + 8 * Vd)[2 * r + h];
    w[16] = v.x;
    w[17] = v.y;
  }
  __device__ void block(int r, int h, float m[36]) const {
    uint32_t w[18];
    block_words(r, h, w);
#pragma unroll
    for (int k = 0; k < 18; ++k) { float2 f = h2f(w[k]); m[2 * k] = f.x; m[2 * k + 1] = f.y; }
  }
  static constexpr int link_bytes_per_site = LINK16_BYTES_PER_SITE;
  static constexpr int mat_bytes_per_site = 9 * 16;
};

template <> struct MatBlock<float> {
  const float2* lk;    // [mu][9][Vd], entries in the order D0, D1, D2
  const float4* cm;    // [18][Vd]
  int Vd;
  __device__ void set_links(const void* p) { lk = reinterpret_cast<const float2*>(p); }
  __device__ void set_mats(const void* p) { cm = reinterpret_cast<const float4*>(p); }
  __device__ void link(int mu, int r, int h, Link<float>& U) const {
    const float2* q = lk + mu * 9 * Vd + r;
    const float2* q1 = q + 3 * h * Vd;    // h = 1: D2 in the place of D1 and
    const float2* q2 = q - 3 * h * Vd;    // D1 in the place of D2
    const uint32_t conj = h ? 0x80000000u : 0u;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const float2 v = (k < 3 ? q : k < 6 ? q1 : q2)[k * Vd];
      U.e[link_row(k)][link_col(k)] = mk(v.x, __uint_as_float(__float_as_uint(v.y) ^ conj));
    }
  }
  __device__ void block(int r, int h, float m[36]) const {
#pragma unroll
    for (int u = 0; u < 9; ++u) {
      const float4 v = cm[(9 * h + u) * Vd + r];
      m[4 * u] = v.x; m[4 * u + 1] = v.y; m[4 * u + 2] = v.z; m[4 * u + 3] = v.w;
    }
  }
  static constexpr int link_bytes_per_site = 4 * 9 * 8;
  static constexpr int mat_bytes_per_site = 18 * 16;
};

template <typename MT>
__device__ inline void site_mat(const MatBlock<MT>& M, int r, float m[72]) {
  M.block(r, 0, m);
  M.block(r, 1, m + 36);
}

// ------------------------------------------------------------------ work buffers
__device__ inline void ld_buf(const float4* buf, int Hd, int i, Spinor<float>& v) {
#pragma unroll
  for (int u = 0; u < 6; ++u) {
    float4 q = buf[u * Hd + i];
    int k = 2 * u;
    v.c[k / 3][k % 3] = mk(q.x, q.y);
    v.c[(k + 1) / 3][(k + 1) % 3] = mk(q.z, q.w);
  }
}
__device__ inline void st_buf(float4* buf, int Hd, int i, const Spinor<float>& v) {
#pragma unroll
  for (int u = 0; u < 6; ++u) {
    int k = 2 * u;
    buf[u * Hd + i] = make_float4(v.c[k / 3][k % 3].re, v.c[k / 3][k % 3].im, v.c[(k + 1) / 3][(k + 1) % 3].re,
                                  v.c[(k + 1) / 3][(k + 1) % 3].im);
  }
}

// Even-site residual store: per domain Hd sites.
template <typename VT> struct EvenStore;
template <> struct EvenStore<float> {
  float4* p;
  float* unused;
  __device__ void load(long long d, int Hd, int i, Spinor<float>& v) const { ld_buf(p + d * 6 * Hd, Hd, i, v); }
  __device__ void store(long long d, int Hd, int i, const Spinor<float>& v) const { st_buf(p + d * 6 * Hd, Hd, i, v); }
};
template <> struct EvenStore<__half> {
  uint4* p;
  float* norm;
  __device__ void load(long long d, int Hd, int i, Spinor<float>& v) const {
    float n = norm[d * Hd + i];
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      uint4 q = p[(d * 3 + u) * Hd + i];
      uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float2 f = h2f(w[e]);
        int k = 4 * u + e;
        v.c[k / 3][k % 3] = mk(f.x * n, f.y * n);
      }
    }
  }
  __device__ void store(long long d, int Hd, int i, const Spinor<float>& v) const {
    float m = 0.f;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) m = fmaxf(m, fmaxf(fabsf(v.c[a][b].re), fabsf(v.c[a][b].im)));
    float inv = m > 0.f ? 1.f / m : 0.f;
    norm[d * Hd + i] = m;
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        int k = 4 * u + e;
        w[e] = f2h(v.c[k / 3][k % 3].re * inv, v.c[k / 3][k % 3].im * inv);
      }
      p[(d * 3 + u) * Hd + i] = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
};

template <typename VT> struct VecPtr;
template <> struct VecPtr<float> {
  typedef SpinorPtr<float> type;
  __device__ static type make(void* p, float*) { return type{(float4*)p}; }
};
template <> struct VecPtr<__half> {
  typedef SpinorPtr<__half> type;
  __device__ static type make(void* p, float* n) { return type{(uint4*)p, n}; }
};

// ------------------------------------------------------------------ hop helpers
// acc += sum of the hops of one site that stay inside its domain (no -1/2 factor).
// src holds the other parity's vector; links come from the domain's block.
template <int MU, typename MT>
__device__ inline void inside_hop_mu(const Geom& g, const int l[4], int lex, int p, int r_self, const float4* src,
                                     const MatBlock<MT>& M, Spinor<float>& acc) {
  Spinor<float> psi;
  Half<float> h, uh;
  Link<float> L;
  if (l[MU] + 1 < g.b[MU]) {
    int j = (lex + g.bstride[MU]) >> 1;
    ld_buf(src, g.Hd, j, psi);
    project<MU, -1>(psi, h);
    M.link(MU, r_self, 0, L);
    su3_mul(L, h, uh);
    accum_recon<MU, -1>(acc, uh);
  }
  if (l[MU] > 0) {
    int j = (lex - g.bstride[MU]) >> 1;
    ld_buf(src, g.Hd, j, psi);
    project<MU, +1>(psi, h);
    M.link(MU, (1 - p) * g.Hd + j, 0, L);
    su3_dag_mul(L, h, uh);
    accum_recon<MU, +1>(acc, uh);
  }
}

template <typename MT>
__device__ inline void inside_hops(const Geom& g, const int l[4], int lex, int p, int r_self, const float4* src,
                                   const MatBlock<MT>& M, Spinor<float>& acc) {
  inside_hop_mu<0>(g, l, lex, p, r_self, src, M, acc);
  inside_hop_mu<1>(g, l, lex, p, r_self, src, M, acc);
  inside_hop_mu<2>(g, l, lex, p, r_self, src, M, acc);
  inside_hop_mu<3>(g, l, lex, p, r_self, src, M, acc);
}

__device__ inline void ld_half(const float4* q, Half<float>& h) {
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    float4 v = q[u];
    int k = 2 * u;
    h.c[k / 3][k % 3] = mk(v.x, v.y);
    h.c[(k + 1) / 3][(k + 1) % 3] = mk(v.z, v.w);
  }
}
__device__ inline void st_half(float4* q, const Half<float>& h) {
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    int k = 2 * u;
    q[u] = make_float4(h.c[k / 3][k % 3].re, h.c[k / 3][k % 3].im, h.c[(k + 1) / 3][(k + 1) % 3].re,
                       h.c[(k + 1) / 3][(k + 1) % 3].im);
  }
}

// acc += hops from the neighbouring domains, read from their face buffers.
//   +mu face of this domain: neighbour d+mu wrote P^-_mu delta on its -mu face;
//     the hop is (1 - gamma_mu) U_mu(x) delta(x + mu).
//   -mu face: neighbour d-mu wrote U_mu(y)^dag P^+_mu delta(y) on its +mu face.
template <int MU, typename MT>
__device__ inline void face_hop_mu(const Geom& g, int d, const int n[4], const int l[4], int r_self,
                                   const float4* faces, const MatBlock<MT>& M, Spinor<float>& acc) {
  Half<float> h, uh;
  if (l[MU] == g.b[MU] - 1) {
    long long dn = neighbour_domain(g, d, n, MU, +1);
    const float4* q = faces + (dn * g.face_block + g.face_off[2 * MU] + face_index(g, l, MU)) * 3;
    ld_half(q, h);
    Link<float> L;
    M.link(MU, r_self, 0, L);
    su3_mul(L, h, uh);
    accum_recon<MU, -1>(acc, uh);
  }
  if (l[MU] == 0) {
    long long dn = neighbour_domain(g, d, n, MU, -1);
    const float4* q = faces + (dn * g.face_block + g.face_off[2 * MU + 1] + face_index(g, l, MU)) * 3;
    ld_half(q, h);
    accum_recon<MU, +1>(acc, h);
  }
}

template <typename MT>
__device__ inline void face_hops(const Geom& g, int d, const int n[4], const int l[4], int r_self,
                                 const float4* faces, const MatBlock<MT>& M, Spinor<float>& acc) {
  face_hop_mu<0>(g, d, n, l, r_self, faces, M, acc);
  face_hop_mu<1>(g, d, n, l, r_self, faces, M, acc);
  face_hop_mu<2>(g, d, n, l, r_self, faces, M, acc);
  face_hop_mu<3>(g, d, n, l, r_self, faces, M, acc);
}

template <int MU, typename MT>
__device__ inline void face_write_mu(const Geom& g, long long d, const int l[4], int r_self, float4* faces,
                                     const MatBlock<MT>& M, const Spinor<float>& dl) {
  Half<float> h, uh;
  if (l[MU] == 0) {
    project<MU, -1>(dl, h);
    st_half(faces + (d * g.face_block + g.face_off[2 * MU] + face_index(g, l, MU)) * 3, h);
  }
  if (l[MU] == g.b[MU] - 1) {
    project<MU, +1>(dl, h);
    Link<float> L;
    M.link(MU, r_self, 0, L);
    su3_dag_mul(L, h, uh);
    st_half(faces + (d * g.face_block + g.face_off[2 * MU + 1] + face_index(g, l, MU)) * 3, uh);
  }
}

template <typename MT>
__device__ inline void face_write(const Geom& g, long long d, const int l[4], int r_self, float4* faces,
                                  const MatBlock<MT>& M, const Spinor<float>& dl) {
  face_write_mu<0>(g, d, l, r_self, faces, M, dl);
  face_write_mu<1>(g, d, l, r_self, faces, M, dl);
  face_write_mu<2>(g, d, l, r_self, faces, M, dl);
  face_write_mu<3>(g, d, l, r_self, faces, M, dl);
}

struct SapArgs {
  Geom g;
  int colour, first, use_faces, last, i_domain;
  const void* links;
  const void* smat;
  void* r_store;
  float* r_norm;
  void* u_store;
  float* u_norm;
  float4* faces;       // face buffers read by the couplings
  float4* faces_out;   // face buffers written (== faces except in the additive form)
  int both_colours;    // additive form: the grid covers the domains of both colours
  const float4* v;
  float4* z;
  const float* vscale;   // if set: the input is v * (*vscale) (a basis vector stored unnormalised)
  const float* const* vscales;   // the same for the inputs of vptr
  const float4* const* vptr;   // if set: input / output of right-hand side r at vptr[r] / zptr[r]
  float4* const* zptr;
  int* err;
  // Bound of the wait for the staged matrices, and extra bytes the barrier is told to
  // expect: 0 normally; a test sets it so the wait runs out and the error path is taken.
  unsigned long long wait_ns;
  unsigned extra_tx;
  // several right-hand sides per launch (two-threads-per-site kernel): strides between
  // consecutive right-hand sides of v / z (float4), faces (float4), residual and solution
  // storage (bytes) and their FP16 norms (floats)
  int nrhs;
  long long v_stride, f_stride, r_bytes, u_bytes, rn_stride, un_stride;
};

constexpr int SAP_MAX_THREADS = 256;

template <typename MT, typename VT, bool MSMEM>
__global__ void __launch_bounds__(SAP_MAX_THREADS, 1) sap_kernel(SapArgs a) {
  const Geom& g = a.g;
  extern __shared__ float4 smem[];
  __shared__ uint64_t mbar, mbar_inj;   // staged copies; injected bytes (test hook)
  __shared__ float4 red[SAP_MAX_THREADS / 32];
  const int tid = threadIdx.x;
  const int Hd = g.Hd, Vd = g.Vd;

  // domain of this CTA: the blockIdx.x-th domain of the given colour
  int n[4];
  {
    int half = g.N[0] >> 1;
    int j = blockIdx.x % half;
    int row = blockIdx.x / half;
    n[1] = row % g.N[1];
    n[2] = (row / g.N[1]) % g.N[2];
    n[3] = row / (g.N[1] * g.N[2]);
    n[0] = 2 * j + ((a.colour + n[1] + n[2] + n[3]) & 1);
  }
  const long long d = n[0] + (long long)g.dstride[1] * n[1] + (long long)g.dstride[2] * n[2] +
                      (long long)g.dstride[3] * n[3];

  const size_t lk_bytes = (size_t)MatBlock<MT>::link_bytes_per_site * Vd;
  const size_t cm_bytes = (size_t)MatBlock<MT>::mat_bytes_per_site * Vd;
  char* sbase = reinterpret_cast<char*>(smem);
  MatBlock<MT> M;
  M.Vd = Vd;
  const char* glk = reinterpret_cast<const char*>(a.links) + d * (long long)lk_bytes;
  const char* gcm = reinterpret_cast<const char*>(a.smat) + d * (long long)cm_bytes;
  float4* sE;
  if (MSMEM) {
    M.set_links(sbase);
    M.set_mats(sbase + lk_bytes);
    sE = reinterpret_cast<float4*>(sbase + lk_bytes + cm_bytes);
    if (tid == 0) {
      mbar_init(&mbar, 1);
      mbar_init(&mbar_inj, 1);
      mbar_init_fence();
    }
    __syncthreads();
    if (tid == 0) {
      mbar_expect_tx(&mbar, (uint32_t)(lk_bytes + cm_bytes));
      bulk_g2s(sbase, glk, (uint32_t)lk_bytes, &mbar);
      bulk_g2s(sbase + lk_bytes, gcm, (uint32_t)cm_bytes, &mbar);
      // test hook: bytes that nobody sends, on a barrier of their own
      if (a.extra_tx) mbar_expect_tx(&mbar_inj, a.extra_tx);
    }
  } else {
    M.set_links(glk);
    M.set_mats(gcm);
    sE = smem;
  }
  float4* sO = sE + 6 * Hd;

  int le[4], lo[4];
  local_coords(g, 0, tid, le);
  local_coords(g, 1, tid, lo);
  const int lex_e = le[0] + g.bstride[1] * le[1] + g.bstride[2] * le[2] + g.bstride[3] * le[3];
  const int lex_o = lo[0] + g.bstride[1] * lo[1] + g.bstride[2] * lo[2] + g.bstride[3] * lo[3];
  const long long s_e = (d << g.lgVd) + tid, s_o = s_e + Hd;
  const int r_e = tid, r_o = Hd + tid;

  // 1. residual
  Spinor<float> re, ro;
  const SpinorPtr<float> vin{const_cast<float4*>(a.v)};
  EvenStore<VT> rst{reinterpret_cast<decltype(EvenStore<VT>::p)>(a.r_store), a.r_norm};
  if (a.first) {
    vin.load(g, s_e, re);
    vin.load(g, s_o, ro);
    if (a.vscale) {
      const float sc = *a.vscale;
#pragma unroll
      for (int sp = 0; sp < 4; ++sp)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          re.c[sp][c] = sc * re.c[sp][c];
          ro.c[sp][c] = sc * ro.c[sp][c];
        }
    }
  } else {
    rst.load(d, Hd, tid, re);
    zero(ro);
  }
  if (MSMEM) {
    bool ok = mbar_wait(&mbar, 0, a.wait_ns);
    if (a.extra_tx) ok = mbar_wait(&mbar_inj, 0, a.wait_ns) && ok;
    if (__syncthreads_or(!ok)) {
      // a wait ran out: flag it; then wait (bounded) for the staged copies themselves,
      // which were issued and will land, so none is left writing into this CTA's shared
      // memory after it exits
      if (tid == 0) atomicExch(a.err, 1);
      mbar_wait(&mbar, 0, a.wait_ns);
      return;
    }
  }
  if (a.use_faces) {
    Spinor<float> ae, ao;
    zero(ae);
    zero(ao);
    face_hops(g, (int)d, n, le, r_e, a.faces, M, ae);
    face_hops(g, (int)d, n, lo, r_o, a.faces, M, ao);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        re.c[s][c] = re.c[s][c] + 0.5f * ae.c[s][c];
        ro.c[s][c] = ro.c[s][c] + 0.5f * ao.c[s][c];
      }
  }

  // 2. even-odd preparation
  float m[72];
  Spinor<float> t, acc, rho, x;
  site_mat(M, r_o, m);
  clover_mul(m, ro, t);
  st_buf(sO, Hd, tid, t);
  __syncthreads();
  zero(acc);
  inside_hops(g, le, lex_e, 0, r_e, sO, M, acc);
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      rho.c[s][c] = re.c[s][c] + 0.5f * acc.c[s][c];
      x.c[s][c] = mk(0.f, 0.f);
    }
  st_buf(sE, Hd, tid, rho);
  __syncthreads();

  // 3. MR on the Schur complement
  const int nwarp = (Hd + 31) >> 5;
  for (int it = 0; it < a.i_domain; ++it) {
    // odd sites: t = A_oo^{-1} H_oe rho
    zero(acc);
    inside_hops(g, lo, lex_o, 1, r_o, sE, M, acc);
    site_mat(M, r_o, m);
    clover_mul(m, acc, t);
    st_buf(sO, Hd, tid, t);
    __syncthreads();
    // even sites: p = A_ee rho - 1/4 H_eo t
    zero(acc);
    inside_hops(g, le, lex_e, 0, r_e, sO, M, acc);
    Spinor<float> pv;
    site_mat(M, r_e, m);
    clover_mul(m, rho, pv);
    float pr_re = 0.f, pr_im = 0.f, pp = 0.f;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        pv.c[s][c] = pv.c[s][c] - 0.25f * acc.c[s][c];
        cx<float> q = cjmul(pv.c[s][c], rho.c[s][c]);
        pr_re += q.re;
        pr_im += q.im;
        pp += pv.c[s][c].re * pv.c[s][c].re + pv.c[s][c].im * pv.c[s][c].im;
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      pr_re += __shfl_xor_sync(0xffffffffu, pr_re, o);
      pr_im += __shfl_xor_sync(0xffffffffu, pr_im, o);
      pp += __shfl_xor_sync(0xffffffffu, pp, o);
    }
    if ((tid & 31) == 0) red[tid >> 5] = make_float4(pr_re, pr_im, pp, 0.f);
    __syncthreads();
    float sr = 0.f, si = 0.f, sp = 0.f;
    for (int w = 0; w < nwarp; ++w) {
      float4 q = red[w];
      sr += q.x;
      si += q.y;
      sp += q.z;
    }
    cx<float> alpha = sp > 0.f ? mk(sr / sp, si / sp) : mk(0.f, 0.f);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        x.c[s][c] = cmac(x.c[s][c], alpha, rho.c[s][c]);
        rho.c[s][c] = cnmac(rho.c[s][c], alpha, pv.c[s][c]);
      }
    st_buf(sE, Hd, tid, rho);
    __syncthreads();
  }

  // 4. odd reconstruction: delta_o = A_oo^{-1} (r_o + 1/2 H_oe x)
  st_buf(sE, Hd, tid, x);
  __syncthreads();
  zero(acc);
  inside_hops(g, lo, lex_o, 1, r_o, sE, M, acc);
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) acc.c[s][c] = ro.c[s][c] + 0.5f * acc.c[s][c];
  Spinor<float> dlo;
  site_mat(M, r_o, m);
  clover_mul(m, acc, dlo);

  // solution and residual
  typename VecPtr<VT>::type ust = VecPtr<VT>::make(a.u_store, a.u_norm);
  Spinor<float> ue, uo;
  if (a.first) {
    ue = x;
    uo = dlo;
  } else {
    ust.load(g, s_e, ue);
    ust.load(g, s_o, uo);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        ue.c[s][c] = ue.c[s][c] + x.c[s][c];
        uo.c[s][c] = uo.c[s][c] + dlo.c[s][c];
      }
  }
  if (a.last) {
    SpinorPtr<float> zo{a.z};
    zo.store(g, s_e, ue);
    zo.store(g, s_o, uo);
  } else {
    ust.store(g, s_e, ue);
    ust.store(g, s_o, uo);
    rst.store(d, Hd, tid, rho);
  }
  // 5. faces for the other colour (not needed after the very last half-sweep)
  if (!(a.last && a.colour == 1)) {
    face_write(g, d, le, r_e, a.faces, M, x);
    face_write(g, d, lo, r_o, a.faces, M, dlo);
  }
}

// ------------------------------------------------------------------ two threads per site
// Same algorithm with 2 Hd threads per domain.  Lanes l and l + 16 of a warp (h = 0, 1) work
// on even site i and odd site i: h = 0 takes the four forward hops of a site, h = 1 the four
// backward hops, and each keeps chirality half h (spins 2h, 2h+1) of x, rho and the odd
// solution.  The clover block and its inverse act within one chirality, so the only exchange
// is of the two lanes' partial hop sums: one shuffle per number.
//
// Both lanes run the same instructions.  In lane h's frame the own spins are 2h, 2h+1 and
// the others follow; with gamma_mu = [[0, B], [B^dag, 0]] a forward hop (1 - gamma) projects to
// own - B other and adds -B^dag U h to the other spins, a backward hop (1 + gamma) in the frame
// of h = 1 to own + B^dag other and +B U^dag h.  B_k^dag = -B_k in space, so the two agree; in
// time B = 1 and they differ by a sign, which is a register.  The adjoint link comes from
// the same loads (MatBlock).
//
// Hops that leave the domain read a zero spinor (eight zero slots behind every unit of the
// work buffers, one per 16-byte bank group), so no hop is conditional and the loads of
// one hop overlap the arithmetic of another.
//
// Measured against the form with the hop directions split over two warps (masked hops, the
// partial sums exchanged through shared memory, faces read site by site from global memory):
// half-sweep of 32^3x64 (8x4x4x4 domains, I_domain 4, FP16 storage) 571 -> 430 us, of 24^3x48
// (4^4, I_domain 3) 162 -> 112 us, FP32 storage 32^3x64 679 -> 474 us; 12.0k -> 10.0k cycles and
// 2029 -> 1860 instructions per warp and MR step, 28k -> 21k cycles a visit outside them (405,
// 103 and 469 us with the launches overlapped and the order inside a phase chosen, below).
// Bound by instruction issue and shared-memory wavefronts together (74 % and 63 % busy in the MR
// steps) and by the latency of staging and output with one CTA per SM.  Cheaper arithmetic
// alone does not help: SU(3) products in packed FP32 multiply-adds measured 445 us.

constexpr int ZERO_SLOTS = 8;

template <int MU>
__device__ __forceinline__ void frame_project(const Spinor<float>& p, float st, Half<float>& o) {
  if constexpr (MU < 3) {
    project<MU, -1>(p, o);
  } else {
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c)
        o.c[s][c] = mk(fmaf(st, p.c[2 + s][c].re, p.c[s][c].re), fmaf(st, p.c[2 + s][c].im, p.c[s][c].im));
  }
}
// the first hop of a sum (MU = 3) sets it
__device__ __forceinline__ void frame_recon_first(Spinor<float>& acc, float st, const Half<float>& u) {
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      acc.c[s][c] = u.c[s][c];
      acc.c[2 + s][c] = st * u.c[s][c];
    }
}
template <int MU>
__device__ __forceinline__ void frame_recon(Spinor<float>& acc, float st, const Half<float>& u) {
  if constexpr (MU < 3) {
    accum_recon<MU, -1>(acc, u);
  } else {
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        acc.c[s][c] = acc.c[s][c] + u.c[s][c];
        acc.c[2 + s][c] = mk(fmaf(st, u.c[s][c].re, acc.c[2 + s][c].re), fmaf(st, u.c[s][c].im, acc.c[2 + s][c].im));
      }
  }
}

// Three units (one chirality half) at site i of a buffer whose units are `stride` apart.
__device__ __forceinline__ void ld_half3(const float4* q, int stride, cx<float> v[6]) {
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    const float4 w = q[u * stride];
    v[2 * u] = mk(w.x, w.y);
    v[2 * u + 1] = mk(w.z, w.w);
  }
}
__device__ __forceinline__ void st_half3(float4* q, int stride, const Half<float>& v) {
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    const int k = 2 * u;
    q[u * stride] = make_float4(v.c[k / 3][k % 3].re, v.c[k / 3][k % 3].im, v.c[(k + 1) / 3][(k + 1) % 3].re,
                                v.c[(k + 1) / 3][(k + 1) % 3].im);
  }
}
__device__ __forceinline__ void ld_half3(const float4* q, int stride, Half<float>& v) {
  cx<float> w[6];
  ld_half3(q, stride, w);
#pragma unroll
  for (int k = 0; k < 6; ++k) v.c[k / 3][k % 3] = w[k];
}

// The same in a work buffer, colour by colour: unit c holds colour c of both spins, so a hop needs
// two units for each colour that it projects and keeps few numbers waiting for their partners.
__device__ __forceinline__ void ld_work(const float4* q, int stride, Half<float>& v) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float4 w = q[c * stride];
    v.c[0][c] = mk(w.x, w.y);
    v.c[1][c] = mk(w.z, w.w);
  }
}
__device__ __forceinline__ void st_work(float4* q, int stride, const Half<float>& v) {
#pragma unroll
  for (int c = 0; c < 3; ++c) q[c * stride] = make_float4(v.c[0][c].re, v.c[0][c].im, v.c[1][c].re, v.c[1][c].im);
}
// a whole site in the frame whose own half starts at `own`
__device__ __forceinline__ void ld_frame(const float4* own, const float4* oth, int stride, Spinor<float>& v) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float4 a = own[c * stride], b = oth[c * stride];
    v.c[0][c] = mk(a.x, a.y);
    v.c[1][c] = mk(a.z, a.w);
    v.c[2][c] = mk(b.x, b.y);
    v.c[3][c] = mk(b.z, b.w);
  }
}

// own half of the sum over the two lanes of a site
__device__ __forceinline__ void join_halves(const Spinor<float>& acc, Half<float>& own) {
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c)
      own.c[s][c] = mk(acc.c[s][c].re + __shfl_xor_sync(0xffffffffu, acc.c[2 + s][c].re, 16),
                       acc.c[s][c].im + __shfl_xor_sync(0xffffffffu, acc.c[2 + s][c].im, 16));
}

// One chirality half of a stored spinor (N sites from p on).  The half-precision form is
// [2][N] 16-byte units (the first four numbers of half h), then [N][2] 8-byte units, scaled
// by the site's norm.
template <typename T> struct HalfField;
template <> struct HalfField<float> {
  float4* p;
  __device__ HalfField(void* base, float*, long long first) : p((float4*)base + first * 6) {}
  __device__ void load(int N, int r, int h, Half<float>& v) const { ld_half3(p + 3 * h * N + r, N, v); }
  __device__ void store(int N, int r, int h, const Half<float>& v) const { st_half3(p + 3 * h * N + r, N, v); }
  __device__ void prefetch(int N, int r, int h) const {
#pragma unroll
    for (int u = 0; u < 3; ++u) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + (3 * h + u) * N + r));
  }
};
template <> struct HalfField<__half> {
  uint4* p;
  float* norm;
  __device__ HalfField(void* base, float* n, long long first) : p((uint4*)base + first * 3), norm(n + first) {}
  __device__ void load(int N, int r, int h, Half<float>& v) const {
    const float n = norm[r];
    const uint4 a = p[h * N + r];
    const uint2 b = reinterpret_cast<const uint2*>(p + 2 * N)[2 * r + h];
    const uint32_t w[6] = {a.x, a.y, a.z, a.w, b.x, b.y};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const float2 f = h2f(w[k]);
      v.c[k / 3][k % 3] = mk(f.x * n, f.y * n);
    }
  }
  __device__ void store(int N, int r, int h, const Half<float>& v) const {
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < 6; ++k) m = fmaxf(m, fmaxf(fabsf(v.c[k / 3][k % 3].re), fabsf(v.c[k / 3][k % 3].im)));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
    const float inv = m > 0.f ? 1.f / m : 0.f;
    if (h == 0) norm[r] = m;
    uint32_t w[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) w[k] = f2h(v.c[k / 3][k % 3].re * inv, v.c[k / 3][k % 3].im * inv);
    p[h * N + r] = make_uint4(w[0], w[1], w[2], w[3]);
    reinterpret_cast<uint2*>(p + 2 * N)[2 * r + h] = make_uint2(w[4], w[5]);
  }
  __device__ void prefetch(int N, int r, int h) const {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p + h * N + r));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const uint2*>(p + 2 * N) + 2 * r + h));
  }
};

// ------------------------------------------------------------------ packed FP16 arithmetic
// Optional form of the domain solve's two products, in half2 arithmetic (two FP16 lanes
// per instruction) straight from the FP16 links and Schwarz matrices in shared memory.
//  - SU(3) times a half-spinor is spin-vectorised: the two spin rows of one colour share
//    a half2 (re = (s0.re, s1.re), im = (s0.im, s1.im)), so each link element, broadcast
//    to both lanes, enters four fused multiply-adds that cover both spins.
//  - A Hermitian 6x6 block times a 6-vector keeps (re, im) in a half2 and a copy of i x
//    per input entry, (-im, re); an entry L enters y_i += Lr x_j + Li (i x_j) and, as
//    conj(L), y_j += Lr x_i - Li (i x_i).
// Hop sums, MR reductions and vector updates stay FP32; values are scaled per domain into
// FP16's range before they meet these products (sap_pair_body).
struct HalfH2 {
  __half2 re[3], im[3];   // colour c: (spin 0, spin 1) of the real and imaginary parts
};

__device__ inline __half2 as_h2(uint32_t w) { return *reinterpret_cast<__half2*>(&w); }

__device__ inline void pack_h2(const Half<float>& h, HalfH2& o) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    o.re[c] = __floats2half2_rn(h.c[0][c].re, h.c[1][c].re);
    o.im[c] = __floats2half2_rn(h.c[0][c].im, h.c[1][c].im);
  }
}
__device__ inline void unpack_h2(const HalfH2& o, Half<float>& h) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float2 r = __half22float2(o.re[c]), i = __half22float2(o.im[c]);
    h.c[0][c] = mk(r.x, i.x);
    h.c[1][c] = mk(r.y, i.y);
  }
}

// o = U h; w: the nine (re, im) words of U in the order D0, D1, D2.
__device__ inline void su3_h2(const uint32_t w[9], const HalfH2& h, HalfH2& o) {
  __half2 U[3][3];
#pragma unroll
  for (int k = 0; k < 9; ++k) U[link_row(k)][link_col(k)] = as_h2(w[k]);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    __half2 re, im;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const __half2 er = __low2half2(U[a][b]), ei = __high2half2(U[a][b]);
      if (b == 0) {
        re = __hmul2(er, h.re[b]);
        im = __hmul2(er, h.im[b]);
      } else {
        re = __hfma2(er, h.re[b], re);
        im = __hfma2(er, h.im[b], im);
      }
      re = __hfma2(__hneg2(ei), h.im[b], re);
      im = __hfma2(ei, h.re[b], im);
    }
    o.re[a] = re;
    o.im[a] = im;
  }
}

// y = H x; the block's 18 words are 3 pairs of diagonal entries and the 15 lower entries
// (re, im) in the order of tri(i, j).
__device__ inline void clover_block_h2(const uint32_t w[18], const __half2 x[6], __half2 y[6]) {
  const __half2 sgn = __floats2half2_rn(-1.f, 1.f);
  __half2 xs[6];   // i x = (-im, re)
#pragma unroll
  for (int j = 0; j < 6; ++j) xs[j] = __hmul2(__lowhigh2highlow(x[j]), sgn);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const __half2 d = as_h2(w[i / 2]);
    y[i] = __hmul2((i & 1) ? __high2half2(d) : __low2half2(d), x[i]);
  }
#pragma unroll
  for (int i = 1; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < i; ++j) {
      const __half2 L = as_h2(w[3 + tri(i, j)]);
      const __half2 lr = __low2half2(L), li = __high2half2(L);
      y[i] = __hfma2(lr, x[j], y[i]);
      y[i] = __hfma2(li, xs[j], y[i]);
      y[j] = __hfma2(lr, x[i], y[j]);
      y[j] = __hfma2(__hneg2(li), xs[i], y[j]);
    }
}

// y = (chirality block h of site r) x
template <typename MT, bool H2>
__device__ __forceinline__ void pair_block(const MatBlock<MT>& M, int r, int h, const Half<float>& x, Half<float>& y) {
  if constexpr (H2) {
    uint32_t w[18];
    M.block_words(r, h, w);
    __half2 xv[6], yv[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) xv[k] = __floats2half2_rn(x.c[k / 3][k % 3].re, x.c[k / 3][k % 3].im);
    clover_block_h2(w, xv, yv);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const float2 f = __half22float2(yv[k]);
      y.c[k / 3][k % 3] = mk(f.x, f.y);
    }
  } else {
    float m[36];
    M.block(r, h, m);
    cx<float> v[6], w[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = x.c[k / 3][k % 3];
    clover_block_mul(m, v, w);
#pragma unroll
    for (int k = 0; k < 6; ++k) y.c[k / 3][k % 3] = w[k];
  }
}

// The geometry of one thread's two sites: nb[mu] holds, for the even (low 16 bits) and the odd
// site, the index of the neighbour this lane's hop reads (x + mu for h = 0, x - mu for h = 1)
// among the sites of the other parity, or of a zero slot when it lies outside the domain.
struct PairSites {
  unsigned nb[4];
  int i, h;
  float st;   // sign of the time direction in this lane's frame
  template <int P> __device__ __forceinline__ int neighbour(int mu) const {
    return P ? (int)(nb[mu] >> 16) : (int)(nb[mu] & 0xffffu);
  }
};

// One hop in direction MU of the site of parity P.
template <int P, int MU, typename MT, bool H2>
__device__ __forceinline__ void pair_hop(const Geom& g, const PairSites& q, const float4* own, const float4* oth,
                                         const MatBlock<MT>& M, Spinor<float>& acc) {
  const int HP = g.Hd + ZERO_SLOTS;
  const int j = q.neighbour<P>(MU);
  // U_mu of the site itself, or of the neighbour (any link where that is a zero slot)
  const int r = q.h ? (1 - P) * g.Hd + (j & (g.Hd - 1)) : P * g.Hd + q.i;
  Spinor<float> psi;
  ld_frame(own + j, oth + j, HP, psi);
  Half<float> hp, uh;
  frame_project<MU>(psi, q.st, hp);
  if constexpr (H2) {
    uint32_t w[9];
    M.words(MU, r, q.h, w);
    HalfH2 hh, oh;
    pack_h2(hp, hh);
    su3_h2(w, hh, oh);
    unpack_h2(oh, uh);
  } else {
    Link<float> U;
    M.link(MU, r, q.h, U);
    su3_mul(U, hp, uh);
  }
  if constexpr (MU == 3) frame_recon_first(acc, q.st, uh);
  else frame_recon<MU>(acc, q.st, uh);
}

// Own half of the sum of all hops inside the domain at the site of parity P (no -1/2 factor).  The
// order of the directions and the place of the block products only move what the compiler
// can overlap: of those tried, t first and y last with the block before the hops was the
// fastest (32^3x64 half-sweep 423 -> 405 us, 24^3x48 106 -> 102.6 us).
template <int P, typename MT, bool H2>
__device__ __forceinline__ void pair_hops(const Geom& g, const PairSites& q, const float4* src, const MatBlock<MT>& M,
                                          Half<float>& out) {
  const int HP = g.Hd + ZERO_SLOTS;
  const float4* own = src + 3 * q.h * HP;
  const float4* oth = src + 3 * (1 - q.h) * HP;
  Spinor<float> acc;
  pair_hop<P, 3, MT, H2>(g, q, own, oth, M, acc);
  pair_hop<P, 0, MT, H2>(g, q, own, oth, M, acc);
  pair_hop<P, 2, MT, H2>(g, q, own, oth, M, acc);
  pair_hop<P, 1, MT, H2>(g, q, own, oth, M, acc);
  join_halves(acc, out);
}

// ---- faces.  The block of face (mu, side) holds [3][face_n] 16-byte units of half-spinors:
// side 0 (written on the -mu face) P^- delta in the upper spins, side 1 (on the +mu face)
// U^dag P^+ delta in the lower spins, the frames in which h = 0 and h = 1 read them.  Only one
// site in four to eight lies on a given face, so the SU(3) products and the output run over
// lists of face sites, one thread each, instead of over the threads' own sites: per warp
// ~800 instead of ~1900 instructions a visit (half-sweep of 32^3x64: 459 -> 430 us).

// The k-th site of the four faces of one side (k < face_block / 2): direction, index in its
// face, and index r among the domain's sites.
struct FaceSite { int mu, idx, r; };
__device__ __forceinline__ FaceSite face_site(const Geom& g, int side, int k) {
  FaceSite f;
  int lo = 0, first = 0, S = 1, lg = g.lgb[0];
  f.mu = 0;
#pragma unroll
  for (int mu = 1; mu < 4; ++mu) {
    lo += g.face_n[mu - 1];
    if (k >= lo) {
      f.mu = mu;
      first = lo;
      S = g.bstride[mu];
      lg = g.lgb[mu];
    }
  }
  f.idx = k - first;
  // the coordinate along mu (0 or b - 1) goes in between the lower and the higher ones
  const int lex = (f.idx & (S - 1)) + (side ? ((S << lg) - S) : 0) + ((f.idx & ~(S - 1)) << lg);
  int p = lex, sh = 0;
#pragma unroll
  for (int mu = 0; mu < 3; ++mu) {
    sh += g.lgb[mu];
    p ^= lex >> sh;
  }
  f.r = (p & 1) * g.Hd + (lex >> 1);
  return f;
}

// Multiply the staged half-spinors of the forward couplings by this domain's links, in place.
template <typename MT>
__device__ __forceinline__ void pair_face_links(const Geom& g, const Geom& gf, float4* sF, const MatBlock<MT>& M) {
  for (int k = threadIdx.x; k < gf.face_block / 2; k += 2 * g.Hd) {
    const FaceSite f = face_site(g, 1, k);
    const int fn = gf.face_n[f.mu];
    float4* q = sF + 3 * gf.face_off[2 * f.mu] + f.idx;
    Half<float> hf, uh;
    Link<float> U;
    ld_half3(q, fn, hf);
    M.link(f.mu, f.r, 0, U);
    su3_mul(U, hf, uh);
    st_half3(q, fn, uh);
  }
}

// Own half of the couplings of the site of parity P to the neighbouring domains.
template <int P>
__device__ __forceinline__ void pair_face_hops(const Geom& g, const Geom& gf, const PairSites& q, const int l[4],
                                               const float4* sF, Half<float>& out) {
  Spinor<float> acc;
  zero(acc);
  auto face = [&](auto mu_c) {
    constexpr int MU = decltype(mu_c)::value;
    if (q.neighbour<P>(MU) >= g.Hd) {
      Half<float> uh;
      ld_half3(sF + 3 * gf.face_off[2 * MU + q.h] + face_index(g, l, MU), g.face_n[MU], uh);
      frame_recon<MU>(acc, q.st, uh);
    }
  };
  face(std::integral_constant<int, 0>());
  face(std::integral_constant<int, 1>());
  face(std::integral_constant<int, 2>());
  face(std::integral_constant<int, 3>());
  join_halves(acc, out);
}

// Face output of one side from delta in the work buffers.
template <int SIDE, typename MT>
__device__ __forceinline__ void pair_face_write(const Geom& g, const Geom& gf, long long d, const float4* sE,
                                                float4* faces, const MatBlock<MT>& M) {
  const int HP = g.Hd + ZERO_SLOTS;
  const float st = SIDE ? 1.f : -1.f;
  for (int k = threadIdx.x; k < gf.face_block / 2; k += 2 * g.Hd) {
    const FaceSite f = face_site(g, SIDE, k);
    const float4* b = sE + (f.r >= g.Hd ? 6 * HP + f.r - g.Hd : f.r);
    Spinor<float> v;
    ld_frame(b + 3 * SIDE * HP, b + 3 * (1 - SIDE) * HP, HP, v);
    Half<float> hp, uh;
    switch (f.mu) {
      case 0: frame_project<0>(v, st, hp); break;
      case 1: frame_project<1>(v, st, hp); break;
      case 2: frame_project<2>(v, st, hp); break;
      default: frame_project<3>(v, st, hp); break;
    }
    uh = hp;
    if (SIDE) {
      Link<float> U;
      M.link(f.mu, f.r, 1, U);
      su3_mul(U, hp, uh);
    }
    st_half3(faces + (d * gf.face_block + gf.face_off[2 * f.mu + SIDE]) * 3 + f.idx, gf.face_n[f.mu], uh);
  }
}

// cta: index of the domain among the domains of the launch's colour.
// MATS: the Schwarz matrices are staged beside the links (else read from global memory).
// H2: hop and clover products in packed FP16 (see su3_h2); the domain's residual is then
// scaled by a power of two, 16 / 2^ceil(log2 max|r|), before it enters the work buffers,
// and everything that leaves them (the new residual, delta) is scaled back.  The MR
// iteration is invariant under that scaling and powers of two are exact in FP32.
//
// The odd solution needs no hop phase of its own: x = sum_k alpha_k rho_k over the MR steps,
// and step k has already formed t_k = A_oo^{-1} H rho_k, so
//   delta_o = A_oo^{-1} (r_o + 1/2 H x) = A_oo^{-1} r_o + 1/2 sum_k alpha_k t_k
// is accumulated beside x: one phase (hops and block) less per visit.
template <typename MT, bool MATS, bool H2, int SHAPE>
__device__ __forceinline__ void sap_pair_body(const SapArgs& a, int cta) {
  // hop phases use g (constant domain fields when SHAPE != 0); face offsets come from a.g
  const Geom g = fixed_shape<SHAPE>(a.g);
  extern __shared__ float4 smem[];
  __shared__ uint64_t bars[3];   // links and faces; Schwarz matrices; injected bytes (test hook)
  __shared__ float4 red[2 * SAP_MAX_THREADS / 32];
  const int tid = threadIdx.x, lane = tid & 31;
  const int Hd = g.Hd, Vd = g.Vd, HP = Hd + ZERO_SLOTS;

  // This CTA's domain: the cta-th of the launch (the additive form runs both colours, colour
  // 0 first).
  const int ndom = a.both_colours ? g.ND : (g.ND >> 1);
  if (cta >= ndom) return;
  int n[4], colour;
  long long d;
  {
    colour = a.both_colours ? (cta >= (g.ND >> 1)) : a.colour;
    const int cidx = a.both_colours ? cta - colour * (g.ND >> 1) : cta;
    int hx = g.N[0] >> 1;
    int j = cidx % hx;
    int row = cidx / hx;
    n[1] = row % g.N[1];
    n[2] = (row / g.N[1]) % g.N[2];
    n[3] = row / (g.N[1] * g.N[2]);
    n[0] = 2 * j + ((colour + n[1] + n[2] + n[3]) & 1);
    d = n[0] + (long long)g.dstride[1] * n[1] + (long long)g.dstride[2] * n[2] + (long long)g.dstride[3] * n[3];
  }

  // Shared memory: links, Schwarz matrices (MATS), then the two work buffers, which first
  // receive the face blocks of the neighbouring domains.
  const uint32_t lk_bytes = (uint32_t)MatBlock<MT>::link_bytes_per_site * Vd;
  const uint32_t cm_bytes = MATS ? (uint32_t)MatBlock<MT>::mat_bytes_per_site * Vd : 0u;
  char* sbase = reinterpret_cast<char*>(smem);
  float4* sE = reinterpret_cast<float4*>(sbase + lk_bytes + cm_bytes);
  float4* sO = sE + 6 * HP;
  const char* glk = reinterpret_cast<const char*>(a.links) + d * lk_bytes;
  const char* gcm = reinterpret_cast<const char*>(a.smat) + d * ((long long)MatBlock<MT>::mat_bytes_per_site * Vd);
  MatBlock<MT> M;
  M.Vd = Vd;
  M.set_links(sbase);
  M.set_mats(MATS ? (const void*)(sbase + lk_bytes) : (const void*)gcm);

  // one thread: the eight face blocks this domain reads, each one contiguous copy
  auto stage_faces = [&](const float4* faces) {
#pragma unroll
    for (int mu = 0; mu < 4; ++mu)
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const long long dn = neighbour_domain(g, (int)d, n, mu, side ? -1 : +1);
        bulk_g2s(sE + 3 * a.g.face_off[2 * mu + side], faces + (dn * a.g.face_block + a.g.face_off[2 * mu + side]) * 3,
                 48u * a.g.face_n[mu], &bars[0]);
      }
  };
  const uint32_t face_bytes = a.use_faces ? 48u * a.g.face_block : 0u;
  if (tid == 0) {
#pragma unroll
    for (int b = 0; b < 3; ++b) mbar_init(&bars[b], 1);
    mbar_init_fence();
    mbar_expect_tx(&bars[0], lk_bytes + face_bytes);
    bulk_g2s(sbase, glk, lk_bytes, &bars[0]);
    if (MATS) {
      mbar_expect_tx(&bars[1], cm_bytes);
      bulk_g2s(sbase + lk_bytes, gcm, cm_bytes, &bars[1]);
    }
    // test hook: bytes that nobody sends, on a barrier of their own
    if (a.extra_tx) mbar_expect_tx(&bars[2], a.extra_tx);
  }

  // This thread's sites.
  PairSites q;
  q.h = lane >> 4;
  q.i = (tid >> 5) * 16 + (lane & 15);
  q.st = q.h ? 1.f : -1.f;
  const int h = q.h, i = q.i;
  int le[4], lo[4];
  local_coords(g, 0, i, le);
  local_coords(g, 1, i, lo);
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    unsigned w = 0;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int* l = p ? lo : le;
      const int lex = l[0] + g.bstride[1] * l[1] + g.bstride[2] * l[2] + g.bstride[3] * l[3];
      const bool out = h ? l[mu] == 0 : l[mu] == g.b[mu] - 1;
      const int step = h ? (out ? g.b[mu] - 1 : -1) : (out ? 1 - g.b[mu] : 1);   // periodic in the domain
      const int j = (lex + step * g.bstride[mu]) >> 1;
      // a zero slot in the bank group that the wrapped neighbour would use
      w |= (unsigned)(out ? Hd + (j & (ZERO_SLOTS - 1)) : j) << (16 * p);
    }
    q.nb[mu] = w;
  }
  const int r_e = i, r_o = Hd + i;
  float4* const eo = sE + 3 * h * HP + i;   // own half of the even / odd site in the work buffers
  float4* const oo = sO + 3 * h * HP + i;
  // Links and matrices were complete before any launch of this stream began (see
  // overlapped_launch); everything from here on may come from the previous launch.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (tid == 0) {
    if (a.use_faces) stage_faces(a.faces);
    // the next half-sweep may start (and stage its links and matrices) where SMs are free
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  __syncthreads();   // barriers initialised

  // Right-hand sides share the staged matrices; each has its own input, output and state.
#pragma unroll 1
  for (int rhs = 0; rhs < a.nrhs; ++rhs) {
    float* const rnr = a.r_norm ? a.r_norm + rhs * a.rn_stride : nullptr;
    float* const unr = a.u_norm ? a.u_norm + rhs * a.un_stride : nullptr;
    const HalfField<MT> rst((char*)a.r_store + rhs * a.r_bytes, rnr, d * Hd);
    const HalfField<MT> ust((char*)a.u_store + rhs * a.u_bytes, unr, d * Vd);
    float inv_sc = 1.f;   // H2: undoes the domain's scaling on the way out
    Half<float> rho, dO, x, t, own;   // residual and solution (even), solution (odd); own halves

    // 1. residual with the couplings to the other colour
    if (a.first) {
      const float4* v = (a.vptr ? a.vptr[rhs] : a.v + rhs * a.v_stride) + d * 6 * Vd + 3 * h * Vd;
      ld_half3(v + r_e, Vd, rho);
      ld_half3(v + r_o, Vd, dO);
      if (a.vscale || a.vscales) {
        const float sc = a.vscales ? *a.vscales[rhs] : *a.vscale;
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            rho.c[s][c] = sc * rho.c[s][c];
            dO.c[s][c] = sc * dO.c[s][c];
          }
      }
    } else {
      rst.load(Hd, i, h, rho);
      ust.prefetch(Vd, r_e, h);
      ust.prefetch(Vd, r_o, h);
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) dO.c[s][c] = mk(0.f, 0.f);
    }
    if (rhs == 0 || a.use_faces) {
      bool ok = mbar_wait(&bars[0], rhs & 1, a.wait_ns);
      if (rhs == 0) {
        if (MATS) ok = mbar_wait(&bars[1], 0, a.wait_ns) && ok;
        if (a.extra_tx) ok = mbar_wait(&bars[2], 0, a.wait_ns) && ok;
      }
      if (__syncthreads_or(!ok)) {
        // a wait ran out: flag it; then wait (bounded) for the staged copies themselves,
        // which were issued and will land, so none is left writing into this CTA's shared
        // memory after it exits
        if (tid == 0) atomicExch(a.err, 1);
        mbar_wait(&bars[0], rhs & 1, a.wait_ns);
        if (MATS && rhs == 0) mbar_wait(&bars[1], 0, a.wait_ns);
        return;
      }
    }
    if (a.use_faces) {
      pair_face_links<MT>(g, a.g, sE, M);
      __syncthreads();
      pair_face_hops<0>(g, a.g, q, le, sE, own);
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) rho.c[s][c] = rho.c[s][c] + 0.5f * own.c[s][c];
      pair_face_hops<1>(g, a.g, q, lo, sE, own);
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) dO.c[s][c] = dO.c[s][c] + 0.5f * own.c[s][c];
    }
    if constexpr (H2) {
      float m = 0.f;
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          m = fmaxf(m, fmaxf(fabsf(rho.c[s][c].re), fabsf(rho.c[s][c].im)));
          m = fmaxf(m, fmaxf(fabsf(dO.c[s][c].re), fabsf(dO.c[s][c].im)));
        }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0) red[tid >> 5].x = m;
      __syncthreads();
      m = 0.f;
      for (int w = 0; w < (2 * Hd + 31) >> 5; ++w) m = fmaxf(m, red[w].x);
      int e = 0;
      frexpf(m, &e);   // m < 2^e
      const float sc = m > 0.f ? ldexpf(1.f, 4 - max(e, -100)) : 1.f;   // finite even for tiny m
      inv_sc = 1.f / sc;
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          rho.c[s][c] = sc * rho.c[s][c];
          dO.c[s][c] = sc * dO.c[s][c];
        }
    }
    pair_block<MT, H2>(M, r_o, h, dO, t);   // t_o = A_oo^{-1} r_o
    dO = t;
    __syncthreads();   // the staged faces have been read: the work buffers may be written
    for (int k = tid; k < 12 * ZERO_SLOTS; k += 2 * Hd)
      sE[(k / ZERO_SLOTS) * HP + Hd + k % ZERO_SLOTS] = make_float4(0.f, 0.f, 0.f, 0.f);
    st_work(oo, HP, t);
    __syncthreads();

    // 2. even-odd preparation: rho = r_e + 1/2 H t_o
    pair_hops<0, MT, H2>(g, q, sO, M, own);
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        rho.c[s][c] = rho.c[s][c] + 0.5f * own.c[s][c];
        x.c[s][c] = mk(0.f, 0.f);
      }
    st_work(eo, HP, rho);
    __syncthreads();

    // 3. MR steps on the Schur complement
    const int nwarp = (2 * Hd + 31) >> 5;
#pragma unroll 1
    for (int it = 0; it < a.i_domain; ++it) {
      // odd sites: t = A_oo^{-1} H rho
      pair_hops<1, MT, H2>(g, q, sE, M, own);
      pair_block<MT, H2>(M, r_o, h, own, t);
      st_work(oo, HP, t);
      __syncthreads();
      // even sites: p = A_ee rho - 1/4 H t
      Half<float> pv;
      pair_block<MT, H2>(M, r_e, h, rho, pv);
      pair_hops<0, MT, H2>(g, q, sO, M, own);
      float pr_re = 0.f, pr_im = 0.f, pp = 0.f;
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          pv.c[s][c] = pv.c[s][c] - 0.25f * own.c[s][c];
          cx<float> z = cjmul(pv.c[s][c], rho.c[s][c]);
          pr_re += z.re;
          pr_im += z.im;
          pp += pv.c[s][c].re * pv.c[s][c].re + pv.c[s][c].im * pv.c[s][c].im;
        }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        pr_re += __shfl_xor_sync(0xffffffffu, pr_re, o);
        pr_im += __shfl_xor_sync(0xffffffffu, pr_im, o);
        pp += __shfl_xor_sync(0xffffffffu, pp, o);
      }
      if (lane == 0) red[tid >> 5] = make_float4(pr_re, pr_im, pp, 0.f);
      __syncthreads();
      // every warp sums the nwarp partial sums the same way (lane l holds entry l, a
      // butterfly over the lanes, lane 0's total broadcast), so all threads get one alpha
      float sr = 0.f, si = 0.f, sp = 0.f;
      if (lane < nwarp) {
        const float4 w = red[lane];
        sr = w.x;
        si = w.y;
        sp = w.z;
      }
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        if (o >= nwarp) break;
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        si += __shfl_xor_sync(0xffffffffu, si, o);
        sp += __shfl_xor_sync(0xffffffffu, sp, o);
      }
      sr = __shfl_sync(0xffffffffu, sr, 0);
      si = __shfl_sync(0xffffffffu, si, 0);
      sp = __shfl_sync(0xffffffffu, sp, 0);
      const cx<float> alpha = sp > 0.f ? mk(sr / sp, si / sp) : mk(0.f, 0.f);
      const cx<float> ah = 0.5f * alpha;
      ld_work(oo, HP, t);   // this step's t of the own odd site
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          x.c[s][c] = cmac(x.c[s][c], alpha, rho.c[s][c]);
          rho.c[s][c] = cnmac(rho.c[s][c], alpha, pv.c[s][c]);
          dO.c[s][c] = cmac(dO.c[s][c], ah, t.c[s][c]);
        }
      if (it + 1 < a.i_domain) {
        st_work(eo, HP, rho);
        __syncthreads();
      }
    }
    if constexpr (H2) {
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          rho.c[s][c] = inv_sc * rho.c[s][c];
          x.c[s][c] = inv_sc * x.c[s][c];
          dO.c[s][c] = inv_sc * dO.c[s][c];
        }
    }

    // 4. faces of delta for the next half-sweep (none after the very last one)
    if (!(a.last && (a.both_colours || colour == 1))) {
      st_work(eo, HP, x);
      st_work(oo, HP, dO);
      __syncthreads();
      float4* const fw = a.faces_out + rhs * a.f_stride;
      pair_face_write<1, MT>(g, a.g, d, sE, fw, M);
      pair_face_write<0, MT>(g, a.g, d, sE, fw, M);
    }
    // the next right-hand side's faces land in the work buffers while this one is stored
    if (rhs + 1 < a.nrhs) {
      __syncthreads();
      if (tid == 0 && a.use_faces) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(&bars[0], face_bytes);
        stage_faces(a.faces + (rhs + 1) * a.f_stride);
      }
    }

    // 5. u += delta and the new residual
    Half<float> ue = x, uo = dO;
    if (!a.first) {
      Half<float> w;
      ust.load(Vd, r_e, h, w);
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) ue.c[s][c] = ue.c[s][c] + w.c[s][c];
      ust.load(Vd, r_o, h, w);
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) uo.c[s][c] = uo.c[s][c] + w.c[s][c];
    }
    if (a.last) {
      float4* z = (a.zptr ? a.zptr[rhs] : a.z + rhs * a.v_stride) + d * 6 * Vd + 3 * h * Vd;
      st_half3(z + r_e, Vd, ue);
      st_half3(z + r_o, Vd, uo);
    } else {
      rst.store(Hd, i, h, rho);
      ust.store(Vd, r_e, h, ue);
      ust.store(Vd, r_o, h, uo);
    }
  }
}

// One CTA per domain.  A persistent grid that walks its domains, each one's copies issued as the
// previous one's buffers fall free, measured the same on 32^3x64 (430 us) and slower on 24^3x48
// (117 instead of 112 us): its loop state spills what the copies gain.
template <typename MT, bool MATS, bool H2, int SHAPE>
__global__ void __launch_bounds__(2 * SAP_MAX_THREADS, 1) sap_kernel_pair(const __grid_constant__ SapArgs a) {
  sap_pair_body<MT, MATS, H2, SHAPE>(a, blockIdx.x);
}

// Several lattices of the same domain shape in one launch: the grid is the concatenation
// of every lattice's domains of the colour; lattice l owns CTAs first[l] .. first[l+1]-1.
constexpr int SAP_MAX_LATTICES = 4;
struct SapLattices {
  SapArgs lat[SAP_MAX_LATTICES];
  int first[SAP_MAX_LATTICES + 1];
  int nlat;
};

__global__ void __launch_bounds__(2 * SAP_MAX_THREADS, 1) sap_kernel_pair_lattices(const __grid_constant__ SapLattices m) {
  int l = 0;
  while (l + 1 < m.nlat && (int)blockIdx.x >= m.first[l + 1]) ++l;
  sap_pair_body<__half, true, false, 0>(m.lat[l], blockIdx.x - m.first[l]);
}

// A half-sweep's blocks may start before the previous launch of the stream has ended: they stage
// their links and matrices and wait (griddepcontrol.wait) before they touch anything else.  What
// they stage is written by dd_load_gauge and dd_build_clover only, which wait for the stream
// before they return, so no launch that writes it can be the previous one.
// Launches of a few blocks are bound by such latencies: Schwarz on 8^4, 32 half-sweeps, 640 -> 562
// us; FP32 storage on 16^3x32, 8 half-sweeps, 309 -> 287 us; 24^3x48, 8 half-sweeps, 868 -> 820 us;
// 32^3x64, 4 half-sweeps, 1638 -> 1621 us by its last wave.
// Where a launch fills a few of each SM's places once, early blocks take the places that are
// free and leave the SMs unevenly loaded: with the next launch let in at a block's start, 256 blocks
// of 128 threads took 28.6 us for 23.7.  So not there: only with one block per SM, with half the
// SMs empty, or with at least two waves.  With the next launch let in after the wait, as now, that case
// gains too (8 half-sweeps of 16^4, 4x4x4x2 domains: 189 us by this rule, 168 without); the
// sizes between have not been measured.
static cudaLaunchAttribute overlapped_launch(const DeviceInfo& dev, int grid, int threads, size_t smem) {
  const int sms = dev.sms;
  // 128 registers a thread; smem and 2 KB of shared memory a block
  const int places = std::max(1, std::min((int)(dev.smem_sm / (smem + 2048)), 2 * SAP_MAX_THREADS / threads));
  cudaLaunchAttribute a = {};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = places == 1 || 2 * grid <= sms || grid >= 2 * sms * places;
  return a;
}

// One thread per site: the work vectors, and links and matrices when both fit.  Two threads
// per site: the links always, the matrices when they fit beside them; the work buffers (with
// their zero slots) share their space with the staged faces.
size_t sap_smem_bytes(const Geom& g, int mat_prec, bool mat_in_smem, int threads_per_site) {
  const size_t lk = mat_prec == P16 ? MatBlock<__half>::link_bytes_per_site : MatBlock<float>::link_bytes_per_site;
  const size_t cm = mat_prec == P16 ? MatBlock<__half>::mat_bytes_per_site : MatBlock<float>::mat_bytes_per_site;
  if (threads_per_site == 1) return (size_t)2 * 6 * g.Hd * 16 + (mat_in_smem ? (lk + cm) * g.Vd : 0);
  const size_t work = (size_t)2 * 6 * (g.Hd + ZERO_SLOTS) * 16, faces = (size_t)48 * g.face_block;
  return (lk + (mat_in_smem ? cm : 0)) * g.Vd + (work > faces ? work : faces);
}

bool sap_mat_fits_smem(const Geom& g, int mat_prec, int threads_per_site) {
  return sap_smem_bytes(g, mat_prec, true, threads_per_site) + 1024 <= (size_t)device_info().smem_block;
}

// Static shared memory (barriers, reduction slots) is below 1 KB; the rest may be dynamic.
static void allow_sap_smem(SmemAllowed& done, const DeviceInfo& dev, const void* kernel) {
  allow_smem(done, dev, kernel, dev.smem_block - 1024);
}

int sap_max_domain_sites() { return 2 * SAP_MAX_THREADS; }

template <typename MT, bool MATS, bool H2, int SHAPE>
static void launch_shape(const SapArgs& a, int grid, size_t smem, cudaStream_t st) {
  static SmemAllowed allowed;
  const DeviceInfo& dev = device_info();
  allow_sap_smem(allowed, dev, (const void*)sap_kernel_pair<MT, MATS, H2, SHAPE>);
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(2 * a.g.Hd);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute early = overlapped_launch(dev, grid, 2 * a.g.Hd, smem);
  c.attrs = &early;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, sap_kernel_pair<MT, MATS, H2, SHAPE>, a);
}

template <typename MT, bool MATS, bool H2 = false>
static int launch_pair(const SapArgs& a, int grid, cudaStream_t st) {
  const size_t smem = sap_smem_bytes(a.g, std::is_same<MT, __half>::value ? P16 : P32, MATS, 2);
  switch (domain_shape_id(a.g)) {
    case 1: launch_shape<MT, MATS, H2, 1>(a, grid, smem, st); break;
    case 2: launch_shape<MT, MATS, H2, 2>(a, grid, smem, st); break;
    default: launch_shape<MT, MATS, H2, 0>(a, grid, smem, st); break;
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

template <typename MT, bool MSMEM>
static int launch_single(const SapArgs& a, int grid, cudaStream_t st) {
  const size_t smem = sap_smem_bytes(a.g, std::is_same<MT, __half>::value ? P16 : P32, MSMEM, 1);
  static SmemAllowed allowed;
  allow_sap_smem(allowed, device_info(), (const void*)sap_kernel<MT, MT, MSMEM>);
  sap_kernel<MT, MT, MSMEM><<<grid, a.g.Hd, smem, st>>>(a);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

static SapArgs make_args(const Geom& g, const SapState& S, int colour, int first, int use_faces, int last,
                         const float4* v, float4* z, int i_domain);

// All lattices' domains of one colour in one launch (FP16 storage, two threads per site,
// same domain shape everywhere).
int sap_half_sweep_lattices(const Geom* gs, const SapState* Ss, int nlat, int colour, int first, int use_faces,
                            int last, const float4* const* v, float4* const* z, int i_domain, cudaStream_t st) {
  if (nlat < 1 || nlat > SAP_MAX_LATTICES) return -1;
  SapLattices m;
  m.nlat = nlat;
  int total = 0;
  for (int l = 0; l < nlat; ++l) {
    const Geom& g = gs[l];
    if (g.Hd != gs[0].Hd || g.Hd > SAP_MAX_THREADS || (g.Hd & 31) || Ss[l].mat_prec != P16 || Ss[l].vec_prec != P16 ||
        Ss[l].mat_in_smem != Ss[0].mat_in_smem)
      return -1;
    m.lat[l] = make_args(g, Ss[l], colour, first, use_faces, last, v[l], z[l], i_domain);
    m.first[l] = total;
    total += g.ND / 2;
  }
  m.first[nlat] = total;
  // the domains may differ in shape: room for the one with the most face sites
  size_t smem = 0;
  for (int l = 0; l < nlat; ++l) smem = std::max(smem, sap_smem_bytes(gs[l], P16, true, 2));
  static SmemAllowed allowed;
  const DeviceInfo& dev = device_info();
  allow_sap_smem(allowed, dev, (const void*)sap_kernel_pair_lattices);
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(total);
  c.blockDim = dim3(2 * gs[0].Hd);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute early = overlapped_launch(dev, total, 2 * gs[0].Hd, smem);
  c.attrs = &early;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, sap_kernel_pair_lattices, m);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

int sap_half_sweep(const Geom& g, const SapState& S, int colour, int first, int use_faces, int last,
                   const float4* v, float4* z, int i_domain, cudaStream_t st) {
  if (g.Hd > SAP_MAX_THREADS || (g.Hd & 31)) return -1;
  // only the pair kernel loops over right-hand sides and reads pointer lists
  if ((S.nrhs > 1 || S.vlist || S.vscales) && S.threads_per_site != 2) return -1;
  if (S.both_colours && S.threads_per_site != 2) return -1;   // the additive form: pair kernel only
  SapArgs a = make_args(g, S, colour, first, use_faces, last, v, z, i_domain);
  int grid = S.both_colours ? g.ND : g.ND / 2;
  bool ms = S.mat_in_smem;
  int pr = S.threads_per_site == 2;
  // matrices and vectors are stored in the same precision (FP16 or FP32)
  if (S.mat_prec != S.vec_prec) return -1;
  if (S.half_arith) {   // packed FP16 products: FP16 storage and the two-thread kernel only
    if (S.mat_prec != P16 || !pr || !ms) return -1;
    return launch_pair<__half, true, true>(a, grid, st);
  }
  if (S.mat_prec == P16) {   // 304 bytes of matrices per site: every allowed domain fits
    if (!ms) return -1;
    return pr ? launch_pair<__half, true>(a, grid, st) : launch_single<__half, true>(a, grid, st);
  }
  if (pr) return ms ? launch_pair<float, true>(a, grid, st) : launch_pair<float, false>(a, grid, st);
  return ms ? launch_single<float, true>(a, grid, st) : launch_single<float, false>(a, grid, st);
}

static SapArgs make_args(const Geom& g, const SapState& S, int colour, int first, int use_faces, int last,
                         const float4* v, float4* z, int i_domain) {
  SapArgs a;
  a.g = g;
  a.colour = colour;
  a.first = first;
  a.use_faces = use_faces;
  a.last = last;
  a.i_domain = i_domain;
  a.links = S.links;
  a.smat = S.smat;
  a.r_store = S.r_store;
  a.r_norm = S.r_norm;
  a.u_store = S.u_store;
  a.u_norm = S.u_norm;
  a.faces = S.faces;
  a.faces_out = S.faces_out ? S.faces_out : S.faces;
  a.both_colours = S.both_colours ? 1 : 0;
  a.v = v;
  a.z = z;
  a.vscale = S.vscale;
  a.vscales = S.vscales;
  a.vptr = S.vlist;
  a.zptr = S.zlist;
  a.err = S.err;
  a.nrhs = S.nrhs;
  a.v_stride = g.V * 6;
  a.f_stride = (long long)g.ND * g.face_block * 3;
  a.r_bytes = S.r_bytes;
  a.u_bytes = S.u_bytes;
  a.rn_stride = g.V / 2;
  a.un_stride = g.V;
  a.extra_tx = S.inject_wait_timeout ? 16u : 0u;
  a.wait_ns = S.inject_wait_timeout ? 50000000ull : 2000000000ull;
  return a;
}

}  // namespace dd

// ------------------------------------------------------------------ allocation-free variant
// Scratch of dd_sap_precondition_noalloc: a fixed array in this module's global memory.
// Every GPU that loads the library holds it until the process exits; every call of the
// allocation-free entry point shares it.
namespace dd {

constexpr size_t SAP_NOALLOC_SCRATCH_BYTES = size_t(64) << 20;   // 64 MiB
static __device__ __align__(256) unsigned char g_sap_noalloc_scratch[SAP_NOALLOC_SCRATCH_BYTES];

size_t sap_noalloc_scratch_bytes() { return SAP_NOALLOC_SCRATCH_BYTES; }

// Device address of the scratch array on the current device.  In host code the array's
// name is only a stand-in, so the address is looked up with cudaGetSymbolAddress, once per
// device, with that device current; a mutex makes the first lookups from several threads
// safe.  The address belongs to the device's context: after cudaDeviceReset the cache is
// stale, and the library (whose contexts are then invalid too) must not be used on that
// device again in this process.  Returns nullptr if the lookup fails.
void* sap_noalloc_scratch() {
  static std::mutex mu;
  static void* addr[64] = {};
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_sap_noalloc_scratch) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    addr[dev] = p;
  }
  return addr[dev];
}

}  // namespace dd
