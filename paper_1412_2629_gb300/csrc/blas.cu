// Vector kernels of the outer solver on FP32 (float4 = two complex numbers) and FP64
// (double2 = one complex number) fields in the internal layout.
//
// Inner products: every thread sums its share of the products in FP32 (a few hundred
// terms at most), converts once, and the block and grid reductions run in FP64.  The grid
// follows from the SM count and the field's size alone, so the order of the final FP64 sum
// is fixed and the result is reproducible run to run.
#include <cuda.h>

#include <algorithm>

#include "dd_kernels.hpp"
#include "dd_tma.cuh"

namespace dd {

constexpr int BT = 256;           // threads per block
constexpr int NCHUNK = 8;         // vectors per pass of the multi-dot

int blas_partials_blocks() { return 4 * device_info().sms; }

__device__ inline cx<float> dot4(float4 v, float4 w) {  // conj(v) . w over two complex numbers
  return mk(v.x * w.x + v.y * w.y + v.z * w.z + v.w * w.w, v.x * w.y - v.y * w.x + v.z * w.w - v.w * w.z);
}

// Basis vectors in FP32 (float4: two complex numbers) or FP16 (uint2: the same two complex
// numbers as two half2); every kernel that reads or writes a basis does its arithmetic in
// FP32 on float4 values.
__device__ inline float4 ldv(const float4* p, long long q) { return p[q]; }
__device__ inline float4 ldv(const uint2* p, long long q) {
  const uint2 u = p[q];
  const float2 a = h2f(u.x), b = h2f(u.y);
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ inline void stv(float4* p, long long q, float4 v, float s) {
  p[q] = make_float4(v.x * s, v.y * s, v.z * s, v.w * s);
}
__device__ inline void stv(uint2* p, long long q, float4 v, float s) {
  p[q] = make_uint2(f2h(v.x * s, v.y * s), f2h(v.z * s, v.w * s));
}

// Blocks of a grid-stride kernel over n4 elements: four per SM, fewer when there are not that
// many elements (an 8^4 field has 96 blocks' worth), where idle threads would only lengthen
// the FP64 reductions below.
static int blas_blocks(long long n4) {
  const long long need = (n4 + BT - 1) / BT;
  const int most = blas_partials_blocks();
  return need < most ? (int)need : most;
}

// Sums of N reals per thread over a warp.  Each butterfly step halves the list: a lane keeps
// one half, sends the other to its partner and adds what it receives, so 32 lanes spend
// N / 2 + N / 4 + ... FP64 additions each instead of 5 N.  GB300 adds two FP64 numbers per
// clock and SM, and with full butterflies the 18 sums of a Gram-Schmidt dot pass took longer
// than its memory traffic on all but the largest lattices.  Returns whether this lane ends
// with a sum, v[0], and which one.
template <int N, int O>
__device__ __forceinline__ void warp_fold(double* v, int& index, int& count) {
  constexpr int half = (N + 1) / 2;
  const bool up = threadIdx.x & O;
#pragma unroll
  for (int i = 0; i < half; ++i) {
    const double lo = v[i], hi = half + i < N ? v[half + i] : 0.0;
    v[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, O);
  }
  index += up ? half : 0;
  count = up ? count - half : min(count, half);
  if constexpr (O > 1) warp_fold<half, O / 2>(v, index, count);
}

// s_out[k] = sum over the block of NT threads of v[k], k < N (shared memory).
template <int NT = BT, int N>
__device__ inline void block_sums(double (&v)[N], double* s_out) {
  __shared__ double sh[NT / 32][N];
  int index = 0, count = N;
  warp_fold<N, 16>(v, index, count);
  if (count > 0) sh[threadIdx.x >> 5][index] = v[0];
  __syncthreads();
  if (threadIdx.x < N) {
    double t = 0;
    for (int k = 0; k < NT / 32; ++k) t += sh[k][threadIdx.x];
    s_out[threadIdx.x] = t;
  }
  __syncthreads();
}

// partial[blockIdx][v0 + i] = sum over this block's share of conj(V_{v0+i}) . w
template <int NV>
__global__ void __launch_bounds__(BT) multi_dot_kernel(const float4* V, int v0, int nv, long long n4, const float4* w,
                                                       double2* partial, int ldp) {
  float re[NV], im[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) re[i] = im[i] = 0.f;
  for (long long q = blockIdx.x * (long long)BT + threadIdx.x; q < n4; q += (long long)gridDim.x * BT) {
    float4 wq = w[q];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      if (v0 + i < nv) {
        cx<float> d = dot4(V[(long long)(v0 + i) * n4 + q], wq);
        re[i] += d.re;
        im[i] += d.im;
      }
    }
  }
  double acc[2 * NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) { acc[2 * i] = re[i]; acc[2 * i + 1] = im[i]; }
  __shared__ double out[2 * NV];
  block_sums(acc, out);
  if (threadIdx.x < NV && v0 + (int)threadIdx.x < nv)
    partial[(long long)blockIdx.x * ldp + v0 + threadIdx.x] = make_double2(out[2 * threadIdx.x], out[2 * threadIdx.x + 1]);
}

int launch_multi_dot(const float4* V, int nv, long long n4, const float4* w, double2* partial, cudaStream_t st) {
  int nb = blas_partials_blocks(), n = 0;
  for (int v0 = 0; v0 < nv; v0 += NCHUNK, ++n) multi_dot_kernel<NCHUNK><<<nb, BT, 0, st>>>(V, v0, nv, n4, w, partial, nv);
  return n;
}

// out[i] (+)= sum over blocks of partial[b][i], fixed order.
__global__ void reduce_partials_kernel(const double2* partial, int nb, int nv, double2* out, int accumulate) {
  int i = blockIdx.x;
  double sx = 0, sy = 0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) { sx += partial[(long long)b * nv + i].x; sy += partial[(long long)b * nv + i].y; }
  __shared__ double shx[256], shy[256];
  shx[threadIdx.x] = sx;
  shy[threadIdx.x] = sy;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) { shx[threadIdx.x] += shx[threadIdx.x + o]; shy[threadIdx.x] += shy[threadIdx.x + o]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (accumulate) { out[i].x += shx[0]; out[i].y += shy[0]; }
    else out[i] = make_double2(shx[0], shy[0]);
  }
}

void launch_reduce_partials(const double2* partial, int nv, double2* out, int accumulate, cudaStream_t st) {
  reduce_partials_kernel<<<nv, 256, 0, st>>>(partial, blas_partials_blocks(), nv, out, accumulate);
}

// |x|^2 of an FP64 field (double2 units); exact FP64 arithmetic throughout.
__global__ void __launch_bounds__(BT) norm2_64_kernel(const double2* x, long long n2, double2* partial) {
  double s = 0;
  for (long long q = blockIdx.x * (long long)BT + threadIdx.x; q < n2; q += (long long)gridDim.x * BT) {
    double2 a = x[q];
    s += a.x * a.x + a.y * a.y;
  }
  double acc[1] = {s};
  __shared__ double out[1];
  block_sums(acc, out);
  if (threadIdx.x == 0) partial[blockIdx.x] = make_double2(out[0], 0.0);
}
void launch_norm2_64(const double2* x, long long n2, double2* partial, cudaStream_t st) {
  norm2_64_kernel<<<blas_partials_blocks(), BT, 0, st>>>(x, n2, partial);
}

// x += sum_i y_i Z_i (Z FP32, x FP64): the sum is formed in FP32, added in FP64.
__global__ void __launch_bounds__(BT) x_update_kernel(double2* x, const float4* Z, int nz, long long n4, const double2* y) {
  __shared__ float2 ys[64];
  if (threadIdx.x < nz) ys[threadIdx.x] = make_float2((float)y[threadIdx.x].x, (float)y[threadIdx.x].y);
  __syncthreads();
  for (long long q = blockIdx.x * (long long)BT + threadIdx.x; q < n4; q += (long long)gridDim.x * BT) {
    float4 a = make_float4(0, 0, 0, 0);
    for (int i = 0; i < nz; ++i) {
      float4 v = Z[(long long)i * n4 + q];
      float2 c = ys[i];
      a.x += c.x * v.x - c.y * v.y;
      a.y += c.x * v.y + c.y * v.x;
      a.z += c.x * v.z - c.y * v.w;
      a.w += c.x * v.w + c.y * v.z;
    }
    double2 x0 = x[2 * q], x1 = x[2 * q + 1];
    x[2 * q] = make_double2(x0.x + a.x, x0.y + a.y);
    x[2 * q + 1] = make_double2(x1.x + a.z, x1.y + a.w);
  }
}
void launch_x_update(double2* x, const float4* Z, int nz, long long n4, const double2* y, cudaStream_t st) {
  x_update_kernel<<<blas_partials_blocks(), BT, 0, st>>>(x, Z, nz, n4, y);
}

// v = r / sqrt(nrm2) in FP32 (the FP64 and FP32 layouts hold the same complex numbers
// in the same order: double2 unit 2q and 2q+1 <-> float4 unit q).
__global__ void r64_to_v32_kernel(float4* v, const double2* r, long long n4, const double2* nrm2, const int* gate) {
  if (gate && *gate != 1) return;
  double s = 1.0 / sqrt(nrm2->x);
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n4; q += (long long)gridDim.x * blockDim.x) {
    double2 a = r[2 * q], b = r[2 * q + 1];
    v[q] = make_float4((float)(a.x * s), (float)(a.y * s), (float)(b.x * s), (float)(b.y * s));
  }
}
void launch_r64_to_v32(float4* v, const double2* r, long long n4, const double2* nrm2, cudaStream_t st,
                       const int* gate) {
  r64_to_v32_kernel<<<blas_partials_blocks(), BT, 0, st>>>(v, r, n4, nrm2, gate);
}

// out_l = sum_i P[i + l ldp] V_i for l < nout (P complex FP64, column-major).  One pass
// produces NO outputs (instantiated for every count up to 16, so a deflated restart with
// k <= 15 reads each basis once and holds no unused accumulators); each loop trip issues
// RU independent input loads per thread, which is what keeps HBM busy here.  out may be
// V itself (in-place recombination): a thread reads all inputs at q before it writes
// the outputs at q, and no other thread touches q.
// Bound by issue and shared-memory reads of the coefficients as much as by HBM: in packed FP32
// multiply-adds 41 -> 9 vectors of 32^3x64 take 2.38 ms (4.2 TB/s), in scalar ones 3.66 ms.
constexpr int RBT = 128, RU = 8;
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
template <int NO, typename VT>
__global__ void __launch_bounds__(RBT) recombine_kernel(VT* out, const VT* V, int nv, int l0, long long n4,
                                                        const double2* P, int ldp, const int* gate,
                                                        const float* vscale, float oscale) {
  if (gate && *gate != 1) return;
  __shared__ float4 ps[64][NO];   // coefficients, each part twice: (re, re, im, im)
  for (int t = threadIdx.x; t < nv * NO; t += RBT) {
    int i = t / NO, l = t % NO;
    const double2 c = P[i + (long long)(l0 + l) * ldp];
    const double sc = vscale ? (double)vscale[i] : 1.0;   // stored V_i = v_i / vscale[i]
    const float cr = (float)(c.x * sc), ci = (float)(c.y * sc);
    ps[i][l] = make_float4(cr, cr, ci, ci);
  }
  __syncthreads();
  for (long long q = blockIdx.x * (long long)RBT + threadIdx.x; q < n4; q += (long long)gridDim.x * RBT) {
    // packed FP32 multiply-adds: (re, im) += cr (v.re, v.im) + ci (-v.im, v.re), four issue slots
    // for an input and an output instead of twelve
    unsigned long long a[NO][2];
#pragma unroll
    for (int l = 0; l < NO; ++l) a[l][0] = a[l][1] = 0;
    auto fma_in = [&](int i, float4 v) {
      const unsigned long long v0 = pack2(v.x, v.y), v1 = pack2(v.z, v.w), w0 = pack2(-v.y, v.x), w1 = pack2(-v.w, v.z);
#pragma unroll
      for (int l = 0; l < NO; ++l) {
        const float4 c = ps[i][l];
        const unsigned long long cr = pack2(c.x, c.y), ci = pack2(c.z, c.w);
        a[l][0] = fma2(ci, w0, fma2(cr, v0, a[l][0]));
        a[l][1] = fma2(ci, w1, fma2(cr, v1, a[l][1]));
      }
    };
    int i = 0;
    for (; i + RU <= nv; i += RU) {
      float4 v[RU];
#pragma unroll
      for (int u = 0; u < RU; ++u) v[u] = ldv(V, (long long)(i + u) * n4 + q);
#pragma unroll
      for (int u = 0; u < RU; ++u) fma_in(i + u, v[u]);
    }
    for (; i < nv; ++i) fma_in(i, ldv(V, (long long)i * n4 + q));
#pragma unroll
    for (int l = 0; l < NO; ++l) {
      const float2 lo = unpack2(a[l][0]), hi = unpack2(a[l][1]);
      stv(out, (long long)(l0 + l) * n4 + q, make_float4(lo.x, lo.y, hi.x, hi.y), oscale);
    }
  }
}

template <int NO, typename VT>
static void recombine_launch(int nl, VT* out, const VT* V, int nv, int l0, long long n4, const double2* P, int ldp,
                             cudaStream_t st, const int* gate, const float* vscale, float oscale) {
  if constexpr (NO > 1) {
    if (nl < NO) return recombine_launch<NO - 1, VT>(nl, out, V, nv, l0, n4, P, ldp, st, gate, vscale, oscale);
  }
  recombine_kernel<NO, VT><<<2 * blas_partials_blocks(), RBT, 0, st>>>(out, V, nv, l0, n4, P, ldp, gate, vscale,
                                                                      oscale);
}

int launch_recombine(float4* out, const float4* V, int nv, int nout, long long n4, const double2* P, int ldp,
                     cudaStream_t st, const int* gate, const float* vscale) {
  int n = 0;
  for (int l0 = 0; l0 < nout; l0 += 16, ++n)
    recombine_launch<16, float4>(nout - l0 < 16 ? nout - l0 : 16, out, V, nv, l0, n4, P, ldp, st, gate, vscale, 1.f);
  return n;
}

int launch_recombine(uint2* out, const uint2* V, int nv, int nout, long long n4, const double2* P, int ldp,
                     cudaStream_t st, const int* gate, const float* vscale, float oscale) {
  int n = 0;
  for (int l0 = 0; l0 < nout; l0 += 16, ++n)
    recombine_launch<16, uint2>(nout - l0 < 16 ? nout - l0 : 16, out, V, nv, l0, n4, P, ldp, st, gate, vscale,
                                oscale);
  return n;
}

// ------------------------------------------------------------------ Gram-Schmidt passes
// Classical Gram-Schmidt with selective reorthogonalisation, gated on the device so no
// host round trip is needed.  Pass 1 forms h = V^H w and |w|^2 in one read of the basis;
// the projection pass writes w - V h and its exact squared norm; a second projection runs
// only when the first cancelled more than half of |w|^2.
//
// One launch covers every basis vector.  Block b takes the chunk b % nch of NV vectors
// and the q-slice b / nch, so blocks that read the same elements of w are adjacent in
// launch order and all but the first find them in L2.  Each loop trip handles U elements
// per vector, (NV + 1) * U independent 16-byte loads per thread, which keeps enough bytes
// in flight for HBM even for the short last chunk.
template <int NV, int U>
__global__ void __launch_bounds__(BT, 2) gs_dot_kernel(const float4* __restrict__ V, int nv, int nch, long long n4,
                                                       const float4* __restrict__ w, double2* partial, int ldp,
                                                       const int* gate, int want, const float* vscale) {
  if (gate && *gate != want) return;
  const int chunk = blockIdx.x % nch, qb = blockIdx.x / nch, nqb = gridDim.x / nch;
  const int v0 = chunk * NV, nvc = min(NV, nv - v0);
  const bool self = chunk == 0;
  float re[NV], im[NV], ww = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) re[i] = im[i] = 0.f;
  const long long stride = (long long)nqb * BT;
  const float4* Vc = V + (long long)v0 * n4;
  long long q = (long long)qb * BT + threadIdx.x;
  for (; q + (U - 1) * stride < n4; q += U * stride) {
    float4 wq[U], vq[NV][U];
#pragma unroll
    for (int u = 0; u < U; ++u) wq[u] = w[q + u * stride];
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (i < nvc)
#pragma unroll
        for (int u = 0; u < U; ++u) vq[i][u] = ldv(Vc, (long long)i * n4 + q + u * stride);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (self) ww += wq[u].x * wq[u].x + wq[u].y * wq[u].y + wq[u].z * wq[u].z + wq[u].w * wq[u].w;
#pragma unroll
      for (int i = 0; i < NV; ++i)
        if (i < nvc) {
          cx<float> d = dot4(vq[i][u], wq[u]);
          re[i] += d.re;
          im[i] += d.im;
        }
    }
  }
  for (; q < n4; q += stride) {
    float4 wq = w[q];
    if (self) ww += wq.x * wq.x + wq.y * wq.y + wq.z * wq.z + wq.w * wq.w;
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (i < nvc) {
        cx<float> d = dot4(ldv(Vc, (long long)i * n4 + q), wq);
        re[i] += d.re;
        im[i] += d.im;
      }
  }
  double acc[2 * NV + 1];
#pragma unroll
  for (int i = 0; i < NV; ++i) { acc[2 * i] = re[i]; acc[2 * i + 1] = im[i]; }
  acc[2 * NV] = ww;
  __shared__ double out[2 * NV + 1];
  block_sums(acc, out);
  if ((int)threadIdx.x < nvc) {
    // stored V_i = v_i / vscale[i]: the product with v_i is the stored one times vscale[i]
    const double sc = vscale ? (double)vscale[v0 + threadIdx.x] : 1.0;
    partial[(long long)qb * ldp + v0 + threadIdx.x] = make_double2(out[2 * threadIdx.x] * sc, out[2 * threadIdx.x + 1] * sc);
  }
  if (self && threadIdx.x == 0) partial[(long long)qb * ldp + nv] = make_double2(out[2 * NV], 0.0);
}

// partial layout [q-slice][nv + 1]: entries 0..nv-1 are V^H w, entry nv is |w|^2.
int launch_gs_dot(const float4* V, int nv, long long n4, const float4* w, double2* partial, const int* gate, int want,
                  cudaStream_t st, const float* vscale) {
  const int nch = nv > 0 ? (nv + 7) / 8 : 1;
  gs_dot_kernel<8, 2><<<blas_blocks(n4) * nch, BT, 0, st>>>(V, nv, nch, n4, w, partial, nv + 1, gate, want,
                                                                   vscale);
  return 1;
}

// The FP16-basis forms read the basis in 16-byte loads of two units (four complex numbers)
// and w as the matching two float4, so each load moves as many bytes as in the FP32 forms.
__device__ inline void unpack_pair(uint4 u, float4& lo, float4& hi) {
  const float2 a = h2f(u.x), b = h2f(u.y), c = h2f(u.z), d = h2f(u.w);
  lo = make_float4(a.x, a.y, b.x, b.y);
  hi = make_float4(c.x, c.y, d.x, d.y);
}

template <int NV, int U>
__global__ void __launch_bounds__(BT, 2) gs_dot16_kernel(const uint4* __restrict__ V, int nv, int nch, long long n8,
                                                         const float4* __restrict__ w, double2* partial, int ldp,
                                                         const int* gate, int want, const float* vscale) {
  if (gate && *gate != want) return;
  const int chunk = blockIdx.x % nch, qb = blockIdx.x / nch, nqb = gridDim.x / nch;
  const int v0 = chunk * NV, nvc = min(NV, nv - v0);
  const bool self = chunk == 0;
  float re[NV], im[NV], ww = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) re[i] = im[i] = 0.f;
  const long long stride = (long long)nqb * BT;
  const uint4* Vc = V + (long long)v0 * n8;
  for (long long q = (long long)qb * BT + threadIdx.x; q < n8; q += U * stride) {
    float4 wl[U], wh[U];
    uint4 vq[NV][U];
    bool ok[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long e = q + u * stride;
      ok[u] = e < n8;
      wl[u] = ok[u] ? w[2 * e] : make_float4(0.f, 0.f, 0.f, 0.f);
      wh[u] = ok[u] ? w[2 * e + 1] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (i < nvc)
#pragma unroll
        for (int u = 0; u < U; ++u) vq[i][u] = ok[u] ? Vc[(long long)i * n8 + q + u * stride] : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (self)
        ww += wl[u].x * wl[u].x + wl[u].y * wl[u].y + wl[u].z * wl[u].z + wl[u].w * wl[u].w +
              wh[u].x * wh[u].x + wh[u].y * wh[u].y + wh[u].z * wh[u].z + wh[u].w * wh[u].w;
#pragma unroll
      for (int i = 0; i < NV; ++i)
        if (i < nvc) {
          float4 lo, hi;
          unpack_pair(vq[i][u], lo, hi);
          const cx<float> d0 = dot4(lo, wl[u]), d1 = dot4(hi, wh[u]);
          re[i] += d0.re + d1.re;
          im[i] += d0.im + d1.im;
        }
    }
  }
  double acc[2 * NV + 1];
#pragma unroll
  for (int i = 0; i < NV; ++i) { acc[2 * i] = re[i]; acc[2 * i + 1] = im[i]; }
  acc[2 * NV] = ww;
  __shared__ double out[2 * NV + 1];
  block_sums(acc, out);
  if ((int)threadIdx.x < nvc) {
    // stored V_i = v_i / vscale[i]: the product with v_i is the stored one times vscale[i]
    const double sc = vscale ? (double)vscale[v0 + threadIdx.x] : 1.0;
    partial[(long long)qb * ldp + v0 + threadIdx.x] = make_double2(out[2 * threadIdx.x] * sc, out[2 * threadIdx.x + 1] * sc);
  }
  if (self && threadIdx.x == 0) partial[(long long)qb * ldp + nv] = make_double2(out[2 * NV], 0.0);
}

int launch_gs_dot(const uint2* V, int nv, long long n4, const float4* w, double2* partial, const int* gate, int want,
                  cudaStream_t st, const float* vscale) {
  const int nch = nv > 0 ? (nv + 7) / 8 : 1;
  // n4 is even (six units per site): the basis is read as n4 / 2 pairs of units
  gs_dot16_kernel<8, 2><<<blas_blocks(n4) * nch, BT, 0, st>>>(reinterpret_cast<const uint4*>(V), nv, nch,
                                                                     n4 / 2, w, partial, nv + 1, gate, want, vscale);
  return 1;
}

__global__ void gs_reduce_kernel(const double2* partial, int nb, int ld, double2* out, const int* gate, int want) {
  if (gate && *gate != want) return;
  int i = blockIdx.x;
  double sx = 0, sy = 0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) { sx += partial[(long long)b * ld + i].x; sy += partial[(long long)b * ld + i].y; }
  __shared__ double shx[256], shy[256];
  shx[threadIdx.x] = sx;
  shy[threadIdx.x] = sy;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) { shx[threadIdx.x] += shx[threadIdx.x + o]; shy[threadIdx.x] += shy[threadIdx.x + o]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) out[i] = make_double2(shx[0], shy[0]);
}

void launch_gs_reduce(const double2* partial, int nv, long long n4, double2* out, const int* gate, int want,
                      cudaStream_t st) {
  gs_reduce_kernel<<<nv + 1, 256, 0, st>>>(partial, blas_blocks(n4), nv + 1, out, gate, want);
}
void launch_gs_reduce_blocks(const double2* partial, int nv, int nb, double2* out, const int* gate, int want,
                             cudaStream_t st) {
  gs_reduce_kernel<<<nv + 1, 256, 0, st>>>(partial, nb, nv + 1, out, gate, want);
}

// The last block of a projection pass to finish (a device-scope ticket taken after a fence;
// nobody waits) sums the blocks' norms in block order in FP64 and takes the pass's decision:
// stage 1, after the first projection, asks for a second one when |out|^2 fell below half
// of |w|^2 = hA[nv] and clears hB; stage 2, after the second, only replaces the norm.  In
// place of two one-block launches per pass: see launch_gs_project.
template <int NT>
__device__ inline void gs_tail(double nrm, double2* norm_partial, const GsTail& tail, int nv) {
  double acc[1] = {nrm};
  __shared__ double o[1];
  __shared__ int last;
  block_sums<NT>(acc, o);
  if (threadIdx.x == 0) norm_partial[blockIdx.x] = make_double2(o[0], 0.0);
  if (tail.stage == 0) return;
  if (threadIdx.x == 0) {
    __threadfence();   // this block's norm is visible before its ticket is taken
    last = atomicAdd(tail.ticket, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  double t = 0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += NT) t += __ldcg(&norm_partial[b].x);
  acc[0] = t;
  block_sums<NT>(acc, o);
  if (tail.stage == 1)
    for (int i = threadIdx.x; i <= nv; i += NT) tail.hB[i] = Z(0.0);
  if (threadIdx.x == 0) {
    *tail.nu2 = o[0];
    if (tail.stage == 1) *tail.flag = o[0] < 0.5 * tail.hA[nv].re ? 1 : 0;
    *tail.ticket = 0;
  }
}

// out = w - V h with |out|^2 partials per block (exact norm of the projected vector).
// in_place: out aliases w (each thread reads w[q] before it writes out[q]).
// Each thread carries GP_U elements and loads GP_B basis vectors for all of them before the
// products, so 8 independent 16-byte loads are in flight per thread (one vector at a time
// reached ~4.9 TB/s; this form reaches the copy bandwidth).  Every element still subtracts
// h_0 v_0, h_1 v_1, ... in that order, so the result does not depend on the unrolling.
constexpr int GP_U = 2, GP_B = 4;
__global__ void __launch_bounds__(BT) gs_project_kernel(float4* out, const float4* w, const float4* __restrict__ V,
                                                        int nv, long long n4, const double2* h,
                                                        double2* norm_partial, const int* gate, int want,
                                                        const float* vscale, GsTail tail) {
  if (gate && *gate != want) return;
  __shared__ float2 hs[64];
  for (int i = threadIdx.x; i < nv; i += BT) {
    const double sc = vscale ? (double)vscale[i] : 1.0;   // h_i v_i = (h_i vscale[i]) V_i
    hs[i] = make_float2((float)(h[i].x * sc), (float)(h[i].y * sc));
  }
  __syncthreads();
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const long long stride = (long long)gridDim.x * BT;
  float nrm = 0.f;
  for (long long q0 = blockIdx.x * (long long)BT + threadIdx.x; q0 < n4; q0 += GP_U * stride) {
    float4 a[GP_U];
    long long q[GP_U];
    bool ok[GP_U];
#pragma unroll
    for (int u = 0; u < GP_U; ++u) {
      q[u] = q0 + u * stride;
      ok[u] = q[u] < n4;
      a[u] = ok[u] ? w[q[u]] : zero;
    }
    int i = 0;
    for (; i + GP_B <= nv; i += GP_B) {
      float4 v[GP_B][GP_U];
#pragma unroll
      for (int b = 0; b < GP_B; ++b)
#pragma unroll
        for (int u = 0; u < GP_U; ++u) v[b][u] = ok[u] ? ldv(V, (long long)(i + b) * n4 + q[u]) : zero;
#pragma unroll
      for (int b = 0; b < GP_B; ++b) {
        const float2 c = hs[i + b];
#pragma unroll
        for (int u = 0; u < GP_U; ++u) {
          a[u].x -= c.x * v[b][u].x - c.y * v[b][u].y;
          a[u].y -= c.x * v[b][u].y + c.y * v[b][u].x;
          a[u].z -= c.x * v[b][u].z - c.y * v[b][u].w;
          a[u].w -= c.x * v[b][u].w + c.y * v[b][u].z;
        }
      }
    }
    for (; i < nv; ++i) {
      const float2 c = hs[i];
#pragma unroll
      for (int u = 0; u < GP_U; ++u) {
        if (!ok[u]) continue;
        const float4 x = ldv(V, (long long)i * n4 + q[u]);
        a[u].x -= c.x * x.x - c.y * x.y;
        a[u].y -= c.x * x.y + c.y * x.x;
        a[u].z -= c.x * x.z - c.y * x.w;
        a[u].w -= c.x * x.w + c.y * x.z;
      }
    }
#pragma unroll
    for (int u = 0; u < GP_U; ++u)
      if (ok[u]) {
        out[q[u]] = a[u];
        nrm += a[u].x * a[u].x + a[u].y * a[u].y + a[u].z * a[u].z + a[u].w * a[u].w;
      }
  }
  gs_tail<BT>(nrm, norm_partial, tail, nv);
}

void launch_gs_project(float4* out, const float4* w, const float4* V, int nv, long long n4, const double2* h,
                       double2* norm_partial, const int* gate, int want, cudaStream_t st, const float* vscale,
                       const GsTail& tail) {
  gs_project_kernel<<<blas_blocks(n4), BT, 0, st>>>(out, w, V, nv, n4, h, norm_partial, gate, want, vscale, tail);
}

// The first projection of a step and the dots of the second one in one pass over the basis:
// out = w - V h with |out|^2, and partial = V^H out.  Wherever the preconditioner is good, A M v
// is close to v, the first projection cancels most of |w|^2 and the second is needed in
// every step; computing its dots here, from the tile that the projection has just read,
// costs no traffic, so a step reads the basis three times instead of four.
//
// One persistent block per SM walks tiles of T float4.  A tile of w and the tiles of all basis
// vectors arrive by two copies, the second a box of a two-dimensional tensor map (vectors by
// elements): one bulk copy per vector costs ~50 cycles more than its bytes and held
// this kernel to 4 TB/s.  A warp of its own issues them several stages ahead.  G groups
// of four warps take turns at the tiles, so one group's latencies (the wait, the barrier between
// the two parts) hide behind the others: a group projects its tile in place, one thread per
// complex number, and then takes the dots, warp u the vectors u, u + 4, ... against the
// finished tile.  The number of stages is a multiple of G, so a stage always belongs to the
// same group: waits on a barrier's phase parity are only sound for a waiter that has seen
// the phase before (copies of different stages may land out of order).
// Basis of 32^3x64 vectors, 16: 533 us (6.8 TB/s) for 1025 us of the two passes apart, 40: 1248
// for 2398 us; 24^3x48, 8: 111 for 196 us.
//
// Sums: a lane adds at most 64 terms in FP32, as the dot kernels do, and hands them to a
// two-float sum (TwoSum, exact to the last bits), which is converted to FP64 at the end.
constexpr int GT = 128;   // threads of a group; 32 more threads issue the copies
struct TwoFloat {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float s = hi + x, b = s - hi;
    lo += (hi - (s - b)) + (x - b);
    hi = s;
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

__device__ __forceinline__ bool group_or(int group, bool p) {   // barrier over one group
  int r;
  asm volatile(
      "{\n .reg .pred P, Q;\n setp.ne.s32 P, %1, 0;\n barrier.cta.red.or.pred Q, %3, %2, P;\n selp.s32 %0, 1, 0, Q;\n}\n"
      : "=r"(r)
      : "r"((int)p), "n"(GT), "r"(group + 1)
      : "memory");
  return r != 0;
}

template <int T, int G, int MOST>   // MOST: the largest number of vectors
__global__ void __launch_bounds__(G* GT + 32, 1)
    gs_project_dot_kernel(const __grid_constant__ CUtensorMap basis, float4* out, const float4* w, int nv, long long n4,
                          const double2* h,
                          const float* vscale, double2* partial, double2* norm_partial, int stages, int* err,
                          unsigned long long wait_ns, unsigned extra_tx, GsTail tail) {
  constexpr int K = (MOST + 3) / 4;            // vectors per warp
  constexpr int E = 2 * T / GT;                // complex numbers per thread
  constexpr int FLUSH = 2048 / T;              // tiles between flushes of the FP32 sums
  extern __shared__ __align__(128) float4 sm[];
  __shared__ float2 hs[64];
  __shared__ uint64_t full[16], empty[16], injected;
  const int tid = threadIdx.x, lane = tid & 31;
  const int piece = (nv + 1) * T;             // float4 per stage
  for (int i = tid; i < nv; i += G * GT + 32) {
    const double sc = vscale ? (double)vscale[i] : 1.0;   // h_i v_i = (h_i vscale[i]) V_i
    hs[i] = make_float2((float)(h[i].x * sc), (float)(h[i].y * sc));
  }
  const long long ntile = n4 / T;
  const int mine = (int)((ntile - blockIdx.x + gridDim.x - 1) / gridDim.x);   // tiles of this block
  if (tid == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], GT / 32);
    }
    mbar_init(&injected, 1);
    mbar_init_fence();
    if (extra_tx) mbar_expect_tx(&injected, extra_tx);   // test hook: bytes that nobody sends
  }
  __syncthreads();

  TwoFloat snrm;
  const int group = tid / GT;
  if (group == G) {
    int issued = 0;
    for (int k = 0, s = 0, turn = 0; k < mine; ++k) {
      // the group has left this stage's previous tile
      if (!__all_sync(0xffffffffu, turn == 0 || mbar_wait(&empty[s], (turn - 1) & 1, wait_ns))) break;
      if (lane == 0) {
        const long long q = (blockIdx.x + (long long)k * gridDim.x) * T;
        mbar_expect_tx(&full[s], (uint32_t)(piece * 16));
        bulk_g2s(sm + s * piece, w + q, T * 16, &full[s]);
        tensor_g2s_2d(sm + s * piece + T, &basis, (int)(2 * q), 0, &full[s]);   // 8-byte elements
      }
      __syncwarp();
      if (++s == stages) {
        s = 0;
        ++turn;
      }
      issued = k + 1;
    }
    // no copy may land in this block's shared memory after it has left (a wait only when a
    // group gave up)
    for (int k = max(0, issued - stages); k < issued; ++k) mbar_wait(&full[k % stages], (k / stages) & 1, wait_ns);
  } else {
    const int gt = tid - group * GT, warp = gt >> 5;
    float re[K], im[K], nrm = 0.f;
    TwoFloat sre[K], sim[K];
#pragma unroll
    for (int k = 0; k < K; ++k) re[k] = im[k] = 0.f;
    int left = FLUSH;
    const bool held = extra_tx && !mbar_wait(&injected, 0, wait_ns);
    for (int k = group, s = group, turn = 0; k < mine; k += G) {
      float4* const st = sm + s * piece;
      const float4* sv = st + T;
      const bool ok = mbar_wait(&full[s], turn & 1, wait_ns) && !held;
      float2 a[E];
#pragma unroll
      for (int e = 0; e < E; ++e) a[e] = reinterpret_cast<const float2*>(st)[gt + GT * e];
#pragma unroll 4
      for (int i = 0; i < nv; ++i) {
        const float2 c = hs[i];
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const float2 v = reinterpret_cast<const float2*>(sv + i * T)[gt + GT * e];
          a[e].x -= c.x * v.x - c.y * v.y;
          a[e].y -= c.x * v.y + c.y * v.x;
        }
      }
      float2* o = reinterpret_cast<float2*>(out + (blockIdx.x + (long long)k * gridDim.x) * T);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        o[gt + GT * e] = a[e];
        reinterpret_cast<float2*>(st)[gt + GT * e] = a[e];
        nrm += a[e].x * a[e].x + a[e].y * a[e].y;
      }
      if (group_or(group, !ok)) {   // a copy did not arrive: flag it and stop
        if (gt == 0) atomicExch(err, 1);
        break;
      }
#pragma unroll 2
      for (int e = 0; e < T / 32; ++e) {
        const float4 p = st[lane + 32 * e];
#pragma unroll
        for (int j = 0; j < K; ++j) {
          const int i = 4 * j + warp;
          if (i < nv) {
            const cx<float> d = dot4(sv[i * T + lane + 32 * e], p);
            re[j] += d.re;
            im[j] += d.im;
          }
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // before copies land here again
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[s]);
      if (--left == 0 || k + G >= mine) {
#pragma unroll
        for (int j = 0; j < K; ++j) {
          sre[j].add(re[j]);
          sim[j].add(im[j]);
          re[j] = im[j] = 0.f;
        }
        snrm.add(nrm);
        nrm = 0.f;
        left = FLUSH;
      }
      s += G;
      if (s >= stages) {
        s -= stages;
        ++turn;
      }
    }
    // each vector's sum over the group's tiles lies in one warp
    double acc[2 * K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
      acc[2 * j] = sre[j].value();
      acc[2 * j + 1] = sim[j].value();
    }
    int index = 0, count = 2 * K;
    warp_fold<2 * K, 16>(acc, index, count);
    const int i = 4 * (index >> 1) + warp;
    double2* row = partial + (long long)(blockIdx.x * G + group) * (nv + 1);
    if (count > 0 && i < nv) {
      const double sc = vscale ? (double)vscale[i] : 1.0;
      reinterpret_cast<double*>(row + i)[index & 1] = acc[0] * sc;
    }
    if (gt == 0) row[nv] = make_double2(0.0, 0.0);
  }
  gs_tail<G * GT + 32>(snrm.value(), norm_partial, tail, nv);
}

// Tensor map of nv basis vectors (rows) of n4 float4, in 8-byte elements (a box holds at most 256
// per dimension): boxes of all rows by T float4.
static bool basis_map(CUtensorMap* m, const float4* V, int nv, long long n4, int T) {
  typedef CUresult (*Encode)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const Encode encode = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult r;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &r) != cudaSuccess ||
        r != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      f = nullptr;
    }
    return (Encode)f;
  }();
  if (!encode) return false;
  const cuuint64_t dim[2] = {(cuuint64_t)n4 * 2, (cuuint64_t)nv}, stride[1] = {(cuuint64_t)n4 * 16};
  const cuuint32_t box[2] = {(cuuint32_t)T * 2, (cuuint32_t)nv}, step[2] = {1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<float4*>(V), dim, stride, box, step,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int T, int G, int MOST>
static int project_dot_launch(float4* out, const float4* w, const float4* V, int nv, long long n4, const double2* h,
                              const float* vscale, double2* partial, double2* norm_partial, const GsWait& wait,
                              cudaStream_t st, const GsTail& tail) {
  const size_t stage = (size_t)(nv + 1) * T * 16, room = (size_t)208 * 1024;
  const int stages = (int)std::min<size_t>(16, room / stage) / G * G;
  const DeviceInfo& dev = device_info();
  const int nb = (int)std::min<long long>(dev.sms, n4 / T);
  CUtensorMap basis;
  if (!wait.tensor_maps || !basis_map(&basis, V, nv, n4, T)) {   // no tensor maps: the two passes apart
    launch_gs_project(out, w, V, nv, n4, h, norm_partial, nullptr, 0, st, vscale, tail);
    launch_gs_dot(V, nv, n4, out, partial, nullptr, 0, st, vscale);
    return blas_blocks(n4);
  }
  static SmemAllowed allowed;
  allow_smem(allowed, dev, (const void*)gs_project_dot_kernel<T, G, MOST>, room);
  gs_project_dot_kernel<T, G, MOST><<<nb, G * GT + 32, stages * stage, st>>>(basis, out, w, nv, n4, h, vscale, partial,
                                                                             norm_partial, stages, wait.err,
                                                                             wait.inject_timeout ? 50000000ull : 2000000000ull,
                                                                             wait.inject_timeout ? 16u : 0u, tail);
  return nb * G;
}

// Tile and groups by the number of vectors: stages of 4 to 64 KB, at least two per group (three
// for the single group), so that copies are in flight while every group works.  n4 is a
// multiple of 6144 (V of 1024), hence of every tile.  Returns the number of rows in partial.
int launch_gs_project_dot(float4* out, const float4* w, const float4* V, int nv, long long n4, const double2* h,
                          const float* vscale, double2* partial, double2* norm_partial, const GsWait& wait,
                          cudaStream_t st, const GsTail& tail) {
  const auto go = [&](auto launch) {
    return launch(out, w, V, nv, n4, h, vscale, partial, norm_partial, wait, st, tail);
  };
  if (nv <= 7) return go(project_dot_launch<128, 4, 7>);
  if (nv <= 15) return go(project_dot_launch<64, 4, 15>);
  if (nv <= 31) return go(project_dot_launch<64, 3, 31>);
  if (nv <= 51) return go(project_dot_launch<64, 2, 51>);
  return go(project_dot_launch<64, 1, 63>);
}

// out = w - V h over an FP16 basis read in unit pairs (see gs_dot16_kernel); in place
// allowed (out aliases w).
__global__ void __launch_bounds__(BT) gs_project16_kernel(float4* out, const float4* w, const uint4* __restrict__ V,
                                                          int nv, long long n8, const double2* h,
                                                          double2* norm_partial, const int* gate, int want,
                                                          const float* vscale, GsTail tail) {
  if (gate && *gate != want) return;
  __shared__ float2 hs[64];
  for (int i = threadIdx.x; i < nv; i += BT) {
    const double sc = vscale ? (double)vscale[i] : 1.0;
    hs[i] = make_float2((float)(h[i].x * sc), (float)(h[i].y * sc));
  }
  __syncthreads();
  auto sub = [](float4& a, float2 c, float4 v) {
    a.x -= c.x * v.x - c.y * v.y;
    a.y -= c.x * v.y + c.y * v.x;
    a.z -= c.x * v.z - c.y * v.w;
    a.w -= c.x * v.w + c.y * v.z;
  };
  const long long stride = (long long)gridDim.x * BT;
  float nrm = 0.f;
  for (long long q0 = blockIdx.x * (long long)BT + threadIdx.x; q0 < n8; q0 += GP_U * stride) {
    float4 al[GP_U], ah[GP_U];
    long long q[GP_U];
    bool ok[GP_U];
#pragma unroll
    for (int u = 0; u < GP_U; ++u) {
      q[u] = q0 + u * stride;
      ok[u] = q[u] < n8;
      al[u] = ok[u] ? w[2 * q[u]] : make_float4(0.f, 0.f, 0.f, 0.f);
      ah[u] = ok[u] ? w[2 * q[u] + 1] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    int i = 0;
    for (; i + GP_B <= nv; i += GP_B) {
      uint4 v[GP_B][GP_U];
#pragma unroll
      for (int b = 0; b < GP_B; ++b)
#pragma unroll
        for (int u = 0; u < GP_U; ++u) v[b][u] = ok[u] ? V[(long long)(i + b) * n8 + q[u]] : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int b = 0; b < GP_B; ++b) {
        const float2 c = hs[i + b];
#pragma unroll
        for (int u = 0; u < GP_U; ++u) {
          float4 lo, hi;
          unpack_pair(v[b][u], lo, hi);
          sub(al[u], c, lo);
          sub(ah[u], c, hi);
        }
      }
    }
    for (; i < nv; ++i) {
      const float2 c = hs[i];
#pragma unroll
      for (int u = 0; u < GP_U; ++u) {
        if (!ok[u]) continue;
        float4 lo, hi;
        unpack_pair(V[(long long)i * n8 + q[u]], lo, hi);
        sub(al[u], c, lo);
        sub(ah[u], c, hi);
      }
    }
#pragma unroll
    for (int u = 0; u < GP_U; ++u)
      if (ok[u]) {
        out[2 * q[u]] = al[u];
        out[2 * q[u] + 1] = ah[u];
        nrm += al[u].x * al[u].x + al[u].y * al[u].y + al[u].z * al[u].z + al[u].w * al[u].w +
               ah[u].x * ah[u].x + ah[u].y * ah[u].y + ah[u].z * ah[u].z + ah[u].w * ah[u].w;
      }
  }
  gs_tail<BT>(nrm, norm_partial, tail, nv);
}

void launch_gs_project(float4* out, const float4* w, const uint2* V, int nv, long long n4, const double2* h,
                       double2* norm_partial, const int* gate, int want, cudaStream_t st, const float* vscale,
                       const GsTail& tail) {
  gs_project16_kernel<<<blas_blocks(n4), BT, 0, st>>>(out, w, reinterpret_cast<const uint4*>(V), nv, n4 / 2, h,
                                                      norm_partial, gate, want, vscale, tail);
}

// v16 = FP16 of s w / sqrt(*nu2) and v32 = w / sqrt(*nu2) (the FP32 copy the next Schwarz
// application reads); with a gate, only when *gate == 1.
__global__ void basis16_store_kernel(uint2* v16, float4* v32, const float4* w, long long n4, const double* nu2,
                                     float s, const int* gate) {
  if (gate && *gate != 1) return;
  const float inv = (float)(1.0 / sqrt(*nu2));
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n4; q += (long long)gridDim.x * blockDim.x) {
    const float4 a = w[q];
    const float4 v = make_float4(a.x * inv, a.y * inv, a.z * inv, a.w * inv);
    if (v32) v32[q] = v;
    stv(v16, q, v, s);
  }
}
void launch_basis16_store(uint2* v16, float4* v32, const float4* w, long long n4, const double* nu2, float s,
                          cudaStream_t st, const int* gate) {
  basis16_store_kernel<<<blas_partials_blocks(), BT, 0, st>>>(v16, v32, w, n4, nu2, s, gate);
}

// v32 = FP32 of v16 * s
__global__ void basis16_load_kernel(float4* v32, const uint2* v16, long long n4, float s) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n4; q += (long long)gridDim.x * blockDim.x) {
    const float4 a = ldv(v16, q);
    v32[q] = make_float4(a.x * s, a.y * s, a.z * s, a.w * s);
  }
}
void launch_basis16_load(float4* v32, const uint2* v16, long long n4, float s, cudaStream_t st) {
  basis16_load_kernel<<<blas_partials_blocks(), BT, 0, st>>>(v32, v16, n4, s);
}

// v *= 1 / sqrt(*nu2)
__global__ void scale_inplace_kernel(float4* v, long long n4, const double* nu2) {
  float s = (float)(1.0 / sqrt(*nu2));
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n4; q += (long long)gridDim.x * blockDim.x) {
    float4 a = v[q];
    v[q] = make_float4(a.x * s, a.y * s, a.z * s, a.w * s);
  }
}
void launch_scale_inplace(float4* v, long long n4, const double* nu2, cudaStream_t st) {
  scale_inplace_kernel<<<blas_partials_blocks(), BT, 0, st>>>(v, n4, nu2);
}

}  // namespace dd
