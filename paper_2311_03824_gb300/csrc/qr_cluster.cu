// Cholesky-QR in one launch: one cluster of eight CTAs holds the n x r matrix in
// shared memory (Algorithm 1, "Set U <- U+": the sum of the gradient's partial
// blocks, Z = U - eta grad and Q(Z)).
//
// The five launches of the separate kernels took 46 us at n = 1000, r = 5
// (FP64 Gram loops and FP64 Cholesky chains, each on a cold SM).  Here a CTA
// keeps n / 8 rows; the Gram is a double-float sum of exact products, exchanged
// through distributed shared memory and added over the CTAs in FP64, and every
// CTA factors it redundantly, in double-float in one warp's registers.  The rows
// times R^{-1} = L^{-T} are sums of exact products with its 48 bits: each entry
// of Q is rounded once.
//
// With cond(Z)^2 <= K^2 = sum over p, l of L^{-1}(l, p)^2 G(p, p) (columns of norm
// one), Q^T Q - I is at most r 2^-45 K^2: one pass is enough up to kOnePass = 4096
// (2^-29 at r = 16, below the rounding of Q), which every step of a solve meets;
// beyond, a second pass takes the rounded rows, whose Gram is near I.  (Two
// passes with FP32 factors left two roundings, 3.5e-8 to 4.9e-8 of Q against
// 2.5e-8; U after two iterations at n = 200, q = 2000, r = 2: 6.1e-8, now 4.9e-8.
// They took 2 us more at r = 3, and 30 us less at r = 16, where the double-float
// factor is a long chain in one warp.)  A Gram that this factor cannot take (a
// pivot below 1e-9 of its diagonal, or outside float32's range: entries of Z
// beyond about 1e-15 .. 1e15) is summed and factored again in FP64, in every CTA
// alike, since all hold the same sums.
#include "lrs_dev.cuh"
#include "lrs_internal.h"

namespace lrs {
namespace {

constexpr int kQT = 512;   // threads per CTA
constexpr int kQC = 8;     // CTAs (portable cluster size)
constexpr int kMaxR = 16;
constexpr float kOnePass = 4096.f;

struct QrArgs {
  int n, r, rows, ldz;
  const float* X;      // n x r row-major
  const float* G;      // nparts blocks n x r whose sum is the gradient (or null)
  int nparts;
  const double* eta;
  float* Q;            // n x r (may be X)
  float* Qpad;         // optional: rows padded to rpad
  int rpad;
  int* err;
};

template <int R>
__global__ void __launch_bounds__(kQT) __cluster_dims__(kQC, 1, 1) qr_cluster_kernel(QrArgs q) {
  extern __shared__ __align__(16) float Zt[];  // [R][ldz], column l of this CTA's rows
  constexpr int NE = R * (R + 1) / 2;
  __shared__ double part[2][NE], part64[NE];
  __shared__ double G[kMaxR * kMaxR], Ld[kMaxR * kMaxR], Li[kMaxR * kMaxR], iL[kMaxR];
  __shared__ float2 LL[kMaxR * kMaxR];  // L^{-1} and what its rounding left
  __shared__ int factored, one;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, r = q.r;
  const unsigned rank = cluster_rank();
  const int lo = min(q.n, static_cast<int>(rank) * q.rows), cnt = min(q.n, lo + q.rows) - lo;
  // Z = X - eta sum of the gradient's blocks
  const float e = q.eta ? static_cast<float>(*q.eta) : 0.f;
  const size_t nr = static_cast<size_t>(q.n) * r, base = static_cast<size_t>(lo) * r;
  for (int u = tid; u < cnt * r; u += kQT) {
    float v = q.X[base + u];
    if (q.G) {
      float s = 0.f;
#pragma unroll 8
      for (int b = 0; b < q.nparts; ++b) s += __ldg(q.G + b * nr + base + u);
      v = fmaf(-e, s, v);
    }
    const int i = u / r, l = u - i * r;
    Zt[l * q.ldz + i] = v;
  }
  __syncthreads();
  for (int pass = 0;; ++pass) {
    // this CTA's part of the Gram: a warp per entry, lanes over the rows
    for (int t = w; t < r * (r + 1) / 2; t += kQT / 32) {
      int a = 0;
      while ((a + 1) * (a + 2) / 2 <= t) ++a;
      const int b = t - a * (a + 1) / 2;
      const float *za = Zt + a * q.ldz, *zb = Zt + b * q.ldz;
      float hi = 0.f, lw = 0.f;
      for (int i = lane; i < cnt; i += 32) df_fma(hi, lw, za[i], zb[i]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        df_add(hi, lw, __shfl_xor_sync(0xffffffffu, hi, o), __shfl_xor_sync(0xffffffffu, lw, o));
      if (lane == 0) part[pass][t] = static_cast<double>(hi) + static_cast<double>(lw);
    }
    auto sum_parts = [&](const double* p) {  // every CTA sums the parts in rank order
      cluster_sync_all();
      if (tid < r * (r + 1) / 2) {
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < kQC; ++c) s += *peer_ptr(p + tid, c);
        int a = 0;
        while ((a + 1) * (a + 2) / 2 <= tid) ++a;
        const int b = tid - a * (a + 1) / 2;
        G[a * kMaxR + b] = s;
        G[b * kMaxR + a] = s;
      }
      __syncthreads();
    };
    sum_parts(part[pass]);
    if (w == 0) {
      float k2 = 0.f;
      const float g = lane < r ? static_cast<float>(G[lane * kMaxR + lane]) : 0.f;
      const bool ok = chol_df<R>(G, r, [&](int i, df x) {
        LL[i * kMaxR + lane] = make_float2(x.h, x.l);
        k2 = fmaf(x.h * x.h, g, k2);
      });
      k2 = warp_sum(k2);
      if (lane == 0) {
        factored = ok;
        one = ok && k2 <= kOnePass;
      }
    }
    __syncthreads();
    if (!factored) {
      for (int t = w; t < r * (r + 1) / 2; t += kQT / 32) {
        int a = 0;
        while ((a + 1) * (a + 2) / 2 <= t) ++a;
        const float *za = Zt + a * q.ldz, *zb = Zt + (t - a * (a + 1) / 2) * q.ldz;
        double s = 0.0;
        for (int i = lane; i < cnt; i += 32) s = __fma_rn(static_cast<double>(za[i]), static_cast<double>(zb[i]), s);
        s = warp_sum(s);
        if (lane == 0) part64[t] = s;
      }
      sum_parts(part64);
      if (w == 0) {
        if (!chol_inverse_warp(G, Ld, Li, iL, r, kMaxR) && lane == 0 && rank == 0)
          report_error(q.err, kErrNotSPD, -1);
        __syncwarp();
        for (int t = lane; t < r * kMaxR; t += 32) {
          const float h = static_cast<float>(Li[t]);
          LL[t] = make_float2(h, static_cast<float>(Li[t] - static_cast<double>(h)));
        }
      }
      __syncthreads();
    }
    const bool last = pass == 1 || one;
    // rows times R^{-1}, a thread per row
    for (int i = tid; i < cnt; i += kQT) {
      float z[R];
#pragma unroll
      for (int l = 0; l < R; ++l) z[l] = l < r ? Zt[l * q.ldz + i] : 0.f;
#pragma unroll
      for (int l = 0; l < R; ++l) {
        if (l >= r) break;
        float h = 0.f, lw = 0.f;
#pragma unroll
        for (int p = 0; p <= l; ++p) {
          const float2 f = LL[l * kMaxR + p];
          df_fma(h, lw, f.x, z[p]);
          lw = fmaf(f.y, z[p], lw);
        }
        Zt[l * q.ldz + i] = h + lw;
      }
    }
    __syncthreads();
    if (last) break;  // (the same in every CTA)
  }
  for (int u = tid; u < cnt * r; u += kQT) {
    const int i = u / r, l = u - i * r;
    const float v = Zt[l * q.ldz + i];
    q.Q[base + u] = v;
    if (q.Qpad) q.Qpad[static_cast<size_t>(lo + i) * q.rpad + l] = v;
  }
  cluster_sync_all();  // no CTA leaves while a peer may still read its partials
}

template <int R>
cudaError_t launch(const QrArgs& q, size_t smem, cudaStream_t s) {
  // A block has 48 KB without asking for more, and the kernel's static arrays
  // (11.6 KB at R = 16) count: the limit of the largest request (idempotent) is
  // set from 32 KB on, every time, since nothing says that this process and
  // device had a larger call before.
  cudaError_t e = cudaSuccess;
  if (smem > 32 * 1024)
    e = cudaFuncSetAttribute(qr_cluster_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kQrSmem);
  if (e != cudaSuccess) return e;
  qr_cluster_kernel<R><<<kQC, kQT, smem, s>>>(q);
  return cudaGetLastError();
}

}  // namespace

bool qr_cluster_fits(int n, int r) {
  const size_t rows = (static_cast<size_t>(n) + kQC - 1) / kQC;
  return (rows | 1) * static_cast<size_t>(r) * 4 <= kQrSmem;
}

cudaError_t qr_cluster(int n, int r, const float* X, const float* Gparts, int nparts,
                       const double* eta, float* Q, float* Qpad, int rpad, int* err,
                       cudaStream_t s) {
  QrArgs q{};
  q.n = n;
  q.r = r;
  q.rows = (n + kQC - 1) / kQC;
  q.ldz = q.rows | 1;
  q.X = X;
  q.G = Gparts;
  q.nparts = nparts;
  q.eta = eta;
  q.Q = Q;
  q.Qpad = Qpad;
  q.rpad = rpad;
  q.err = err;
  const size_t smem = static_cast<size_t>(q.ldz) * r * 4;
  if (r <= 2) return launch<2>(q, smem, s);
  if (r <= 4) return launch<4>(q, smem, s);
  if (r <= 6) return launch<6>(q, smem, s);
  if (r <= 8) return launch<8>(q, smem, s);
  if (r <= 12) return launch<12>(q, smem, s);
  return launch<16>(q, smem, s);
}

}  // namespace lrs
