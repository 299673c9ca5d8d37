// Cholesky-QR2 in one launch: one cluster of eight CTAs holds the n x r matrix
// in shared memory through both passes (Algorithm 1, "Set U <- U+": the sum of
// the gradient's partial blocks, Z = U - eta grad and Q(Z)).
//
// The five launches of the separate kernels took 46 us at n = 1000, r = 5
// (FP64 Gram loops and FP64 Cholesky chains, each on a cold SM).  Here a CTA
// keeps n / 8 rows; the two Grams are exchanged through distributed shared
// memory (two cluster barriers) and every CTA factors them redundantly.
//   Pass 1: Gram in double-float from exact products, summed over the CTAs in
//     FP64; Cholesky in FP32 when every pivot is above 1e-3 of its diagonal
//     (R1 needs to be good enough only for the second pass to start from a Gram
//     near I: any upper triangular R1 leaves Q unchanged).
//   Pass 2: the Gram is I + E; Cholesky and inverse are carried as deviations
//     from I in FP32 (relative to E), so that Q = Q1 + Q1 H adds a correction
//     known to about 1e-7 |E|, where a rounded R2^{-1} would put 6e-8 on every
//     entry.
//   When a factor fails (small pivots, E not small, a Gram outside float32's
//   range: entries of Z beyond about 1e-15 .. 1e15) Gram and factor are done
//   again in FP64, in every CTA alike, since all hold the same sums.
#include "lrs_dev.cuh"
#include "lrs_internal.h"

namespace lrs {
namespace {

constexpr int kQT = 512;   // threads per CTA
constexpr int kQC = 8;     // CTAs (portable cluster size)
constexpr int kMaxR = 16;

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

// One warp: FP32 Cholesky of the r x r matrix G (dev: of G = I + E, in
// deviations), lane i <-> row i, and its inverse, lane c <-> column c:
// Rinv[c * 16 + i] = (L^{-1})(i, c), the entry (c, i) of R^{-1} = L^{-T}
// (dev: minus the identity).  False when a pivot asks for FP64.
template <int R>
__device__ bool chol_f32(const double* G, float* Rinv, int r, bool dev) {
  const int lane = threadIdx.x & 31;
  float a[R], inv[R], dinv[R];
#pragma unroll
  for (int k = 0; k < R; ++k) {
    double g = lane < r && k < r ? G[lane * kMaxR + k] : 0.0;
    if (dev && k == lane) g -= 1.0;
    a[k] = static_cast<float>(g);
  }
  bool ok = true;
#pragma unroll
  for (int j = 0; j < R; ++j) {
    inv[j] = 1.f;
    dinv[j] = 0.f;
    if (j >= r || !ok) continue;
    const float p = __shfl_sync(0xffffffffu, a[j], j);
    if (dev) {
      ok = fabsf(p) < 0.25f;
      const float l1 = p / (1.f + sqrtf(1.f + p));  // L_jj - 1
      inv[j] = 1.f / (1.f + l1);
      dinv[j] = -l1 * inv[j];
    } else {
      ok = p > 1e-3f * static_cast<float>(G[j * kMaxR + j]) && p > 1e-30f && p < 1e30f;
      inv[j] = rsqrtf(p);
    }
    a[j] *= inv[j];
#pragma unroll
    for (int k = j + 1; k < R; ++k) {
      const float lk = __shfl_sync(0xffffffffu, a[j], k);
      a[k] = fmaf(-a[j], lk, a[k]);  // used for rows >= k only
    }
  }
  if (!ok) return false;
  float x[R];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    float t = 0.f;
#pragma unroll
    for (int p = 0; p < i; ++p) t = fmaf(-__shfl_sync(0xffffffffu, a[p], i), x[p], t);
    x[i] = i < lane ? 0.f : i == lane ? inv[i] : t * inv[i];
  }
  if (lane < r)
#pragma unroll
    for (int i = 0; i < R; ++i)
      if (i >= lane && i < r) Rinv[lane * kMaxR + i] = dev && i == lane ? dinv[i] : x[i];
  __syncwarp();
  return true;
}

template <int R>
__global__ void __launch_bounds__(kQT) __cluster_dims__(kQC, 1, 1) qr_cluster_kernel(QrArgs q) {
  extern __shared__ __align__(16) float Zt[];  // [R][ldz], column l of this CTA's rows
  constexpr int NE = R * (R + 1) / 2;
  __shared__ double part[2][NE], part64[NE];
  __shared__ double G[kMaxR * kMaxR], Ld[kMaxR * kMaxR], Li[kMaxR * kMaxR], iL[kMaxR];
  __shared__ float Rinv[kMaxR * kMaxR];
  __shared__ int factored;
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
  for (int pass = 0; pass < 2; ++pass) {
    // this CTA's part of the Gram: a warp per entry, lanes over the rows
    for (int t = w; t < r * (r + 1) / 2; t += kQT / 32) {
      int a = 0;
      while ((a + 1) * (a + 2) / 2 <= t) ++a;
      const int b = t - a * (a + 1) / 2;
      const float *za = Zt + a * q.ldz, *zb = Zt + b * q.ldz;
      float hi = 0.f, lw = 0.f;
      for (int i = lane; i < cnt; i += 32) {
        const float x = za[i], y = zb[i], p = x * y;
        float s, d;
        two_sum(hi, p, s, d);
        hi = s;
        lw += d + fmaf(x, y, -p);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float bh = __shfl_xor_sync(0xffffffffu, hi, o), bl = __shfl_xor_sync(0xffffffffu, lw, o);
        float s, d;
        two_sum(hi, bh, s, d);
        hi = s;
        lw += bl + d;
      }
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
      const bool ok = chol_f32<R>(G, Rinv, r, pass == 1);
      if (lane == 0) factored = ok;
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
        for (int t = lane; t < r * r; t += 32) {
          const int a = t / r, b = t - a * r;
          Rinv[a * kMaxR + b] = static_cast<float>(Li[b * kMaxR + a] - (pass == 1 && a == b ? 1.0 : 0.0));
        }
      }
      __syncthreads();
    }
    // rows times R^{-1} (pass 1) or I + H (pass 2), a thread per row
    for (int i = tid; i < cnt; i += kQT) {
      float z[R];
#pragma unroll
      for (int l = 0; l < R; ++l) z[l] = l < r ? Zt[l * q.ldz + i] : 0.f;
#pragma unroll
      for (int l = R - 1; l >= 0; --l) {
        if (l >= r) continue;
        float s = 0.f;
#pragma unroll
        for (int p = 0; p <= l; ++p) s = fmaf(z[p], Rinv[p * kMaxR + l], s);
        if (pass == 1) s += z[l];
        Zt[l * q.ldz + i] = s;
      }
    }
    __syncthreads();
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
  // (10.6 KB at R = 16) count: the limit of the largest request (idempotent) is
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
