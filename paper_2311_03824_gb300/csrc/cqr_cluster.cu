// Complex Cholesky-QR in one launch: one cluster of eight CTAs holds the r x n
// matrix (column-major) in shared memory (Z = U - eta grad and Q(Z), Algorithm 1).
//
// The cooperative launch of 152 blocks that it replaces where the matrix fits
// took 82 us at n = 16384, r = 6 and 44 us at n = 400, r = 4: FP64 Gram loops,
// two FP64 factors and two grid barriers; this one takes 35 and 14 us (44 and 17
// with two passes always).  The
// Gram is a double-float sum of exact products, exchanged through distributed
// shared memory, and every CTA factors it redundantly in one warp's registers,
// also in double-float.  The rows times L^{-H} are sums of exact products with
// its 48 bits, so that each entry of Z L^{-H} is rounded once, as the FP64
// products round it (float32 products lose cond(Z) 2^-24).
//
// With cond(Z)^2 <= K^2 = sum over p, l of |L^{-1}(l, p)|^2 M(p, p) (columns of
// norm one), Q^H Q - I is at most r 2^-45 K^2: one pass is enough up to
// kOnePass = 4096 (2^-29 at r = 16, below the rounding of Q), which every step
// of a solve meets; beyond, a second pass takes the rounded rows, whose Gram is
// near I.  A Gram that the double-float factor cannot take (a pivot below 1e-9
// of its diagonal, or outside float32's range) is summed and factored again in
// FP64, in every CTA alike, since all hold the same sums.
#include "fourier_dev.cuh"

namespace lrs {
namespace {
using namespace fourier;

constexpr int kQT = 512;   // threads per CTA
constexpr int kQC = 8;     // CTAs (portable cluster size)
constexpr float kOnePass = 4096.f;

struct CqrArgs {
  int n, r, rows, ldz;
  const float2* X;     // r x n (rank l at X + l n)
  const float2* G;     // gradient, same layout (or null)
  const double* eta;
  float2* Q;           // r x n (may be X)
  int* err;
};

template <int R>
__global__ void __launch_bounds__(kQT) __cluster_dims__(kQC, 1, 1) cqr_cluster_kernel(CqrArgs q) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ float2 mine[2][R * R], Gd[R * R];
  __shared__ double2 Li[kMaxR * kMaxR], mine64[kMaxR * kMaxR];
  __shared__ float4 LL[kMaxR * kMaxR];  // L^{-1}: real and imaginary part, and what their rounding left
  __shared__ int ready, one;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, r = q.r, nw = kQT / 32;
  float2* Z = reinterpret_cast<float2*>(sm);                  // [r][ldz]
  float2* part = Z + (r * q.ldz + 1) / 2 * 2;                 // the warps' sums, then FP64 scratch
  double2* scratch = reinterpret_cast<double2*>(part + nw * R * R);
  const unsigned rank = cluster_rank();
  const int lo = min(q.n, static_cast<int>(rank) * q.rows), cnt = min(q.n, lo + q.rows) - lo;
  const float e = q.eta ? static_cast<float>(*q.eta) : 0.f;
  for (int l = 0; l < r; ++l) {
    const size_t at = static_cast<size_t>(l) * q.n + lo;
    for (int i = tid; i < cnt; i += kQT) {
      float2 v = q.X[at + i];
      if (q.G) {
        const float2 g = __ldg(q.G + at + i);
        v = make_float2(fmaf(-e, g.x, v.x), fmaf(-e, g.y, v.y));
      }
      Z[l * q.ldz + i] = v;
    }
  }
  __syncthreads();
  for (int pass = 0;; ++pass) {
    cgram_warp<R>(Z, q.ldz, cnt, r, nw, part + w * R * R);
    __syncthreads();
    for (int t = tid; t < r * r; t += kQT) {
      float h = 0.f, lw = 0.f;
      for (int ww = 0; ww < nw; ++ww) df_add(h, lw, part[ww * R * R + t].x, part[ww * R * R + t].y);
      mine[pass][t] = make_float2(h, lw);
    }
    cluster_sync_all();
    for (int t = tid; t < r * r; t += kQT) {  // every CTA sums the parts in rank order
      float h = 0.f, lw = 0.f;
#pragma unroll
      for (int c = 0; c < kQC; ++c) {
        const float2 x = *peer_ptr(&mine[pass][t], c);
        df_add(h, lw, x.x, x.y);
      }
      Gd[t] = make_float2(h, lw);
    }
    __syncthreads();
    if (w == 0) {
      const bool ok = cchol_df<R>(Gd, r, Li, reinterpret_cast<float2*>(LL));
      float k2 = 0.f;
      if (ok && lane < r)
        for (int l = lane; l < r; ++l) {
          const float x = static_cast<float>(Li[l * kMaxR + lane].x), y = static_cast<float>(Li[l * kMaxR + lane].y);
          k2 = fmaf(fmaf(x, x, y * y), Gd[lane * lane + 2 * lane].x, k2);
        }
      k2 = warp_sum(k2);
      if (lane == 0) {
        ready = ok;
        one = ok && k2 <= kOnePass;
      }
    }
    __syncthreads();
    if (!ready) {
      for (int t = w; t < r * (r + 1) / 2; t += nw) {  // conj(z_a) z_b
        int a = 0;
        while ((a + 1) * (a + 2) / 2 <= t) ++a;
        const int b = t - a * (a + 1) / 2;
        double sx = 0.0, sy = 0.0;
        for (int i = lane; i < cnt; i += 32) {
          const float2 x = Z[a * q.ldz + i], y = Z[b * q.ldz + i];
          sx += static_cast<double>(x.x) * y.x + static_cast<double>(x.y) * y.y;
          sy += static_cast<double>(x.x) * y.y - static_cast<double>(x.y) * y.x;
        }
        sx = warp_sum(sx);
        sy = warp_sum(sy);
        if (lane == 0) mine64[a * kMaxR + b] = make_double2(sx, sy);
      }
      cluster_sync_all();
      for (int t = tid; t < kMaxR * kMaxR; t += kQT) {
        const int a = t / kMaxR, b = t - a * kMaxR;
        if (a >= r || b > a) continue;
        double2 s = make_double2(0.0, 0.0);
        for (int c = 0; c < kQC; ++c) {
          const double2 x = *peer_ptr(&mine64[t], c);
          s.x += x.x;
          s.y += x.y;
        }
        scratch[t] = s;
      }
      __syncthreads();
      if (w == 0 && !cchol_f64(r, scratch, Li, reinterpret_cast<float2*>(LL)) && lane == 0 && rank == 0)
        report_error(q.err, kErrNotSPD, -1);
      __syncthreads();
    }
    for (int t = tid; t < r * kMaxR; t += kQT) {
      const double2 x = Li[t];
      const float hx = static_cast<float>(x.x), hy = static_cast<float>(x.y);
      LL[t] = make_float4(hx, hy, static_cast<float>(x.x - static_cast<double>(hx)),
                          static_cast<float>(x.y - static_cast<double>(hy)));
    }
    __syncthreads();
    const bool last = pass == 1 || one;
    // rows times L^{-H}, a thread per row
    for (int i = tid; i < cnt; i += kQT) {
      float2 z[R];
#pragma unroll
      for (int l = 0; l < R; ++l) z[l] = l < r ? Z[l * q.ldz + i] : make_float2(0.f, 0.f);
#pragma unroll
      for (int l = 0; l < R; ++l) {
        if (l >= r) break;
        float xh = 0.f, xl = 0.f, yh = 0.f, yl = 0.f;
#pragma unroll
        for (int p = 0; p <= l; ++p) {
          const float4 f = LL[l * kMaxR + p];
          df_fma(xh, xl, f.x, z[p].x);
          df_fma(yh, yl, f.x, z[p].y);
          xl = fmaf(f.z, z[p].x, xl);
          yl = fmaf(f.z, z[p].y, yl);
          if (p < l) {  // the diagonal is real
            df_fma(xh, xl, f.y, z[p].y);
            df_fma(yh, yl, -f.y, z[p].x);
            xl = fmaf(f.w, z[p].y, xl);
            yl = fmaf(-f.w, z[p].x, yl);
          }
        }
        const float2 s = make_float2(xh + xl, yh + yl);
        if (last) q.Q[static_cast<size_t>(l) * q.n + lo + i] = s;
        else Z[l * q.ldz + i] = s;
      }
    }
    if (last) break;  // (the same in every CTA)
    __syncthreads();
  }
  cluster_sync_all();  // no CTA leaves while a peer may still read its sums
}

// shared memory of a CTA for rank width R
size_t cqr_smem(int n, int r, int R) {
  const size_t rows = (static_cast<size_t>(n) + kQC - 1) / kQC;
  const size_t z = ((rows | 1) * r + 1) / 2 * 2 + static_cast<size_t>(kQT / 32) * R * R;
  return z * 8 + (2 * kMaxR * kMaxR + kMaxR) * 16;
}
int width(int r) { return r <= 2 ? 2 : r <= 4 ? 4 : r <= 6 ? 6 : r <= 8 ? 8 : r <= 12 ? 12 : 16; }

template <int R>
cudaError_t launch(const CqrArgs& q, size_t smem, cudaStream_t s) {
  // the limit is that of the largest request (the call is idempotent)
  const cudaError_t e =
      cudaFuncSetAttribute(cqr_cluster_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, kQrSmem);
  if (e != cudaSuccess) return e;
  cqr_cluster_kernel<R><<<kQC, kQT, smem, s>>>(q);
  return cudaGetLastError();
}

}  // namespace

bool cqr_cluster_fits(int n, int r) { return cqr_smem(n, r, width(r)) <= kQrSmem; }

cudaError_t cqr_cluster(int n, int r, const float2* X, const float2* G, const double* eta, float2* Q,
                        int* err, cudaStream_t s) {
  CqrArgs q{};
  q.n = n;
  q.r = r;
  q.rows = (n + kQC - 1) / kQC;
  q.ldz = q.rows | 1;
  q.X = X;
  q.G = G;
  q.eta = eta;
  q.Q = Q;
  q.err = err;
  const size_t smem = cqr_smem(n, r, width(r));
  switch (width(r)) {
    case 2: return launch<2>(q, smem, s);
    case 4: return launch<4>(q, smem, s);
    case 6: return launch<6>(q, smem, s);
    case 8: return launch<8>(q, smem, s);
    case 12: return launch<12>(q, smem, s);
    default: return launch<16>(q, smem, s);
  }
}

}  // namespace lrs
