// Complex Cholesky-QR2 in one launch: one cluster of eight CTAs holds the r x n
// matrix (column-major) in shared memory through both passes (Z = U - eta grad
// and Q(Z), Algorithm 1).
//
// The cooperative launch of 152 blocks that it replaces where the matrix fits
// took 82 us at n = 16384, r = 6 and 44 us at n = 400, r = 4: FP64 Gram loops,
// two FP64 factors and two grid barriers; this one takes 44 and 17 us.  Both
// Grams are double-float sums of exact products, exchanged through distributed
// shared memory, and every CTA factors them redundantly in one warp's registers.
// The second Gram is I + E: its inverse factor is applied as Q1 + Q1 H with H
// known to about 1e-7 |E|.
#include "fourier_dev.cuh"

namespace lrs {
namespace {
using namespace fourier;

constexpr int kQT = 512;   // threads per CTA
constexpr int kQC = 8;     // CTAs (portable cluster size)

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
  __shared__ double2 Li[kMaxR * kMaxR];
  __shared__ float2 Lf[kMaxR * kMaxR];
  const int tid = threadIdx.x, w = tid >> 5, r = q.r, nw = kQT / 32;
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
  for (int pass = 0; pass < 2; ++pass) {
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
    if (w == 0 && !cchol_warp<R>(Gd, r, pass == 1, scratch, Li, Lf) && tid == 0 && rank == 0)
      report_error(q.err, kErrNotSPD, -1);
    __syncthreads();
    // rows times L^{-H} (pass 1) or I + H (pass 2), a thread per row
    for (int i = tid; i < cnt; i += kQT) {
      float2 z[R];
#pragma unroll
      for (int l = 0; l < R; ++l) z[l] = l < r ? Z[l * q.ldz + i] : make_float2(0.f, 0.f);
#pragma unroll
      for (int l = 0; l < R; ++l) {
        if (l >= r) break;
        float2 s = make_float2(0.f, 0.f);
#pragma unroll
        for (int p = 0; p <= l; ++p) s = ccfma(Lf[l * kMaxR + p], z[p], s);
        if (pass == 1) {
          s = cadd(s, z[l]);
          q.Q[static_cast<size_t>(l) * q.n + lo + i] = s;
        } else {
          Z[l * q.ldz + i] = s;
        }
      }
    }
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
