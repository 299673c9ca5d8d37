// AltGDmin-LR+S for the row-masked 2D DFT operator (the Fourier / dynamic-MRI
// case of Section I-A): A_k x = (F2 x)[Omega_k], A_k^H v = F2^H(zero-fill_k v),
// F2 the unitary 2D DFT of an nx x ny frame, rows indexed kx*ny + ky in natural
// order.  Complex throughout: transposes become conjugate transposes and
// HardThreshold ranks by the modulus.
//
// Per GDmin iteration (Algorithm 1):
//   FU = F2 U                      r forward 2D FFTs (shared by all frames),
//                                  so W_k = A_k U = FU[Omega_k, :]
//   sweep (one CTA per frame k)    fourier_sweep.cuh: W_k's orthonormal basis,
//                                  the IHT sweeps, then b_k and res_k = W_k b_k
//                                  + A_k s_k - y_k
//   K = sum_k zero-fill_k(res_k) b_k^H   k-space accumulation through the
//                                  inverse index of the masks (fixed order)
//   grad = F2^H K                  r inverse 2D FFTs (linearity of F2)
//   eta at t = 1, U <- Q(U - eta grad) by complex Cholesky-QR (cqr_cluster.cu;
//                                  cqr2 below for what one cluster does not hold).
// The initialisation forms L0 = [A_k^H (y_k - A_k s_k)] and its top-r left
// singular subspace by FP64 complex subspace iteration.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "fourier_sweep.cuh"

namespace lrs {
#define LRS_FSWEEP_R(X) X(2) X(4) X(6) X(8) X(12) X(16)
#define LRS_DECL(R) void* fsweep_kernel_r##R(bool pow2);  // fsweep_r*.cu
LRS_FSWEEP_R(LRS_DECL)
#undef LRS_DECL
namespace fourier {

// g = log2 G consecutive radix-2 decimation-in-time stages s .. s + g - 1 on
// the G elements x[t] at positions i0 + t h (h = 2^s, i0 = j mod h) of a block
// of G h along a side of length N.  Stage s + u pairs x[t] with x[t + d]
// (d = 2^u, bit u of t clear) with twiddle tw[(j + (t mod d) h) N / 2^(s+u+1)]:
// the butterflies of g single-stage passes, in the same order, on registers.
template <int G>
__device__ __forceinline__ void dit_group(float2 (&x)[G], int j, int h, int s, int N,
                                          const float2* tw, bool inverse) {
#pragma unroll
  for (int d = 1; d < G; d <<= 1) {
    const int sig = s + __ffs(d) - 1;  // the global stage
    const int step = N >> (sig + 1);
#pragma unroll
    for (int t = 0; t < G; ++t) {
      if (t & d) continue;
      float2 w = tw[(j + (t & (d - 1)) * h) * step];
      if (inverse) w.y = -w.y;
      const float2 a = x[t], c = cmul(x[t + d], w);
      x[t] = cadd(a, c);
      x[t + d] = csub(a, c);
    }
  }
}

// One pass of g stages over every line of one side: nl lines of N elements,
// element p of line l at X[l * ls + p * es].  Consecutive threads take the
// same group of consecutive lines (distinct banks for the row stride ny + 1,
// contiguous for columns; the twiddles are broadcasts).  With brev (the first
// pass, when a round of the CTA's threads holds whole lines) the inputs come
// from the bit-reversed positions: a round's reads all end before its writes.
// f scales the outputs.
template <int G>
__device__ void dit_pass(float2* X, int nl, int ls, int es, int N, int lN, int s,
                         const float2* tw, bool inverse, float f, bool brev) {
  const int h = 1 << s, gpl = N / G, g = __ffs(G) - 1, bd = blockDim.x;
  if (!brev) {
    for (int b = threadIdx.x; b < nl * gpl; b += bd) {
      const int line = b % nl, t = b / nl, j = t & (h - 1);
      const int i0 = ((t >> s) << (s + g)) + j;
      float2* L = X + line * ls;
      float2 x[G];
#pragma unroll
      for (int u = 0; u < G; ++u) x[u] = L[(i0 + u * h) * es];
      dit_group<G>(x, j, h, s, N, tw, inverse);
#pragma unroll
      for (int u = 0; u < G; ++u) L[(i0 + u * h) * es] = make_float2(x[u].x * f, x[u].y * f);
    }
    __syncthreads();
    return;
  }
  const int lpr = min(nl, bd / gpl);  // lines per round (>= 1: checked by the caller)
  for (int l0 = 0; l0 < nl; l0 += lpr) {
    const int b = threadIdx.x;
    const bool on = b < lpr * gpl && l0 + b % lpr < nl;
    float2 x[G];
    int line = 0, i0 = 0;
    if (on) {
      line = l0 + b % lpr;
      i0 = (b / lpr) << g;  // s = 0: h = 1, j = 0
      float2* L = X + line * ls;
#pragma unroll
      for (int u = 0; u < G; ++u) {
        const int src = static_cast<int>(__brev(static_cast<unsigned>(i0 + u)) >> (32 - lN));
        x[u] = L[src * es];
      }
      dit_group<G>(x, 0, 1, 0, N, tw, inverse);
    }
    __syncthreads();
    if (on) {
      float2* L = X + line * ls;
#pragma unroll
      for (int u = 0; u < G; ++u) L[(i0 + u) * es] = make_float2(x[u].x * f, x[u].y * f);
    }
    __syncthreads();
  }
}

// Radix-2 DIT transform of every line of one power-of-two side (lN = log2 N),
// in passes of up to kDitMax stages (a register budget: 3 in the FFT kernel,
// 2 inside the sweep); the last pass scales by f.  The bit reversal is read
// by the first pass, or (lines longer than the CTA's threads hold) swapped in
// a pass of its own.
template <int kDitMax>
__device__ __forceinline__ void dit_side(float2* X, int nl, int ls, int es, int N, int lN, const float2* tw,
                         bool inverse, float f) {
  if (lN <= 0) return;
  const bool fused = (N >> min(kDitMax, lN)) <= static_cast<int>(blockDim.x);
  if (!fused) {
    for (int e = threadIdx.x; e < nl * N; e += blockDim.x) {
      const int line = e % nl, p = e / nl;
      const int q = static_cast<int>(__brev(static_cast<unsigned>(p)) >> (32 - lN));
      if (q > p) {
        float2* L = X + line * ls;
        const float2 t = L[p * es];
        L[p * es] = L[q * es];
        L[q * es] = t;
      }
    }
    __syncthreads();
  }
  for (int s = 0; s < lN;) {
    const int g = min(kDitMax, lN - s);
    const float fs = (s + g == lN) ? f : 1.f;
    const bool br = fused && s == 0;
    switch (g) {
      case 1: dit_pass<2>(X, nl, ls, es, N, lN, s, tw, inverse, fs, br); break;
      case 2: dit_pass<4>(X, nl, ls, es, N, lN, s, tw, inverse, fs, br); break;
      default: dit_pass<(kDitMax >= 3 ? 8 : 4)>(X, nl, ls, es, N, lN, s, tw, inverse, fs, br); break;
    }
    s += g;
  }
}

// out[f] = F2(in[f]) (or F2^H) for frames f; frames are n-vectors in natural
// row-major order (pixel kx*ny + ky), frame f at in + f*n; its pixel e goes to
// out[e * es + f * fs].  One cluster of eight CTAs per frame: a CTA transforms
// its rows, then gathers its columns from the peers' shared memory and
// transforms them.  A power-of-two side by register passes, any other by a
// direct DFT.
//
// One CTA per frame kept r of the 152 SMs busy (26 us at 128 x 128, r = 6; with
// the k-space sums 53 us per iteration, now 26). A launch per side was faster
// there (39 us) and slower on frames up to 64 x 64 (22 us against 20; now 17).
constexpr int kFC = 8;    // CTAs per frame
constexpr int kFCT = 256;

struct FftCarve {
  size_t X1, X1b, X2, tx, ty, total;
  int rl, cl;  // rows and columns of a CTA
};
__host__ __device__ inline FftCarve fft_carve(const Geo& g) {
  FftCarve c;
  size_t o = 0;
  auto put = [&](size_t bytes) {
    const size_t at = o;
    o += al16(bytes);
    return at;
  };
  c.rl = (g.nx + kFC - 1) / kFC;
  c.cl = (g.ny + kFC - 1) / kFC;
  const size_t rows = static_cast<size_t>(c.rl) * (g.ny + 1) * 8;
  c.X1 = put(rows);
  c.X1b = put(g.lny < 0 ? rows : 0);
  c.X2 = put(static_cast<size_t>(c.cl) * (g.nx + 1) * 8);
  c.tx = put(static_cast<size_t>(g.nx) * 8);
  c.ty = put(static_cast<size_t>(g.ny) * 8);
  c.total = o;
  return c;
}

// entry p of the direct DFT of the line X (N elements)
__device__ __forceinline__ float2 dft_entry(const float2* X, const float2* t, int N, int p, bool inverse) {
  float2 v = make_float2(0.f, 0.f);
  int idx = 0;  // p k mod N
  for (int k = 0; k < N; ++k) {
    float2 w = t[idx];
    if (inverse) w.y = -w.y;
    v = cfma(X[k], w, v);
    idx += p;
    if (idx >= N) idx -= N;
  }
  return v;
}

__global__ void __launch_bounds__(kFCT) __cluster_dims__(kFC, 1, 1)
    fft_frames_kernel(Geo g, const float2* __restrict__ in, float2* __restrict__ out, size_t es, size_t fs,
                      int inverse, const float2* __restrict__ twx, const float2* __restrict__ twy) {
  extern __shared__ __align__(16) unsigned char sm[];
  const FftCarve c = fft_carve(g);
  float2* X1 = reinterpret_cast<float2*>(sm + c.X1);
  float2* X2 = reinterpret_cast<float2*>(sm + c.X2);
  float2* tx = reinterpret_cast<float2*>(sm + c.tx);
  float2* ty = reinterpret_cast<float2*>(sm + c.ty);
  const int rank = static_cast<int>(cluster_rank()), nx = g.nx, ny = g.ny;
  const size_t f = blockIdx.x / kFC;
  const int r0 = min(nx, rank * c.rl), nr = min(nx, r0 + c.rl) - r0;
  const int c0 = min(ny, rank * c.cl), nc = min(ny, c0 + c.cl) - c0;
  for (int k = threadIdx.x; k < nx; k += kFCT) tx[k] = __ldg(twx + k);
  for (int k = threadIdx.x; k < ny; k += kFCT) ty[k] = __ldg(twy + k);
  const float2* src = in + f * g.n + static_cast<size_t>(r0) * ny;
#pragma unroll 4
  for (int u = threadIdx.x; u < nr * ny; u += kFCT) {
    const int l = frow(g, u);
    X1[l * (ny + 1) + (u - l * ny)] = src[u];
  }
  __syncthreads();
  if (g.lny >= 0) {
    if (nr > 0) dit_side<3>(X1, nr, ny + 1, 1, ny, g.lny, ty, inverse != 0, 1.f);
  } else {
    float2* Xb = reinterpret_cast<float2*>(sm + c.X1b);
    for (int u = threadIdx.x; u < nr * ny; u += kFCT) {
      const int l = u / ny, p = u - l * ny;
      Xb[l * (ny + 1) + p] = dft_entry(X1 + l * (ny + 1), ty, ny, p, inverse != 0);
    }
    X1 = Xb;
  }
  cluster_sync_all();
#pragma unroll 4
  for (int u = threadIdx.x; u < nx * nc; u += kFCT) {
    const int x = u / nc, l = u - x * nc, from = x / c.rl;
    X2[l * (nx + 1) + x] = *peer_ptr(X1 + (x - from * c.rl) * (ny + 1) + c0 + l, from);
  }
  cluster_sync_all();  // also: no CTA leaves while a peer reads its rows
  if (g.lnx >= 0 && nc > 0) dit_side<3>(X2, nc, nx + 1, 1, nx, g.lnx, tx, inverse != 0, 1.f);
  const float sc = rsqrtf(static_cast<float>(g.n));
  for (int u = threadIdx.x; u < nx * nc; u += kFCT) {
    const int x = u / nc, l = u - x * nc;
    const float2* L = X2 + l * (nx + 1);
    const float2 v = g.lnx >= 0 ? L[x] : dft_entry(L, tx, nx, x, inverse != 0);
    out[(static_cast<size_t>(x) * ny + c0 + l) * es + f * fs] = make_float2(v.x * sc, v.y * sc);
  }
}

// K[l][w] = sum over the (k, i) with mask_k[i] = w of res_k[i] conj(b_k[l]).
// One warp per frequency w (a frequency every frame samples has q entries,
// most have a few): lanes take entries lane, lane + 32, ... of its list, then the
// 2 R sums at once by halving exchanges (fixed order; a butterfly per sum was
// 120 of the 200 instructions of a frequency with 32 entries at R = 6).
template <int R>
__global__ void __launch_bounds__(256) kspace_kernel(int n, int m, int r, const int* __restrict__ ptr,
                                                     const int* __restrict__ list,
                                                     const float2* __restrict__ RES,
                                                     const float2* __restrict__ B, float2* __restrict__ K) {
  constexpr int N = R <= 2 ? 4 : R <= 4 ? 8 : R <= 8 ? 16 : 32, G = 32 / N;
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (w >= n) return;  // uniform over the warp
  float v[N];
#pragma unroll
  for (int j = 0; j < N; ++j) v[j] = 0.f;
  const int t1 = ptr[w + 1];
  for (int t = ptr[w] + lane; t < t1; t += 32) {
    const int ki = list[t];
    const float2* b = B + static_cast<size_t>(ki / m) * r;
    const float2 rv = RES[ki];
#pragma unroll
    for (int l = 0; l < R; ++l)
      if (l < r) {
        const float2 s = cfma(rv, cconj(b[l]), make_float2(v[2 * l], v[2 * l + 1]));
        v[2 * l] = s.x;
        v[2 * l + 1] = s.y;
      }
  }
  const float s = reduce_multi<N>(v);
  const int j = lane / G;
  if (lane % G == 0 && j < 2 * r) reinterpret_cast<float*>(K + static_cast<size_t>(j >> 1) * n + w)[j & 1] = s;
}

// ---- complex column-reduced ops on r x n column-major matrices (l-major) ----
// partial Hermitian Grams: part[blk][a][b] = sum_j conj(X_ja) X_jb (a >= b)
// Gram partials of the rows [lo, hi) of the block Y (r x n column-major):
// out[a * r + b] = sum_j conj(y_a[j]) y_b[j] (a >= b) in FP64.  Entry p of the
// lower triangle (row-major) and row group g: the rows g, g + ng, ... of the
// range; the groups are added in order afterwards.  All threads of the block.
__device__ void cgram_rows(int n, int r, const float2* __restrict__ Y, int lo, int hi,
                           double2* __restrict__ out) {
  __shared__ double2 red[256];
  const int npair = r * (r + 1) / 2, ng = max(1, static_cast<int>(blockDim.x) / npair);
  const int t = threadIdx.x, p = t % npair, g = t / npair;
  int a = 0, b = p;
  while (b > a) b -= ++a;
  double sx = 0, sy = 0;
  if (g < ng && t < 256) {
    for (int j = lo + g; j < hi; j += ng) {
      const float2 xa = Y[static_cast<size_t>(a) * n + j], xb = Y[static_cast<size_t>(b) * n + j];
      sx += static_cast<double>(xa.x) * xb.x + static_cast<double>(xa.y) * xb.y;  // conj(x_a) x_b
      sy += static_cast<double>(xa.x) * xb.y - static_cast<double>(xa.y) * xb.x;
    }
    red[t] = make_double2(sx, sy);
  }
  __syncthreads();
  if (t < npair) {
    double2 s = red[t];
    for (int gg = 1; gg < ng; ++gg) {
      s.x += red[gg * npair + t].x;
      s.y += red[gg * npair + t].y;
    }
    out[a * r + b] = s;
  }
  __syncthreads();
}
// Z = X - eta G2 on the rows [lo, hi) (float32, as the sweep's update)
__device__ void cstep_rows(int n, int r, const float2* __restrict__ X, const float2* __restrict__ G2,
                           float e, float2* __restrict__ Xout, int lo, int hi) {
  for (int j = lo + threadIdx.x; j < hi; j += blockDim.x)
    for (int l = 0; l < r; ++l) {
      float2 v = X[static_cast<size_t>(l) * n + j];
      if (G2) {
        const float2 g = G2[static_cast<size_t>(l) * n + j];
        v = make_float2(fmaf(-e, g.x, v.x), fmaf(-e, g.y, v.y));
      }
      Xout[static_cast<size_t>(l) * n + j] = v;
    }
  __syncthreads();
}
__global__ void cgram_part_kernel(int n, int r, const float2* __restrict__ X,
                                  const float2* __restrict__ G2, const double* __restrict__ eta,
                                  float2* __restrict__ Xout, double2* __restrict__ part) {
  const int rows = (n + gridDim.x - 1) / gridDim.x;
  const int lo = blockIdx.x * rows, hi = min(n, lo + rows);
  if (Xout) cstep_rows(n, r, X, G2, eta ? static_cast<float>(*eta) : 0.f, Xout, lo, hi);
  cgram_rows(n, r, Xout ? Xout : X, lo, hi, part + static_cast<size_t>(blockIdx.x) * r * r);
}
// M = sum of partials (M[a][b] for a >= b = sum conj(x_a) x_b), Hermitian;
// M = R^H R with R = L^H (L lower from the Cholesky of M^T... we factor the
// matrix N[i][j] = sum conj(x_i) x_j directly: N = L L^H), Rinv = L^{-H}.
// (All threads of the block; the partials read through L2.)
__device__ void cchol_block(int r, int nblk, const double2* __restrict__ part,
                            double2* __restrict__ Rinv, int* err) {
  __shared__ double2 N[kMaxR * kMaxR], Lw[kMaxR * kMaxR], Li[kMaxR * kMaxR];
  __shared__ double iL[kMaxR];
  // the partials of each entry: one warp per entry, lanes over the blocks,
  // butterfly sum (fixed order); then warp 0 factors
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int t = threadIdx.x >> 5; t < r * r; t += nw) {
    const int a = t / r, b = t - a * r;
    if (b > a) continue;
    double sx = 0, sy = 0;
    for (int k = lane; k < nblk; k += 32) {
      const double2 v = __ldcg(part + static_cast<size_t>(k) * r * r + a * r + b);
      sx += v.x;
      sy += v.y;
    }
    sx = warp_sum(sx);
    sy = warp_sum(sy);
    if (lane == 0) {
      // N[a][b] = sum conj(x_a) x_b ; N[b][a] = conj(N[a][b])
      N[a * kMaxR + b] = make_double2(sx, sy);
      N[b * kMaxR + a] = make_double2(sx, -sy);
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    // (X^H X)[i][j] = sum conj(x_i) x_j = N[i][j]: factor N = L L^H, column j
    // by the lanes i >= j at once (lane j's entry is the pivot)
    bool ok = true;
    for (int j = 0; j < r; ++j) {
      double2 t = make_double2(0.0, 0.0);
      if (lane >= j && lane < r) {
        t = N[lane * kMaxR + j];
        for (int p = 0; p < j; ++p) {
          const double2 a = Lw[lane * kMaxR + p], b = Lw[j * kMaxR + p];
          t.x -= a.x * b.x + a.y * b.y;
          t.y -= a.y * b.x - a.x * b.y;
        }
      }
      const double s = __shfl_sync(0xffffffffu, t.x, j);
      if (!(s > 1e-13 * N[j * kMaxR + j].x) || !(s < 1e300)) {
        ok = false;
        break;
      }
      const double ij = rsqrt_newton(s);
      if (lane == j) {
        Lw[j * kMaxR + j] = make_double2(s * ij, 0);
        iL[j] = ij;
      } else if (lane > j && lane < r) {
        Lw[lane * kMaxR + j] = make_double2(t.x * ij, t.y * ij);
      }
      __syncwarp();
    }
    if (!ok) {
      if (lane == 0) {
        report_error(err, kErrNotSPD, -1);
        for (int i = 0; i < r; ++i) {
          for (int p = 0; p < r; ++p) Lw[i * kMaxR + p] = make_double2(i == p ? 1.0 : 0.0, 0);
          iL[i] = 1.0;
        }
      }
    }
    __syncwarp();
    if (lane < r) {
      const int cc = lane;
      for (int i = 0; i < r; ++i) {
        double2 t = make_double2(i == cc ? 1.0 : 0.0, 0.0);
        for (int p = cc; p < i; ++p) {
          const double2 q = dcmul(Lw[i * kMaxR + p], Li[p * kMaxR + cc]);
          t.x -= q.x;
          t.y -= q.y;
        }
        Li[i * kMaxR + cc] = (i < cc) ? make_double2(0, 0) : make_double2(t.x * iL[i], t.y * iL[i]);
      }
    }
    __syncwarp();
    // X^H X = L L^H  ->  with R = L^H (upper), Q = X R^{-1} = X L^{-H}:
    // Rinv[a][b] = (L^{-H})[a][b] = conj(Li[b][a])
    for (int t = lane; t < r * r; t += 32) {
      const int a = t / r, b = t - a * r;
      const double2 v = Li[b * kMaxR + a];
      Rinv[a * r + b] = make_double2(v.x, -v.y);
    }
  }
  __syncthreads();
}
__global__ void cchol_fin_kernel(int r, int nblk, const double2* __restrict__ part,
                                 double2* __restrict__ Rinv, int* err) {
  cchol_block(r, nblk, part, Rinv, err);
}
// Y = X Rinv (column-major complex, FP64 accumulation) for the entries
// (l, j), j in [lo, hi), of the block's range; Rinv r x r (row-major).
__device__ __forceinline__ float2 capply_one(int n, int r, const float2* __restrict__ X,
                                             const double2* __restrict__ Rinv, int l, int j) {
  double sx = 0, sy = 0;
  for (int p = 0; p <= l; ++p) {
    const float2 x = X[static_cast<size_t>(p) * n + j];
    const double2 q = Rinv[p * r + l];
    sx += x.x * q.x - x.y * q.y;
    sy += x.x * q.y + x.y * q.x;
  }
  return make_float2(static_cast<float>(sx), static_cast<float>(sy));
}
__global__ void capply_kernel(int n, int r, const float2* __restrict__ X,
                              const double2* __restrict__ Rinv, float2* __restrict__ Y) {
  const size_t t = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  if (t >= static_cast<size_t>(n) * r) return;
  const int l = static_cast<int>(t / n), j = static_cast<int>(t - static_cast<size_t>(l) * n);
  Y[t] = capply_one(n, r, X, Rinv, l, j);
}

// Grid barrier of a cooperative launch (every block resident): thread 0
// counts in and waits, bounded by wait_ns on the global timer, for
// `target` arrivals; on expiry the launch's error flag records a timeout and
// the block goes on (its results are then void, the host reports the error).
__device__ void grid_barrier(unsigned* ctr, unsigned target, int* err, unsigned long long wait_ns) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1u);
    unsigned long long t0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (;;) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
      if (v >= target) break;
      unsigned long long t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (t - t0 > wait_ns) {
        report_error(err, kErrTimeout, -1);
        break;
      }
      __nanosleep(64);
    }
    __threadfence();
  }
  __syncthreads();
}

// The whole complex Cholesky-QR2 of Z = X - eta G2 (G2 null: Z = X) in one
// cooperative launch of nblk blocks, block b on the same rows in every
// phase: Z and its Gram partials; barrier; every block factors the Gram
// (the same sums in the same order, so the same R^{-1}) and forms its rows of
// Z2 = Z R^{-1} and their Gram partials; barrier; R2^{-1} and U = Z2 R2^{-1}.
// The arithmetic is that of the separate kernels (gram, chol, apply twice).
__global__ void __launch_bounds__(256) cqr2_fused_kernel(int n, int r, const float2* X,
                                                         const float2* __restrict__ G2,
                                                         const double* __restrict__ eta,
                                                         float2* __restrict__ Z, float2* __restrict__ Z2,
                                                         float2* Uout, double2* __restrict__ part,
                                                         double2* __restrict__ part2, unsigned* bar,
                                                         int* err, unsigned long long wait_ns) {
  __shared__ double2 Rs[kMaxR * kMaxR];
  const int nb = gridDim.x, rows = (n + nb - 1) / nb;
  const int lo = blockIdx.x * rows, hi = min(n, lo + rows);
  const float2* Y = X;
  if (G2) {
    cstep_rows(n, r, X, G2, static_cast<float>(*eta), Z, lo, hi);
    Y = Z;
  }
  cgram_rows(n, r, Y, lo, hi, part + static_cast<size_t>(blockIdx.x) * r * r);
  grid_barrier(bar, static_cast<unsigned>(nb), err, wait_ns);
  cchol_block(r, nb, part, Rs, err);
  for (int t = threadIdx.x; t < (hi - lo) * r; t += blockDim.x) {
    const int l = t / (hi - lo), j = lo + (t - l * (hi - lo));
    Z2[static_cast<size_t>(l) * n + j] = capply_one(n, r, Y, Rs, l, j);
  }
  __syncthreads();
  cgram_rows(n, r, Z2, lo, hi, part2 + static_cast<size_t>(blockIdx.x) * r * r);
  grid_barrier(bar, 2u * static_cast<unsigned>(nb), err, wait_ns);
  cchol_block(r, nb, part2, Rs, err);
  for (int t = threadIdx.x; t < (hi - lo) * r; t += blockDim.x) {
    const int l = t / (hi - lo), j = lo + (t - l * (hi - lo));
    Uout[static_cast<size_t>(l) * n + j] = capply_one(n, r, Z2, Rs, l, j);
  }
}

// eta = c / sqrt(lambda_max(grad^H grad)), from the real 2r x 2r symmetric
// embedding [[Re, -Im], [Im, Re]] of the Hermitian Gram (every eigenvalue of
// the Gram appears twice).  The embedding is summed in FP64; a cyclic Jacobi
// in FP32 (normalised by the largest diagonal entry) gives an eigenvector v of
// the largest eigenvalue, and lambda_max is the FP64 Rayleigh quotient
// v^T A v / v^T v, whose error is second order in v's error.
__global__ void ceta_kernel(int r, int nblk, const double2* __restrict__ part, double c_eta,
                            double* __restrict__ eta) {
  __shared__ double A[2 * kMaxR][2 * kMaxR];
  __shared__ float Af[2 * kMaxR][2 * kMaxR + 1], V[2 * kMaxR][2 * kMaxR + 1];
  __shared__ int best;
  const int R2 = 2 * r, lane = threadIdx.x;
  if (lane >= 32) return;
  // entries of the lower triangle, each summed over the blocks in order
  for (int t = lane; t < r * r; t += 32) {
    const int a = t / r, b = t - a * r;
    if (b > a) continue;
    double sx = 0, sy = 0;
    for (int k = 0; k < nblk; ++k) {
      const double2 v = part[static_cast<size_t>(k) * r * r + a * r + b];
      sx += v.x;
      sy += v.y;
    }
    // N[a][b] = sx + i sy, N[b][a] = sx - i sy
    A[a][b] = sx; A[b][a] = sx; A[a + r][b + r] = sx; A[b + r][a + r] = sx;
    A[a + r][b] = sy; A[b][a + r] = sy; A[a][b + r] = -sy; A[b + r][a] = -sy;
  }
  __syncwarp();
  if (lane == 0) {
    double dmax = 0.0;
    for (int a = 0; a < R2; ++a) dmax = fmax(dmax, A[a][a]);
    const double sc = dmax > 0.0 ? 1.0 / dmax : 0.0;
    for (int a = 0; a < R2; ++a)
      for (int b = 0; b < R2; ++b) {
        Af[a][b] = static_cast<float>(A[a][b] * sc);
        V[a][b] = a == b ? 1.f : 0.f;
      }
    for (int sweep = 0; sweep < 30; ++sweep) {
      float off = 0.f, diag = 0.f;
      for (int a = 0; a < R2; ++a)
        for (int b = 0; b < R2; ++b) (a == b ? diag : off) += Af[a][b] * Af[a][b];
      if (off <= 1e-13f * diag) break;
      for (int p = 0; p < R2 - 1; ++p)
        for (int q2 = p + 1; q2 < R2; ++q2) {
          const float apq = Af[p][q2];
          if (apq == 0.f) continue;
          const float th = (Af[q2][q2] - Af[p][p]) / (2.f * apq);
          const float t = (th >= 0.f ? 1.f : -1.f) / (fabsf(th) + sqrtf(th * th + 1.f));
          const float cs = 1.f / sqrtf(t * t + 1.f), sn = t * cs;
          for (int kk = 0; kk < R2; ++kk) {
            const float akp = Af[kk][p], akq = Af[kk][q2];
            Af[kk][p] = cs * akp - sn * akq;
            Af[kk][q2] = sn * akp + cs * akq;
            const float vkp = V[kk][p], vkq = V[kk][q2];
            V[kk][p] = cs * vkp - sn * vkq;
            V[kk][q2] = sn * vkp + cs * vkq;
          }
          for (int kk = 0; kk < R2; ++kk) {
            const float apk = Af[p][kk], aqk = Af[q2][kk];
            Af[p][kk] = cs * apk - sn * aqk;
            Af[q2][kk] = sn * apk + cs * aqk;
          }
        }
    }
    int bi = 0;
    for (int a = 1; a < R2; ++a)
      if (Af[a][a] > Af[bi][bi]) bi = a;
    best = bi;
  }
  __syncwarp();
  // Rayleigh quotient in FP64: lane a holds (A v)_a v_a and v_a^2
  double num = 0.0, den = 0.0;
  if (lane < R2) {
    double y = 0.0;
    for (int b = 0; b < R2; ++b) y += A[lane][b] * static_cast<double>(V[b][best]);
    const double va = V[lane][best];
    num = y * va;
    den = va * va;
  }
  num = warp_sum(num);
  den = warp_sum(den);
  if (lane == 0) {
    const double lmax = den > 0.0 ? fmax(0.0, num / den) : 0.0;
    const double nrm = sqrt(lmax);
    *eta = (nrm > 0.0) ? c_eta / nrm : 0.0;
  }
}

// ---- subspace iteration of the initialisation: float32 products -----------
// P[k][l] = sum_j conj(H[k][j]) U[l][j] (U column-major: column l contiguous),
// in two steps.  Partials: block (kb, c) takes the 8 columns k = 8 kb + w (one
// per warp) over the chunk c of cs rows j; the chunk's U is staged in shared
// memory 256 rows at a time and serves all 8 warps (H read once, U once per 8
// columns); lanes over j, then a warp butterfly.  Then the chunks' partials
// are added in chunk order.
constexpr int kProjRows = 256;
__global__ void __launch_bounds__(256) cproject_part_kernel(int n, int q, int r, int cs,
                                                            const float2* __restrict__ H,
                                                            const float2* __restrict__ U,
                                                            float2* __restrict__ part) {
  __shared__ float2 Us[kMaxR][kProjRows];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int k = blockIdx.x * 8 + w, c = blockIdx.y;
  const int j0 = c * cs, j1 = min(n, j0 + cs);
  float2 acc[kMaxR];
#pragma unroll
  for (int l = 0; l < kMaxR; ++l) acc[l] = make_float2(0.f, 0.f);
  for (int jb = j0; jb < j1; jb += kProjRows) {
    const int nj = min(kProjRows, j1 - jb);
    __syncthreads();
    for (int t = threadIdx.x; t < r * kProjRows; t += blockDim.x) {
      const int l = t / kProjRows, jj = t - l * kProjRows;
      Us[l][jj] = jj < nj ? U[static_cast<size_t>(l) * n + jb + jj] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    if (k < q)
      for (int jj = lane; jj < nj; jj += 32) {
        const float2 h = H[static_cast<size_t>(k) * n + jb + jj];
#pragma unroll
        for (int l = 0; l < kMaxR; ++l)
          if (l < r) acc[l] = ccfma(h, Us[l][jj], acc[l]);
      }
  }
#pragma unroll
  for (int l = 0; l < kMaxR; ++l) {
    if (l >= r) break;
    const float sx = warp_sumf(acc[l].x), sy = warp_sumf(acc[l].y);
    if (lane == 0 && k < q) part[(static_cast<size_t>(c) * q + k) * r + l] = make_float2(sx, sy);
  }
}
__global__ void cproject_sum_kernel(int q, int r, int nc, const float2* __restrict__ part,
                                    float2* __restrict__ P) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= q * r) return;
  float2 s = make_float2(0.f, 0.f);
  for (int c = 0; c < nc; ++c) s = cadd(s, part[static_cast<size_t>(c) * q * r + t]);
  P[t] = s;
}
// Z[l][j] = sum_k H[k][j] P[k][l]: a block holds 32 columns j; its 8 warps
// take contiguous runs of k, and their sums are added in warp (k) order
__global__ void __launch_bounds__(256) cgrad_kernel(int n, int q, int r,
                                                    const float2* __restrict__ H,
                                                    const float2* __restrict__ P,
                                                    float2* __restrict__ Z) {
  __shared__ float2 red[8][kMaxR][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int j = blockIdx.x * 32 + lane;
  const int per = (q + 7) / 8, k0 = w * per, k1 = min(q, k0 + per);
  float2 acc[kMaxR];
#pragma unroll
  for (int l = 0; l < kMaxR; ++l) acc[l] = make_float2(0.f, 0.f);
  if (j < n)
    for (int k = k0; k < k1; ++k) {
      const float2 h = H[static_cast<size_t>(k) * n + j];
#pragma unroll
      for (int l = 0; l < kMaxR; ++l)
        if (l < r) acc[l] = cfma(h, P[static_cast<size_t>(k) * r + l], acc[l]);
    }
#pragma unroll
  for (int l = 0; l < kMaxR; ++l)
    if (l < r) red[w][l][lane] = acc[l];
  __syncthreads();
  // thread (l, lane) of the first r warps adds the 8 runs in order
  if (w < 8 && j < n)
    for (int l = w; l < r; l += 8) {
      float2 s = red[0][l][lane];
      for (int ww = 1; ww < 8; ++ww) s = cadd(s, red[ww][l][lane]);
      Z[static_cast<size_t>(l) * n + j] = s;
    }
}
// subspace change ||Un - Uo (Uo^H Un)||_F^2 of float32 blocks, in FP64:
// partials of D = Uo^H Un per row block, then per row block the residual
// (every block adds the partials of D in block order), then their sum
__global__ void coverlap_part_kernel(int n, int r, const float2* __restrict__ Uo,
                                     const float2* __restrict__ Un, double2* __restrict__ part) {
  const int rows = (n + gridDim.x - 1) / gridDim.x;
  const int lo = blockIdx.x * rows, hi = min(n, lo + rows);
  const int t = threadIdx.x, a = t / kMaxR, b = t - (t / kMaxR) * kMaxR;
  if (a >= r || b >= r) return;
  double sx = 0, sy = 0;
  for (int j = lo; j < hi; ++j) {
    const float2 x = Uo[static_cast<size_t>(a) * n + j], y = Un[static_cast<size_t>(b) * n + j];
    sx += static_cast<double>(x.x) * y.x + static_cast<double>(x.y) * y.y;
    sy += static_cast<double>(x.x) * y.y - static_cast<double>(x.y) * y.x;
  }
  part[static_cast<size_t>(blockIdx.x) * r * r + a * r + b] = make_double2(sx, sy);
}
__global__ void cresid_part_kernel(int n, int r, int nblk, const double2* __restrict__ part,
                                   const float2* __restrict__ Uo, const float2* __restrict__ Un,
                                   double* __restrict__ rpart) {
  __shared__ double2 D[kMaxR * kMaxR];
  __shared__ double red[32];
  for (int t = threadIdx.x; t < r * r; t += blockDim.x) {
    double2 s = make_double2(0, 0);
    for (int k = 0; k < nblk; ++k) {
      s.x += part[static_cast<size_t>(k) * r * r + t].x;
      s.y += part[static_cast<size_t>(k) * r * r + t].y;
    }
    D[t] = s;
  }
  __syncthreads();
  const int rows = (n + gridDim.x - 1) / gridDim.x;
  const int lo = blockIdx.x * rows, hi = min(n, lo + rows);
  double acc = 0.0;
  for (int e = threadIdx.x; e < (hi - lo) * r; e += blockDim.x) {
    const int l = e / (hi - lo), j = lo + (e - l * (hi - lo));
    const float2 un = Un[static_cast<size_t>(l) * n + j];
    double sx = un.x, sy = un.y;
    for (int p = 0; p < r; ++p) {
      const float2 u = Uo[static_cast<size_t>(p) * n + j];
      const double2 d = D[p * r + l];
      sx -= u.x * d.x - u.y * d.y;
      sy -= u.x * d.y + u.y * d.x;
    }
    acc += sx * sx + sy * sy;
  }
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s2 = 0;
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) s2 += red[w];
    rpart[blockIdx.x] = s2;
  }
}
__global__ void csum_fin_kernel(int nblk, const double* __restrict__ rpart, double* __restrict__ out) {
  if (threadIdx.x != 0) return;
  double s2 = 0;
  for (int k = 0; k < nblk; ++k) s2 += rpart[k];
  *out = s2;
}

}  // namespace fourier

using namespace fourier;

// --------------------------------------------------------------- driver --
struct FourierSolver {
  Geo g{};
  int m = 0, q = 0, r = 0, rho = 0;
  int tau0 = 10, tau = 3;
  double c_eta = 0.14;
  int power_iters = 1000;
  double power_tol = 1e-11;
  uint64_t seed = 0;
  cudaStream_t s = nullptr;
  int nblk = 1;
  int t = 0;
  bool have_eta = false;
  // device
  float2 *y = nullptr, *U = nullptr, *FU = nullptr, *B = nullptr, *S_val = nullptr, *RES = nullptr,
         *H = nullptr, *K = nullptr, *grad = nullptr, *Z = nullptr, *Z2 = nullptr, *twx = nullptr,
         *twl = nullptr,
         *twy = nullptr;
  int *mask = nullptr, *S_idx = nullptr, *iptr = nullptr, *ilist = nullptr, *err = nullptr;
  double2* part = nullptr;
  double2* part2 = nullptr;  // second Gram partials of the fused Cholesky-QR2
  unsigned* qbar = nullptr;  // its grid-barrier counter
  bool cluster = false;      // the matrix fits the cluster Cholesky-QR2
  bool coop = false;         // the fused Cholesky-QR2 fits one cooperative launch
  double2* rfac = nullptr;
  double* eta = nullptr;
  double* scal = nullptr;
  float2* vecs = nullptr;  // the sweep's m-vectors in global memory (large m)
  float2* Wk = nullptr;    // q x r x m: the sweep's W_k and Q_k (not when in shared memory)
  float2* AS = nullptr;    // q x m: A_k s_k - y_k from the last sweep's final stage
  int* asv = nullptr;      // q flags: AS[k] matches the current s_k
  unsigned long long* prof = nullptr;  // kFProf sweep cycle counters (profiling)
  void* sweep = nullptr;   // fsweep_kernel of the rank width
  bool lean = false;       // no room for its tables
  float fft_err = 0.f;     // FArgs
  int tb = 0, qmode = 0;   // its table's columns and Q_k's place (FArgs)
  size_t smem = 0;
};

// by_sample: out is n x nframes (frame f at out[e * nframes + f]), so that the
// sweep reads the values of a sampled frequency from one or two sectors, not
// from nframes
static cudaError_t fft_frames(FourierSolver* F, const float2* in, float2* out, int nframes,
                              bool inverse, bool by_sample) {
  const size_t es = by_sample ? nframes : 1, fs = by_sample ? 1 : F->g.n;
  fft_frames_kernel<<<kFC * nframes, kFCT, fft_carve(F->g).total, F->s>>>(F->g, in, out, es, fs, inverse ? 1 : 0,
                                                                          F->twx, F->twy);
  return cudaGetLastError();
}

// log2 of a power of two, -1 for any other side (direct DFT)
static int ilog2(int v) {
  int l = 0;
  while ((1 << l) < v) ++l;
  return (1 << l) == v ? l : -1;
}

FourierSolver* fourier_create(int nx, int ny, int m, int q, int r, int rho, int tau0, int tau,
                              double c_eta, int power_iters, double power_tol, uint64_t seed,
                              cudaStream_t s, std::string* msg) {
  FourierSolver* F = new FourierSolver();
  F->g.nx = nx;
  F->g.ny = ny;
  F->g.lnx = ilog2(nx);
  F->g.lny = ilog2(ny);
  F->g.n = nx * ny;
  {
    int a = nx, b = ny;  // L = lcm(nx, ny) by Euclid's gcd
    while (b) {
      const int t = a % b;
      a = b;
      b = t;
    }
    F->g.L = nx / a * ny;
    F->g.sxL = F->g.L / nx;
    F->g.syL = F->g.L / ny;
    F->g.lL = ilog2(F->g.L);
    const double span = 2.0 * std::max(nx, ny) * F->g.L * F->g.L;
    F->g.magic = span < 4294967296.0 ? static_cast<unsigned>((0x100000000ull + F->g.L - 1) / F->g.L) : 0u;
  }
  {  // 7 roundings a radix-2 stage; a direct DFT of N terms: (N + 4) |F| |x|, || |F| || = sqrt(N)
    auto side = [](int len, int l) { return l >= 0 ? 7.0 * l : (len + 4) * std::sqrt(static_cast<double>(len)); };
    F->fft_err = static_cast<float>(0x1p-24 * (side(nx, F->g.lnx) + side(ny, F->g.lny)));
  }
  F->m = m;
  F->q = q;
  F->r = r;
  F->rho = rho;
  F->tau0 = tau0;
  F->tau = tau;
  F->c_eta = c_eta;
  F->power_iters = power_iters;
  F->power_tol = power_tol;
  F->seed = seed;
  F->s = s;
  const int n = F->g.n;
  F->nblk = std::max(1, std::min(152, (n + 63) / 64));
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  F->cluster = cqr_cluster_fits(n, r);
  {  // the cooperative Cholesky-QR2 needs all its blocks resident at once
    int coop = 0, nsm = 0, per_sm = 0;
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cqr2_fused_kernel, 256, 0) != cudaSuccess)
      cudaGetLastError();
    F->coop = coop != 0 && per_sm * nsm >= F->nblk;
  }
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  // Shared memory of the sweep: what lets as many frames run at once as its
  // threads and the frames there are allow, else one frame's limit.  First the
  // sparse DFT's table (every column a support can have), then Q_k; the m-vectors
  // go to global memory when less than four columns of it fit beside them.
  // (The sweep also holds kFStaticSmem bytes of static shared memory.)
  const size_t room = static_cast<size_t>(optin) - kFStaticSmem;
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int ctas = std::max(1, std::min(kFT / fsweep_threads(n), (q + nsm - 1) / std::max(1, nsm)));
  const size_t share = ctas == 1 ? room : (room + 1024) / ctas - 1024 - kFStaticSmem;
  const int want = m >= 2 * nx ? std::min(std::max(1, rho), ny) : 0;
  bool vglob = false;
  auto total = [&](bool vg, int tb, bool qs) { return fcarve(F->g, m, r, rho, vg, tb, qs, false).total; };
  auto plan = [&](size_t limit, int least) {  // the most that fits, or false
    for (int vg = 0; vg < 2; ++vg) {
      int tb = want;
      while (tb > least && total(vg, tb, false) > limit) --tb;
      if (total(vg, tb, false) > limit) continue;
      vglob = vg != 0;
      F->tb = tb;
      const size_t frame = static_cast<size_t>(nx) * (ny + 1);
      F->qmode = tb == want && total(vg, tb, true) <= limit ? 1 : static_cast<size_t>(r) * m <= frame ? 2 : 0;
      F->smem = total(vg, tb, F->qmode == 1);
      return true;
    }
    return false;
  };
  if (!plan(share, std::min(want, 4)) && !plan(room, std::min(want, 4))) {
    F->lean = vglob = true;
    F->tb = F->qmode = 0;
    F->smem = fcarve(F->g, m, r, rho, true, 0, false, true).total;
  }
  if (F->smem > room || fft_carve(F->g).total > static_cast<size_t>(optin)) {
    *msg = "frame too large for one CTA's shared memory (n <= 16384 fits)";
    delete F;
    return nullptr;
  }
  switch (r <= 2 ? 2 : r <= 4 ? 4 : r <= 6 ? 6 : r <= 8 ? 8 : r <= 12 ? 12 : 16) {
#define LRS_CASE(R) case R: F->sweep = fsweep_kernel_r##R(F->g.lnx >= 0 && F->g.lny >= 0); break;
    LRS_FSWEEP_R(LRS_CASE)
#undef LRS_CASE
  }
  cudaFuncSetAttribute(F->sweep, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       smem_optin_limit() - static_cast<int>(kFStaticSmem));
  cudaFuncSetAttribute(fft_frames_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       smem_optin_limit());
  const size_t rr = static_cast<size_t>(r) * r;
  bool ok = cudaMallocAsync(reinterpret_cast<void**>(&F->y), sizeof(float2) * m * q, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->mask), sizeof(int) * m * q, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->U), sizeof(float2) * n * r, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->FU), sizeof(float2) * n * r, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->B), sizeof(float2) * q * r, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->S_idx), sizeof(int) * q * std::max(1, rho), F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->S_val), sizeof(float2) * q * std::max(1, rho), F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->RES), sizeof(float2) * m * q, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->H), sizeof(float2) * static_cast<size_t>(n) * q, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->K), sizeof(float2) * n * r, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->grad), sizeof(float2) * n * r, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->Z), sizeof(float2) * n * r, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->Z2), sizeof(float2) * n * r, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->twx), sizeof(float2) * nx, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->twl), sizeof(float2) * F->g.L, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->twy), sizeof(float2) * ny, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->iptr), sizeof(int) * (n + 1), F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->ilist), sizeof(int) * m * q, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->err), sizeof(int) * 2, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->part), sizeof(double2) * F->nblk * rr, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->part2), sizeof(double2) * F->nblk * rr, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->qbar), sizeof(unsigned), F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->rfac), sizeof(double2) * 2 * rr, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->eta), sizeof(double), F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->scal), sizeof(double) * 4, F->s) == cudaSuccess &&
            (F->qmode == 1 || cudaMallocAsync(reinterpret_cast<void**>(&F->Wk),
                                       sizeof(float2) * static_cast<size_t>(r) * m * q, F->s) == cudaSuccess) &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->AS),
                            sizeof(float2) * static_cast<size_t>(m) * q, F->s) == cudaSuccess &&
            cudaMallocAsync(reinterpret_cast<void**>(&F->asv), sizeof(int) * q, F->s) == cudaSuccess &&
            (!vglob || cudaMallocAsync(reinterpret_cast<void**>(&F->vecs),
                                       sizeof(float2) * 2 * static_cast<size_t>(m) * q, F->s) == cudaSuccess);
  if (!ok) {
    *msg = "device allocation failed";
    return F;  // caller frees
  }
  std::vector<float2> tw(std::max(nx, ny));
  for (int k = 0; k < nx; ++k) {
    const double a = -2.0 * M_PI * k / nx;
    tw[k] = make_float2(static_cast<float>(std::cos(a)), static_cast<float>(std::sin(a)));
  }
  cudaMemcpyAsync(F->twx, tw.data(), sizeof(float2) * nx, cudaMemcpyHostToDevice, F->s);
  for (int k = 0; k < ny; ++k) {
    const double a = -2.0 * M_PI * k / ny;
    tw[k] = make_float2(static_cast<float>(std::cos(a)), static_cast<float>(std::sin(a)));
  }
  cudaMemcpyAsync(F->twy, tw.data(), sizeof(float2) * ny, cudaMemcpyHostToDevice, F->s);
  std::vector<float2> twl(F->g.L);
  for (int k = 0; k < F->g.L; ++k) {
    const double a = -2.0 * M_PI * k / F->g.L;
    twl[k] = make_float2(static_cast<float>(std::cos(a)), static_cast<float>(std::sin(a)));
  }
  cudaMemcpyAsync(F->twl, twl.data(), sizeof(float2) * F->g.L, cudaMemcpyHostToDevice, F->s);
  cudaMemsetAsync(F->err, 0, 8, F->s);
  cudaMemsetAsync(F->asv, 0, sizeof(int) * q, F->s);
  cudaMemsetAsync(F->S_idx, 0, sizeof(int) * q * std::max(1, rho), F->s);
  cudaMemsetAsync(F->S_val, 0, sizeof(float2) * q * std::max(1, rho), F->s);
  cudaStreamSynchronize(F->s);  // the twiddle tables' host staging ends here
  return F;
}

void fourier_destroy(FourierSolver* F) {
  if (!F) return;
  void* ps[] = {F->y, F->mask, F->U, F->FU, F->B, F->S_idx, F->S_val, F->RES, F->H, F->K, F->grad,
                F->Z, F->Z2, F->twx, F->twy, F->twl, F->iptr, F->ilist, F->err, F->part, F->rfac, F->eta,
                F->scal,
                F->vecs, F->Wk, F->AS, F->asv, F->part2, F->qbar, F->prof};
  for (void* p : ps)
    if (p) cudaFreeAsync(p, F->s);
  cudaStreamSynchronize(F->s);
  delete F;
}

// masks: host int32 q x m (each column ascending, in [0, n)); y host or device
int fourier_set_measurements(FourierSolver* F, const void* y, const void* mask, int mem_kind,
                             std::string* msg) {
  const int n = F->g.n, m = F->m, q = F->q;
  std::vector<int> hm(static_cast<size_t>(m) * q);
  if (mem_kind) {
    if (cudaMemcpyAsync(hm.data(), mask, sizeof(int) * hm.size(), cudaMemcpyDeviceToHost, F->s) !=
            cudaSuccess ||
        cudaStreamSynchronize(F->s) != cudaSuccess) {
      *msg = "mask copy failed";
      return 4;
    }
  } else {
    std::memcpy(hm.data(), mask, sizeof(int) * hm.size());
  }
  for (int k = 0; k < q; ++k)
    for (int i = 0; i < m; ++i) {
      const int v = hm[static_cast<size_t>(k) * m + i];
      if (v < 0 || v >= n || (i > 0 && v <= hm[static_cast<size_t>(k) * m + i - 1])) {
        *msg = "mask row indices must be strictly ascending in [0, n)";
        return 1;
      }
    }
  // inverse index: for each frequency the (k, i) that sample it, k ascending
  std::vector<int> ptr(n + 1, 0), list(static_cast<size_t>(m) * q);
  for (int v : hm) ptr[v + 1]++;
  for (int w = 0; w < n; ++w) ptr[w + 1] += ptr[w];
  std::vector<int> fill(ptr.begin(), ptr.end() - 1);
  for (int k = 0; k < q; ++k)
    for (int i = 0; i < m; ++i) list[fill[hm[static_cast<size_t>(k) * m + i]]++] = k * m + i;
  cudaError_t e = cudaMemcpyAsync(F->mask, hm.data(), sizeof(int) * hm.size(), cudaMemcpyHostToDevice, F->s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(F->iptr, ptr.data(), sizeof(int) * ptr.size(), cudaMemcpyHostToDevice, F->s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(F->ilist, list.data(), sizeof(int) * list.size(), cudaMemcpyHostToDevice, F->s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(F->y, y, sizeof(float2) * m * q,
                        mem_kind ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, F->s);
  if (e == cudaSuccess) e = cudaMemsetAsync(F->asv, 0, sizeof(int) * q, F->s);  // new A_k
  if (e == cudaSuccess) e = cudaStreamSynchronize(F->s);
  if (e != cudaSuccess) {
    *msg = cudaGetErrorString(e);
    return 4;
  }
  F->t = 0;
  F->have_eta = false;
  return 0;
}

static cudaError_t launch_fsweep(FourierSolver* F, int mode, int tau) {
  FArgs a{};
  a.g = F->g;
  a.m = F->m;
  a.q = F->q;
  a.r = F->r;
  a.rho = F->rho;
  a.tau = tau;
  a.mode = mode;
  a.y = F->y;
  a.mask = F->mask;
  a.FU = F->FU;
  a.S_idx = F->S_idx;
  a.S_val = F->S_val;
  a.B = F->B;
  a.RES = F->RES;
  a.H = F->H;
  a.twx = F->twx;
  a.twy = F->twy;
  a.twl = F->twl;
  a.err = F->err;
  a.vecs = F->vecs;
  a.Wk = F->Wk;
  a.AS = F->AS;
  a.asv = F->asv;
  a.prof = F->prof;
  a.tb = F->tb;
  a.lean = F->lean;
  a.fft_err = F->fft_err;
  a.qmode = F->qmode;
  void* args[] = {&a};
  return cudaLaunchKernel(F->sweep, dim3(F->q), dim3(fsweep_threads(F->g.n)), args, F->smem, F->s);
}

// complex Cholesky-QR2 of Zin (r x n column-major) into Uout
static cudaError_t ccholqr2(FourierSolver* F, const float2* Zin, float2* Uout) {
  const int n = F->g.n, r = F->r;
  const unsigned nb = static_cast<unsigned>((static_cast<size_t>(n) * r + 255) / 256);
  cgram_part_kernel<<<F->nblk, 256, 0, F->s>>>(n, r, Zin, nullptr, nullptr, nullptr, F->part);
  cchol_fin_kernel<<<1, 256, 0, F->s>>>(r, F->nblk, F->part, F->rfac, F->err);
  capply_kernel<<<nb, 256, 0, F->s>>>(n, r, Zin, F->rfac, F->Z2);
  cgram_part_kernel<<<F->nblk, 256, 0, F->s>>>(n, r, F->Z2, nullptr, nullptr, nullptr, F->part);
  cchol_fin_kernel<<<1, 256, 0, F->s>>>(r, F->nblk, F->part, F->rfac + r * r, F->err);
  capply_kernel<<<nb, 256, 0, F->s>>>(n, r, F->Z2, F->rfac + r * r, Uout);
  return cudaGetLastError();
}

// Z = X - eta G2 (G2 null: Z = X), then Uout = its Cholesky-QR2: one cluster
// launch when the matrix fits its shared memory (r up to 11 at n = 16384), else
// one cooperative launch when every block fits on the device at once, else the
// separate kernels.  Uout may be X.
static cudaError_t cqr2(FourierSolver* F, const float2* X, const float2* G2, const double* eta,
                        float2* Uout) {
  const int n = F->g.n, r = F->r;
  if (F->cluster) return cqr_cluster(n, r, X, G2, eta, Uout, F->err, F->s);
  if (F->coop) {
    cudaError_t e = cudaMemsetAsync(F->qbar, 0, sizeof(unsigned), F->s);
    if (e != cudaSuccess) return e;
    float2* Z = F->Z;
    float2* Z2 = F->Z2;
    unsigned long long wait_ns = 10ull * 1000 * 1000 * 1000;
    int nn = n, rr = r;
    void* args[] = {&nn, &rr, const_cast<float2**>(&X), const_cast<float2**>(&G2),
                    const_cast<double**>(&eta), &Z, &Z2, &Uout, &F->part, &F->part2, &F->qbar,
                    &F->err, &wait_ns};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(cqr2_fused_kernel),
                                       dim3(F->nblk), dim3(256), args, 0, F->s);
  }
  if (G2) {
    cgram_part_kernel<<<F->nblk, 256, 0, F->s>>>(n, r, X, G2, eta, F->Z, F->part);
    return ccholqr2(F, F->Z, Uout);
  }
  return ccholqr2(F, X, Uout);
}

int fourier_check_error(FourierSolver* F, std::string* msg) {
  int e[2] = {0, 0};
  cudaMemcpyAsync(e, F->err, sizeof(e), cudaMemcpyDeviceToHost, F->s);
  if (cudaStreamSynchronize(F->s) != cudaSuccess) {
    *msg = "CUDA error";
    return 4;
  }
  if (e[0]) {
    cudaMemsetAsync(F->err, 0, 8, F->s);
    *msg = e[0] == kErrNotSPD ? "r x r Gram matrix not positive definite" : "NaN/Inf in the iteration";
    if (e[1] >= 0) *msg += " (frame " + std::to_string(e[1]) + ")";
    return 5;
  }
  return 0;
}

int fourier_init(FourierSolver* F, std::string* msg) {
  const int n = F->g.n, q = F->q, r = F->r;
  cudaError_t e = launch_fsweep(F, kModeInit, F->tau0);  // s_k and the L0 columns in H
  // Complex subspace iteration for the top-r left singular vectors of L0:
  // float32 products P = L0^H U and Z = L0 P, complex Cholesky-QR2 of Z with
  // FP64 r x r factors, until the subspace moves by less than power_tol or by
  // less than the float32 resolution of U (4 eps sqrt(n r): a converged
  // float32 iteration moves U by its rounding).
  const size_t nr = static_cast<size_t>(n) * r;
  float2 *Uo = nullptr, *Zf = nullptr, *Pf = nullptr;
  double* rpart = nullptr;
  if (e == cudaSuccess) e = cudaMallocAsync(reinterpret_cast<void**>(&Uo), nr * 8, F->s);
  if (e == cudaSuccess) e = cudaMallocAsync(reinterpret_cast<void**>(&Zf), nr * 8, F->s);
  if (e == cudaSuccess) e = cudaMallocAsync(reinterpret_cast<void**>(&Pf), static_cast<size_t>(q) * r * 8, F->s);
  // the projection's row chunks: about two blocks per SM in all
  const int kb = (q + 7) / 8;
  int cs = (n + std::max(1, 304 / kb) - 1) / std::max(1, 304 / kb);
  cs = (cs + kProjRows - 1) / kProjRows * kProjRows;
  const int nc = (n + cs - 1) / cs;
  float2* Pp = nullptr;
  if (e == cudaSuccess) e = cudaMallocAsync(reinterpret_cast<void**>(&Pp), static_cast<size_t>(nc) * q * r * 8, F->s);
  if (e == cudaSuccess) e = cudaMallocAsync(reinterpret_cast<void**>(&rpart), F->nblk * sizeof(double), F->s);
  // start: deterministic complex Gaussian block
  std::vector<float2> st(nr);
  uint64_t sd = F->seed * 0x9E3779B97F4A7C15ull + 0x2545F4914F6CDD1Dull;
  auto nxt = [&]() {
    uint64_t z = (sd += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
  };
  for (auto& v : st) {
    const double u1 = ((nxt() >> 11) + 1.0) * 0x1.0p-53, u2 = (nxt() >> 11) * 0x1.0p-53;
    const double rad = std::sqrt(-2.0 * std::log(u1));
    v = make_float2(static_cast<float>(rad * std::cos(6.283185307179586 * u2)),
                    static_cast<float>(rad * std::sin(6.283185307179586 * u2)));
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(Zf, st.data(), nr * 8, cudaMemcpyHostToDevice, F->s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(F->s);  // the host block may go
  if (e == cudaSuccess) e = cqr2(F, Zf, nullptr, nullptr, F->U);
  const double floor_tol = 4.0 * 0x1.0p-24 * std::sqrt(static_cast<double>(nr));
  const double tol = std::max(F->power_tol, floor_tol);
  for (int it = 0; it < F->power_iters && e == cudaSuccess; ++it) {
    e = cudaMemcpyAsync(Uo, F->U, nr * 8, cudaMemcpyDeviceToDevice, F->s);
    cproject_part_kernel<<<dim3(kb, nc), 256, 0, F->s>>>(n, q, r, cs, F->H, Uo, Pp);
    cproject_sum_kernel<<<(q * r + 255) / 256, 256, 0, F->s>>>(q, r, nc, Pp, Pf);
    cgrad_kernel<<<(n + 31) / 32, 256, 0, F->s>>>(n, q, r, F->H, Pf, Zf);
    if (e == cudaSuccess) e = cqr2(F, Zf, nullptr, nullptr, F->U);
    if (e == cudaSuccess && ((it % 5) == 4 || it + 1 == F->power_iters)) {
      coverlap_part_kernel<<<F->nblk, 256, 0, F->s>>>(n, r, Uo, F->U, F->part);
      cresid_part_kernel<<<F->nblk, 256, 0, F->s>>>(n, r, F->nblk, F->part, Uo, F->U, rpart);
      csum_fin_kernel<<<1, 32, 0, F->s>>>(F->nblk, rpart, F->scal);
      double chg2 = 0;
      e = cudaGetLastError();
      if (e == cudaSuccess) e = cudaMemcpyAsync(&chg2, F->scal, sizeof(double), cudaMemcpyDeviceToHost, F->s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(F->s);
      if (e == cudaSuccess && std::sqrt(std::max(0.0, chg2)) < tol) break;
    }
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(F->s);
  for (void* p : {static_cast<void*>(Uo), static_cast<void*>(Zf), static_cast<void*>(Pf),
                  static_cast<void*>(Pp), static_cast<void*>(rpart)})
    if (p) cudaFreeAsync(p, F->s);
  // b_k = (A_k U0)^+ (y_k - A_k s_k)
  if (e == cudaSuccess) e = fft_frames(F, F->U, F->FU, r, false, true);
  if (e == cudaSuccess) e = launch_fsweep(F, kModeLS, 0);
  if (e != cudaSuccess) {
    *msg = cudaGetErrorString(e);
    return 4;
  }
  F->t = 0;
  F->have_eta = false;
  return fourier_check_error(F, msg);
}

// evs (optional): 4 events per iteration, recorded before FU = F2 U, after
// the per-frame sweep, after the gradient and after the QR.
int fourier_iterate(FourierSolver* F, int iters, std::string* msg, cudaEvent_t* evs) {
  const int n = F->g.n, r = F->r;
  for (int i = 0; i < iters; ++i) {
    cudaEvent_t* ev = evs ? evs + 4 * static_cast<size_t>(i) : nullptr;
    if (ev) cudaEventRecord(ev[0], F->s);
    cudaError_t e = fft_frames(F, F->U, F->FU, r, false, true);            // FU = F2 U
    if (e == cudaSuccess) e = launch_fsweep(F, kModeIter, F->tau);   // per-frame work
    if (ev) cudaEventRecord(ev[1], F->s);
    {
      const dim3 nb((n + 7) / 8), nt(256);
      switch (r <= 2 ? 2 : r <= 4 ? 4 : r <= 6 ? 6 : r <= 8 ? 8 : r <= 12 ? 12 : 16) {
#define LRS_CASE(R) \
  case R: kspace_kernel<R><<<nb, nt, 0, F->s>>>(n, F->m, r, F->iptr, F->ilist, F->RES, F->B, F->K); break;
        LRS_FSWEEP_R(LRS_CASE)
#undef LRS_CASE
      }
    }
    if (e == cudaSuccess) e = fft_frames(F, F->K, F->grad, r, true, false);  // grad = F2^H K
    if (e == cudaSuccess && F->t == 0) {
      cgram_part_kernel<<<F->nblk, 256, 0, F->s>>>(n, r, F->grad, nullptr, nullptr, nullptr, F->part);
      ceta_kernel<<<1, 32, 0, F->s>>>(r, F->nblk, F->part, F->c_eta, F->eta);
    }
    if (ev) cudaEventRecord(ev[2], F->s);
    // Z = U - eta grad, then complex Cholesky-QR2
    if (e == cudaSuccess) e = cqr2(F, F->U, F->grad, F->eta, F->U);
    if (ev) cudaEventRecord(ev[3], F->s);
    if (e != cudaSuccess) {
      *msg = cudaGetErrorString(e);
      return 4;
    }
    F->t += 1;
  }
  return fourier_check_error(F, msg);
}

// host/device copies of U (n x r column-major = our layout), B, S
int fourier_get(FourierSolver* F, void* U, void* B, int* S_idx, void* S_val, int mem_kind) {
  const cudaMemcpyKind k = mem_kind ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  const size_t n = F->g.n;
  if (U) cudaMemcpyAsync(U, F->U, sizeof(float2) * n * F->r, k, F->s);
  if (B) cudaMemcpyAsync(B, F->B, sizeof(float2) * F->q * F->r, k, F->s);
  if (S_idx && F->rho) cudaMemcpyAsync(S_idx, F->S_idx, sizeof(int) * F->q * F->rho, k, F->s);
  if (S_val && F->rho) cudaMemcpyAsync(S_val, F->S_val, sizeof(float2) * F->q * F->rho, k, F->s);
  return cudaStreamSynchronize(F->s) == cudaSuccess ? 0 : 4;
}

int fourier_set_state(FourierSolver* F, const void* U, const void* B, const int* S_idx,
                      const void* S_val, int t, double eta, int mem_kind) {
  const cudaMemcpyKind k = mem_kind ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  const size_t n = F->g.n;
  cudaMemcpyAsync(F->U, U, sizeof(float2) * n * F->r, k, F->s);
  cudaMemcpyAsync(F->B, B, sizeof(float2) * F->q * F->r, k, F->s);
  if (F->rho) {
    const int* si = S_idx;
    const float* sv = static_cast<const float*>(S_val);
    if (!mem_kind) {
      cudaMemcpyAsync(F->S_idx, S_idx, sizeof(int) * F->q * F->rho, k, F->s);
      cudaMemcpyAsync(F->S_val, S_val, sizeof(float2) * F->q * F->rho, k, F->s);
      si = F->S_idx;
      sv = reinterpret_cast<const float*>(F->S_val);
    }
    if (set_support(F->g.n, F->q, F->rho, 2, si, sv, F->S_idx, reinterpret_cast<float*>(F->S_val), F->s) !=
        cudaSuccess)
      return 4;
  }
  cudaMemsetAsync(F->asv, 0, sizeof(int) * F->q, F->s);  // a new s_k
  cudaMemcpyAsync(F->eta, &eta, sizeof(double), cudaMemcpyHostToDevice, F->s);
  F->t = t;
  return cudaStreamSynchronize(F->s) == cudaSuccess ? 0 : 4;
}

double fourier_eta(FourierSolver* F) {
  double v = 0;
  cudaMemcpyAsync(&v, F->eta, sizeof(double), cudaMemcpyDeviceToHost, F->s);
  cudaStreamSynchronize(F->s);
  return F->t ? v : 0.0;
}
int fourier_t(FourierSolver* F) { return F->t; }

// Kernels one steady iteration launches: F2 U, the sweep, the k-space
// reduction, F2^H K, and the step with its Cholesky-QR2 (one launch, else the
// Gram partials and two factorisations and applications).
int fourier_launches_per_iteration(FourierSolver* F) { return 4 + (F->cluster || F->coop ? 1 : 6); }
int fourier_fused_qr(FourierSolver* F) { return F->cluster || F->coop ? 1 : 0; }

// Sweep cycle counters: enable (allocate, zero) and read-and-zero.
int fourier_prof_enable(FourierSolver* F) {
  if (F->prof) return 0;
  if (cudaMallocAsync(reinterpret_cast<void**>(&F->prof), sizeof(unsigned long long) * kFProf, F->s) !=
      cudaSuccess)
    return 3;  // LRS_ERR_OOM
  return cudaMemsetAsync(F->prof, 0, sizeof(unsigned long long) * kFProf, F->s) == cudaSuccess
             ? 0
             : 4;  // LRS_ERR_CUDA
}
int fourier_prof_read(FourierSolver* F, unsigned long long* out, int len) {
  if (!F->prof) return 2;  // LRS_ERR_STATE
  const int n = len < kFProf ? len : kFProf;
  if (cudaMemcpyAsync(out, F->prof, sizeof(unsigned long long) * n, cudaMemcpyDeviceToHost, F->s) !=
          cudaSuccess ||
      cudaMemsetAsync(F->prof, 0, sizeof(unsigned long long) * kFProf, F->s) != cudaSuccess ||
      cudaStreamSynchronize(F->s) != cudaSuccess)
    return 4;  // LRS_ERR_CUDA
  return 0;
}

}  // namespace lrs
