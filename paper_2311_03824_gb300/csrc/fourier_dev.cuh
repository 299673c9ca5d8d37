// Shared by the DFT operator's kernels: complex and double-float arithmetic,
// the frame geometry and the 2D FFT of a frame in shared memory.
#pragma once

#include <cuda_runtime.h>

#include "lrs_dev.cuh"
#include "lrs_internal.h"

namespace lrs {
namespace fourier {

// sweep profile slots: set-up and Gram, sparse DFTs, norms and vector
// updates, 2D FFTs with the frame's fills, HardThreshold, final stage,
// projections' Q^H v, projections' v - Q c
constexpr int kFProf = 8;
// static shared memory of the sweep (its profile counters), an upper bound
constexpr size_t kFStaticSmem = 256;
constexpr int kMaxR = 16;

// ------------------------------------------------------------ complex --
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
// acc += a * b
__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 acc) {
  acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
  acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
  return acc;
}
// acc += conj(a) * b
__device__ __forceinline__ float2 ccfma(float2 a, float2 b, float2 acc) {
  acc.x = fmaf(a.x, b.x, fmaf(a.y, b.y, acc.x));
  acc.y = fmaf(a.x, b.y, fmaf(-a.y, b.x, acc.y));
  return acc;
}
__device__ __forceinline__ double2 dcmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 dccmul(double2 a, double2 b) {  // conj(a) * b
  return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float cabs2(float2 a) { return fmaf(a.x, a.x, a.y * a.y); }

__device__ __forceinline__ float warp_sumf(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ------------------------------------------------------------ 2D FFT --
// Sides that are not powers of two take a direct DFT (frames of at most
// kDirectPer * blockDim.x pixels): each thread keeps its outputs in
// registers until every thread has read the frame.
constexpr int kDirectPer = 8;

__device__ inline void dft_direct_smem(float2* X, int nx, int ny, bool rows, const float2* tw,
                                bool inverse) {
  const int ld = ny + 1, n = nx * ny, len = rows ? ny : nx;
  float2 acc[kDirectPer];
#pragma unroll
  for (int u = 0; u < kDirectPer; ++u) {
    const int e = threadIdx.x + u * blockDim.x;
    float2 s = make_float2(0.f, 0.f);
    if (e < n) {
      const int row = e / ny, col = e - row * ny;
      const int j = rows ? col : row;  // output frequency along the transformed side
      int idx = 0;                     // j * k mod len
      for (int k = 0; k < len; ++k) {
        float2 w = tw[idx];
        if (inverse) w.y = -w.y;
        s = cfma(rows ? X[row * ld + k] : X[k * ld + col], w, s);
        idx += j;
        if (idx >= len) idx -= len;
      }
    }
    acc[u] = s;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kDirectPer; ++u) {
    const int e = threadIdx.x + u * blockDim.x;
    if (e < n) {
      const int row = e / ny, col = e - row * ny;
      X[row * ld + col] = acc[u];
    }
  }
  __syncthreads();
}

// Two radix-2 decimation-in-time stages s and s + 1 on the quad x0, x1, x2,
// x3 at offsets 0, h, 2h, 3h (h = 2^s) of a block of 4h: stage s pairs
// (x0, x1) and (x2, x3) with twiddle w1, stage s + 1 pairs (x0, x2) with w2a
// and (x1, x3) with w2b.  Every element gets the operations of the two
// stages run one after the other, in the same order, so the result is that
// of two single-stage passes, with one shared-memory round trip instead of two.
__device__ __forceinline__ void stage_pair(float2& x0, float2& x1, float2& x2, float2& x3,
                                           float2 w1, float2 w2a, float2 w2b, bool inverse) {
  if (inverse) {
    w1.y = -w1.y;
    w2a.y = -w2a.y;
    w2b.y = -w2b.y;
  }
  const float2 a0 = x0, a2 = x2;
  const float2 c1 = cmul(x1, w1), c3 = cmul(x3, w1);
  const float2 b0 = cadd(a0, c1), b1 = csub(a0, c1), b2 = cadd(a2, c3), b3 = csub(a2, c3);
  const float2 d2 = cmul(b2, w2a), d3 = cmul(b3, w2b);
  x0 = cadd(b0, d2);
  x2 = csub(b0, d2);
  x1 = cadd(b1, d3);
  x3 = csub(b1, d3);
}

// ------------------------------------------- Gram and Cholesky, complex --
// Entries (a, b <= a), A0 <= a < A1, of the Gram conj(W_b) W_a over this warp's
// rows, in double-float from exact products; the warp's sums to part.
// Sixteen warps share the rows, not the entries (21 entries of r = 6 on 16
// warps took two rounds), and a row of W is read once for several entries.
template <int A0, int A1>
__device__ __forceinline__ void cgram_part(const float2* W, size_t ld, int m, int r, int nw, float2* part) {
  if (A0 >= r) return;
  constexpr int NE = (A1 * (A1 + 1) - A0 * (A0 + 1)) / 2;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float xh[NE], xl[NE], yh[NE], yl[NE];
#pragma unroll
  for (int t = 0; t < NE; ++t) xh[t] = xl[t] = yh[t] = yl[t] = 0.f;
  for (int i = 32 * w + lane; i < m; i += 32 * nw) {
    float2 x[A1];
#pragma unroll
    for (int l = 0; l < A1; ++l) x[l] = l < r ? W[l * ld + i] : make_float2(0.f, 0.f);
    int t = 0;
#pragma unroll
    for (int a = A0; a < A1; ++a)
#pragma unroll
      for (int b = 0; b <= a; ++b, ++t) {
        df_fma(xh[t], xl[t], x[b].x, x[a].x);
        df_fma(xh[t], xl[t], x[b].y, x[a].y);
        if (b < a) {  // the diagonal is real
          df_fma(yh[t], yl[t], x[b].x, x[a].y);
          df_fma(yh[t], yl[t], -x[b].y, x[a].x);
        }
      }
  }
  // the real parts, then the imaginary parts of the entries off the diagonal,
  // in blocks of sixteen values: halving exchanges leave one per lane pair
  constexpr int NV = 2 * NE - (A1 - A0);
#pragma unroll
  for (int v0 = 0; v0 < NV; v0 += 16) {
    float h[16], l[16];
#pragma unroll
    for (int z = 0; z < 16; ++z) {
      h[z] = l[z] = 0.f;
      int v = 0;
#pragma unroll
      for (int a = A0; a < A1; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) {
          const int t = (a * (a + 1) - A0 * (A0 + 1)) / 2 + b;
          if (v == v0 + z) { h[z] = xh[t]; l[z] = xl[t]; }
          ++v;
          if (b < a) {
            if (v == v0 + z) { h[z] = yh[t]; l[z] = yl[t]; }
            ++v;
          }
        }
    }
#pragma unroll
    for (int k = 8, off = 16; k >= 1; k >>= 1, off >>= 1) {
      const bool up = lane & off;
#pragma unroll
      for (int z = 0; z < k; ++z) {
        const float sh = up ? h[z] : h[z + k], sl = up ? l[z] : l[z + k];
        const float kh = up ? h[z + k] : h[z], kl = up ? l[z + k] : l[z];
        h[z] = kh;
        l[z] = kl;
        df_add(h[z], l[z], __shfl_xor_sync(0xffffffffu, sh, off), __shfl_xor_sync(0xffffffffu, sl, off));
      }
    }
    df_add(h[0], l[0], __shfl_xor_sync(0xffffffffu, h[0], 1), __shfl_xor_sync(0xffffffffu, l[0], 1));
    // lane 2 z holds value v0 + z: row a's values start at a^2 (2 b and 2 b + 1,
    // the diagonal's real part last)
    if ((lane & 1) == 0 && v0 + (lane >> 1) < NV) part[A0 * A0 + v0 + (lane >> 1)] = make_float2(h[0], l[0]);
  }
}

// double-float complex
struct cdf {
  df x, y;
};
__device__ __forceinline__ cdf cdf_shfl(const cdf& a, int src) { return cdf{df_shfl(a.x, src), df_shfl(a.y, src)}; }
// c - a b, and c - a conj(b)
__device__ __forceinline__ cdf cdf_sub_mul(const cdf& c, const cdf& a, const cdf& b) {
  return cdf{df_sub(df_sub(c.x, df_mul(a.x, b.x)), df_mul(df{-a.y.h, -a.y.l}, b.y)),
             df_sub(df_sub(c.y, df_mul(a.x, b.y)), df_mul(a.y, b.x))};
}
__device__ __forceinline__ cdf cdf_sub_mulc(const cdf& c, const cdf& a, const cdf& b) {
  return cdf_sub_mul(c, a, cdf{b.x, df{-b.y.h, -b.y.l}});
}

// every entry of the lower triangle
template <int R>
__device__ __forceinline__ void cgram_warp(const float2* W, size_t ld, int m, int r, int nw, float2* part) {
  cgram_part<0, (R < 4 ? R : 4)>(W, ld, m, r, nw, part);
  if constexpr (R > 4) cgram_part<4, 6>(W, ld, m, r, nw, part);
  if constexpr (R > 6) cgram_part<6, 8>(W, ld, m, r, nw, part);
  if constexpr (R > 8) {
    cgram_part<8, 9>(W, ld, m, r, nw, part);
    cgram_part<9, 10>(W, ld, m, r, nw, part);
    cgram_part<10, 11>(W, ld, m, r, nw, part);
    cgram_part<11, 12>(W, ld, m, r, nw, part);
  }
  if constexpr (R > 12) {
    cgram_part<12, 13>(W, ld, m, r, nw, part);
    cgram_part<13, 14>(W, ld, m, r, nw, part);
    cgram_part<14, 15>(W, ld, m, r, nw, part);
    cgram_part<15, 16>(W, ld, m, r, nw, part);
  }
}

// One warp: the complex Cholesky factor L of M (Gd: the sums of cgram_warp) and
// L^{-1} in double-float in registers (lane = row, then lane = column; an FP64
// factor through shared memory took 31 K cycles at r = 6); Lf is L^{-1} rounded,
// with what the rounding of its (real) diagonal left in the imaginary part.
// False, and nothing written, when a pivot is below 1e-9 of its diagonal or
// outside float32's range (a NaN is).
template <int R>
__device__ bool cchol_df(const float2* Gd, int r, double2* Li, float2* Lf) {
  const int lane = threadIdx.x & 31;
  bool done = true;
  // M[i][q] = conj(W_i) W_q, q <= i: the conjugate of the sums
  cdf a[R];
  df inv[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    a[q] = cdf{df{0.f, 0.f}, df{0.f, 0.f}};
    if (q <= lane && lane < r) {
      const float2 x = Gd[lane * lane + 2 * q];
      a[q].x = df_norm(x.x, x.y);
      if (q < lane) {
        const float2 yv = Gd[lane * lane + 2 * q + 1];
        a[q].y = df_norm(-yv.x, -yv.y);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < R; ++j) {
    inv[j] = df{1.f, 0.f};
    if (j >= r || !done) continue;
    const df pv = df_shfl(a[j].x, j);
    const float dj = Gd[j * j + 2 * j].x;
    done = pv.h > 1e-9f * dj && pv.h > 1e-30f && pv.h < 1e30f;
    inv[j] = df_rsqrt(pv);
    a[j].x = df_mul(a[j].x, inv[j]);
    a[j].y = df_mul(a[j].y, inv[j]);
#pragma unroll
    for (int q = j + 1; q < R; ++q) a[q] = cdf_sub_mulc(a[q], a[j], cdf_shfl(a[j], q));
  }
  if (!done) return false;
  {
    cdf x[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {  // column lane of L^{-1}
      cdf t = cdf{df{0.f, 0.f}, df{0.f, 0.f}};
#pragma unroll
      for (int q = 0; q < i; ++q) t = cdf_sub_mul(t, cdf_shfl(a[q], i), x[q]);
      t.x = df_mul(t.x, inv[i]);
      t.y = df_mul(t.y, inv[i]);
      const df z = df{0.f, 0.f};
      x[i] = i < lane ? cdf{z, z} : i == lane ? cdf{inv[i], z} : t;
      if (lane < kMaxR && i < r) {
        Li[i * kMaxR + lane] = make_double2(static_cast<double>(x[i].x.h) + static_cast<double>(x[i].x.l),
                                              static_cast<double>(x[i].y.h) + static_cast<double>(x[i].y.l));
        Lf[i * kMaxR + lane] = make_float2(x[i].x.h, i == lane ? x[i].x.l : x[i].y.h);
      }
    }
  }
  __syncwarp();
  return true;
}

// The same in FP64 from the lower triangle G of M (ld kMaxR), the first part of
// scratch (2 kMaxR^2 + kMaxR / 2 values).  False when M is not positive
// definite; L is then I.
__device__ inline bool cchol_f64(int r, double2* scratch, double2* Li, float2* Lf) {
  const int lane = threadIdx.x & 31;
  const double2* G = scratch;
  double2* Lc = scratch + kMaxR * kMaxR;
  double* iL = reinterpret_cast<double*>(scratch + 2 * kMaxR * kMaxR);
  bool ok = true;
  for (int j = 0; j < r; ++j) {
    double2 t = make_double2(0.0, 0.0);
    if (lane >= j && lane < r) {
      t = G[lane * kMaxR + j];
      for (int p = 0; p < j; ++p) {
        const double2 x = Lc[lane * kMaxR + p], y = Lc[j * kMaxR + p];
        // t -= L[i][p] * conj(L[j][p])
        t.x -= x.x * y.x + x.y * y.y;
        t.y -= x.y * y.x - x.x * y.y;
      }
    }
    const double sj = __shfl_sync(0xffffffffu, t.x, j);
    if (!(sj > 1e-13 * G[j * kMaxR + j].x) || !(sj < 1e300)) {
      ok = false;
      break;
    }
    const double ij = rsqrt_newton(sj);
    if (lane == j) {
      Lc[j * kMaxR + j] = make_double2(sj * ij, 0.0);
      iL[j] = ij;
    } else if (lane > j && lane < r) {
      Lc[lane * kMaxR + j] = make_double2(t.x * ij, t.y * ij);
    }
    __syncwarp();
  }
  if (!ok && lane == 0) {
    for (int i = 0; i < r; ++i) {
      for (int p = 0; p < r; ++p) Lc[i * kMaxR + p] = make_double2(i == p ? 1.0 : 0.0, 0.0);
      iL[i] = 1.0;
    }
  }
  __syncwarp();
  if (lane < kMaxR) {  // column lane of L^{-1}
    const int cc = lane;
    for (int i = 0; i < r; ++i) {
      double2 t = make_double2(i == cc ? 1.0 : 0.0, 0.0);
      for (int p = cc; p < i; ++p) {
        const double2 q = dcmul(Lc[i * kMaxR + p], Li[p * kMaxR + cc]);
        t.x -= q.x;
        t.y -= q.y;
      }
      t = i < cc ? make_double2(0, 0) : make_double2(t.x * iL[i], t.y * iL[i]);
      Li[i * kMaxR + cc] = t;
      const float h = static_cast<float>(t.x);
      Lf[i * kMaxR + cc] =
          make_float2(h, static_cast<float>(i == cc ? t.x - static_cast<double>(h) : t.y));
    }
  }
  __syncwarp();
  return ok;
}

// ---------------------------------------------------------------- frames --
struct Geo {
  int nx, ny, lnx, lny, n;  // lnx / lny: log2 of a power-of-two side, else -1
  int L, sxL, syL, lL;      // L = lcm(nx, ny), L / nx, L / ny, log2 L (or -1)
  unsigned magic;           // ceil(2^32 / L) when v mod L may use it (below), else 0
};

// row, column of pixel e = row * ny + column, and an index modulo nx (ny)
__device__ __forceinline__ int frow(const Geo& g, int e) { return g.lny >= 0 ? e >> g.lny : e / g.ny; }
__device__ __forceinline__ int fcol(const Geo& g, int e) {
  return g.lny >= 0 ? e & (g.ny - 1) : e - (e / g.ny) * g.ny;
}
__device__ __forceinline__ int fwrapx(const Geo& g, int v) { return g.lnx >= 0 ? v & (g.nx - 1) : v % g.nx; }
__device__ __forceinline__ int fwrapy(const Geo& g, int v) { return g.lny >= 0 ? v & (g.ny - 1) : v % g.ny; }
// v mod L, 0 <= v < 2 max(nx, ny) L.  floor(v / L) = (v magic) >> 32 while
// v (magic L - 2^32) < 2^32, which v L < 2^32 ensures; the host sets magic
// only when 2 max(nx, ny) L^2 < 2^32 (an integer division costs about 20
// instructions, and the sparse DFTs take one per term).
__device__ __forceinline__ int fwrapL(const Geo& g, int v) {
  if (g.lL >= 0) return v & (g.L - 1);
  if (g.magic) return v - static_cast<int>(__umulhi(static_cast<unsigned>(v), g.magic)) * g.L;
  return v % g.L;
}
// where pixel or frequency e of a frame goes before fft2_smem
__device__ __forceinline__ int frev(const Geo& g, int e) {
  int x = frow(g, e), y = fcol(g, e);
  if (g.lnx > 0) x = static_cast<int>(__brev(static_cast<unsigned>(x)) >> (32 - g.lnx));
  if (g.lny > 0) y = static_cast<int>(__brev(static_cast<unsigned>(y)) >> (32 - g.lny));
  return x * (g.ny + 1) + y;
}

// In-place unitary 2D FFT of the frame X (nx rows x ny columns, row stride
// ny + 1 complex) in shared memory: along the rows, then along the columns,
// each by radix-2 decimation in time (a power-of-two side, lny / lnx its
// log2) or a direct DFT (lny / lnx = -1).  The input lies bit-reversed along
// the power-of-two sides (frev: the sweep scatters its samples there, which
// saves the two reversal passes); the output is in natural order.  tx[k] = exp(-2 pi i k / nx),
// k < nx (same for ty); inverse uses the conjugate twiddles.  All threads of
// the CTA call it.
__device__ inline void fft2_smem(float2* X, int nx, int ny, int lnx, int lny, const float2* tx,
                          const float2* ty, bool inverse) {
  const int ld = ny + 1, n = nx * ny;
  if (lny < 0) {
    dft_direct_smem(X, nx, ny, true, ty, inverse);
  } else {
    // consecutive threads take the same position in consecutive rows: the row
    // stride ny + 1 puts them in distinct banks, and they share the twiddle (a
    // broadcast)
    int s = 0;
    for (; s + 1 < lny; s += 2) {  // stages s and s + 1 in one pass
      const int h = 1 << s;
      for (int b = threadIdx.x; b < n / 4; b += blockDim.x) {
        const int t = lnx >= 0 ? b >> lnx : b / nx, row = b - t * nx;
        const int j = t & (h - 1), i0 = ((t >> s) << (s + 2)) + j;
        float2* x = X + row * ld;
        stage_pair(x[i0], x[i0 + h], x[i0 + 2 * h], x[i0 + 3 * h], ty[j * (ny >> (s + 1))],
                   ty[j * (ny >> (s + 2))], ty[(j + h) * (ny >> (s + 2))], inverse);
      }
      __syncthreads();
    }
    if (s < lny) {  // a last single stage
      const int half = 1 << s, step = ny >> (s + 1);
      for (int b = threadIdx.x; b < n / 2; b += blockDim.x) {
        const int t = lnx >= 0 ? b >> lnx : b / nx, row = b - t * nx;
        const int j = t & (half - 1), i1 = ((t >> s) << (s + 1)) + j, i2 = i1 + half;
        float2 w = ty[j * step];
        if (inverse) w.y = -w.y;
        const float2 a = X[row * ld + i1], c = cmul(X[row * ld + i2], w);
        X[row * ld + i1] = cadd(a, c);
        X[row * ld + i2] = csub(a, c);
      }
      __syncthreads();
    }
  }
  // the unitary scale 1/sqrt(n) is applied by the last column pass as it
  // stores (the same multiply as a separate pass), else by a pass of its own
  const float sc = rsqrtf(static_cast<float>(n));
  bool scaled = false;
  if (lnx < 0) {
    dft_direct_smem(X, nx, ny, false, tx, inverse);
  } else {
    int s = 0;
    for (; s + 1 < lnx; s += 2) {  // stages s and s + 1 in one pass
      const int h = 1 << s;
      const float f = (s + 2 == lnx) ? sc : 1.f;  // the last pass scales
      for (int b = threadIdx.x; b < n / 4; b += blockDim.x) {
        const int t = lny >= 0 ? b >> lny : b / ny, col = b - t * ny;
        const int j = t & (h - 1), i0 = ((t >> s) << (s + 2)) + j;
        float2* p0 = X + i0 * ld + col;
        float2 x0 = p0[0], x1 = p0[h * ld], x2 = p0[2 * h * ld], x3 = p0[3 * h * ld];
        stage_pair(x0, x1, x2, x3, tx[j * (nx >> (s + 1))], tx[j * (nx >> (s + 2))],
                   tx[(j + h) * (nx >> (s + 2))], inverse);
        if (s + 2 == lnx) {
          x0 = make_float2(x0.x * f, x0.y * f);
          x1 = make_float2(x1.x * f, x1.y * f);
          x2 = make_float2(x2.x * f, x2.y * f);
          x3 = make_float2(x3.x * f, x3.y * f);
        }
        p0[0] = x0;
        p0[h * ld] = x1;
        p0[2 * h * ld] = x2;
        p0[3 * h * ld] = x3;
      }
      __syncthreads();
    }
    if (s < lnx) {  // a last single stage
      const int half = 1 << s, step = nx >> (s + 1);
      for (int b = threadIdx.x; b < n / 2; b += blockDim.x) {
        const int t = lny >= 0 ? b >> lny : b / ny, col = b - t * ny;
        const int j = t & (half - 1), i1 = ((t >> s) << (s + 1)) + j, i2 = i1 + half;
        float2 w = tx[j * step];
        if (inverse) w.y = -w.y;
        const float2 a = X[i1 * ld + col], c = cmul(X[i2 * ld + col], w);
        const float2 o1 = cadd(a, c), o2 = csub(a, c);
        X[i1 * ld + col] = make_float2(o1.x * sc, o1.y * sc);
        X[i2 * ld + col] = make_float2(o2.x * sc, o2.y * sc);
      }
      __syncthreads();
    }
    scaled = lnx > 0;
  }
  if (!scaled) {
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
      const int row = e / ny, j = e - row * ny;
      X[row * ld + j].x *= sc;
      X[row * ld + j].y *= sc;
    }
    __syncthreads();
  }
}

}  // namespace fourier
}  // namespace lrs
