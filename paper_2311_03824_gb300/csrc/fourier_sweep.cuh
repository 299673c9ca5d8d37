// The per-frame sweep of the DFT operator (Algorithm 1's column work with the
// IHT of Algorithm 2), one CTA per frame with the frame in shared memory.
//
// Projection.  W_k = (F2 U)[Omega_k] is orthonormalised once per frame: Q = W
// L^{-H} with W^H W = L L^H, so P_perp v = v - Q (Q^H v), b = L^{-H} Q^H (y -
// A s), and the sweeps hold no r x r solve (FP64 solves with four barriers
// each took 23 of 244 K cycles at 64 x 64, r = 4).
//
// Sparse DFTs.  A x of a support in few frame columns goes column by column:
// T(kx, c) = sum of x over the column's pixels, then one term per column at
// every sampled frequency, rho nx + columns m terms in the place of rho m (128
// x 128 blob supports: 66 K, not 168 K).  Both steps are bound by shared-memory
// wavefronts, so the second one reads T as broadcasts (the samples of a warp
// share kx) and looks a twiddle up once per run of up to four adjacent columns,
// stepping it by exp(-2 pi i ky / ny) along the run.  (A^H u) on the support is
// the transpose.
//
// Sweeps without a 2D FFT.  A column of A_k has norm N = sqrt(m / n), so
// |(A^H u)_j| <= N ||u||; after a pass has computed g at u_ref with the
// support kept, also <= max_{j off the support} |g_j| + N ||u - u_ref||, and
// ||u - u_ref|| <= sum of mu ||P A g_G|| over the sweeps since.  When mu times
// that bound (1 + 1e-3) is below the smallest new |v_i| on the support,
// HardThreshold keeps the support whatever g is off it, and the sweep needs g
// on the support alone: no 2D FFT (the 1e-3 covers the rounding of mu and the
// norms; the FFT's own, at most fft_err ||u_ref||, is added to the max |g_j|,
// however small).  The test is made on the
// sweep's own mu and v; a sweep that fails it takes the FFT.
//
// Bound: instruction issue (593 K warp instructions per 128 x 128 frame, issue
// slots 43 % used, shared-memory wavefronts 28 % of peak). A sweep with an FFT
// costs 31 K cycles for it and about 12 K for HardThreshold, one without 20 K for
// the adjoint. n = 128 x 128, q = 256, r = 6, m = 2048, rho = 82, relative error
// 2e-2: 497 -> 353 us with F2 U; 64 x 64, q = 99, r = 4: 145 -> 112; 20 x 20, q =
// 400: 215 -> 55.
#pragma once

#include "fourier_dev.cuh"

namespace lrs {
namespace fourier {

struct FArgs {
  Geo g;
  int m, q, r, rho, tau, mode;
  int tb;               // support columns of the sparse DFT's table beside the frame
  int lean;             // no room for the tables (fcarve)
  float fft_err;        // bound of the 2D FFT's rounding error in the 2-norm
  int qmode;            // Q_k: 0 in Wk, 1 in shared memory, 2 in the frame's place
                        // while no FFT needs it (kept in Wk meanwhile)
  const float2* y;      // q x m
  const int* mask;      // q x m
  const float2* FU;     // n x r (row e: F2 u_l at frequency e)
  int* S_idx;           // q x rho
  float2* S_val;        // q x rho
  float2* B;            // q x r
  float2* RES;          // q x m: W b + A s - y (iteration)
  float2* H;            // q x n: L0 columns A^H (y - A s) (initialisation)
  const float2* twx;
  const float2* twy;
  const float2* twl;    // exp(-2 pi i j / L), j < L = lcm(nx, ny)
  int* err;
  float2* vecs;         // q x 2m: the two m-vectors of the sweep, when they do
                        // not fit shared memory beside the frame
  float2* Wk;           // q x r x m: W_k, then Q_k (row l of frame k
                        // contiguous), unless qmode is 1
  float2* AS;           // q x m: A_k s_k - y_k of the last sweep's final stage
  int* asv;             // q: 1 while AS[k] belongs to the current s_k
  unsigned long long* prof;  // optional kFProf cycle counters (thread 0 of each CTA)
};

// Threads per frame, by its size: a 20 x 20 frame has 400 pixels and a few
// hundred samples, and four 128-thread CTAs per SM (128 registers) take the
// place of one of 512 threads that mostly waits at barriers (a 20 x 20 solve of
// 400 frames: with the rest of this sweep 215 -> 55 us).  On the largest frames 768 and 1024
// threads were slower (128 x 128: 353 us per sweep with 512, 382 with 768, 449
// with 1024: spills and more redundant work per warp).
constexpr int kFT = 512;  // at most
__host__ __device__ constexpr int fsweep_threads(int n) { return n <= 512 ? 128 : n < 2048 ? 256 : kFT; }

struct FCarve {
  size_t X, tx, ty, tl, dv, ev, msk, rptr, sp, sv, gv, vn, ord, ent, cs, ccol, pcs, Li, Lf, red,
      scal, hist, cand, cl, T, Q, total;
};

// HardThreshold candidates of the threshold filter
constexpr int kCandCap = 512;
// what the squares of a norm lose below float32's range
constexpr float kTinySq = 4e-41f;

__host__ __device__ inline size_t al16(size_t x) { return (x + 15) & ~size_t(15); }

// Shared-memory carve of the sweep; with vglob the two m-vectors live in global
// memory (FArgs::vecs) and take no space.  T for tb support columns, Q when own_q.
// lean (tall frames, or m near n, that leave no room): no T (tb is 0, sparse
// products term by term), the Gram's scratch in the frame's place.
__host__ __device__ inline FCarve fcarve(const Geo& g, int m, int r, int rho, bool vglob, int tb, bool own_q, bool lean) {
  FCarve c;
  size_t o = 0;
  const size_t rh = rho > 0 ? rho : 1;
  const int nw = fsweep_threads(g.n) / 32;
  const size_t mv = vglob ? 0 : al16(static_cast<size_t>(m) * 8);
  const size_t frame = static_cast<size_t>(g.nx) * (g.ny + 1) * 8;
  const int rw = r <= 2 ? 2 : r <= 4 ? 4 : r <= 6 ? 6 : r <= 8 ? 8 : r <= 12 ? 12 : 16;  // rank width
  const size_t gram = (2 * kMaxR * kMaxR + kMaxR) * 16 + static_cast<size_t>(nw + 1) * rw * rw * 8;
  auto put = [&](size_t bytes) {
    const size_t at = o;
    o += al16(bytes);
    return at;
  };
  c.X = put(lean && gram > frame ? gram : frame);
  c.tx = put(static_cast<size_t>(g.nx) * 8);
  c.ty = put(static_cast<size_t>(g.ny) * 8);
  c.tl = put(static_cast<size_t>(g.L) * 8);
  c.dv = put(mv);
  c.ev = put(mv);
  c.msk = put(static_cast<size_t>(m) * 4);
  c.rptr = put(tb ? static_cast<size_t>(g.nx + 1) * 4 : 0);
  c.sp = put(rh * 4);
  c.sv = put(rh * 8);
  c.gv = put(rh * 8);
  c.vn = put(rh * 8);
  c.ord = put(tb ? rh * 2 : 0);
  c.ent = put(tb ? rh * 4 : 0);
  c.cs = put(tb ? (rh + 1) * 2 : 0);
  c.ccol = put(tb ? rh * 2 : 0);
  c.pcs = put(tb ? (rh + 1) * 2 : 0);
  c.Li = put(kMaxR * kMaxR * 16);
  c.Lf = put(kMaxR * kMaxR * 8);
  c.red = put(static_cast<size_t>(nw) * 2 * kMaxR * 4);
  c.scal = put(static_cast<size_t>(4) * nw * 4);
  c.hist = put(256 * 4 + 64);
  c.cand = put((rh + 72) * 4);
  c.cl = put(static_cast<size_t>(kCandCap) * 8);
  // T; before the first sweep, the Gram's partial sums, G and L
  const size_t tab = tb ? static_cast<size_t>(tb | 1) * g.nx * 8 : 0;
  c.T = put(lean ? 0 : tab > gram ? tab : gram);
  c.Q = put(own_q ? static_cast<size_t>(r) * m * 8 : 0);
  c.total = o;
  return c;
}

struct FCtx {
  Geo g;
  int m, r, rho, k, nw;
  float2* X;
  float2* tx;      // full-period twiddles exp(-2 pi i k / nx), k < nx
  float2* ty;
  float2* tl;      // exp(-2 pi i j / L), j < L = lcm(nx, ny)
  float2* dv;
  float2* ev;
  int* msk;
  int* rptr;       // samples of frequency row kx: rptr[kx] .. rptr[kx + 1]
  int* sp;         // support pixels
  float2* sv;      // support values
  float2* gv;      // g on the support
  int* spo;        // the support before the last HardThreshold, in the place
                   // of gv (read before it)
  float2* vn;      // s - mu g on the support
  // the support by (column, row): entry of each position, its row and (above 16
  // bits) column index; the distinct columns' first positions (and the end), and
  // the columns; the first column of each piece (at most four adjacent columns;
  // and the end)
  unsigned short *ord, *cs, *ccol, *pcs;
  int* ent;
  double2* Li;     // L^{-1} (ld kMaxR)
  float2* Lf;
  float* red;
  float* scal;     // 4 slots of warp sums
  int* hist;
  int* cand;
  unsigned long long* cl;  // threshold-filter candidates: key, then ~pixel
  float2* T;       // tables of the sparse DFTs
  float2* Q;       // W_k, then Q_k (r x m, row l contiguous)
  int* err;
};

// block sums of one float: fput, a barrier, fget on every thread (the warps'
// partials in warp order)
__device__ __forceinline__ void fput(const FCtx& C, int slot, float v) {
  v = warp_sumf(v);
  if ((threadIdx.x & 31) == 0) C.scal[slot * C.nw + (threadIdx.x >> 5)] = v;
}
__device__ __forceinline__ float fget(const FCtx& C, int slot) {
  const float4* from = reinterpret_cast<const float4*>(C.scal + slot * C.nw);
  float s = 0.f;
#pragma unroll 4
  for (int w = 0; w < C.nw / 4; ++w) {
    const float4 x = from[w];
    s += x.x;
    s += x.y;
    s += x.z;
    s += x.w;
  }
  return s;
}
// and block maxima of nonnegative floats
__device__ __forceinline__ void fput_max(const FCtx& C, int slot, float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) C.scal[slot * C.nw + (threadIdx.x >> 5)] = v;
}
__device__ __forceinline__ float fget_max(const FCtx& C, int slot) {
  float s = 0.f;
  for (int w = 0; w < C.nw; ++w) s = fmaxf(s, C.scal[slot * C.nw + w]);
  return s;
}

// ------------------------------------------------------------ sparse DFTs --
constexpr int kSdPer = 4;  // frequencies a thread takes at once

// out = A x for the pixels sp[e], values v[e], term by term: frames with fewer
// samples than two per row, where a table over kx is no saving, and those that
// leave no room for it.  Ends with a barrier.
__device__ inline void sparse_direct(const FCtx& C, const float2* v, int nnz, float2* out) {
  const float sc = rsqrtf(static_cast<float>(C.g.n));
  const int bd = blockDim.x;
  for (int i0 = threadIdx.x; i0 < C.m; i0 += kSdPer * bd) {
    int kx[kSdPer], ky[kSdPer];
    float2 acc[kSdPer];
#pragma unroll
    for (int u = 0; u < kSdPer; ++u) {
      const int i = i0 + u * bd, om = i < C.m ? C.msk[i] : 0;
      kx[u] = frow(C.g, om);
      ky[u] = fcol(C.g, om);
      acc[u] = make_float2(0.f, 0.f);
    }
    for (int e = 0; e < nnz; ++e) {
      const int p = C.sp[e], qx = frow(C.g, p) * C.g.sxL, qy = fcol(C.g, p) * C.g.syL;
      const float2 ve = v[e];
#pragma unroll
      for (int u = 0; u < kSdPer; ++u)
        acc[u] = cfma(C.tl[fwrapL(C.g, kx[u] * qx + ky[u] * qy)], ve, acc[u]);
    }
#pragma unroll
    for (int u = 0; u < kSdPer; ++u) {
      const int i = i0 + u * bd;
      if (i < C.m) out[i] = make_float2(acc[u].x * sc, acc[u].y * sc);
    }
  }
  __syncthreads();
}

// out = A x by support columns (head of the file); T holds cap columns (four
// or all of them at least).  Scratch: vn.  Ends with a barrier.
__device__ inline void sparse_cols(const FCtx& C, int np, const float2* v, float2* out, int cap) {
  float2* T = C.T;
  const float sc = rsqrtf(static_cast<float>(C.g.n));
  const int bd = blockDim.x, nx = C.g.nx, ng = max(1, bd / nx);
  for (int e = threadIdx.x; e < C.rho; e += bd) C.vn[e] = v[C.ord[e]];  // in column order
  __syncthreads();
  int j0 = 0;
  do {
    int j1 = j0;
    while (j1 < np && C.pcs[j1 + 1] - C.pcs[j0] <= cap) ++j1;
    const bool last = j1 >= np;
    const int cA = np ? C.pcs[j0] : 0, nc = np ? C.pcs[j1] - cA : 0, ldc = nc | 1;
    // T: a thread takes kx and a block of columns, its pixels in one flat loop
    for (int t = threadIdx.x; t < nx * ng; t += bd) {
      const int grp = t / nx, kx = t - grp * nx, kxL = kx * C.g.sxL;
      const int c0 = nc * grp / ng, c1 = nc * (grp + 1) / ng;
      if (c0 == c1) continue;
      float2* Tk = T + kx * ldc - cA;
      const int p1 = C.cs[cA + c1];
      int p = C.cs[cA + c0], c = cA + c0;
      float2 acc = make_float2(0.f, 0.f);
      for (; p < p1; p += 4) {
        int cc[4];
        float2 w[4], x[4];
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const int at = min(p + z, p1 - 1);
          cc[z] = C.ent[at];
          x[z] = C.vn[at];
          w[z] = C.tl[fwrapL(C.g, kxL * (cc[z] & 0xffff))];
          cc[z] >>= 16;
        }
#pragma unroll
        for (int z = 0; z < 4; ++z)
          if (p + z < p1) {
            if (cc[z] != c) {
              Tk[c] = acc;
              acc = make_float2(0.f, 0.f);
              c = cc[z];
            }
            acc = cfma(w[z], x[z], acc);
          }
      }
      Tk[c] = acc;
    }
    __syncthreads();
    for (int i0 = threadIdx.x; i0 < C.m; i0 += kSdPer * bd) {
      const float2* Tk[kSdPer];
      int ky[kSdPer];
      float2 acc[kSdPer], wy[kSdPer];
#pragma unroll
      for (int u = 0; u < kSdPer; ++u) {
        const int i = i0 + u * bd, om = i < C.m ? C.msk[i] : 0;
        Tk[u] = T + frow(C.g, om) * ldc - cA;
        ky[u] = fcol(C.g, om) * C.g.syL;
        wy[u] = C.tl[fwrapL(C.g, ky[u])];
        acc[u] = j0 && i < C.m ? out[i] : make_float2(0.f, 0.f);
      }
      for (int j = j0; j < j1; ++j) {
        const int c0 = C.pcs[j], len = C.pcs[j + 1] - c0, py = C.ccol[c0];
        float2 w[kSdPer];
#pragma unroll
        for (int u = 0; u < kSdPer; ++u) {
          w[u] = C.tl[fwrapL(C.g, ky[u] * py)];
          acc[u] = cfma(w[u], Tk[u][c0], acc[u]);
        }
#pragma unroll
        for (int z = 1; z < 4; ++z)
          if (z < len)
#pragma unroll
            for (int u = 0; u < kSdPer; ++u) {
              w[u] = cmul(w[u], wy[u]);
              acc[u] = cfma(w[u], Tk[u][c0 + z], acc[u]);
            }
      }
#pragma unroll
      for (int u = 0; u < kSdPer; ++u) {
        const int i = i0 + u * bd;
        if (i < C.m) out[i] = last ? make_float2(acc[u].x * sc, acc[u].y * sc) : acc[u];
      }
    }
    __syncthreads();
    j0 = j1;
  } while (j0 < np);
}

// gv = (A^H u) on the support, by its columns: V(kx, c) = sum over the samples
// of row kx (four lanes share a row's samples for one piece of columns, and the
// rows go from the lowest frequency up: a variable-density mask has most of its
// samples there), then one term per kx and pixel.  V takes T, cap columns at a time.  Ends with a barrier.
__device__ inline void sparse_adjoint(const FCtx& C, int np, const float2* u, int cap) {
  const int nx = C.g.nx, ny = C.g.ny, lane = threadIdx.x & 31, w = threadIdx.x >> 5, part = lane & 3;
  const float sc = rsqrtf(static_cast<float>(C.g.n));
  for (int j0 = 0; j0 < np;) {
    int j1 = j0;
    while (j1 < np && C.pcs[j1 + 1] - C.pcs[j0] <= cap) ++j1;
    const int nj = j1 - j0, cA = C.pcs[j0], cB = C.pcs[j1], ldc = (cB - cA) | 1, total = 4 * nx * nj;
    float2* V = C.T - cA;
    for (int t = threadIdx.x; t - lane < total; t += blockDim.x) {
      const int tt = min(t >> 2, nx * nj - 1), kq = tt / nj, j = j0 + tt - kq * nj;
      const int kx = kq & 1 ? nx - 1 - (kq >> 1) : kq >> 1;
      const int c0 = C.pcs[j], len = C.pcs[j + 1] - c0, py = C.ccol[c0];
      const int e1 = C.rptr[kx + 1], kb = kx * ny;
      float2 acc[4];
#pragma unroll
      for (int z = 0; z < 4; ++z) acc[z] = make_float2(0.f, 0.f);
      for (int i = C.rptr[kx] + part; i < e1; i += 8) {
        float2 ui[2], wy[2], x[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const bool in = i + 4 * h < e1;
          const int at = in ? i + 4 * h : i, ky = (C.msk[at] - kb) * C.g.syL;
          ui[h] = u[at];
          if (!in) ui[h] = make_float2(0.f, 0.f);
          wy[h] = C.tl[ky];
          x[h] = C.tl[fwrapL(C.g, ky * py)];
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) acc[0] = ccfma(x[h], ui[h], acc[0]);
#pragma unroll
        for (int z = 1; z < 4; ++z)
          if (z < len)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              x[h] = cmul(x[h], wy[h]);
              acc[z] = ccfma(x[h], ui[h], acc[z]);
            }
      }
#pragma unroll
      for (int z = 0; z < 4; ++z)
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
          acc[z].x += __shfl_xor_sync(0xffffffffu, acc[z].x, o);
          acc[z].y += __shfl_xor_sync(0xffffffffu, acc[z].y, o);
        }
      if (t < total && part < len)
        V[kx * ldc + c0 + part] = part == 0 ? acc[0] : part == 1 ? acc[1] : part == 2 ? acc[2] : acc[3];
    }
    __syncthreads();
    const int pB = C.cs[cB];
    for (int e0 = C.cs[cA] + 4 * w; e0 < pB; e0 += 4 * C.nw) {
      float v[8];
      int p[4], c[4];
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        const int e = min(e0 + z, pB - 1);
        p[z] = (C.ent[e] & 0xffff) * C.g.sxL;
        c[z] = C.ent[e] >> 16;
        v[2 * z] = v[2 * z + 1] = 0.f;
      }
      for (int kx = lane; kx < nx; kx += 32)
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const float2 s = ccfma(C.tl[fwrapL(C.g, kx * p[z])], V[kx * ldc + c[z]],
                                 make_float2(v[2 * z], v[2 * z + 1]));
          v[2 * z] = s.x;
          v[2 * z + 1] = s.y;
        }
      const float s = reduce_multi<8>(v) * sc;  // lane 4 j: value j
      const int e = e0 + (lane >> 3);
      if ((lane & 3) == 0 && e < pB) reinterpret_cast<float*>(C.gv + C.ord[e])[(lane >> 2) & 1] = s;
    }
    __syncthreads();
    j0 = j1;
  }
}

// The (distinct) support by columns; returns the number of pieces.  Ends with a
// barrier.
__device__ inline int support_cols(const FCtx& C, int* np_s) {
  int* key = C.cand;
  const int rho = C.rho;
  for (int e = threadIdx.x; e < rho; e += blockDim.x)
    key[e] = (fcol(C.g, C.sp[e]) << 16) | frow(C.g, C.sp[e]);
  __syncthreads();
  for (int e = threadIdx.x; e < rho; e += blockDim.x) {
    const int mine = key[e];
    int pos = 0;
#pragma unroll 8
    for (int f = 0; f < rho; ++f) pos += key[f] < mine;
    C.ord[pos] = static_cast<unsigned short>(e);
    C.ent[pos] = mine;  // the column's index in its place below
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int nc = 0, np = 0, run = 0, before = -2;  // run: index of the last run's first column
    for (int e0 = 0; e0 < rho; e0 += 32) {
      const int e = e0 + lane, col = e < rho ? C.ent[e] >> 16 : -1;
      int prev = __shfl_up_sync(0xffffffffu, col, 1);
      if (lane == 0) prev = before;
      before = __shfl_sync(0xffffffffu, col, 31);
      const bool st = e < rho && col != prev;
      const unsigned b = __ballot_sync(0xffffffffu, st), upto = (2u << lane) - 1u;
      const int c = nc + __popc(b & upto) - 1;  // this entry's column index
      const unsigned rb = __ballot_sync(0xffffffffu, st && col != prev + 1) & upto;
      // the run's first column: that of the last run start at or before this lane
      const int at = rb ? 31 - __clz(rb) : 0;
      const int cr = __shfl_sync(0xffffffffu, c, at);
      const int r0 = rb ? cr : run;
      const bool ps = st && ((c - r0) & 3) == 0;
      const unsigned pb = __ballot_sync(0xffffffffu, ps);
      __syncwarp();
      if (e < rho) C.ent[e] = (c << 16) | (C.ent[e] & 0xffff);
      if (st) {
        C.cs[c] = static_cast<unsigned short>(e);
        C.ccol[c] = static_cast<unsigned short>(col);
      }
      if (ps) C.pcs[np + __popc(pb & upto) - 1] = static_cast<unsigned short>(c);
      nc += __popc(b);
      np += __popc(pb);
      run = __shfl_sync(0xffffffffu, r0, 31);
    }
    if (lane == 0) {
      C.cs[nc] = static_cast<unsigned short>(rho);
      C.pcs[np] = static_cast<unsigned short>(nc);
      *np_s = np;
    }
  }
  __syncthreads();
  return *np_s;
}

// ------------------------------------------------------------- projection --
// rows of Q a thread takes at once
constexpr int kApPer = 4;

// cf = Q^H v on every thread (float32, the warps' partials in warp order).  One
// barrier; the caller has another one before the next call.
template <int R>
__device__ void fcoefs(const FCtx& C, const float2* v, float2 (&cf)[R]) {
  constexpr int N = R <= 2 ? 4 : R <= 4 ? 8 : R <= 8 ? 16 : 32;
  const int bd = blockDim.x, m = C.m, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float2 acc[R];
#pragma unroll
  for (int l = 0; l < R; ++l) acc[l] = make_float2(0.f, 0.f);
  for (int i0 = threadIdx.x; i0 < m; i0 += kApPer * bd) {
    float2 vi[kApPer];
#pragma unroll
    for (int u = 0; u < kApPer; ++u) vi[u] = i0 + u * bd < m ? v[i0 + u * bd] : make_float2(0.f, 0.f);
#pragma unroll
    for (int l = 0; l < R; ++l) {
      const float2* q = C.Q + static_cast<size_t>(l < C.r ? l : 0) * m + i0;
#pragma unroll
      for (int u = 0; u < kApPer; ++u)
        if (l < C.r && i0 + u * bd < m) acc[l] = ccfma(q[u * bd], vi[u], acc[l]);
    }
  }
  float x[N];
#pragma unroll
  for (int j = 0; j < N; ++j) x[j] = j < 2 * R ? (j & 1 ? acc[j / 2 < R ? j / 2 : 0].y : acc[j / 2 < R ? j / 2 : 0].x) : 0.f;
  const float t = reduce_multi<N>(x);
  constexpr int G = 32 / N;
  if (lane % G == 0) C.red[w * 2 * kMaxR + lane / G] = t;
  __syncthreads();
  // every warp adds the partials, lane = value, and hands them round
  float s = 0.f;
#pragma unroll 8
  for (int ww = 0; ww < C.nw; ++ww) s += C.red[ww * 2 * kMaxR + lane];
#pragma unroll
  for (int l = 0; l < R; ++l)
    cf[l] = make_float2(__shfl_sync(0xffffffffu, s, 2 * l), __shfl_sync(0xffffffffu, s, 2 * l + 1));
}

// v <- v + sign Q cf; returns this thread's part of ||v||^2
template <int R>
__device__ float fapply(const FCtx& C, float2* v, const float2 (&cf)[R], float sign) {
  const int bd = blockDim.x, m = C.m;
  float nn = 0.f;
  for (int i0 = threadIdx.x; i0 < m; i0 += kApPer * bd) {
    float2 s[kApPer];
#pragma unroll
    for (int u = 0; u < kApPer; ++u) s[u] = i0 + u * bd < m ? v[i0 + u * bd] : make_float2(0.f, 0.f);
#pragma unroll
    for (int l = 0; l < R; ++l) {
      const float2* q = C.Q + static_cast<size_t>(l < C.r ? l : 0) * m + i0;
      const float2 x = make_float2(sign * cf[l].x, sign * cf[l].y);
#pragma unroll
      for (int u = 0; u < kApPer; ++u)
        if (l < C.r && i0 + u * bd < m) s[u] = cfma(q[u * bd], x, s[u]);
    }
#pragma unroll
    for (int u = 0; u < kApPer; ++u)
      if (i0 + u * bd < m) {
        v[i0 + u * bd] = s[u];
        nn += cabs2(s[u]);
      }
  }
  return nn;
}

// M = W^H W (double-float sums) = L L^H, L^{-1}, and Q = W L^{-H} in place of W.
// Scratch: T.  Ends with a barrier.
template <int R>
__device__ void ffactor(const FCtx& C) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, r = C.r;
  double2* G = reinterpret_cast<double2*>(C.T);
  float2* part = reinterpret_cast<float2*>(G + 2 * kMaxR * kMaxR + kMaxR);
  float2* Gd = part + C.nw * R * R;  // value layout of cgram_part, summed over the warps
  float2* mine = part + w * R * R;
  cgram_warp<R>(C.Q, C.m, C.m, r, C.nw, mine);
  __syncthreads();
  for (int t = threadIdx.x; t < r * r; t += blockDim.x) {
    float h = 0.f, l = 0.f;
#pragma unroll 4
    for (int ww = 0; ww < C.nw; ++ww) df_add(h, l, part[ww * R * R + t].x, part[ww * R * R + t].y);
    Gd[t] = make_float2(h, l);
  }
  __syncthreads();
  if (threadIdx.x < 32 && !cchol_df<R>(Gd, r, C.Li, C.Lf)) {
    if (lane < r)
      for (int q = 0; q <= lane; ++q) {
        const float2 x = Gd[lane * lane + 2 * q], y = q < lane ? Gd[lane * lane + 2 * q + 1] : make_float2(0.f, 0.f);
        G[lane * kMaxR + q] = make_double2(static_cast<double>(x.x) + static_cast<double>(x.y),
                                           -(static_cast<double>(y.x) + static_cast<double>(y.y)));
      }
    __syncwarp();
    if (!cchol_f64(r, G, C.Li, C.Lf) && lane == 0) report_error(C.err, kErrNotSPD, C.k);
  }
  __syncthreads();
  // Q_l = sum_{p <= l} W_p conj(L^{-1}[l][p]), the diagonal with its remainder: a
  // column that is off by a common factor of 1 + 3e-8 puts the error into b and the
  // residual whole, where the rounding of its entries averages out
  for (int i = threadIdx.x; i < C.m; i += blockDim.x) {
    float2 x[R];
#pragma unroll
    for (int l = 0; l < R; ++l) x[l] = l < r ? C.Q[static_cast<size_t>(l) * C.m + i] : make_float2(0.f, 0.f);
#pragma unroll
    for (int l = 0; l < R; ++l) {
      if (l >= r) break;
      float2 s = make_float2(0.f, 0.f);
#pragma unroll
      for (int p = 0; p < l; ++p) s = ccfma(C.Lf[l * kMaxR + p], x[p], s);
      const float2 d = C.Lf[l * kMaxR + l];
      s.x = fmaf(d.x, x[l].x, fmaf(d.y, x[l].x, s.x));
      s.y = fmaf(d.x, x[l].y, fmaf(d.y, x[l].y, s.y));
      C.Q[static_cast<size_t>(l) * C.m + i] = s;
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------- HardThreshold --
// The rho entries of largest modulus of the frame (ties to the lower pixel
// index) by an 8-bit radix select -> pixels ascending, and values when
// keep_values.
__device__ inline void fhard_threshold(const FCtx& C, bool keep_values) {
  const int n = C.g.n, ld = C.g.ny + 1, rho = C.rho, lane = threadIdx.x & 31;
  int* info = C.hist + 256;
  int* sel = C.cand;            // rho entries
  unsigned prefix = 0, mask = 0;
  if (threadIdx.x == 0) info[1] = rho;
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int t = threadIdx.x; t < 256; t += blockDim.x) C.hist[t] = 0;
    __syncthreads();
    for (int e0 = threadIdx.x - lane; e0 < n; e0 += blockDim.x) {
      const int e = e0 + lane;
      unsigned key = 0u;
      if (e < n) {
        const int row = frow(C.g, e), col = fcol(C.g, e);
        key = __float_as_uint(cabs2(C.X[row * ld + col]));
      }
      const bool in = e < n && (key & mask) == prefix;
      const unsigned digit = in ? ((key >> shift) & 255u) : 256u;
      const unsigned peers = __match_any_sync(0xffffffffu, digit);
      if (in && (__ffs(peers) - 1) == lane) atomicAdd(&C.hist[digit], __popc(peers));
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      const int need = info[1];
      int own[8], tot = 0;
#pragma unroll
      for (int z = 0; z < 8; ++z) { own[z] = C.hist[255 - 8 * lane - z]; tot += own[z]; }
      int incl = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      const int excl = incl - tot;
      if (excl < need && incl >= need) {
        int acc = excl;
        for (int z = 0; z < 8; ++z) {
          if (acc + own[z] >= need) {
            info[0] = 255 - 8 * lane - z;
            info[1] = need - acc;
            break;
          }
          acc += own[z];
        }
      }
    }
    __syncthreads();
    prefix |= static_cast<unsigned>(info[0]) << shift;
    mask |= 255u << shift;
  }
  const unsigned T = prefix;
  const int need = info[1];
  int* ties = C.cand + rho + 8; // tie candidates (bounded below)
  const int tie_cap = 56;
  if (threadIdx.x == 0) { info[2] = 0; info[3] = 0; }
  __syncthreads();
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int row = frow(C.g, e), col = fcol(C.g, e);
    const unsigned key = __float_as_uint(cabs2(C.X[row * ld + col]));
    if (key > T) sel[atomicAdd(&info[3], 1)] = e;
    else if (key == T) {
      const int s = atomicAdd(&info[2], 1);
      if (s < tie_cap) ties[s] = e;
    }
  }
  __syncthreads();
  const int nt = min(info[2], tie_cap), ngt = info[3];
  if (info[2] > tie_cap && threadIdx.x == 0) report_error(C.err, kErrNaN, C.k);
  for (int t = threadIdx.x; t < nt; t += blockDim.x) {
    const int e = ties[t];
    int rank = 0;
    for (int u = 0; u < nt; ++u) rank += ties[u] < e;
    if (rank < need) sel[ngt + rank] = e;
  }
  __syncthreads();
  // store ascending by pixel (fixed order for every later sum over the support)
  for (int t = threadIdx.x; t < rho; t += blockDim.x) {
    const int e = sel[t];
    int pos = 0;
    for (int u = 0; u < rho; ++u) pos += sel[u] < e;
    const int row = frow(C.g, e), col = fcol(C.g, e);
    C.sp[pos] = e;
    C.sv[pos] = keep_values ? C.X[row * ld + col] : make_float2(0.f, 0.f);
  }
  __syncthreads();
}

// HardThreshold of v = s - mu g for a strictly ascending support, from g in the
// frame and v on the support in vn.  The support's entries have keys >= T0,
// their smallest, so the rho largest of all are among the support and the
// entries off it at or above T0: none of these, and the support stays; else
// the candidates are sorted by (key descending, pixel ascending), the order
// of the radix select, unless there are more than kCandCap of them.  gmax2:
// max |g|^2 off the support (each thread's part).  Returns whether the support
// stays.  Ends with a barrier.
__device__ inline bool fthreshold(const FCtx& C, float mu, float& gmax2) {
  const int n = C.g.n, ld = C.g.ny + 1, rho = C.rho, lane = threadIdx.x & 31;
  int* info = C.hist + 256;
  if (threadIdx.x < 32) {
    unsigned mn = 0xffffffffu;
    for (int e = lane; e < rho; e += 32) mn = min(mn, __float_as_uint(cabs2(C.vn[e])));
    mn = __reduce_min_sync(0xffffffffu, mn);
    if (lane == 0) {
      info[4] = static_cast<int>(mn);
      info[5] = 0;
    }
  }
  for (int e = threadIdx.x; e < rho; e += blockDim.x) {
    const int p = C.sp[e];
    C.X[frow(C.g, p) * ld + fcol(C.g, p)] = make_float2(0.f, 0.f);
  }
  __syncthreads();
  const unsigned T0 = static_cast<unsigned>(info[4]);
  gmax2 = 0.f;
  if (T0 != 0u) {
#pragma unroll 4
    for (int e0 = threadIdx.x - lane; e0 < n; e0 += blockDim.x) {
      const int e = e0 + lane;
      unsigned key = 0u;
      if (e < n) {
        const float2 x = C.X[frow(C.g, e) * ld + fcol(C.g, e)];
        gmax2 = fmaxf(gmax2, cabs2(x));
        key = __float_as_uint(cabs2(make_float2(x.x * -mu, x.y * -mu)));
      }
      if (__any_sync(0xffffffffu, key >= T0) && key >= T0) {
        const int pos = atomicAdd(&info[5], 1) + rho;
        if (pos < kCandCap)
          C.cl[pos] = (static_cast<unsigned long long>(key) << 32) | (0xffffffffu - static_cast<unsigned>(e));
      }
    }
  }
  __syncthreads();
  const int cnt = info[5] + rho;
  if (T0 != 0u && cnt == rho) {
    for (int e = threadIdx.x; e < rho; e += blockDim.x) C.sv[e] = C.vn[e];
    __syncthreads();
    return true;
  }
  for (int e = threadIdx.x; e < rho; e += blockDim.x) C.spo[e] = C.sp[e];
  if (T0 == 0u || cnt > kCandCap) {  // v in the frame, radix select
    for (int e = threadIdx.x; e < C.g.nx * ld; e += blockDim.x) {
      C.X[e].x *= -mu;
      C.X[e].y *= -mu;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < rho; e += blockDim.x) {
      const int p = C.sp[e];
      C.X[frow(C.g, p) * ld + fcol(C.g, p)] = C.vn[e];
    }
    __syncthreads();
    fhard_threshold(C, true);
    int same = 1;
    for (int e = threadIdx.x; e < rho; e += blockDim.x) same &= C.spo[e] == C.sp[e];
    return __syncthreads_and(same) != 0;
  }
  int P = 1;
  while (P < cnt) P <<= 1;
  for (int t = threadIdx.x; t < P; t += blockDim.x)
    if (t < rho || t >= cnt)
      C.cl[t] = t >= cnt ? 0ull
                         : (static_cast<unsigned long long>(__float_as_uint(cabs2(C.vn[t]))) << 32) |
                               (0xffffffffu - static_cast<unsigned>(C.sp[t]));
  __syncthreads();
  for (int kk = 2; kk <= P; kk <<= 1)
    for (int j = kk >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < P; t += blockDim.x) {
        const int o = t ^ j;
        if (o > t) {
          const unsigned long long x = C.cl[t], y = C.cl[o];
          if (((t & kk) == 0) ? (x < y) : (x > y)) {
            C.cl[t] = y;
            C.cl[o] = x;
          }
        }
      }
      __syncthreads();
    }
  // ascending by pixel; the value from vn (entries of the old support, by
  // binary search) or from g
  for (int t = threadIdx.x; t < rho; t += blockDim.x) {
    const unsigned e = 0xffffffffu - static_cast<unsigned>(C.cl[t]);
    int pos = 0;
    for (int u = 0; u < rho; ++u) pos += 0xffffffffu - static_cast<unsigned>(C.cl[u]) < e;
    int lo = 0, hi = rho;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (static_cast<unsigned>(C.spo[mid]) < e) lo = mid + 1;
      else hi = mid;
    }
    C.sp[pos] = static_cast<int>(e);
    if (lo < rho && static_cast<unsigned>(C.spo[lo]) == e) {
      C.sv[pos] = C.vn[lo];
    } else {
      const float2 x = C.X[frow(C.g, e) * ld + fcol(C.g, e)];
      C.sv[pos] = make_float2(x.x * -mu, x.y * -mu);
    }
  }
  __syncthreads();
  return false;
}

// ------------------------------------------------------------- the kernel --
// P2: both sides are powers of two (indices by shifts and masks, without the
// tests; a third of the instructions of the sparse DFTs otherwise).
template <int R, bool P2>
__global__ void __launch_bounds__(kFT, 1) fsweep_kernel(const FArgs a) {
  extern __shared__ __align__(16) unsigned char sm[];
  const FCarve cv = fcarve(a.g, a.m, a.r, a.rho, a.vecs != nullptr, a.tb, a.qmode == 1, a.lean != 0);
  FCtx C;
  C.g = a.g;
  if constexpr (P2) {
    __builtin_assume(C.g.lnx >= 0);
    __builtin_assume(C.g.lny >= 0);
    __builtin_assume(C.g.lL >= 0);
  }
  C.m = a.m;
  C.r = a.r;
  C.rho = a.rho;
  C.k = blockIdx.x;
  C.nw = blockDim.x >> 5;
  C.X = reinterpret_cast<float2*>(sm + cv.X);
  C.tx = reinterpret_cast<float2*>(sm + cv.tx);
  C.ty = reinterpret_cast<float2*>(sm + cv.ty);
  C.tl = reinterpret_cast<float2*>(sm + cv.tl);
  const int k = C.k, m = C.m, r = C.r, rho = C.rho, n = C.g.n, ld = C.g.ny + 1;
  C.dv = a.vecs ? a.vecs + static_cast<size_t>(k) * 2 * m : reinterpret_cast<float2*>(sm + cv.dv);
  C.ev = a.vecs ? C.dv + m : reinterpret_cast<float2*>(sm + cv.ev);
  C.msk = reinterpret_cast<int*>(sm + cv.msk);
  C.rptr = reinterpret_cast<int*>(sm + cv.rptr);
  C.sp = reinterpret_cast<int*>(sm + cv.sp);
  C.sv = reinterpret_cast<float2*>(sm + cv.sv);
  C.gv = reinterpret_cast<float2*>(sm + cv.gv);
  C.spo = reinterpret_cast<int*>(sm + cv.gv);
  C.vn = reinterpret_cast<float2*>(sm + cv.vn);
  C.ord = reinterpret_cast<unsigned short*>(sm + cv.ord);
  C.ent = reinterpret_cast<int*>(sm + cv.ent);
  C.cs = reinterpret_cast<unsigned short*>(sm + cv.cs);
  C.ccol = reinterpret_cast<unsigned short*>(sm + cv.ccol);
  C.pcs = reinterpret_cast<unsigned short*>(sm + cv.pcs);
  C.Li = reinterpret_cast<double2*>(sm + cv.Li);
  C.Lf = reinterpret_cast<float2*>(sm + cv.Lf);
  C.red = reinterpret_cast<float*>(sm + cv.red);
  C.scal = reinterpret_cast<float*>(sm + cv.scal);
  C.hist = reinterpret_cast<int*>(sm + cv.hist);
  C.cand = reinterpret_cast<int*>(sm + cv.cand);
  C.cl = reinterpret_cast<unsigned long long*>(sm + cv.cl);
  C.T = a.lean ? C.X : reinterpret_cast<float2*>(sm + cv.T);
  float2* const Qg = a.qmode == 1 ? nullptr : a.Wk + static_cast<size_t>(k) * r * m;
  C.Q = a.qmode == 0 ? Qg : a.qmode == 1 ? reinterpret_cast<float2*>(sm + cv.Q) : C.X;
  C.err = a.err;
  __shared__ int np_s;
  // phase cycle counters (profile): thread 0's clock between the CTA's phases
  // (kept in shared memory: registers are scarce in this kernel)
  __shared__ unsigned long long pc[kFProf];
  __shared__ long long tl;
  if (a.prof && threadIdx.x == 0) {
    for (int slot = 0; slot < kFProf; ++slot) pc[slot] = 0ull;
    tl = clock64();
  }
  auto mark = [&](int slot) {
    if (a.prof && threadIdx.x == 0) {
      const long long t = clock64();
      pc[slot] += static_cast<unsigned long long>(t - tl);
      tl = t;
    }
  };
  const float2* y = a.y + static_cast<size_t>(k) * m;
  const bool init = a.mode == kModeInit, project = !init;
  for (int t = threadIdx.x; t < C.g.nx; t += blockDim.x) C.tx[t] = __ldg(a.twx + t);
  for (int t = threadIdx.x; t < C.g.ny; t += blockDim.x) C.ty[t] = __ldg(a.twy + t);
  for (int t = threadIdx.x; t < C.g.L; t += blockDim.x) C.tl[t] = __ldg(a.twl + t);
  {
    const int bd = blockDim.x;
    const int* mask = a.mask + static_cast<size_t>(k) * m;
    constexpr int kG = 4;  // samples in flight per thread
    for (int i0 = threadIdx.x; i0 < m; i0 += kG * bd) {
      int om[kG];
#pragma unroll
      for (int u = 0; u < kG; ++u) om[u] = i0 + u * bd < m ? __ldg(mask + i0 + u * bd) : 0;
#pragma unroll
      for (int u = 0; u < kG; ++u)
        if (i0 + u * bd < m) C.msk[i0 + u * bd] = om[u];
      if (project) {  // W_k = (F2 U)[Omega_k]
        float2 x[kG][R];
#pragma unroll
        for (int u = 0; u < kG; ++u) {
          const float2* from = a.FU + static_cast<size_t>(om[u]) * r;
          if (r == R) {  // R is even: 16-byte loads (rows are 8 R bytes)
#pragma unroll
            for (int l = 0; l < R; l += 2) {
              const float4 w = __ldg(reinterpret_cast<const float4*>(from + l));
              x[u][l] = make_float2(w.x, w.y);
              x[u][l + 1] = make_float2(w.z, w.w);
            }
          } else {
#pragma unroll
            for (int l = 0; l < R; ++l) x[u][l] = l < r ? __ldg(from + l) : make_float2(0.f, 0.f);
          }
        }
#pragma unroll
        for (int u = 0; u < kG; ++u)
#pragma unroll
          for (int l = 0; l < R; ++l)
            if (l < r && i0 + u * bd < m) C.Q[static_cast<size_t>(l) * m + i0 + u * bd] = x[u][l];
      }
    }
  }
  // the support, sorted by pixel
  for (int e = threadIdx.x; e < rho; e += blockDim.x) C.spo[e] = init ? e : a.S_idx[static_cast<size_t>(k) * rho + e];
  __syncthreads();
  {
    int inorder = 1;
    for (int e = threadIdx.x; e + 1 < rho; e += blockDim.x) inorder &= C.spo[e] < C.spo[e + 1];
    inorder = __syncthreads_and(inorder);
    for (int e = threadIdx.x; e < rho; e += blockDim.x) {
      const int p = C.spo[e];
      int pos = e;
      if (!inorder) {
        pos = 0;
        for (int f = 0; f < rho; ++f) pos += C.spo[f] < p;  // (distinct: lrs_set_state)
      }
      C.sp[pos] = p;
      C.sv[pos] = init ? make_float2(0.f, 0.f) : a.S_val[static_cast<size_t>(k) * rho + e];
    }
    for (int i = threadIdx.x; a.tb > 0 && i <= m; i += blockDim.x) {  // samples by frequency row (ascending)
      const int x0 = i > 0 ? frow(C.g, C.msk[i - 1]) : -1, x1 = i < m ? frow(C.g, C.msk[i]) : C.g.nx;
      for (int x = x0 + 1; x <= x1; ++x) C.rptr[x] = i;
    }
    __syncthreads();
  }
  const bool by_cols = a.tb > 0;
  int np = by_cols ? support_cols(C, &np_s) : 0;
  // A x for values v on the support
  auto forward = [&](const float2* v, float2* out) {
    if (!by_cols) sparse_direct(C, v, rho, out);
    else sparse_cols(C, np, v, out, a.tb);
  };
  if (project) ffactor<R>(C);
  // Q_k in the frame's place (qmode 2): saved before the first FFT, back before
  // the next projection without one
  bool q_saved = a.qmode != 2, q_home = true;
  auto copy_q = [&](float2* to, const float2* from) {
    __syncthreads();
    for (int t = threadIdx.x; t < r * m; t += blockDim.x) to[t] = from[t];
    __syncthreads();
  };
  auto frame_taken = [&]() {
    if (!project || a.qmode != 2 || !q_home) return;
    if (!q_saved) copy_q(Qg, C.X);
    q_saved = true;
    q_home = false;
    C.Q = Qg;
  };
  auto frame_free = [&]() {
    if (!project || q_home) return;
    copy_q(C.X, Qg);
    q_home = true;
    C.Q = C.X;
  };
  mark(0);
  const int tau = (a.mode == kModeLS || rho == 0) ? 0 : a.tau;
  const float N = sqrtf(static_cast<float>(m) / static_cast<float>(n));  // column norms
  // u = P_perp (A s - y) in dv; c = Q^H (A s - y) in cu when it was formed from s
  float2 cu[R];
  const bool as_ok = a.asv[k] != 0;
  float2* const D = a.AS + static_cast<size_t>(k) * m;
  auto residual = [&](bool stored) {  // returns this thread's part of ||u||^2
    if (!stored) forward(C.sv, C.dv);
    float nn = 0.f;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
      const float2 u = stored ? D[i] : csub(C.dv[i], y[i]);
      if (!stored) D[i] = u;
      C.dv[i] = u;
      nn += cabs2(u);
    }
    mark(1);
    if (project) {
      __syncthreads();
      frame_free();
      fcoefs<R>(C, C.dv, cu);

      mark(6);
      nn = fapply<R>(C, C.dv, cu, -1.f);
      mark(7);
    }
    return nn;
  };
  bool valid = false;  // dv belongs to the present s
  bool have_ref = false;
  float mu_prev = 1.f / (N * N), nn = 0.f, dist = 0.f, gmax = 0.f;
  for (int it = 0; it < tau; ++it) {
    const bool zero_start = init && it == 0;
    if (zero_start) {
      for (int i = threadIdx.x; i < m; i += blockDim.x) C.dv[i] = make_float2(-y[i].x, -y[i].y);
    } else if (!valid) {
      nn = residual(it == 0 && as_ok);
    }
    valid = true;
    fput(C, 0, nn);
    float smin = INFINITY;
    for (int e = threadIdx.x & 31; e < rho; e += 32) smin = fminf(smin, cabs2(C.sv[e]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) smin = fminf(smin, __shfl_xor_sync(0xffffffffu, smin, o));
    __syncthreads();
    const float un = sqrtf(fget(C, 0) + kTinySq);
    float bound = N * un;
    if (have_ref) bound = fminf(bound, fmaf(N, dist, gmax));
    mark(2);
    // worth trying without the FFT: the bound with the last mu and the present s
    bool cert = !zero_start && by_cols && bound * mu_prev < sqrtf(smin);
    bool stop = false;
    float mu = 0.f, den = 0.f;
    for (;;) {
      if (cert) {
        frame_free();
        sparse_adjoint(C, np, C.dv, a.tb);
        mark(1);
      } else {
        frame_taken();
        // g = A^H u: zero-filled frame, inverse 2D FFT
        for (int e = threadIdx.x; e < C.g.nx * ld; e += blockDim.x) C.X[e] = make_float2(0.f, 0.f);
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += blockDim.x) C.X[frev(C.g, C.msk[i])] = C.dv[i];
        __syncthreads();
        fft2_smem(C.X, C.g.nx, C.g.ny, C.g.lnx, C.g.lny, C.tx, C.ty, true);
        mark(3);
        if (zero_start) {  // support of the zero start: the rho largest |g|
          fhard_threshold(C, false);
          if (by_cols) np = support_cols(C, &np_s);
          mark(4);
        }
        for (int e = threadIdx.x; e < rho; e += blockDim.x) {
          const int p = C.sp[e];
          C.gv[e] = C.X[frow(C.g, p) * ld + fcol(C.g, p)];
        }
        __syncthreads();
      }
      // mu = ||g_G||^2 / ||P_perp A g_G||^2
      if (threadIdx.x < 32) {
        float s = 0.f;
        for (int e = threadIdx.x; e < rho; e += 32) s += cabs2(C.gv[e]);
        s = warp_sumf(s);
        if (threadIdx.x == 0) C.scal[1 * C.nw] = s;
      }
      forward(C.gv, C.ev);
      mark(1);
      float nd = 0.f;
      if (project) {
        float2 cf[R];
        fcoefs<R>(C, C.ev, cf);
        mark(6);
        nd = fapply<R>(C, C.ev, cf, -1.f);
        mark(7);
      } else {
        for (int i = threadIdx.x; i < m; i += blockDim.x) nd += cabs2(C.ev[i]);
      }
      fput(C, 2, nd);
      __syncthreads();
      den = fget(C, 2);
      if (!(den > 0.f)) {
        stop = true;
        break;
      }
      mu = C.scal[1 * C.nw] / den;
      if (!isfinite(mu)) {
        if (threadIdx.x == 0) report_error(a.err, kErrNaN, k);
        mu = 0.f;
      }
      int ok = 1;
      for (int e = threadIdx.x; e < rho; e += blockDim.x) {
        const float2 s = C.sv[e], g = C.gv[e];
        const float2 v = make_float2(fmaf(-mu, g.x, s.x), fmaf(-mu, g.y, s.y));
        C.vn[e] = v;
        ok &= bound * mu * 1.001f < sqrtf(cabs2(v));  // false for NaN
      }
      ok = __syncthreads_and(ok);
      mark(2);
      if (!cert || ok) break;
      cert = false;
    }
    if (stop) break;
    mu_prev = mu;
    if (cert) {
      for (int e = threadIdx.x; e < rho; e += blockDim.x) C.sv[e] = C.vn[e];
      dist = fmaf(mu, sqrtf(den), dist);
    } else {
      float g2 = 0.f;
      valid = fthreshold(C, mu, g2);
      have_ref = valid;
      if (valid) {
        fput_max(C, 3, g2);
        __syncthreads();
        gmax = fmaf(a.fft_err, un, sqrtf(fget_max(C, 3) + kTinySq));
        dist = mu * sqrtf(den);
      }
    }
    if (valid) {  // s_new = s - mu g_G on the same support
      nn = 0.f;
      for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const float2 d = C.dv[i], e = C.ev[i];
        const float2 u = make_float2(fmaf(-mu, e.x, d.x), fmaf(-mu, e.y, d.y));
        C.dv[i] = u;
        nn += cabs2(u);
      }
      __syncthreads();
    } else if (by_cols) {
      np = support_cols(C, &np_s);
    }
    mark(4);
  }
  // ---- final stage ----
  // from s itself: its rounding in the sweeps is then part of b and res
  const bool as_kept = tau == 0 && as_ok;  // s unchanged by this sweep
  __syncthreads();
  residual(as_kept);
  if (init) {  // h = A^H (y - A s)
    for (int e = threadIdx.x; e < C.g.nx * ld; e += blockDim.x) C.X[e] = make_float2(0.f, 0.f);
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x) C.X[frev(C.g, C.msk[i])] = make_float2(-C.dv[i].x, -C.dv[i].y);
    __syncthreads();
    fft2_smem(C.X, C.g.nx, C.g.ny, C.g.lnx, C.g.lny, C.tx, C.ty, true);
    float2* Hk = a.H + static_cast<size_t>(k) * n;
    for (int e = threadIdx.x; e < n; e += blockDim.x) Hk[e] = C.X[frow(C.g, e) * ld + fcol(C.g, e)];
  } else {
    if (threadIdx.x < r) {  // b = L^{-H} Q^H (y - A s)
      double2 b = make_double2(0.0, 0.0);
#pragma unroll
      for (int l = 0; l < R; ++l) {
        if (l >= r) break;
        const double2 p = dccmul(C.Li[l * kMaxR + threadIdx.x],
                                 make_double2(-static_cast<double>(cu[l].x), -static_cast<double>(cu[l].y)));
        b.x += p.x;
        b.y += p.y;
      }
      a.B[static_cast<size_t>(k) * r + threadIdx.x] = make_float2(static_cast<float>(b.x), static_cast<float>(b.y));
    }
    if (a.mode == kModeIter)  // res = W b - (y - A s) = u
      for (int i = threadIdx.x; i < m; i += blockDim.x) a.RES[static_cast<size_t>(k) * m + i] = C.dv[i];
  }
  if (threadIdx.x == 0) a.asv[k] = 1;
  if (a.mode != kModeLS)
    for (int e = threadIdx.x; e < rho; e += blockDim.x) {  // S_k, ascending by pixel
      a.S_idx[static_cast<size_t>(k) * rho + e] = C.sp[e];
      a.S_val[static_cast<size_t>(k) * rho + e] = C.sv[e];
    }
  mark(5);
  if (a.prof && threadIdx.x == 0)
    for (int slot = 0; slot < kFProf; ++slot) atomicAdd(a.prof + slot, pc[slot]);
}

}  // namespace fourier
}  // namespace lrs
