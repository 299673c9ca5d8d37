// Streaming engine of the Gaussian sweep (Algorithm 1's per-column work with
// the IHT of Algorithm 2): the phases of an iteration run over all columns of
// a launch, one kernel each.
//
//   w_kernel      W_k = A_k U, and the columns of A_k on the support (AG_k)
//   step_kernel   per column, on W_k and AG_k alone: Gram and inverse, then
//                 the IHT sweeps as far as they need no pass over A_k; either
//                 b_k and the residual e_k, or u_k and an entry in the list
//   g_kernel      g = A_k^T u_k for the listed columns
//   step_kernel   (next) HardThreshold with g, then the sweeps as before
//   g_kernel      (final) h_k = A_k^T e_k for every column
//
// Which sweeps need a pass.  An IHT sweep reads A_k only to learn whether an
// entry outside the support G beats one inside: the new values on G,
// v_i = s_i - mu g_i with g_G = AG^T u, need the support's columns alone.
// Outside G, v_j = -mu a_j^T u and |a_j^T u| <= N_k ||u||, N_k = max_j ||a_j||
// (kept per column, set with the operator).  So when
//     mu N_k ||u|| (1 + 1e-3) < min_{i in G} |v_i|
// HardThreshold returns G whatever g is, and the sweep is done without it
// (the 1e-3 covers the rounding of u, mu and of the pass's own float32 sums,
// m 2^-24 N ||u|| at most).  After a pass at u_ref has given g, the same
// holds with max_{j not in G} |g_j| + N_k ||u - u_ref|| in the place of
// N_k ||u||.  Every other sweep goes through g_kernel and the full
// HardThreshold.  A solve's error e_k enters the test as about ||e_k|| <
// min |s_i|: it holds from a relative error of about 1/sqrt(n) on, after which
// an iteration streams A_k twice (W, h) and not 2 + tau times.
//
// Streaming.  A_k stays in the tiled slab layout of the sweep (one slab).  In
// w_kernel and g_kernel every warp is its own pipeline: it issues TMA bulk
// copies of its next pieces into its own ring of stages and consumes them
// itself, so no warp ever waits for another one and a kernel's work units
// (rows x columns of one A_k) need no queue: warp i takes units i, i + warps,
// ....  Sixteen warps per SM with three stages of about 4 KB keep 200 KB per SM
// in flight (45 KB cover the memory's latency at full rate).
// What a unit sums, and in what order, does not depend on the number of
// CTAs or on the other problems of the launch, so results are the same alone,
// in a batch, under any grid and in a column-sharded solve.
//
// Every wait is bounded by wait_ns; on expiry the warp records kErrTimeout,
// drains its own copies (bounded) and leaves.
#pragma once

#include "sweep_gauss_impl.cuh"

namespace lrs {
namespace stream {

using sweep::a16;
using sweep::elem1s;
using sweep::ht_key;
using sweep::kTW;

constexpr int kSW = 8;            // warps per streaming CTA
constexpr int kStreamNT = 32 * kSW;
constexpr int kStepNT = 128;      // threads per column step
constexpr int kStepNW = kStepNT / 32;
constexpr int kMaxStage = 4;

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ------------------------------------------------------------- warp pipeline --
// One warp's ring: `S` stages, full barriers only (the warp that refills a
// stage is the one that has read it).
struct Pipe {
  unsigned char* base;
  uint64_t* full;
  unsigned stage;        // bytes
  int S;
  unsigned issued, taken;
  bool dead;
  int* err;
  unsigned long long wait_ns;

  __device__ void init(unsigned char* b, uint64_t* f, unsigned stg, int s, unsigned long long w) {
    base = b;
    full = f;
    stage = stg;
    S = s;
    issued = taken = 0;
    dead = false;
    err = nullptr;
    wait_ns = w;
    if ((threadIdx.x & 31) == 0)
      for (int i = 0; i < S; ++i) mbar_init(&full[i], 1);
    __syncwarp();
  }
  __device__ bool wait(uint64_t* bar, unsigned parity) const {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = gtimer();
    while (!mbar_try_wait(bar, parity))
      if (gtimer() - t0 > wait_ns) return false;
    return true;
  }
  // the oldest piece in flight (every lane waits)
  __device__ const unsigned char* take() {
    const unsigned s = taken % S;
    bool ok = wait(&full[s], (taken / S) & 1u);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) {
      dead = true;
      if ((threadIdx.x & 31) == 0) report_error(err, kErrTimeout, -1);
    }
    return base + static_cast<size_t>(s) * stage;
  }
  // before leaving after an expired wait: no copy may land in this CTA's
  // shared memory once it is gone
  __device__ void drain() {
    for (; taken < issued; ++taken) wait(&full[taken % S], (taken / S) & 1u);
  }
};

__device__ __forceinline__ int prob_of(const StreamTable& T, int c) {
  int p = 0;
  while (p + 1 < T.nprob && T.probs[p + 1].col0 <= c) ++p;
  return p;
}

// ------------------------------------------------------------------ W = A U --
// Rows of a unit (a multiple of 8): accumulators rows/4 x R per lane and
// 4 R registers of U at a time leave 128 registers, two CTAs per SM.
__host__ __device__ constexpr int w_rows(int R) { return R <= 6 ? 32 : 16; }

// Unit: RB rows x one chunk of `tbw` tiles of one column.  A CTA keeps its
// chunk of U in shared memory for all its units (a lane reads U of its four
// columns once per tile), so U costs no streaming.  Lane (ro, q) accumulates
// rows 4 t + ro over columns 4 q .. 4 q + 3 of each tile; the 8 lanes of a row
// are added at the end of the unit.  Bound by memory for R up to about 8 in
// float32 (2 R flops per 4 bytes), by the FMA pipe above and for the 16- and
// 8-bit forms.
template <int R, int ET>
__global__ void __launch_bounds__(kStreamNT, 2)
    w_kernel(const StreamTable T, const StreamAssign* __restrict__ asg, int nasg, int S, int tpp,
             unsigned us_bytes) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int RB = w_rows(R), RT = RB / 4;
  constexpr int pb = ET == 0 ? 4 : ET == 1 ? 2 : 1;
  constexpr int planes = ET == 3 ? 2 : 1;
  constexpr int CP = R > 12 ? 2 : 4;  // columns of U held in registers at a time
  constexpr unsigned sub = RB * kTW * pb * planes;  // bytes of one tile of a piece
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int q = lane & 7, ro = lane >> 3;
  float* Us = reinterpret_cast<float*>(smem);
  const unsigned stage = sub * tpp;
  Pipe P;
  P.init(smem + us_bytes + static_cast<size_t>(wid) * S * stage,
         reinterpret_cast<uint64_t*>(smem + us_bytes + static_cast<size_t>(kSW) * S * stage) +
             wid * kMaxStage,
         stage, S, T.wait_ns);
  if (blockIdx.x == 0 && threadIdx.x < T.ncnt) T.cnt[threadIdx.x] = 0;
  for (int a = blockIdx.x; a < nasg; a += gridDim.x) {
    const StreamAssign as = asg[a];
    const StreamProblem& pr = T.probs[as.prob];
    const int m = pr.L.m, n = pr.L.n, rho = pr.te > 0 || pr.L.rho > 0 ? pr.L.rho : 0;
    const int ntile = pr.L.ns / kTW, b0 = as.cc * pr.tbw, b1 = min(ntile, b0 + pr.tbw);
    const int nrb = pr.nrb, nunits = pr.L.q * nrb;
    const size_t tb = static_cast<size_t>(m) * kTW * elem_bytes(ET);
    const unsigned char* A = static_cast<const unsigned char*>(pr.A);
    P.err = pr.err;
    __syncthreads();
    // U of a tile as [z][q]: the 4 R floats of the four columns of lane group q
    // are R 16-byte chunks z, chunk z of the eight groups side by side, so that
    // a warp's read is one conflict-free wavefront for every R (row-major, the
    // groups lie 16 R bytes apart: 8-way conflicts at R = 8 and 16)
    for (int t = threadIdx.x; t < (b1 - b0) * kTW * R / 4; t += kStreamNT) {
      const int b = t / (8 * R), w = t - b * 8 * R, g = w / R, z = w - g * R;
      reinterpret_cast<float4*>(Us)[b * 8 * R + z * 8 + g] =
          reinterpret_cast<const float4*>(pr.Upad + static_cast<size_t>(b0) * kTW * R)[t];
    }
    __syncthreads();
    const int u0 = as.idx * kSW + wid, ustep = as.cnt * kSW;
    int pu = u0, pbt = b0;  // next piece to issue: unit, first tile
    auto issue = [&]() {
      if (pu >= nunits) return;
      const int k = pu / nrb, i0 = (pu - k * nrb) * RB, nr = min(RB, m - i0);
      const int nt = min(tpp, b1 - pbt);
      const unsigned s = P.issued % S;
      const unsigned hb = static_cast<unsigned>(nr * kTW * pb);
      unsigned char* dst = P.base + static_cast<size_t>(s) * stage;
      if (lane == 0) mbar_arrive_expect_tx(&P.full[s], hb * planes * nt);
      __syncwarp();
      if (lane < nt * planes) {
        const int t = lane / planes, pl = lane - t * planes;
        const unsigned char* src = A + (static_cast<size_t>(k) * ntile + pbt + t) * tb +
                                   static_cast<size_t>(pl) * m * kTW +
                                   static_cast<size_t>(i0) * kTW * pb;
        bulk_copy_g2s(dst + t * sub + pl * hb, src, hb, &P.full[s]);
      }
      ++P.issued;
      pbt += nt;
      if (pbt >= b1) {
        pbt = b0;
        pu += ustep;
      }
    };
    for (int i = 0; i < S; ++i) issue();
    for (int u = u0; u < nunits && !P.dead; u += ustep) {
      const int k = u / nrb, i0 = (u - k * nrb) * RB, nr = min(RB, m - i0);
      float s1[RT], s2[RT];
#pragma unroll
      for (int t = 0; t < RT; ++t) {
        s1[t] = s2[t] = 0.f;
        if (ET >= 2 && 4 * t + ro < nr) {
          const size_t o = (static_cast<size_t>(k) * m + i0 + 4 * t + ro) * planes;
          s1[t] = pr.rscale[o];
          if (ET == 3) s2[t] = pr.rscale[o + 1];
        }
      }
      const int* sidx = pr.S_idx + static_cast<size_t>(k) * rho;
      const int j0 = lane < rho ? sidx[lane] : -1;
      float acc[RT][R];
#pragma unroll
      for (int t = 0; t < RT; ++t)
#pragma unroll
        for (int l = 0; l < R; ++l) acc[t][l] = 0.f;
      for (int b = b0; b < b1; b += tpp) {
        const unsigned char* st = P.take();
        if (P.dead) break;
        const int nt = min(tpp, b1 - b);
        for (int tt = 0; tt < nt; ++tt, st += sub) {
          const float4* Ut = reinterpret_cast<const float4*>(Us) + (b + tt - b0) * 8 * R + q;
          float4 av[RT];
#pragma unroll
          for (int c0 = 0; c0 < 4; c0 += CP) {
            float uu[CP * R];
#pragma unroll
            for (int z = 0; z < CP * R / 4; ++z) {
              const float4 w = Ut[(c0 * R / 4 + z) * 8];
              uu[4 * z] = w.x; uu[4 * z + 1] = w.y; uu[4 * z + 2] = w.z; uu[4 * z + 3] = w.w;
            }
#pragma unroll
            for (int t = 0; t < RT; ++t) {
              const int i = 4 * t + ro;
              if (c0 == 0) {
                if (i < nr) {
                  const int off = i * kTW + ((q ^ (i & 7)) << 2);
                  if constexpr (ET == 2) {  // raw values; the row's scale multiplies the sum
                    av[t] = static_cast<float4>(*reinterpret_cast<const __nv_fp8x4_e4m3*>(st + off));
                  } else if constexpr (ET == 3) {
                    const float4 fh = static_cast<float4>(*reinterpret_cast<const __nv_fp8x4_e4m3*>(st + off));
                    const float4 fl = static_cast<float4>(
                        *reinterpret_cast<const __nv_fp8x4_e4m3*>(st + nr * kTW + off));
                    av[t] = make_float4(fmaf(fl.x, s2[t], fh.x * s1[t]), fmaf(fl.y, s2[t], fh.y * s1[t]),
                                        fmaf(fl.z, s2[t], fh.z * s1[t]), fmaf(fl.w, s2[t], fh.w * s1[t]));
                  } else {
                    av[t] = sweep::load4<ET>(st, nr, i, q, nullptr, nullptr);
                  }
                } else {
                  av[t] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
              }
#pragma unroll
              for (int c = 0; c < CP; ++c) {
                const int cc = c0 + c;
                const float x = cc == 0 ? av[t].x : cc == 1 ? av[t].y : cc == 2 ? av[t].z : av[t].w;
#pragma unroll
                for (int l = 0; l < R; ++l) acc[t][l] = fmaf(x, uu[c * R + l], acc[t][l]);
              }
            }
          }
          // support columns that lie in this tile -> AG_k (entry e of the input support)
          for (int e0 = 0; e0 < rho; e0 += 32) {
            const int j = e0 == 0 ? j0 : (e0 + lane < rho ? sidx[e0 + lane] : -1);
            unsigned in = __ballot_sync(0xffffffffu, j >= 0 && j < n && (j >> 5) == b + tt);
            while (in) {
              const int src = __ffs(in) - 1;
              in &= in - 1;
              const int jj = __shfl_sync(0xffffffffu, j, src) & 31;
              float* ag = pr.AG + (static_cast<size_t>(k) * rho + e0 + src) * pr.astride + i0;
              if (lane < nr) {
                float r1 = 0.f, r2 = 0.f;
                if (ET >= 2) {
                  const size_t o = (static_cast<size_t>(k) * m + i0 + lane) * planes;
                  r1 = pr.rscale[o];
                  if (ET == 3) r2 = pr.rscale[o + 1];
                }
                ag[lane] = elem1s<ET>(st, nr, lane, jj, r1, r2);
              }
            }
          }
        }
        ++P.taken;
        __syncwarp();
        issue();
      }
      if (P.dead) break;
      float* out = pr.Wp + (static_cast<size_t>(k) * pr.ncw + as.cc) * pr.wstride +
                   static_cast<size_t>(i0) * R;
#pragma unroll
      for (int t = 0; t < RT; ++t) {
        const int i = 4 * t + ro;
#pragma unroll
        for (int l = 0; l < R; ++l) {
          float v = acc[t][l];
          v += __shfl_xor_sync(0xffffffffu, v, 1);
          v += __shfl_xor_sync(0xffffffffu, v, 2);
          v += __shfl_xor_sync(0xffffffffu, v, 4);
          if (ET == 2) v *= s1[t];
          if ((l & 7) == q && i < nr) out[static_cast<size_t>(i) * R + l] = v;
        }
      }
    }
    if (P.dead) break;
  }
  P.drain();
}

// A_k(i, j) of the stored form
__device__ __forceinline__ float stream_elem(const StreamProblem& pr, int k, int i, int j) {
  const int m = pr.L.m, et = pr.L.et;
  const size_t tb = static_cast<size_t>(m) * kTW * elem_bytes(et);
  const unsigned char* slab =
      static_cast<const unsigned char*>(pr.A) + static_cast<size_t>(k) * (pr.L.ns / kTW) * tb;
  if (et == 0) return elem1s<0>(slab, m, i, j, 0.f, 0.f);
  if (et == 1) return elem1s<1>(slab, m, i, j, 0.f, 0.f);
  const size_t o = (static_cast<size_t>(k) * m + i) * (et == 3 ? 2 : 1);
  if (et == 2) return elem1s<2>(slab, m, i, j, pr.rscale[o], 0.f);
  return elem1s<3>(slab, m, i, j, pr.rscale[o], pr.rscale[o + 1]);
}

// ------------------------------------------------------------- column steps --
// double-float: a value carried as the unevaluated sum hi + lo of two floats
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float z = s - a;
  e = (a - (s - z)) + (b - z);
}

struct StepCarve {
  unsigned W, d, u, v, p, uref, gG, sv, sj, src, red, gi, dbl, ag, vv, tie, hist, lists, total;
  int ms;
};
// Shared memory of a column step; ag: the support's columns are staged too;
// next: the arrays of the full HardThreshold.
__host__ __device__ inline StepCarve step_carve(int R, int m, int n, int rho, int astride, bool ag,
                                                bool next) {
  StepCarve c;
  size_t o = 0;
  const size_t rp = rho > 0 ? rho : 1;
  auto put = [&](size_t bytes) {
    const unsigned at = static_cast<unsigned>(o);
    o += a16(bytes);
    return at;
  };
  c.ms = m | 1;
  c.dbl = put(static_cast<size_t>(3) * 16 * 16 * 8);
  c.W = put(static_cast<size_t>(R) * c.ms * 4);
  c.d = put(static_cast<size_t>(m) * 4);
  c.u = put(static_cast<size_t>(m) * 4);
  c.v = put(static_cast<size_t>(m) * 4);
  c.p = put(static_cast<size_t>(m) * 4);
  c.uref = put(next ? static_cast<size_t>(m) * 4 : 0);
  c.gG = put(rp * 4);
  c.sv = put(2 * rp * 4);
  c.sj = put(rp * 4);
  c.src = put(rp * 4);
  c.red = put((kStepNW * 16 + 4 * kStepNW + 16) * 4);
  c.gi = put(static_cast<size_t>(2) * 16 * 16 * 4);
  c.ag = put(ag ? rp * static_cast<size_t>(astride) * 4 : 0);
  c.vv = put(next ? static_cast<size_t>(n) * 4 : 0);
  c.tie = put(next ? (static_cast<size_t>(n) + 2 * rp + 8) * 4 : 0);
  c.hist = put(next ? (256 + 16) * 4 : 0);
  c.lists = put(next ? 2 * rp * 4 : 0);
  c.total = static_cast<unsigned>(o);
  return c;
}

template <int R>
struct Step {
  const StreamTable& T;
  const StreamProblem& pr;
  int k, c, m, n, r, rho, te, ms, nl, par;
  float *Wt, *d, *u, *v, *p, *uref, *gG, *svb, *red, *gi;
  int *sj, *src;
  double* G;
  float* agsm;       // staged support columns, or nullptr (read from AG_k)
  bool project;

  __device__ Step(const StreamTable& t, const StreamProblem& prob, unsigned char* smem,
                  const StepCarve& cv, bool ag)
      : T(t), pr(prob) {
    m = pr.L.m;
    n = pr.L.n;
    r = pr.L.r;
    rho = pr.L.rho;
    te = pr.te;
    ms = cv.ms;
    par = 0;
    nl = 0;
    auto f = [&](unsigned o) { return reinterpret_cast<float*>(smem + o); };
    Wt = f(cv.W); d = f(cv.d); u = f(cv.u); v = f(cv.v); p = f(cv.p); uref = f(cv.uref); gG = f(cv.gG);
    svb = f(cv.sv); red = f(cv.red); gi = f(cv.gi);
    sj = reinterpret_cast<int*>(smem + cv.sj);
    src = reinterpret_cast<int*>(smem + cv.src);
    G = reinterpret_cast<double*>(smem + cv.dbl);
    agsm = ag ? f(cv.ag) : nullptr;
    project = pr.mode != kModeInit;
  }
  __device__ float* sv(int p) const { return svb + p * max(rho, 1); }
  // column of A_k of support slot e
  __device__ const float* ag(int e) const {
    return agsm ? agsm + static_cast<size_t>(e) * pr.astride
                : pr.AG + (static_cast<size_t>(k) * rho + src[e]) * pr.astride;
  }
  // AG_k into shared memory (rows beyond m are never used)
  __device__ void stage_support() const {
    if (!agsm) return;
    const int a4 = pr.astride / 4;
#pragma unroll 4
    for (int t = threadIdx.x; t < nl * a4; t += kStepNT) {
      const int e = t / a4, i4 = t - e * a4;
      reinterpret_cast<float4*>(agsm)[t] = __ldcg(
          reinterpret_cast<const float4*>(pr.AG + (static_cast<size_t>(k) * rho + src[e]) * pr.astride) + i4);
    }
  }
  __device__ float* coefs() const { return red; }
  __device__ float* scal(int s) const { return red + kStepNW * 16 + s * kStepNW; }

  __device__ void put_coefs(const float (&acc)[R]) const {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int l = 0; l < R; ++l) {
      const float t = warp_sum(acc[l]);
      if (lane == 0) coefs()[w * 16 + l] = t;
    }
  }
  __device__ void put_scal(int s, float x) const {
    x = warp_sum(x);
    if ((threadIdx.x & 31) == 0) scal(s)[threadIdx.x >> 5] = x;
  }
  __device__ float get_scal(int s) const {
    float x = 0.f;
#pragma unroll
    for (int w = 0; w < kStepNW; ++w) x += scal(s)[w];
    return x;
  }
  // x = G^{-1} c from the warps' partial sums of c (after a barrier), in
  // double-float; every warp computes it.  Returns this lane's own x_lane.
  __device__ float solve(float (&x)[R]) const {
    const int lane = threadIdx.x & 31;
    float cl = 0.f;
    if (lane < r)
#pragma unroll
      for (int w = 0; w < kStepNW; ++w) cl += coefs()[w * 16 + lane];
    float xh = 0.f, xl = 0.f;
    for (int b = 0; b < r; ++b) {
      const float cb = __shfl_sync(0xffffffffu, cl, b);
      if (lane < r) {
        const float gh = gi[lane * 16 + b], gl = gi[256 + lane * 16 + b];
        const float p = gh * cb;
        const float e = fmaf(gl, cb, fmaf(gh, cb, -p));
        float s, t;
        two_sum(xh, p, s, t);
        xh = s;
        xl += t + e;
      }
    }
    const float own = lane < r ? xh + xl : 0.f;
#pragma unroll
    for (int l = 0; l < R; ++l) x[l] = __shfl_sync(0xffffffffu, own, l);
    return own;
  }
  __device__ void load_inverse(const double* Gi) const {
    for (int t = threadIdx.x; t < 256; t += kStepNT) {
      const double g = (t >> 4) < r && (t & 15) < r ? Gi[t] : 0.0;
      const float h = static_cast<float>(g);
      gi[t] = h;
      gi[256 + t] = static_cast<float>(g - static_cast<double>(h));
    }
  }

  // Gram W^T W summed in double-float from exact products (two floats hold a
  // product exactly), then its inverse into G + 512 (16 x 16): Cholesky in
  // FP32 and one Newton-Schulz step in FP64, or all in FP64 when a pivot is
  // too small for FP32 (which also reports a Gram that is not positive).
  __device__ void gram_inverse() const {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int t = w; t < r * (r + 1) / 2; t += kStepNW) {
      int p = 0;
      while ((p + 1) * (p + 2) / 2 <= t) ++p;
      const int q2 = t - p * (p + 1) / 2;
      const float *wp = Wt + p * ms, *wq = Wt + q2 * ms;
      float hi = 0.f, lo = 0.f;
      for (int i = lane; i < m; i += 32) {
        const float a = wp[i], b = wq[i], pdt = a * b;
        float s, e;
        two_sum(hi, pdt, s, e);
        hi = s;
        lo += e + fmaf(a, b, -pdt);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float bh = __shfl_xor_sync(0xffffffffu, hi, o), bl = __shfl_xor_sync(0xffffffffu, lo, o);
        float s, e;
        two_sum(hi, bh, s, e);
        hi = s;
        lo += bl + e;
      }
      if (lane == 0) {
        const double s = static_cast<double>(hi) + static_cast<double>(lo);
        G[p * 16 + q2] = s;
        G[q2 * 16 + p] = s;
      }
    }
    __syncthreads();
    float* Lf = reinterpret_cast<float*>(G + 256);
    float* Lif = Lf + 256;
    double* X = G + 512;
    int ok = 1;
    if (threadIdx.x < 32) {
      float ij_own = 0.f;
      for (int j = 0; j < r; ++j) {  // column j of L, a row per lane
        float t = 0.f;
        if (lane >= j && lane < r) {
          t = static_cast<float>(G[lane * 16 + j]);
          for (int p = 0; p < j; ++p) t = fmaf(-Lf[lane * 16 + p], Lf[j * 16 + p], t);
        }
        const float s = __shfl_sync(0xffffffffu, t, j);
        if (!(s > 1e-5f * static_cast<float>(G[j * 16 + j])) || !(s < 1e30f)) { ok = 0; break; }
        const float ij = rsqrtf(s);
        if (lane == j) ij_own = ij;
        if (lane >= j && lane < r) Lf[lane * 16 + j] = lane == j ? s * ij : t * ij;
        __syncwarp();
      }
      if (ok) {
        for (int i = 0; i < r; ++i) {  // L^{-1}, a column per lane
          const float ii = __shfl_sync(0xffffffffu, ij_own, i);
          if (lane < r) {
            float t = i == lane ? 1.f : 0.f;
            for (int p = lane; p < i; ++p) t = fmaf(-Lf[i * 16 + p], Lif[p * 16 + lane], t);
            Lif[i * 16 + lane] = i < lane ? 0.f : t * ii;
          }
          __syncwarp();
        }
      }
    }
    ok = __syncthreads_and(ok);
    if (!ok) {
      if (threadIdx.x < 32) {
        double* L = G + 256;
        __shared__ double iL[16];
        if (!chol_inverse_warp(G, L, X, iL, r, 16) && lane == 0) report_error(pr.err, kErrNotSPD, k);
        __syncwarp();
        for (int t = lane; t < r * r; t += 32) {  // G^{-1} = L^{-T} L^{-1} into G
          const int a = t / r, b = t - a * r;
          double s = 0.0;
          for (int p = max(a, b); p < r; ++p) s = __fma_rn(X[p * 16 + a], X[p * 16 + b], s);
          G[a * 16 + b] = s;
        }
        __syncwarp();
        for (int t = lane; t < r * r; t += 32) X[(t / r) * 16 + t % r] = G[(t / r) * 16 + t % r];
      }
      __syncthreads();
      return;
    }
    for (int t = threadIdx.x; t < r * r; t += kStepNT) {
      const int a = t / r, b = t - a * r;
      float x = 0.f;
      for (int p = max(a, b); p < r; ++p) x = fmaf(Lif[p * 16 + a], Lif[p * 16 + b], x);
      X[a * 16 + b] = x;
    }
    __syncthreads();
    double* Tm = G + 256;
    double t1[2];
    for (int t = threadIdx.x, z = 0; t < r * r; t += kStepNT, ++z) {  // T = G X0
      const int a = t / r, b = t - a * r;
      double x = 0.0;
      for (int p = 0; p < r; ++p) x = __fma_rn(G[a * 16 + p], X[p * 16 + b], x);
      t1[z & 1] = x;
    }
    for (int t = threadIdx.x, z = 0; t < r * r; t += kStepNT, ++z) Tm[(t / r) * 16 + t % r] = t1[z & 1];
    __syncthreads();
    for (int t = threadIdx.x, z = 0; t < r * r; t += kStepNT, ++z) {  // X1 = 2 X0 - X0 T
      const int a = t / r, b = t - a * r;
      double x = 2.0 * X[a * 16 + b];
      for (int p = 0; p < r; ++p) x = __fma_rn(-X[a * 16 + p], Tm[p * 16 + b], x);
      t1[z & 1] = x;
    }
    __syncthreads();
    for (int t = threadIdx.x, z = 0; t < r * r; t += kStepNT, ++z) X[(t / r) * 16 + t % r] = t1[z & 1];
    __syncthreads();
  }

  // u = P_perp d (or d); ||u||^2 partial sums into scalar slot `slot`.
  // Barriers inside; callers read the slot after their next barrier.
  __device__ void residual(int slot) const {
    float x[R];
    if (project) {
      float acc[R];
#pragma unroll
      for (int l = 0; l < R; ++l) acc[l] = 0.f;
      for (int i = threadIdx.x; i < m; i += kStepNT) {
        const float di = d[i];
#pragma unroll
        for (int l = 0; l < R; ++l) acc[l] = fmaf(Wt[l * ms + i], di, acc[l]);
      }
      put_coefs(acc);
      __syncthreads();
      solve(x);
    }
    float nn = 0.f;
    for (int i = threadIdx.x; i < m; i += kStepNT) {
      float s = d[i];
      if (project)
#pragma unroll
        for (int l = 0; l < R; ++l) s = fmaf(-Wt[l * ms + i], x[l], s);
      u[i] = s;
      nn = fmaf(s, s, nn);
    }
    put_scal(slot, nn);
  }

  // d = A_G s - y from the support's columns (own rows; no barrier inside)
  __device__ void fresh_d() const {
    const float* y = pr.y + static_cast<size_t>(k) * m;
    const float* s = sv(par);
    for (int i = threadIdx.x; i < m; i += kStepNT) {
      float t = 0.f;
      for (int e = 0; e < nl; ++e) t = fmaf(ag(e)[i], s[e], t);
      d[i] = t - y[i];
    }
  }

  // gG_e = (column e)^T u, a warp per entry, four entries at a time
  __device__ void support_gradient() const {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int e0 = 4 * w; e0 < nl; e0 += 4 * kStepNW) {
      const float* c0 = ag(e0);
      const float* c1 = ag(min(e0 + 1, nl - 1));
      const float* c2 = ag(min(e0 + 2, nl - 1));
      const float* c3 = ag(min(e0 + 3, nl - 1));
      float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
      for (int i = lane; i < m; i += 32) {
        const float ui = u[i];
        a0 = fmaf(c0[i], ui, a0);
        a1 = fmaf(c1[i], ui, a1);
        a2 = fmaf(c2[i], ui, a2);
        a3 = fmaf(c3[i], ui, a3);
      }
      a0 = warp_sum(a0); a1 = warp_sum(a1); a2 = warp_sum(a2); a3 = warp_sum(a3);
      if (lane < 4 && e0 + lane < nl) gG[e0 + lane] = lane == 0 ? a0 : lane == 1 ? a1 : lane == 2 ? a2 : a3;
    }
  }

  // With gG ready (after a barrier): v = A_G g_G, p = P_perp v (own
  // rows), num = ||g_G||^2, den = ||p||^2.  Two barriers.
  __device__ void curvature(float& num, float& den) const {
    const int lane = threadIdx.x & 31;
    float acc[R], x[R];
#pragma unroll
    for (int l = 0; l < R; ++l) acc[l] = 0.f;
    for (int i = threadIdx.x; i < m; i += kStepNT) {
      float t = 0.f;
      for (int e = 0; e < nl; ++e) t = fmaf(ag(e)[i], gG[e], t);
      v[i] = t;
      if (project)
#pragma unroll
        for (int l = 0; l < R; ++l) acc[l] = fmaf(Wt[l * ms + i], t, acc[l]);
    }
    if (project) put_coefs(acc);
    float t = 0.f;
    for (int e = lane; e < nl; e += 32) t = fmaf(gG[e], gG[e], t);
    num = warp_sum(t);
    __syncthreads();
    if (project) solve(x);
    float nn = 0.f;
    for (int i = threadIdx.x; i < m; i += kStepNT) {
      float s = v[i];
      if (project)
#pragma unroll
        for (int l = 0; l < R; ++l) s = fmaf(-Wt[l * ms + i], x[l], s);
      p[i] = s;
      nn = fmaf(s, s, nn);
    }
    put_scal(0, nn);
    __syncthreads();
    den = get_scal(0);
  }

  // The IHT sweeps sw .. te-1 that need no pass over A_k (see the head of
  // the file); ||u||^2 lies in scalar slot 1 + (sw & 1).  have_ref: gmax and
  // uref of an earlier pass.  Returns the first sweep that needs a pass, or te.
  __device__ int sweeps(int sw, bool have_ref, float gmax) {
    const int lane = threadIdx.x & 31;
    const float N = pr.nmax[k];
    for (; sw < te; ++sw) {
      __syncthreads();
      const float nu = sqrtf(get_scal(1 + (sw & 1)));
      support_gradient();
      __syncthreads();
      float num, den;
      float nd = 0.f;
      if (have_ref) {
        for (int i = threadIdx.x; i < m; i += kStepNT) nd = fmaf(u[i] - uref[i], u[i] - uref[i], nd);
        put_scal(3, nd);
      }
      curvature(num, den);
      if (!(den > 0.f)) return te;  // s is stationary: the remaining sweeps keep it
      const float mu = num / den;
      const float* s = sv(par);
      float vmin = INFINITY;
      for (int e = lane; e < nl; e += 32) vmin = fminf(vmin, fabsf(fmaf(-mu, gG[e], s[e])));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
      float bound = N * nu;
      if (have_ref) bound = fminf(bound, fmaf(N, sqrtf(get_scal(3)), gmax));
      bound = bound * mu * 1.001f;
      // all comparisons are false for NaN: such a column takes the full path
      if (!(nl == rho && isfinite(mu) && (bound < vmin || rho >= n))) return sw;
      float* s2 = sv(par ^ 1);
      for (int e = threadIdx.x; e < nl; e += kStepNT) s2[e] = fmaf(-mu, gG[e], s[e]);
      par ^= 1;
      float nn = 0.f;
      for (int i = threadIdx.x; i < m; i += kStepNT) {
        d[i] = fmaf(-mu, v[i], d[i]);
        const float t = fmaf(-mu, p[i], u[i]);
        u[i] = t;
        nn = fmaf(t, t, nn);
      }
      put_scal(1 + ((sw + 1) & 1), nn);
    }
    return te;
  }

  // vector of the column's next pass: x_i, times the row scales of the FP8 forms
  __device__ void store_vec(int i, float x) const {
    const int planes = pr.L.et == 3 ? 2 : 1;
    float* out = pr.uvec + static_cast<size_t>(k) * planes * pr.astride;
    if (pr.L.et < 2) {
      out[i] = x;
    } else {
      const size_t o = (static_cast<size_t>(k) * m + i) * planes;
      out[i] = x * pr.rscale[o];
      if (planes == 2) out[pr.astride + i] = x * pr.rscale[o + 1];
    }
  }

  // the column waits for g: its state, and its entry in the next list
  __device__ void need_pass(int sw, int list, bool first) const {
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += kStepNT) {
      store_vec(i, u[i]);
      pr.dvec[static_cast<size_t>(k) * pr.astride + i] = d[i];
    }
    const float* s = sv(par);
    for (int e = threadIdx.x; e < nl; e += kStepNT) {
      pr.supj[static_cast<size_t>(k) * rho + e] = sj[e];
      pr.supv[static_cast<size_t>(k) * rho + e] = s[e];
    }
    if (first) {
      for (int t = threadIdx.x; t < m * R; t += kStepNT) {
        const int i = t / R, l = t - i * R;
        pr.Wk[static_cast<size_t>(k) * pr.wstride + t] = Wt[l * ms + i];
      }
      for (int t = threadIdx.x; t < 256; t += kStepNT)
        pr.Gi[static_cast<size_t>(k) * 256 + t] =
            (t >> 4) < r && (t & 15) < r ? G[512 + t] : 0.0;
      // AG_k keyed by support slot from here on (slots move only when entries
      // of the given support were dropped)
      for (int e = 0; e < nl; ++e) {
        if (src[e] == e) continue;
        const float* from = pr.AG + (static_cast<size_t>(k) * rho + src[e]) * pr.astride;
        float* to = pr.AG + (static_cast<size_t>(k) * rho + e) * pr.astride;
        for (int i = threadIdx.x; i < m; i += kStepNT) to[i] = from[i];
      }
    }
    if (threadIdx.x == 0) {
      pr.nsup[k] = nl;
      pr.sweep[k] = sw;
      T.list[static_cast<size_t>(list & 1) * T.ncols + atomicAdd(&T.cnt[list], 1)] = c;
    }
  }

  // b_k, the vector of the final pass and S_k (ascending by index)
  __device__ void finish(bool store_s) const {
    __syncthreads();
    if (pr.mode == kModeInit) {
      for (int i = threadIdx.x; i < m; i += kStepNT) store_vec(i, -d[i]);
    } else {
      float acc[R], x[R];
#pragma unroll
      for (int l = 0; l < R; ++l) acc[l] = 0.f;
      for (int i = threadIdx.x; i < m; i += kStepNT) {
        const float di = -d[i];
#pragma unroll
        for (int l = 0; l < R; ++l) acc[l] = fmaf(Wt[l * ms + i], di, acc[l]);
      }
      put_coefs(acc);
      __syncthreads();
      const float own = solve(x);
      if (threadIdx.x < r) pr.B[static_cast<size_t>(k) * r + threadIdx.x] = own;
      if (pr.mode == kModeIter)
        for (int i = threadIdx.x; i < m; i += kStepNT) {
          float s = d[i];
#pragma unroll
          for (int l = 0; l < R; ++l) s = fmaf(Wt[l * ms + i], x[l], s);
          store_vec(i, s);
        }
    }
    if (store_s) {
      const float* s = sv(par);
      for (int e = threadIdx.x; e < nl; e += kStepNT) {
        const int je = sj[e];
        int pos = 0;
        for (int f = 0; f < nl; ++f) pos += sj[f] < je;
        pr.S_idx[static_cast<size_t>(k) * rho + pos] = je;
        pr.S_val[static_cast<size_t>(k) * rho + pos] = s[e];
      }
    }
  }
};

// The first step of a column (modes ITER and LS): W_k from the column chunks'
// partial sums, Gram and inverse, u, and the sweeps.  Latency-bound (about a
// dozen barriers and r x r chains per column), so the column gets 128 threads
// and as many columns as fit run at once.
template <int R>
__global__ void __launch_bounds__(kStepNT, 8)
    step_first_kernel(const StreamTable T, int use_ag) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int lane = threadIdx.x & 31;
  for (int c = blockIdx.x; c < T.ncols; c += gridDim.x) {
    const StreamProblem& pr = T.probs[prob_of(T, c)];
    const StepCarve cv = step_carve(R, pr.L.m, pr.L.n, pr.L.rho, pr.astride, use_ag, false);
    Step<R> s(T, pr, smem, cv, use_ag);
    s.c = c;
    s.k = c - pr.col0;
    const int m = s.m, rho = s.rho, k = s.k;
    __syncthreads();  // the previous column is done with the buffers
    // the given support, entries outside the column dropped
    __shared__ int snl;
    if (threadIdx.x < 32) {
      int cnt = 0;
      for (int e0 = 0; e0 < rho; e0 += 32) {
        const int e = e0 + lane;
        const int j = e < rho ? pr.S_idx[static_cast<size_t>(k) * rho + e] : -1;
        const float x = e < rho ? pr.S_val[static_cast<size_t>(k) * rho + e] : 0.f;
        const bool in = j >= 0 && j < s.n;
        const unsigned b = __ballot_sync(0xffffffffu, in);
        if (in) {
          const int at = cnt + __popc(b & ((1u << lane) - 1));
          s.sj[at] = j;
          s.svb[at] = x;
          s.src[at] = e;
        }
        cnt += __popc(b);
      }
      if (lane == 0) snl = cnt;
    }
    const float* wp = pr.Wp + static_cast<size_t>(k) * pr.ncw * pr.wstride;
    for (int t4 = threadIdx.x; t4 < pr.wstride / 4; t4 += kStepNT) {
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
      for (int cc = 0; cc < pr.ncw; ++cc) {
        const float4 a = __ldcg(reinterpret_cast<const float4*>(wp + static_cast<size_t>(cc) * pr.wstride) + t4);
        x.x += a.x; x.y += a.y; x.z += a.z; x.w += a.w;
      }
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        const int t = 4 * t4 + z, i = t / R, l = t - i * R;
        if (i < m) s.Wt[l * s.ms + i] = z == 0 ? x.x : z == 1 ? x.y : z == 2 ? x.z : x.w;
      }
    }
    __syncthreads();
    s.nl = snl;
    s.stage_support();
    s.gram_inverse();
    s.load_inverse(s.G + 512);
    s.fresh_d();
    if (pr.mode == kModeLS || s.te == 0) {
      s.finish(pr.mode == kModeIter);
      continue;
    }
    __syncthreads();
    s.residual(1);
    const int sw = s.sweeps(0, false, 0.f);
    if (sw < s.te) s.need_pass(sw, 0, true);
    else s.finish(true);
  }
}

// ---- HardThreshold of v (n entries) on one CTA --------------------------------
// The rho largest keys (|v|, then the lower index) of vv into sel[0..K),
// K = min(rho, n): 8-bit radix select on the float bits, ties by index.
__device__ __forceinline__ int topk_radix(const float* vv, int n, int rho, int* hist, int* ties,
                                          int* sel) {
  const int K = min(rho, n), lane = threadIdx.x & 31;
  int* info = hist + 256;  // [0] digit, [1] remaining, [2] ties, [3] selected
  unsigned prefix = 0, mask = 0;
  if (threadIdx.x == 0) info[1] = K;
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int t = threadIdx.x; t < 256; t += kStepNT) hist[t] = 0;
    __syncthreads();
    for (int j0 = threadIdx.x - lane; j0 < n; j0 += kStepNT) {
      const int j = j0 + lane;
      const unsigned key = j < n ? __float_as_uint(fabsf(vv[j])) : 0u;
      const bool in = j < n && (key & mask) == prefix;
      const unsigned digit = in ? ((key >> shift) & 255u) : 256u;
      const unsigned peers = __match_any_sync(0xffffffffu, digit);
      if (in && (__ffs(peers) - 1) == lane) atomicAdd(&hist[digit], __popc(peers));
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      const int need = info[1];
      int own[8], tot = 0;  // bins 255 - 8 lane .. 248 - 8 lane
#pragma unroll
      for (int z = 0; z < 8; ++z) { own[z] = hist[255 - 8 * lane - z]; tot += own[z]; }
      int incl = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += up;
      }
      const int excl = incl - tot;
      if (excl < need && incl >= need) {
        int acc = excl;
#pragma unroll
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
  const int need = info[1];
  __syncthreads();
  if (threadIdx.x == 0) { info[2] = 0; info[3] = 0; }
  __syncthreads();
  for (int j = threadIdx.x; j < n; j += kStepNT) {
    const unsigned key = __float_as_uint(fabsf(vv[j]));
    if (key > prefix) sel[atomicAdd(&info[3], 1)] = j;
    else if (key == prefix) ties[atomicAdd(&info[2], 1)] = j;
  }
  __syncthreads();
  const int nt = info[2];
  for (int t = threadIdx.x; t < nt; t += kStepNT) {
    int rank = 0;
    for (int z = 0; z < nt; ++z) rank += ties[z] < ties[t];
    if (rank < need) sel[info[3] + rank] = ties[t];
  }
  __syncthreads();
  // in key order: the order in which the threads found them is arbitrary
  for (int t = threadIdx.x; t < K; t += kStepNT) {
    const uint64_t kj = ht_key(vv[sel[t]], sel[t]);
    int rank = 0;
    for (int z = 0; z < K; ++z) rank += ht_key(vv[sel[z]], sel[z]) > kj;
    ties[rank] = sel[t];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < K; t += kStepNT) sel[t] = ties[t];
  __syncthreads();
  return K;
}

// One listed column after its pass: HardThreshold with g, then the sweeps
// that need no further pass.  zero: the first sweep of the initialisation
// (s = 0: the support is the rho largest |g_j|, its values still 0).
template <int R>
__global__ void __launch_bounds__(kStepNT, 6)
    step_next_kernel(const StreamTable T, int round, int zero, int use_ag) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int lane = threadIdx.x & 31;
  const int count = zero ? T.ncols : T.cnt[round];
  for (int at = blockIdx.x; at < count; at += gridDim.x) {
    const int c = zero ? at : T.list[static_cast<size_t>(round & 1) * T.ncols + at];
    const StreamProblem& pr = T.probs[prob_of(T, c)];
    const StepCarve cv = step_carve(R, pr.L.m, pr.L.n, pr.L.rho, pr.astride, use_ag, true);
    Step<R> s(T, pr, smem, cv, use_ag);
    s.c = c;
    s.k = c - pr.col0;
    const int m = s.m, n = s.n, rho = s.rho, k = s.k;
    float* vv = reinterpret_cast<float*>(smem + cv.vv);
    int* ties = reinterpret_cast<int*>(smem + cv.tie);
    int* sel = ties + n;                               // 2 rho + 8 entries
    int* hist = reinterpret_cast<int*>(smem + cv.hist);
    int* info = hist + 256;
    int* removed = reinterpret_cast<int*>(smem + cv.lists);
    int* added = removed + max(rho, 1);
    const float* g = pr.g + static_cast<size_t>(k) * pr.L.ns;
    if (s.te == 0) continue;  // (a problem of the batch without IHT)
    __syncthreads();
    const int sw = zero ? 0 : pr.sweep[k];
    s.nl = zero ? 0 : pr.nsup[k];
    for (int e = threadIdx.x; e < rho; e += kStepNT) {
      s.src[e] = e;
      if (e < s.nl) {
        s.sj[e] = pr.supj[static_cast<size_t>(k) * rho + e];
        s.svb[e] = pr.supv[static_cast<size_t>(k) * rho + e];
      }
    }
    for (int i = threadIdx.x; i < m; i += kStepNT)
      s.d[i] = zero ? -pr.y[static_cast<size_t>(k) * m + i]
                    : pr.dvec[static_cast<size_t>(k) * pr.astride + i];
    if (s.project) {
      for (int t = threadIdx.x; t < m * R; t += kStepNT) {
        const int i = t / R, l = t - i * R;
        s.Wt[l * s.ms + i] = pr.Wk[static_cast<size_t>(k) * pr.wstride + t];
      }
      s.load_inverse(pr.Gi + static_cast<size_t>(k) * 256);
    }
    for (int j = threadIdx.x; j < n; j += kStepNT) vv[j] = __ldcg(g + j);
    __syncthreads();
    s.stage_support();
    bool stopped = false;
    float mu = 0.f;
    if (zero) {
      // support of the zero start
      const int K = topk_radix(vv, n, rho, hist, ties, sel);
      for (int e = threadIdx.x; e < K; e += kStepNT) {
        s.sj[e] = sel[e];
        s.svb[e] = 0.f;
      }
      s.nl = K;
      __syncthreads();
      for (int t = threadIdx.x; t < K * m; t += kStepNT) {
        const int e = t / m, i = t - e * m;
        const float a = stream_elem(pr, k, i, s.sj[e]);
        if (s.agsm) s.agsm[static_cast<size_t>(e) * pr.astride + i] = a;
        pr.AG[(static_cast<size_t>(k) * rho + e) * pr.astride + i] = a;
      }
    }
    s.residual(1);  // u (the vector of the pass), ||u||^2 not needed here
    for (int e = threadIdx.x; e < s.nl; e += kStepNT) s.gG[e] = vv[s.sj[e]];
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += kStepNT) s.uref[i] = s.u[i];
    float num, den, gmax = 0.f;
    s.curvature(num, den);
    bool kept = true;
    if (!(den > 0.f)) {
      stopped = true;
    } else {
      mu = num / den;
      if (!isfinite(mu)) {
        if (threadIdx.x == 0) report_error(pr.err, kErrNaN, k);
        mu = 0.f;
      }
      for (int j = threadIdx.x; j < n; j += kStepNT) vv[j] = -mu * vv[j];
      if (threadIdx.x == 0) info[3] = 0;
      __syncthreads();
      float* snew = s.sv(1);
      const int nl = s.nl;
      for (int e = threadIdx.x; e < nl; e += kStepNT) {
        const float x = fmaf(-mu, s.gG[e], s.svb[e]);
        snew[e] = x;
        vv[s.sj[e]] = x;
      }
      __syncthreads();
      s.par = 1;
      // candidates: when the support holds rho entries, nothing below the
      // smallest of them can enter
      int K = -1;
      if (nl == rho) {
        float t0 = INFINITY;
        for (int e = lane; e < nl; e += 32) t0 = fminf(t0, fabsf(snew[e]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t0 = fminf(t0, __shfl_xor_sync(0xffffffffu, t0, o));
        const int cap = 2 * rho + 8;
        for (int j = threadIdx.x; j < n; j += kStepNT)
          if (fabsf(vv[j]) >= t0) {
            const int slot = atomicAdd(&info[3], 1);
            if (slot < cap) sel[slot] = j;
          }
        __syncthreads();
        const int cn = info[3];
        if (cn == rho) {
          K = 0;  // the support itself: kept
        } else if (cn <= cap && cn > rho) {
          for (int t = threadIdx.x; t < cn; t += kStepNT) {
            const uint64_t kj = ht_key(vv[sel[t]], sel[t]);
            int rank = 0;
            for (int z = 0; z < cn; ++z) rank += ht_key(vv[sel[z]], sel[z]) > kj;
            if (rank < rho) ties[rank] = sel[t];
          }
          __syncthreads();
          for (int t = threadIdx.x; t < rho; t += kStepNT) sel[t] = ties[t];
          __syncthreads();
          K = rho;
        }
      }
      if (K < 0) K = topk_radix(vv, n, rho, hist, ties, sel);
      if (K > 0) {
        // slots of the entries that left take the ones that entered (both in
        // slot / selection order)
        int nrem = 0, nadd = 0;
        if (threadIdx.x < 32) {
          for (int e0 = 0; e0 < rho; e0 += 32) {
            const int e = e0 + lane;
            bool gone = e < K && e >= nl;  // an unused slot
            if (e < nl) {
              gone = true;
              for (int f = 0; f < K; ++f) gone = gone && sel[f] != s.sj[e];
            }
            const unsigned b = __ballot_sync(0xffffffffu, gone);
            if (gone) removed[nrem + __popc(b & ((1u << lane) - 1))] = e;
            nrem += __popc(b);
          }
          for (int f0 = 0; f0 < K; f0 += 32) {
            const int f = f0 + lane;
            bool in = f < K;
            if (in)
              for (int e = 0; e < nl; ++e) in = in && s.sj[e] != sel[f];
            const unsigned b = __ballot_sync(0xffffffffu, in);
            if (in) added[nadd + __popc(b & ((1u << lane) - 1))] = sel[f];
            nadd += __popc(b);
          }
          if (lane == 0) { info[4] = nrem; info[5] = nadd; }
        }
        __syncthreads();
        nadd = min(info[5], info[4]);
        s.nl = K;
        kept = nadd == 0 && K == nl;
        for (int t = threadIdx.x; t < nadd; t += kStepNT) {
          s.sj[removed[t]] = added[t];
          snew[removed[t]] = vv[added[t]];
        }
        for (int t = threadIdx.x; t < nadd * m; t += kStepNT) {
          const int z = t / m, i = t - z * m;
          const float a = stream_elem(pr, k, i, added[z]);
          if (s.agsm) s.agsm[static_cast<size_t>(removed[z]) * pr.astride + i] = a;
          pr.AG[(static_cast<size_t>(k) * rho + removed[z]) * pr.astride + i] = a;
        }
      }
      __syncthreads();
      // largest |g| outside the new support
      for (int e = threadIdx.x; e < s.nl; e += kStepNT) vv[s.sj[e]] = INFINITY;
      __syncthreads();
      for (int j = threadIdx.x; j < n; j += kStepNT)
        if (!isinf(vv[j])) gmax = fmaxf(gmax, fabsf(__ldcg(g + j)));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
      if (lane == 0) s.scal(0)[threadIdx.x >> 5] = gmax;
      __syncthreads();
#pragma unroll
      for (int w = 0; w < kStepNW; ++w) gmax = fmaxf(gmax, s.scal(0)[w]);
      if (kept) {
        float nn = 0.f;
        for (int i = threadIdx.x; i < m; i += kStepNT) {
          s.d[i] = fmaf(-mu, s.v[i], s.d[i]);
          const float t = fmaf(-mu, s.p[i], s.u[i]);
          s.u[i] = t;
          nn = fmaf(t, t, nn);
        }
        s.put_scal(1 + ((sw + 1) & 1), nn);
      } else {
        s.fresh_d();
        __syncthreads();
        s.residual(1 + ((sw + 1) & 1));
      }
    }
    const int nx = stopped ? s.te : s.sweeps(sw + 1, true, gmax);
    if (nx < s.te) s.need_pass(nx, round + 1, false);
    else s.finish(true);
  }
}

}  // namespace stream
}  // namespace lrs
