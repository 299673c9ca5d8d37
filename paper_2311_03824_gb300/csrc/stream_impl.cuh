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
// (the 1e-3 covers the rounding of mu and of the norms, m / 4 2^-24 with m at
// most 11000; kTinySq what the squares lose below float32's range).  After a pass
// at u_ref has given g, the same holds with max_{j not in G} |g_j| + N_k (||u -
// u_ref|| + (m + 4) 2^-24 ||u_ref||) in the place of N_k ||u||: the last term
// bounds the rounding of the pass's sums, which a small max |g_j| says nothing
// about.  Every other sweep goes through g_kernel and the full
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
// Every wait is bounded by wait_ns; on expiry the warp (of a column step: the
// CTA) records kErrTimeout, drains its own copies (bounded) and leaves, with no
// barrier armed again.
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
constexpr int kMaxStage = 4;
// half the spacing below float32's normal range, for 2^15 squares of a sum
constexpr float kTinySq = 4e-41f;

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ bool wait_phase(uint64_t* bar, unsigned parity, unsigned long long wait_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = gtimer();
  while (!mbar_try_wait(bar, parity))
    if (gtimer() - t0 > wait_ns) return false;
  return true;
}

// ------------------------------------------------------------- warp pipeline --
// One warp's ring: `S` stages, full barriers only (the warp that refills a
// stage is the one that has read it).
// Places are byte offsets in the CTA's dynamic shared memory: an access through
// the array itself stays a shared-memory load (a pointer kept in the ring is a
// generic one, with 64-bit addresses).
struct Pipe {
  unsigned base;
  uint64_t* full;
  unsigned stage;        // bytes
  int S;
  int si, st;            // stage of the next piece to issue, to take
  unsigned ph;           // phase bit of the next piece to take
  int flying;            // pieces issued and not taken
  bool dead;
  int* err;
  unsigned long long wait_ns;

  // withhold (test aid): the first stage expects an arrival that never comes
  __device__ void init(unsigned b, uint64_t* f, unsigned stg, int s, unsigned long long w, bool withhold = false) {
    base = b;
    full = f;
    stage = stg;
    S = s;
    si = st = 0;
    ph = 0;
    flying = 0;
    dead = false;
    err = nullptr;
    wait_ns = w;
    if ((threadIdx.x & 31) == 0)
      for (int i = 0; i < S; ++i) mbar_init(&full[i], withhold && i == 0 ? 2 : 1);
    __syncwarp();
  }
  __device__ uint64_t* issue_bar() const { return full + si; }
  __device__ unsigned issue_at() const { return base + static_cast<unsigned>(si) * stage; }
  __device__ void issued() {
    ++flying;
    si = si + 1 == S ? 0 : si + 1;
  }
  __device__ bool wait() const { return wait_phase(full + st, ph, wait_ns); }
  // the oldest piece in flight (every lane waits); taken() when it has been read
  __device__ unsigned take() {
    if (!__all_sync(0xffffffffu, wait())) {
      dead = true;
      if ((threadIdx.x & 31) == 0) report_error(err, kErrTimeout, -1);
    }
    return base + static_cast<unsigned>(st) * stage;
  }
  __device__ void taken() {
    --flying;
    if (++st == S) {
      st = 0;
      ph ^= 1u;
    }
  }
  // before leaving after an expired wait: no copy may land in this CTA's
  // shared memory once it is gone
  __device__ void drain() {
    for (; flying > 0; taken()) wait();
  }
};

__device__ __forceinline__ int prob_of(const StreamTable& T, int c) {
  int p = 0;
  while (p + 1 < T.nprob && T.probs[p + 1].col0 <= c) ++p;
  return p;
}

// ------------------------------------------------------------------ W = A U --
// Rows of a unit (a multiple of 8), rows / 4 x R accumulators per lane.
__host__ __device__ constexpr int w_rows(int R) { return R <= 6 ? 32 : 16; }
// 16-byte chunks of one column's R ranks in the shared copy of U
__host__ __device__ constexpr int w_chunks4(int R) { return (R + 3) / 4; }

// Two multiply-adds in one instruction: (a.x b.x + c.x, a.y b.y + c.y).  The
// pass is bound by instruction issue (R multiply-adds per element), so a pair
// of ranks shares one; rounding is that of two fmaf.
__device__ __forceinline__ void ffma2(unsigned long long& c, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

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
  constexpr int RB = w_rows(R), RT = RB / 4, R2 = (R + 1) / 2, R4 = w_chunks4(R);
  constexpr int pb = ET == 0 ? 4 : ET == 1 ? 2 : 1;
  constexpr int planes = ET == 3 ? 2 : 1;
  constexpr unsigned sub = RB * kTW * pb * planes;  // bytes of one tile of a piece
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int q = lane & 7, ro = lane >> 3;
  // element offsets of this lane's chunk in rows 8 z + ro and 8 z + 4 + ro
  const int off0 = ro * kTW + ((q ^ ro) << 2), off1 = (4 + ro) * kTW + ((q ^ (4 + ro)) << 2);
  float* Us = reinterpret_cast<float*>(smem);
  const unsigned stage = sub * tpp;
  Pipe P;
  P.init(us_bytes + static_cast<unsigned>(wid * S) * stage,
         reinterpret_cast<uint64_t*>(smem + us_bytes + static_cast<size_t>(kSW) * S * stage) +
             wid * kMaxStage,
         stage, S, T.wait_ns, T.withhold == 2 && blockIdx.x == 0 && wid == 0);
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
    // U of a tile as [c][z][q]: ranks 4 z .. 4 z + 3 of column 4 q + c in one
    // 16-byte chunk (zero beyond R), the eight lane groups side by side: a
    // warp's read is one conflict-free wavefront for every R (row-major, the
    // groups lie 16 R bytes apart: 8-way conflicts at R = 8 and 16)
    for (int t = threadIdx.x; t < (b1 - b0) * 32 * R4; t += kStreamNT) {
      const int g = t & 7, z = (t >> 3) % R4, cb = (t >> 3) / R4, c = cb & 3, b = cb >> 2;
      const float* from = pr.Upad + (static_cast<size_t>(b0 + b) * kTW + 4 * g + c) * R + 4 * z;
      float4 x = make_float4(from[0], 0.f, 0.f, 0.f);
      if (4 * z + 1 < R) x.y = from[1];
      if (4 * z + 2 < R) x.z = from[2];
      if (4 * z + 3 < R) x.w = from[3];
      reinterpret_cast<float4*>(Us)[t] = x;
    }
    __syncthreads();
    const int u0 = as.idx * kSW + wid, ustep = as.cnt * kSW;
    const int dk = ustep / nrb, db = ustep - dk * nrb;  // a unit step in (column, row block)
    int pu = u0, pk = u0 / nrb, prb = u0 - pk * nrb, pbt = b0;  // next piece to issue
    auto issue = [&]() {
      if (pu >= nunits) return;
      const int i0 = prb * RB, nr = min(RB, m - i0);
      const int nt = min(tpp, b1 - pbt);
      const unsigned hb = static_cast<unsigned>(nr * kTW * pb);
      unsigned char* dst = smem + P.issue_at();
      if (lane == 0) mbar_arrive_expect_tx(P.issue_bar(), hb * planes * nt);
      __syncwarp();
      if (lane < nt * planes) {
        const int t = lane / planes, pl = lane - t * planes;
        const unsigned char* src = A + (static_cast<size_t>(pk) * ntile + pbt + t) * tb +
                                   static_cast<size_t>(pl) * m * kTW +
                                   static_cast<size_t>(i0) * kTW * pb;
        bulk_copy_g2s(dst + t * sub + pl * hb, src, hb, P.issue_bar());
      }
      P.issued();
      pbt += nt;
      if (pbt >= b1) {
        pbt = b0;
        pu += ustep;
        pk += dk;
        prb += db;
        if (prb >= nrb) {
          prb -= nrb;
          ++pk;
        }
      }
    };
    for (int i = 0; i < S; ++i) issue();
    int k = u0 / nrb, rb = u0 - k * nrb;
    auto next_unit = [&]() {
      k += dk;
      rb += db;
      if (rb >= nrb) {
        rb -= nrb;
        ++k;
      }
    };
    for (int u = u0; u < nunits; u += ustep, next_unit()) {
      const int i0 = rb * RB, nr = min(RB, m - i0);
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
      // the column's support: entries 0..63 in registers, their tiles beside them
      const int* sidx = pr.S_idx + static_cast<size_t>(k) * rho;
      const int j0 = lane < rho ? sidx[lane] : -1, j1 = 32 + lane < rho ? sidx[32 + lane] : -1;
      const int jt0 = j0 < n ? j0 >> 5 : -1, jt1 = j1 < n ? j1 >> 5 : -1;  // (-1 >> 5 = -1)
      unsigned long long acc[RT][R2];  // pairs of ranks
#pragma unroll
      for (int t = 0; t < RT; ++t)
#pragma unroll
        for (int p = 0; p < R2; ++p) acc[t][p] = 0ull;
      for (int b = b0; b < b1; b += tpp) {
        unsigned so = P.take();
        if (P.dead) break;
        const int nt = min(tpp, b1 - b);
        for (int tt = 0; tt < nt; ++tt, so += sub) {
          const unsigned char* st = smem + so;
          const float4* Ut = reinterpret_cast<const float4*>(smem) + (b + tt - b0) * 32 * R4 + q;
          float4 av[RT];
#pragma unroll
          for (int t = 0; t < RT; ++t) {
            // rows at or beyond nr hold stale data: their sums are not stored
            const int off = (t & 1 ? off1 : off0) + (t >> 1) * 8 * kTW;
            if constexpr (ET == 0) {
              av[t] = *reinterpret_cast<const float4*>(st + static_cast<size_t>(off) * 4);
            } else if constexpr (ET == 1) {
              const uint2 raw = *reinterpret_cast<const uint2*>(st + static_cast<size_t>(off) * 2);
              av[t] = make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u),
                                  __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xffff0000u));
            } else if constexpr (ET == 2) {  // raw values; the row's scale multiplies the sum
              av[t] = static_cast<float4>(*reinterpret_cast<const __nv_fp8x4_e4m3*>(st + off));
            } else {
              const float4 fh = static_cast<float4>(*reinterpret_cast<const __nv_fp8x4_e4m3*>(st + off));
              const float4 fl = static_cast<float4>(
                  *reinterpret_cast<const __nv_fp8x4_e4m3*>(st + nr * kTW + off));
              av[t] = make_float4(fmaf(fl.x, s2[t], fh.x * s1[t]), fmaf(fl.y, s2[t], fh.y * s1[t]),
                                  fmaf(fl.z, s2[t], fh.z * s1[t]), fmaf(fl.w, s2[t], fh.w * s1[t]));
            }
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            unsigned long long uu[2 * R4];
#pragma unroll
            for (int z = 0; z < R4; ++z) {
              const float4 w = Ut[(c * R4 + z) * 8];
              uu[2 * z] = pack2(w.x, w.y);
              uu[2 * z + 1] = pack2(w.z, w.w);
            }
#pragma unroll
            for (int t = 0; t < RT; ++t) {
              const float x = c == 0 ? av[t].x : c == 1 ? av[t].y : c == 2 ? av[t].z : av[t].w;
              const unsigned long long xx = pack2(x, x);
#pragma unroll
              for (int p = 0; p < R2; ++p) ffma2(acc[t][p], xx, uu[p]);
            }
          }
          // support columns that lie in this tile -> AG_k (entry e of the input support)
          auto extract = [&](unsigned in, int j, int e0) {
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
          };
          if (const unsigned in = __ballot_sync(0xffffffffu, jt0 == b + tt)) extract(in, j0, 0);
          if (rho > 32) {
            if (const unsigned in = __ballot_sync(0xffffffffu, jt1 == b + tt)) extract(in, j1, 32);
            for (int e0 = 64; e0 < rho; e0 += 32) {
              const int j = e0 + lane < rho ? sidx[e0 + lane] : -1;
              extract(__ballot_sync(0xffffffffu, j < n && j >> 5 == b + tt), j, e0);
            }
          }
        }
        P.taken();
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
          const float2 pr2 = unpack2(acc[t][l >> 1]);
          float v = l & 1 ? pr2.y : pr2.x;
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
// Column steps come in three variants by the column's size (stream_plan):
// 128 threads with the support's columns in shared memory, 256 threads with
// them, 256 threads reading them from AG_k.
__host__ __device__ constexpr int step_threads(int variant) { return variant == 0 ? 128 : 256; }
__host__ __device__ constexpr bool step_staged(int variant) { return variant < 2; }

struct StepCarve {
  unsigned dbl, Lf, Q, u, p, uref, gG, sv, sj, red, ag, vv, tie, hist, lists, total;
  int ms, rp;
};
// Shared memory of a column step; next: the arrays of the full HardThreshold.
__host__ __device__ inline StepCarve step_carve(int R, int m, int n, int rho, int astride,
                                                int variant, bool next) {
  StepCarve c;
  size_t o = 0;
  c.rp = ((rho > 0 ? rho : 1) + 3) & ~3;
  const size_t rp = c.rp;
  auto put = [&](size_t bytes) {
    const unsigned at = static_cast<unsigned>(o);
    o += a16(bytes);
    return at;
  };
  c.ms = m | 1;
  c.dbl = put(static_cast<size_t>(3) * 256 * 8);
  c.Lf = put(256 * 4);
  c.ag = put(step_staged(variant) ? rp * static_cast<size_t>(astride) * 4 : 0);
  c.Q = put(static_cast<size_t>(R) * c.ms * 4);
  c.u = put(static_cast<size_t>(m) * 4);
  c.p = put(static_cast<size_t>(m) * 4);
  c.uref = put(next ? static_cast<size_t>(m) * 4 : 0);
  c.gG = put(rp * 4);
  c.sv = put(2 * rp * 4);
  c.sj = put(rp * 4);
  c.red = put((8 * 16 + 5 * 8) * 4);
  c.vv = put(next ? static_cast<size_t>(n) * 4 : 0);
  c.tie = put(next ? (static_cast<size_t>(n) + 2 * rp + 8) * 4 : 0);
  c.hist = put(next ? (256 + 16) * 4 : 0);
  c.lists = put(next ? 2 * rp * 4 : 0);
  c.total = static_cast<unsigned>(o);
  return c;
}

// Gram of W (columns at Q + l ms) and its factor in FP64, one warp: L^{-1} at
// G + 512, rounded in Lf, its diagonal's remainder at G + 256.  Out of line: the
// column steps are short and run on cold instruction caches.
static __device__ __noinline__ void factor_f64(const float* Q, int ms, int m, int r, int k, double* G, float* Lf, int* err) {
  __shared__ double iL[16];
  const int lane = threadIdx.x & 31, ne = r * (r + 1) / 2;
  double *L = G + 256, *Li = G + 512;
  float* dlo = reinterpret_cast<float*>(L);
  for (int t = 0; t < ne; ++t) {
    int a = 0;
    while ((a + 1) * (a + 2) / 2 <= t) ++a;
    const int b = t - a * (a + 1) / 2;
    double g = 0.0;
    for (int i = lane; i < m; i += 32)
      g = __fma_rn(static_cast<double>(Q[a * ms + i]), static_cast<double>(Q[b * ms + i]), g);
    g = warp_sum(g);
    if (lane == 0) G[a * 16 + b] = G[b * 16 + a] = g;
  }
  __syncwarp();
  if (!chol_inverse_warp(G, L, Li, iL, r, 16) && lane == 0) report_error(err, kErrNotSPD, k);
  __syncwarp();
  for (int t = lane; t < 256; t += 32) {
    const int i = t >> 4, q = t & 15;
    if (q > i || i >= r) Li[t] = 0.0;
    Lf[t] = static_cast<float>(Li[t]);
    if (q == i) dlo[i] = static_cast<float>(Li[t] - static_cast<double>(Lf[t]));
  }
}

// One column on one CTA.  P_perp is applied through an orthonormal basis Q of
// range(W_k): Q = W L^{-T} with G = W^T W = L L^T, so P v = v - Q (Q^T v), the
// residual of the LS step is e = Q Q^T r - r and b = L^{-T} (Q^T r): one matrix
// in shared memory and no r x r solve inside the sweeps.
// Slots of scal: 0 ||g_G||^2, 1 / 2 ||u||^2 (by sweep parity), 3 ||u - uref||^2,
// 4 ||P A_G g_G||^2.
template <int R, int V>
struct Step {
  static constexpr int NT = step_threads(V), NW = NT / 32;
  static constexpr int RN = R <= 2 ? 2 : R <= 4 ? 4 : R <= 8 ? 8 : 16;
  const StreamTable& T;
  const StreamProblem& pr;  // shared-memory copy
  int k, c, m, n, r, rho, te, ms, rp, nl, par, as;
  float *Q, *u, *p, *uref, *gG, *svb, *red, *Lf;
  int* sj;
  double* G;     // Gram, then L (fallback), L^{-1} at G + 512 (16 x 16 each)
  float* ag;     // support columns: slot e at ag + e as
  bool project;

  __device__ Step(const StreamTable& t, const StreamProblem& prob, unsigned char* smem,
                  const StepCarve& cv)
      : T(t), pr(prob) {
    m = pr.L.m;
    n = pr.L.n;
    r = pr.L.r;
    rho = pr.L.rho;
    te = pr.te;
    as = pr.astride;
    ms = cv.ms;
    rp = cv.rp;
    par = 0;
    nl = 0;
    auto f = [&](unsigned o) { return reinterpret_cast<float*>(smem + o); };
    Q = f(cv.Q); u = f(cv.u); p = f(cv.p); uref = f(cv.uref); gG = f(cv.gG);
    svb = f(cv.sv); red = f(cv.red); Lf = f(cv.Lf);
    sj = reinterpret_cast<int*>(smem + cv.sj);
    G = reinterpret_cast<double*>(smem + cv.dbl);
    project = pr.mode != kModeInit;
  }
  __device__ void at_column(int col, unsigned char* smem, const StepCarve& cv) {
    c = col;
    k = col - pr.col0;
    if constexpr (step_staged(V)) ag = reinterpret_cast<float*>(smem + cv.ag);
    else ag = pr.AG + static_cast<size_t>(k) * rho * as;
  }
  __device__ float* sv(int q) const { return svb + q * rp; }
  __device__ float* ag_global() const { return pr.AG + static_cast<size_t>(k) * rho * as; }

  // ---- staging of AG_k by one bulk copy ----
  __device__ void stage_begin(uint64_t* bar) const {
    if constexpr (step_staged(V)) {
      if (threadIdx.x == 0 && rho > 0) {
        asm volatile("fence.proxy.async;" ::: "memory");  // earlier reads of the buffer first
        const unsigned bytes = static_cast<unsigned>(rho * as * 4);
        mbar_arrive_expect_tx(bar, bytes);
        bulk_copy_g2s(ag, ag_global(), bytes, bar);
      }
    }
  }
  // Every thread waits for the copy; false when the wait ran out: the CTA then
  // leaves by stage_abandon.
  __device__ bool stage_end(uint64_t* bar, unsigned& phase) const {
    bool ok = true;
    if constexpr (step_staged(V)) {
      if (rho > 0) {
        ok = wait_phase(bar, phase, T.wait_ns);
        phase ^= 1u;
      }
    }
    return ok;
  }
  // the copy may still be under way: one more bounded wait, after which the CTA
  // goes without touching the barrier or the buffer again
  __device__ void stage_abandon(uint64_t* bar, unsigned phase) const {
    if (threadIdx.x == 0) {
      report_error(pr.err, kErrTimeout, -1);
      wait_phase(bar, phase ^ 1u, T.wait_ns);
    }
  }

  // ---- reductions ----
  __device__ void put_coefs(const float (&acc)[R]) const {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float v[RN];
#pragma unroll
    for (int l = 0; l < RN; ++l) v[l] = l < R ? acc[l < R ? l : 0] : 0.f;
    const float t = reduce_multi<RN>(v);
    constexpr int step = 32 / RN;
    if (lane % step == 0) red[w * 16 + lane / step] = t;
  }
  // (after a barrier) the coefficients in every thread; returns this lane's own
  __device__ float get_coefs(float (&cf)[R]) const {
    const int lane = threadIdx.x & 31;
    float own = 0.f;
    if (lane < R)
#pragma unroll
      for (int w = 0; w < NW; ++w) own += red[w * 16 + lane];
#pragma unroll
    for (int l = 0; l < R; ++l) cf[l] = __shfl_sync(0xffffffffu, own, l);
    return own;
  }
  __device__ float* scal(int s) const { return red + 8 * 16 + s * 8; }
  __device__ void put_scal(int s, float x) const {
    x = warp_sum(x);
    if ((threadIdx.x & 31) == 0) scal(s)[threadIdx.x >> 5] = x;
  }
  __device__ float get_scal(int s) const {
    float x = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) x += scal(s)[w];
    return x;
  }
  // sum_e AG(i, e) x_e over the support in two interleaved sums; where the
  // columns come from memory, in one such pair per sixteen entries (one sum of
  // 400 put half as much again into U's error), whose loads are in flight
  // together: 3.54 -> 2.65 ms for 4 iterations of n = 2000, q = 100, m = 600,
  // rho = 400.  Staged columns have fewer entries and pay for the longer code
  // (per iteration 47 -> 49 us at n = q = 200, 315 -> 320 at n = 1537, q = 301).
  __device__ float support_row(int i, const float* x) const {
    constexpr int B = 16;
    const float* a = ag + i;
    float t = 0.f, t0 = 0.f, t1 = 0.f;
    int e = 0;
    for (; !step_staged(V) && e + B <= nl; e += B, a += B * as) {
      float v[B];
#pragma unroll
      for (int z = 0; z < B; ++z) v[z] = a[z * as];
      t0 = t1 = 0.f;
#pragma unroll
      for (int z = 0; z < B; z += 4) {
        const float4 xe = *reinterpret_cast<const float4*>(x + e + z);
        t0 = fmaf(v[z], xe.x, t0);
        t1 = fmaf(v[z + 1], xe.y, t1);
        t0 = fmaf(v[z + 2], xe.z, t0);
        t1 = fmaf(v[z + 3], xe.w, t1);
      }
      t += t0 + t1;
    }
    t0 = t1 = 0.f;
    for (; e + 4 <= nl; e += 4, a += 4 * as) {
      const float4 xe = *reinterpret_cast<const float4*>(x + e);
      t0 = fmaf(a[0], xe.x, t0);
      t1 = fmaf(a[as], xe.y, t1);
      t0 = fmaf(a[2 * as], xe.z, t0);
      t1 = fmaf(a[3 * as], xe.w, t1);
    }
    for (; e < nl; ++e, a += as) t0 = fmaf(a[0], x[e], t0);
    return t + (t0 + t1);
  }

  // ---- Gram of W (in Q's buffer), its inverse factor, Q = W L^{-T} in place ----
  // The Gram is summed in double-float from exact products; the factor and
  // its inverse are double-float in one warp's registers (lane = row, then
  // lane = column).  A pivot below 1e-9 of its diagonal or outside float32's
  // range sends Gram and factor to FP64, which also reports a Gram that is not
  // positive.
  // Q's rows take L^{-1} rounded, but the diagonal with what its rounding left
  // (dlo): a column of Q that is off by a common factor of 1 + 3e-8 puts the
  // error into b and e whole, where the rounding of its entries averages out.
  __device__ void factor() const {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ne = r * (r + 1) / 2;
    for (int t0 = 4 * w; t0 < ne; t0 += 4 * NW) {
      const float *pa[4], *pb[4];
      float hi[4], lo[4];
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        const int t = min(t0 + z, ne - 1);
        int a = 0;
        while ((a + 1) * (a + 2) / 2 <= t) ++a;
        pa[z] = Q + a * ms;
        pb[z] = Q + (t - a * (a + 1) / 2) * ms;
        hi[z] = lo[z] = 0.f;
      }
      for (int i = lane; i < m; i += 32)
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const float x = pa[z][i], y = pb[z][i], q = x * y;
          float s, e;
          two_sum(hi[z], q, s, e);
          hi[z] = s;
          lo[z] += e + fmaf(x, y, -q);
        }
      // two halvings leave one entry per lane group of eight, then its sum
#pragma unroll
      for (int h = 2, off = 16; h >= 1; h >>= 1, off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int z = 0; z < h; ++z) {
          const float sh = up ? hi[z] : hi[z + h], sl = up ? lo[z] : lo[z + h];
          const float kh = up ? hi[z + h] : hi[z], kl = up ? lo[z + h] : lo[z];
          float s, e;
          two_sum(kh, __shfl_xor_sync(0xffffffffu, sh, off), s, e);
          hi[z] = s;
          lo[z] = kl + __shfl_xor_sync(0xffffffffu, sl, off) + e;
        }
      }
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) {
        float s, e;
        two_sum(hi[0], __shfl_xor_sync(0xffffffffu, hi[0], off), s, e);
        hi[0] = s;
        lo[0] += __shfl_xor_sync(0xffffffffu, lo[0], off) + e;
      }
      const int t = t0 + (lane >> 3);
      if ((lane & 7) == 0 && t < ne) {
        int a = 0;
        while ((a + 1) * (a + 2) / 2 <= t) ++a;
        const int b = t - a * (a + 1) / 2;
        const double g = static_cast<double>(hi[0]) + static_cast<double>(lo[0]);
        G[a * 16 + b] = g;
        G[b * 16 + a] = g;
      }
    }
    __syncthreads();
    double* Li = G + 512;
    float* dlo = reinterpret_cast<float*>(G + 256);
    if (w == 0) {
      const bool ok = chol_df<R>(G, r, [&](int i, df x) {
        Li[i * 16 + lane] = static_cast<double>(x.h) + static_cast<double>(x.l);
        Lf[i * 16 + lane] = x.h;
        if (i == lane) dlo[i] = x.l;
      });
      if (!ok) {
        factor_f64(Q, ms, m, r, k, G, Lf, pr.err);
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += NT) {
      float x[R];
#pragma unroll
      for (int l = 0; l < R; ++l) x[l] = Q[l * ms + i];
#pragma unroll
      for (int l = 0; l < R; ++l) {
        float s = x[l] * dlo[l];
#pragma unroll
        for (int q = 0; q <= l; ++q) s = fmaf(x[q], Lf[l * 16 + q], s);
        Q[l * ms + i] = s;
      }
    }
    // (every thread goes on with its own rows; other rows after the next barrier)
  }

  // u = P_perp (A_G s - y) for the values sv(par); ||u||^2 into slot `slot`
  // (ready after the caller's next barrier).
  __device__ void residual(int slot) const {
    const float* y = pr.y + static_cast<size_t>(k) * m;
    const float* s = sv(par);
    float acc[R], nn = 0.f;
#pragma unroll
    for (int l = 0; l < R; ++l) acc[l] = 0.f;
    for (int i = threadIdx.x; i < m; i += NT) {
      const float t = support_row(i, s) - y[i];
      u[i] = t;
      if (project) {
#pragma unroll
        for (int l = 0; l < R; ++l) acc[l] = fmaf(Q[l * ms + i], t, acc[l]);
      } else {
        nn = fmaf(t, t, nn);
      }
    }
    if (project) {
      float cf[R];
      put_coefs(acc);
      __syncthreads();
      get_coefs(cf);
      for (int i = threadIdx.x; i < m; i += NT) {
        float t = u[i];
#pragma unroll
        for (int l = 0; l < R; ++l) t = fmaf(-Q[l * ms + i], cf[l], t);
        u[i] = t;
        nn = fmaf(t, t, nn);
      }
    }
    put_scal(slot, nn);
  }

  // gG_e = (column e)^T u, a warp per four entries; ||g_G||^2 into slot 0
  __device__ void support_gradient() const {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float sq = 0.f;
    for (int e0 = 4 * w; e0 < nl; e0 += 4 * NW) {
      const float* a0 = ag + e0 * as;
      const float* a1 = ag + min(e0 + 1, nl - 1) * as;
      const float* a2 = ag + min(e0 + 2, nl - 1) * as;
      const float* a3 = ag + min(e0 + 3, nl - 1) * as;
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      for (int i = lane; i < m; i += 32) {
        const float ui = u[i];
        v[0] = fmaf(a0[i], ui, v[0]);
        v[1] = fmaf(a1[i], ui, v[1]);
        v[2] = fmaf(a2[i], ui, v[2]);
        v[3] = fmaf(a3[i], ui, v[3]);
      }
      const float t = reduce_multi<4>(v);
      const int e = e0 + (lane >> 3);
      if ((lane & 7) == 0 && e < nl) {
        gG[e] = t;
        sq = fmaf(t, t, sq);
      }
    }
    put_scal(0, sq);
  }

  // With gG and slot 0 ready (after a barrier): p = P_perp A_G g_G, num =
  // ||g_G||^2, den = ||p||^2.  Two barriers.
  __device__ void curvature(float& num, float& den, bool have_ref) const {
    num = get_scal(0);
    float acc[R], nd = 0.f;
#pragma unroll
    for (int l = 0; l < R; ++l) acc[l] = 0.f;
    for (int i = threadIdx.x; i < m; i += NT) {
      const float t = support_row(i, gG);
      p[i] = t;
      if (project) {
#pragma unroll
        for (int l = 0; l < R; ++l) acc[l] = fmaf(Q[l * ms + i], t, acc[l]);
      }
      if (have_ref) {
        const float x = u[i] - uref[i];
        nd = fmaf(x, x, nd);
      }
    }
    if (project) put_coefs(acc);
    if (have_ref) put_scal(3, nd);
    __syncthreads();
    float cf[R];
    if (project) get_coefs(cf);
    float nn = 0.f;
    for (int i = threadIdx.x; i < m; i += NT) {
      float t = p[i];
      if (project) {
#pragma unroll
        for (int l = 0; l < R; ++l) t = fmaf(-Q[l * ms + i], cf[l], t);
        p[i] = t;
      }
      nn = fmaf(t, t, nn);
    }
    put_scal(4, nn);
    __syncthreads();
    den = get_scal(4);
  }

  // The IHT sweeps sw .. te-1 that need no pass over A_k (see the head of
  // the file), from u and ||u||^2 in slot 1 + (sw & 1).  have_ref: gmax and
  // uref of an earlier pass.  Returns the first sweep that needs a pass (u is
  // then that of sv(par)), or te.  The last barrier of a sweep is the first
  // of the next one.
  __device__ int sweeps(int sw, bool have_ref, float gmax) {
    const float N = pr.nmax[k];
    __syncthreads();
    for (; sw < te; ++sw) {
      const float nu = sqrtf(get_scal(1 + (sw & 1)) + kTinySq);
      support_gradient();
      __syncthreads();
      float num, den;
      curvature(num, den, have_ref);
      if (!(den > 0.f)) return te;  // s is stationary: the remaining sweeps keep it
      const float mu = num / den;
      float bound = N * nu;
      if (have_ref) bound = fminf(bound, fmaf(N, sqrtf(get_scal(3) + kTinySq), gmax));
      bound = bound * mu * 1.001f;
      // all comparisons are false for NaN: such a column takes the full path
      bool ok = nl == rho && isfinite(mu) && (bound >= 0.f || rho >= n);
      const float* s = sv(par);
      float* s2 = sv(par ^ 1);
      for (int e = threadIdx.x; e < nl; e += NT) {
        const float v = fmaf(-mu, gG[e], s[e]);
        s2[e] = v;
        ok = ok && (bound < fabsf(v) || rho >= n);
      }
      float nn = 0.f;
      for (int i = threadIdx.x; i < m; i += NT) {
        const float t = fmaf(-mu, p[i], u[i]);
        u[i] = t;
        nn = fmaf(t, t, nn);
      }
      put_scal(1 + ((sw + 1) & 1), nn);
      if (!__syncthreads_and(ok)) {
        residual(1 + (sw & 1));  // back to the u of sv(par), as the next step forms it
        return sw;
      }
      par ^= 1;
    }
    return te;
  }

  // vector of the column's next pass: x_i, times the row scales of the FP8 forms
  __device__ void store_vec(int i, float x) const {
    const int planes = pr.L.et == 3 ? 2 : 1;
    float* out = pr.uvec + static_cast<size_t>(k) * planes * as;
    if (pr.L.et < 2) {
      out[i] = x;
    } else {
      const size_t o = (static_cast<size_t>(k) * m + i) * planes;
      out[i] = x * pr.rscale[o];
      if (planes == 2) out[as + i] = x * pr.rscale[o + 1];
    }
  }

  // the column waits for g: its state, and its entry in the next list
  __device__ void need_pass(int sw, int list, bool first) const {
    for (int i = threadIdx.x; i < m; i += NT) store_vec(i, u[i]);
    const float* s = sv(par);
    for (int e = threadIdx.x; e < nl; e += NT) {
      pr.supj[static_cast<size_t>(k) * rho + e] = sj[e];
      pr.supv[static_cast<size_t>(k) * rho + e] = s[e];
    }
    if (first) {
      float* out = pr.Wk + static_cast<size_t>(k) * pr.wstride;
      for (int i = threadIdx.x; i < m; i += NT)
#pragma unroll
        for (int l = 0; l < R; ++l) out[static_cast<size_t>(l) * m + i] = Q[l * ms + i];
      for (int t = threadIdx.x; t < 256; t += NT) pr.Li[static_cast<size_t>(k) * 256 + t] = G[512 + t];
    }
    if (threadIdx.x == 0) {
      pr.nsup[k] = nl;
      pr.sweep[k] = sw;
      T.list[static_cast<size_t>(list & 1) * T.ncols + atomicAdd(&T.cnt[list], 1)] = c;
    }
  }

  // b_k, the vector of the final pass and S_k (ascending by index)
  __device__ void finish(bool store_s) const {
    const float* y = pr.y + static_cast<size_t>(k) * m;
    const float* s = sv(par);
    float acc[R];
#pragma unroll
    for (int l = 0; l < R; ++l) acc[l] = 0.f;
    for (int i = threadIdx.x; i < m; i += NT) {
      const float t = y[i] - support_row(i, s);
      if (project) {
        p[i] = t;
#pragma unroll
        for (int l = 0; l < R; ++l) acc[l] = fmaf(Q[l * ms + i], t, acc[l]);
      } else {
        store_vec(i, t);
      }
    }
    if (project) {
      float cf[R];
      put_coefs(acc);
      __syncthreads();
      get_coefs(cf);
      if (threadIdx.x < 32 && threadIdx.x < r) {  // b = L^{-T} (Q^T (y - A s))
        double b = 0.0;
#pragma unroll
        for (int l = 0; l < R; ++l) b = __fma_rn(G[512 + l * 16 + threadIdx.x], static_cast<double>(cf[l]), b);
        pr.B[static_cast<size_t>(k) * r + threadIdx.x] = static_cast<float>(b);
      }
      if (pr.mode == kModeIter)
        for (int i = threadIdx.x; i < m; i += NT) {  // e = W b + A s - y
          float t = -p[i];
#pragma unroll
          for (int l = 0; l < R; ++l) t = fmaf(Q[l * ms + i], cf[l], t);
          store_vec(i, t);
        }
    }
    if (store_s) {
      for (int e = threadIdx.x; e < nl; e += NT) {
        const int je = sj[e];
        int pos = 0;
        for (int f = 0; f < nl; ++f) pos += sj[f] < je;
        pr.S_idx[static_cast<size_t>(k) * rho + pos] = je;
        pr.S_val[static_cast<size_t>(k) * rho + pos] = s[e];
      }
    }
  }
};

// The problem of column c into shared memory (every thread; ends with a
// barrier, which also separates the previous column's use of the buffers).
__device__ __forceinline__ void load_problem(const StreamTable& T, int c, StreamProblem* spr, int& cur) {
  const int p = T.nprob == 1 ? 0 : prob_of(T, c);
  __syncthreads();
  if (p != cur) {
    const int* from = reinterpret_cast<const int*>(T.probs + p);
    int* to = reinterpret_cast<int*>(spr);
    for (int t = threadIdx.x; t < static_cast<int>(sizeof(StreamProblem) / 4); t += blockDim.x) to[t] = from[t];
    cur = p;
    __syncthreads();
  }
}

// The first step of a column (modes ITER and LS): W_k from the column chunks'
// partial sums, its Gram, Q, u, and the sweeps.  Instruction- and barrier-
// bound (four barriers a sweep), so as many columns as fit run at once: at
// n = q = 1000, r = 5, m = 150, rho = 10 all of them.
template <int R, int V>
__global__ void __launch_bounds__(step_threads(V), V == 0 ? 8 : 3)
    step_first_kernel(const StreamTable T) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ StreamProblem spr;
  __shared__ int snl;
  __shared__ uint64_t abar;
  constexpr int NT = step_threads(V);
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) mbar_init(&abar, T.withhold == 3 ? 2 : 1);  // (2: test aid)
  unsigned phase = 0;
  int cur = -1;
  for (int c = blockIdx.x; c < T.ncols; c += gridDim.x) {
    load_problem(T, c, &spr, cur);
    if (spr.fvar != V) continue;
    const StepCarve cv = step_carve(R, spr.L.m, spr.L.n, spr.L.rho, spr.astride, V, false);
    Step<R, V> s(T, spr, smem, cv);
    s.at_column(c, smem, cv);
    s.stage_begin(&abar);
    const int m = s.m, rho = s.rho, k = s.k;
    // the given support, entries outside the column dropped
    if (threadIdx.x < 32) {
      int cnt = 0;
      for (int e0 = 0; e0 < rho; e0 += 32) {
        const int e = e0 + lane;
        const int j = e < rho ? spr.S_idx[static_cast<size_t>(k) * rho + e] : -1;
        const float x = e < rho ? spr.S_val[static_cast<size_t>(k) * rho + e] : 0.f;
        const bool in = j >= 0 && j < s.n;
        const unsigned b = __ballot_sync(0xffffffffu, in);
        if (in) {
          const int at = cnt + __popc(b & ((1u << lane) - 1));
          s.sj[at] = j;
          s.svb[at] = x;
        }
        cnt += __popc(b);
      }
      if (lane == 0) snl = cnt;
    }
    const float* wp = spr.Wp + static_cast<size_t>(k) * spr.ncw * spr.wstride;
    for (int t4 = threadIdx.x; t4 < spr.wstride / 4; t4 += NT) {
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
      for (int cc = 0; cc < spr.ncw; ++cc) {
        const float4 a = __ldcg(reinterpret_cast<const float4*>(wp + static_cast<size_t>(cc) * spr.wstride) + t4);
        x.x += a.x; x.y += a.y; x.z += a.z; x.w += a.w;
      }
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        const int t = 4 * t4 + z, i = t / R, l = t - i * R;
        if (i < m) s.Q[l * s.ms + i] = z == 0 ? x.x : z == 1 ? x.y : z == 2 ? x.z : x.w;
      }
    }
    __syncthreads();
    s.nl = snl;
    s.factor();
    if (!__syncthreads_and(s.stage_end(&abar, phase))) {
      s.stage_abandon(&abar, phase);
      break;
    }
    if (s.nl != rho) {
      // entries of the given support were dropped: the columns of the others
      // move down to their slots (in AG_k too, where the next step finds them)
      for (int i = threadIdx.x; i < m; i += NT) {
        int at = 0;
        for (int e = 0; e < rho; ++e) {
          const int j = spr.S_idx[static_cast<size_t>(k) * rho + e];
          if (j < 0 || j >= s.n) continue;
          const float a = s.ag_global()[static_cast<size_t>(e) * s.as + i];
          s.ag_global()[static_cast<size_t>(at) * s.as + i] = a;
          s.ag[static_cast<size_t>(at) * s.as + i] = a;
          ++at;
        }
      }
      __syncthreads();
    }
    if (spr.mode == kModeLS || s.te == 0) {
      s.finish(spr.mode == kModeIter);
      continue;
    }
    s.residual(1);
    const int sw = s.sweeps(0, false, 0.f);
    if (sw < s.te) s.need_pass(sw, 0, true);
    else s.finish(true);
  }
}

// ---- HardThreshold of v (n entries) on one CTA --------------------------------
// The rho largest keys (|v|, then the lower index) of vv into sel[0..K),
// K = min(rho, n): 8-bit radix select on the float bits, ties by index.
template <int NT>
__device__ __forceinline__ int topk_radix(const float* vv, int n, int rho, int* hist, int* ties,
                                          int* sel) {
  const int K = min(rho, n), lane = threadIdx.x & 31;
  int* info = hist + 256;  // [0] digit, [1] remaining, [2] ties, [3] selected
  unsigned prefix = 0, mask = 0;
  if (threadIdx.x == 0) info[1] = K;
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int t = threadIdx.x; t < 256; t += NT) hist[t] = 0;
    __syncthreads();
    for (int j0 = threadIdx.x - lane; j0 < n; j0 += NT) {
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
  for (int j = threadIdx.x; j < n; j += NT) {
    const unsigned key = __float_as_uint(fabsf(vv[j]));
    if (key > prefix) sel[atomicAdd(&info[3], 1)] = j;
    else if (key == prefix) ties[atomicAdd(&info[2], 1)] = j;
  }
  __syncthreads();
  const int nt = info[2];
  for (int t = threadIdx.x; t < nt; t += NT) {
    int rank = 0;
    for (int z = 0; z < nt; ++z) rank += ties[z] < ties[t];
    if (rank < need) sel[info[3] + rank] = ties[t];
  }
  __syncthreads();
  // in key order: the order in which the threads found them is arbitrary
  for (int t = threadIdx.x; t < K; t += NT) {
    const uint64_t kj = ht_key(vv[sel[t]], sel[t]);
    int rank = 0;
    for (int z = 0; z < K; ++z) rank += ht_key(vv[sel[z]], sel[z]) > kj;
    ties[rank] = sel[t];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < K; t += NT) sel[t] = ties[t];
  __syncthreads();
  return K;
}

// One listed column after its pass: HardThreshold with g, then the sweeps
// that need no further pass.  zero: the first sweep of the initialisation
// (s = 0: the support is the rho largest |g_j|, its values still 0).
template <int R, int V>
__global__ void __launch_bounds__(step_threads(V), V == 0 ? 6 : 3)
    step_next_kernel(const StreamTable T, int round, int zero) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ StreamProblem spr;
  __shared__ uint64_t abar;
  constexpr int NT = step_threads(V);
  const int lane = threadIdx.x & 31;
  const int count = zero ? T.ncols : T.cnt[round];
  if (count == 0) return;
  if (threadIdx.x == 0) mbar_init(&abar, T.withhold == 3 ? 2 : 1);  // (2: test aid)
  unsigned phase = 0;
  int cur = -1;
  for (int at = blockIdx.x; at < count; at += gridDim.x) {
    const int c = zero ? at : T.list[static_cast<size_t>(round & 1) * T.ncols + at];
    load_problem(T, c, &spr, cur);
    if (spr.nvar != V || spr.te == 0) continue;
    const StepCarve cv = step_carve(R, spr.L.m, spr.L.n, spr.L.rho, spr.astride, V, true);
    Step<R, V> s(T, spr, smem, cv);
    s.at_column(c, smem, cv);
    if (!zero) s.stage_begin(&abar);
    const int m = s.m, n = s.n, rho = s.rho, k = s.k;
    float* vv = reinterpret_cast<float*>(smem + cv.vv);
    int* ties = reinterpret_cast<int*>(smem + cv.tie);
    int* sel = ties + n;                               // 2 rho + 8 entries
    int* hist = reinterpret_cast<int*>(smem + cv.hist);
    int* info = hist + 256;
    int* removed = reinterpret_cast<int*>(smem + cv.lists);
    int* added = removed + cv.rp;
    const float* g = spr.g + static_cast<size_t>(k) * spr.L.ns;
    const int sw = zero ? 0 : spr.sweep[k];
    s.nl = zero ? 0 : spr.nsup[k];
    for (int e = threadIdx.x; e < s.nl; e += NT) {
      s.sj[e] = spr.supj[static_cast<size_t>(k) * rho + e];
      s.svb[e] = spr.supv[static_cast<size_t>(k) * rho + e];
    }
    if (s.project) {
      const float* w = spr.Wk + static_cast<size_t>(k) * spr.wstride;
      for (int i = threadIdx.x; i < m; i += NT)
#pragma unroll
        for (int l = 0; l < R; ++l) s.Q[l * s.ms + i] = __ldcg(w + static_cast<size_t>(l) * m + i);
      for (int t = threadIdx.x; t < 256; t += NT) s.G[512 + t] = spr.Li[static_cast<size_t>(k) * 256 + t];
    }
    for (int j = threadIdx.x; j < n; j += NT) vv[j] = __ldcg(g + j);
    if (!__syncthreads_and(zero || s.stage_end(&abar, phase))) {
      s.stage_abandon(&abar, phase);
      break;
    }
    if (zero) {
      // support of the zero start
      const int K = topk_radix<NT>(vv, n, rho, hist, ties, sel);
      for (int e = threadIdx.x; e < K; e += NT) {
        s.sj[e] = sel[e];
        s.svb[e] = 0.f;
      }
      s.nl = K;
      __syncthreads();
      for (int t = threadIdx.x; t < K * m; t += NT) {
        const int e = t / m, i = t - e * m;
        const float a = stream_elem(spr, k, i, s.sj[e]);
        s.ag[static_cast<size_t>(e) * s.as + i] = a;
        if (step_staged(V)) s.ag_global()[static_cast<size_t>(e) * s.as + i] = a;
      }
      __syncthreads();
    }
    s.residual(1);  // u, the vector of the pass
    float sq = 0.f;
    for (int e = threadIdx.x; e < s.nl; e += NT) {
      const float x = vv[s.sj[e]];
      s.gG[e] = x;
      sq = fmaf(x, x, sq);
    }
    s.put_scal(0, sq);
    __syncthreads();
    const float nref = sqrtf(s.get_scal(1));
    for (int i = threadIdx.x; i < m; i += NT) s.uref[i] = s.u[i];
    float num, den, gmax = 0.f;
    s.curvature(num, den, false);
    if (!(den > 0.f)) {  // stationary: the remaining sweeps keep s
      s.finish(true);
      continue;
    }
    float mu = num / den;
    if (!isfinite(mu)) {
      if (threadIdx.x == 0) report_error(spr.err, kErrNaN, k);
      mu = 0.f;
    }
    for (int j = threadIdx.x; j < n; j += NT) vv[j] = -mu * vv[j];
    if (threadIdx.x == 0) info[3] = 0;
    __syncthreads();
    float* snew = s.sv(1);
    const int nl = s.nl;
    for (int e = threadIdx.x; e < nl; e += NT) {
      const float x = fmaf(-mu, s.gG[e], s.svb[e]);
      snew[e] = x;
      vv[s.sj[e]] = x;
    }
    __syncthreads();
    s.par = 1;
    bool kept = true;
    // candidates: when the support holds rho entries, nothing below the
    // smallest of them can enter
    int K = -1;
    if (nl == rho) {
      float t0 = INFINITY;
      for (int e = lane; e < nl; e += 32) t0 = fminf(t0, fabsf(snew[e]));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t0 = fminf(t0, __shfl_xor_sync(0xffffffffu, t0, o));
      const int cap = 2 * rho + 8;
      for (int j = threadIdx.x; j < n; j += NT)
        if (fabsf(vv[j]) >= t0) {
          const int slot = atomicAdd(&info[3], 1);
          if (slot < cap) sel[slot] = j;
        }
      __syncthreads();
      const int cn = info[3];
      if (cn == rho) {
        K = 0;  // the support itself: kept
      } else if (cn <= cap && cn > rho) {
        for (int t = threadIdx.x; t < cn; t += NT) {
          const uint64_t kj = ht_key(vv[sel[t]], sel[t]);
          int rank = 0;
          for (int z = 0; z < cn; ++z) rank += ht_key(vv[sel[z]], sel[z]) > kj;
          if (rank < rho) ties[rank] = sel[t];
        }
        __syncthreads();
        for (int t = threadIdx.x; t < rho; t += NT) sel[t] = ties[t];
        __syncthreads();
        K = rho;
      }
    }
    if (K < 0) K = topk_radix<NT>(vv, n, rho, hist, ties, sel);
    if (K > 0) {
      // slots of the entries that left take the ones that entered (both in
      // slot / key order)
      if (threadIdx.x < 32) {
        int nrem = 0, nadd = 0;
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
        if (lane == 0) info[4] = min(nrem, nadd);
      }
      __syncthreads();
      const int nadd = info[4];
      s.nl = K;
      kept = nadd == 0 && K == nl;
      for (int t = threadIdx.x; t < nadd; t += NT) {
        s.sj[removed[t]] = added[t];
        snew[removed[t]] = vv[added[t]];
      }
      for (int t = threadIdx.x; t < nadd * m; t += NT) {
        const int z = t / m, i = t - z * m;
        const float a = stream_elem(spr, k, i, added[z]);
        s.ag[static_cast<size_t>(removed[z]) * s.as + i] = a;
        if (step_staged(V)) s.ag_global()[static_cast<size_t>(removed[z]) * s.as + i] = a;
      }
    }
    __syncthreads();
    if (sw + 1 >= s.te) {
      s.finish(true);
      continue;
    }
    // largest |g| outside the new support
    for (int e = threadIdx.x; e < s.nl; e += NT) vv[s.sj[e]] = INFINITY;
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += NT)
      if (!isinf(vv[j])) gmax = fmaxf(gmax, fabsf(__ldcg(g + j)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
    if (lane == 0) s.scal(0)[threadIdx.x >> 5] = gmax;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) gmax = fmaxf(gmax, s.scal(0)[w]);
    gmax = fmaf(spr.nmax[k] * nref, (m + 4) * 0x1p-24f, gmax);  // rounding of the pass's sums
    const int slot = 1 + ((sw + 1) & 1);
    if (kept) {
      float nn = 0.f;
      for (int i = threadIdx.x; i < m; i += NT) {
        const float t = fmaf(-mu, s.p[i], s.u[i]);
        s.u[i] = t;
        nn = fmaf(t, t, nn);
      }
      s.put_scal(slot, nn);
    } else {
      s.residual(slot);
    }
    const int nx = s.sweeps(sw + 1, true, gmax);
    if (nx < s.te) s.need_pass(nx, round + 1, false);
    else s.finish(true);
  }
}

}  // namespace stream
}  // namespace lrs
