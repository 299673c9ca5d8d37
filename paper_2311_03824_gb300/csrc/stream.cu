// Launch side of the streaming engine (kernels in stream_impl.cuh; W and the
// column steps are compiled per rank width in stream_r*.cu), the A^T pass and
// the column norms.
#include <algorithm>
#include <vector>

#include "stream_impl.cuh"

namespace lrs {
#define LRS_STREAM_R(X) X(2) X(3) X(4) X(5) X(6) X(8) X(10) X(12) X(16)
#define LRS_DECL(R) void* stream_w_kernel_r##R(int et); void* stream_step_kernel_r##R(int next, int variant);
LRS_STREAM_R(LRS_DECL)
#undef LRS_DECL

namespace {
using namespace stream;

void* pick_w(int R, int et) {
#define LRS_CASE(X) case X: return stream_w_kernel_r##X(et);
  switch (R) { LRS_STREAM_R(LRS_CASE) }
#undef LRS_CASE
  return nullptr;
}
void* pick_step(int R, int next, int variant) {
#define LRS_CASE(X) case X: return stream_step_kernel_r##X(next, variant);
  switch (R) { LRS_STREAM_R(LRS_CASE) }
#undef LRS_CASE
  return nullptr;
}

// g = A_k^T u_k (or h_k, final) for the listed columns (all when list is
// null).  Unit: one 32-column tile of one column, all m rows, in pieces of rp
// rows with their part of u; lane (ro, q) sums columns 4 q .. 4 q + 3 over rows
// 16 t + 4 ro + s, the four row groups are added by shuffles at the end.  Two
// flops per element: bound by memory.  The final pass takes the columns in
// reverse, so that it starts on what the W pass of the sweep has left in L2
// (and the next sweep's W pass on what this one leaves).
template <int ET>
__global__ void __launch_bounds__(kStreamNT, 2)
    g_kernel(const StreamTable T, const int* __restrict__ list, const int* __restrict__ count,
             int final, int maxtile, int S, int rp) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int pb = ET == 0 ? 4 : ET == 1 ? 2 : 1;
  constexpr int planes = ET == 3 ? 2 : 1;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int q = lane & 7, ro = lane >> 3;
  // element offsets of this lane's chunk in rows 4 ro + s of a 16-row group
  int off4[4];
#pragma unroll
  for (int z = 0; z < 4; ++z) off4[z] = (4 * ro + z) * kTW + ((q ^ ((4 * ro + z) & 7)) << 2);
  const int ncol = count ? *count : T.ncols;
  if (ncol == 0) return;
  const unsigned abytes = static_cast<unsigned>(rp * kTW * pb * planes);
  const unsigned stage = abytes + static_cast<unsigned>(planes * rp * 4);
  Pipe P;
  P.init(static_cast<unsigned>(wid * S) * stage,
         reinterpret_cast<uint64_t*>(smem + static_cast<size_t>(kSW) * S * stage) + wid * kMaxStage,
         stage, S, T.wait_ns);
  const int wk = blockIdx.x * kSW + wid, nw = gridDim.x * kSW;
  auto column = [&](int i) { return list ? list[i] : (final ? ncol - 1 - i : i); };
  // units (entry i of the list, tile b) in steps of all warps
  const int di = nw / maxtile, db = nw - di * maxtile;
  const int i_first = wk / maxtile, b_first = wk - i_first * maxtile;
  auto step = [&](int& i, int& b) {
    i += di;
    b += db;
    if (b >= maxtile) {
      b -= maxtile;
      ++i;
    }
  };
  // producer cursor: unit, its problem data, next row
  int pu = i_first, pb_ = b_first, pi = 0, pm = 0, pas = 0;
  const unsigned char* ptile = nullptr;
  const float* pvec = nullptr;
  auto open = [&]() {  // the next unit from the cursor on that exists
    for (; pu < ncol; step(pu, pb_)) {
      const int c = column(pu);
      const StreamProblem& pr = T.probs[prob_of(T, c)];
      const int ntile = pr.L.ns / kTW;
      if (pb_ >= ntile) continue;
      const int k = c - pr.col0;
      pm = pr.L.m;
      pas = pr.astride;
      ptile = static_cast<const unsigned char*>(pr.A) +
              (static_cast<size_t>(k) * ntile + pb_) * (static_cast<size_t>(pm) * kTW * elem_bytes(ET));
      pvec = pr.uvec + static_cast<size_t>(k) * planes * pas;
      pi = 0;
      return;
    }
  };
  auto issue = [&]() {
    if (pu >= ncol) return;
    const int nr = min(rp, pm - pi);
    const unsigned hb = static_cast<unsigned>(nr * kTW * pb);
    const unsigned ub = static_cast<unsigned>(((nr + 3) & ~3) * 4);
    unsigned char* dst = smem + P.issue_at();
    if (lane == 0) {
      uint64_t* bar = P.issue_bar();
      mbar_arrive_expect_tx(bar, (hb + ub) * planes);
#pragma unroll
      for (int pl = 0; pl < planes; ++pl) {
        bulk_copy_g2s(dst + pl * hb, ptile + static_cast<size_t>(pl) * pm * kTW + static_cast<size_t>(pi) * kTW * pb,
                      hb, bar);
        bulk_copy_g2s(dst + abytes + pl * rp * 4, pvec + pl * pas + pi, ub, bar);
      }
    }
    P.issued();
    pi += nr;
    if (pi >= pm) {
      step(pu, pb_);
      open();
    }
  };
  open();
  for (int i = 0; i < S; ++i) issue();
  for (int u = i_first, b = b_first; u < ncol && !P.dead; step(u, b)) {
    const int c = column(u);
    const StreamProblem& pr = T.probs[prob_of(T, c)];
    if (b >= pr.L.ns / kTW) continue;
    const int k = c - pr.col0, m = pr.L.m;
    P.err = pr.err;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i0 = 0; i0 < m; i0 += rp) {
      const unsigned char* st = smem + P.take();
      if (P.dead) break;
      const int nr = min(rp, m - i0);
      const float* w1 = reinterpret_cast<const float*>(st + abytes);
      const float* w2 = w1 + rp;
      auto row = [&](int off, float a1, float a2) {  // off: element offset of the chunk
        float4 a;
        if constexpr (ET >= 2) {
          a = static_cast<float4>(*reinterpret_cast<const __nv_fp8x4_e4m3*>(st + off));
        } else {
          if constexpr (ET == 0) {
            a = *reinterpret_cast<const float4*>(st + static_cast<size_t>(off) * 4);
          } else {
            const uint2 raw = *reinterpret_cast<const uint2*>(st + static_cast<size_t>(off) * 2);
            a = make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u),
                            __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xffff0000u));
          }
        }
        acc.x = fmaf(a.x, a1, acc.x);
        acc.y = fmaf(a.y, a1, acc.y);
        acc.z = fmaf(a.z, a1, acc.z);
        acc.w = fmaf(a.w, a1, acc.w);
        if constexpr (ET == 3) {
          const float4 l =
              static_cast<float4>(*reinterpret_cast<const __nv_fp8x4_e4m3*>(st + nr * kTW + off));
          acc.x = fmaf(l.x, a2, acc.x);
          acc.y = fmaf(l.y, a2, acc.y);
          acc.z = fmaf(l.z, a2, acc.z);
          acc.w = fmaf(l.w, a2, acc.w);
        }
      };
      int t = 0;
#pragma unroll 2
      for (; t + 16 <= nr; t += 16) {
        const int r = t + 4 * ro;
        const float4 a1 = *reinterpret_cast<const float4*>(w1 + r);
        float4 a2 = make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (ET == 3) a2 = *reinterpret_cast<const float4*>(w2 + r);
        row(t * kTW + off4[0], a1.x, a2.x);
        row(t * kTW + off4[1], a1.y, a2.y);
        row(t * kTW + off4[2], a1.z, a2.z);
        row(t * kTW + off4[3], a1.w, a2.w);
      }
      for (int r = t + ro; r < nr; r += 4)
        row(r * kTW + ((q ^ (r & 7)) << 2), w1[r], ET == 3 ? w2[r] : 0.f);
      P.taken();
      __syncwarp();
      issue();
    }
    if (P.dead) break;
#pragma unroll
    for (int o = 8; o <= 16; o <<= 1) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
      acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o);
      acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
    }
    const float v = ro == 0 ? acc.x : ro == 1 ? acc.y : ro == 2 ? acc.z : acc.w;
    const int j = b * kTW + 4 * q + ro;
    if (final) {
      if (j < pr.L.n) pr.H[static_cast<size_t>(k) * pr.L.n + j] = v;
    } else {
      pr.g[static_cast<size_t>(k) * pr.L.ns + j] = v;
    }
  }
  P.drain();
}

void* pick_g(int et) {
  switch (et) {
    case 1: return reinterpret_cast<void*>(&g_kernel<1>);
    case 2: return reinterpret_cast<void*>(&g_kernel<2>);
    case 3: return reinterpret_cast<void*>(&g_kernel<3>);
    default: return reinterpret_cast<void*>(&g_kernel<0>);
  }
}

// Vectors of the initialisation's first pass: -y_k (its IHT starts at s = 0),
// or y_k when no IHT runs; the list counters start at zero.
__global__ void init_vec_kernel(const StreamTable T) {
  if (blockIdx.x == 0 && threadIdx.x < T.ncnt) T.cnt[threadIdx.x] = 0;
  for (int c = blockIdx.x; c < T.ncols; c += gridDim.x) {
    const StreamProblem& pr = T.probs[prob_of(T, c)];
    const int k = c - pr.col0, m = pr.L.m, planes = pr.L.et == 3 ? 2 : 1;
    float* out = pr.uvec + static_cast<size_t>(k) * planes * pr.astride;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
      const float yi = pr.y[static_cast<size_t>(k) * m + i];
      const float x = pr.te > 0 ? -yi : yi;
      if (pr.L.et < 2) {
        out[i] = x;
      } else {
        const size_t o = (static_cast<size_t>(k) * m + i) * planes;
        out[i] = x * pr.rscale[o];
        if (planes == 2) out[pr.astride + i] = x * pr.rscale[o + 1];
      }
    }
  }
}

// max_j ||a_j||: a warp per tile, lanes as in g_kernel; the maximum over a
// column's tiles on the float bits (sums of squares are not negative; a NaN's
// bits are above every number's, so it survives).
template <int ET>
__global__ void __launch_bounds__(256) norms_kernel(GaussLayout L, const unsigned char* __restrict__ A,
                                                    const float* __restrict__ rscale, int k0, int kc,
                                                    int* __restrict__ nmax2) {
  const int lane = threadIdx.x & 31, q = lane & 7, ro = lane >> 3;
  const int ntile = L.ns / kTW, m = L.m;
  const size_t tb = static_cast<size_t>(m) * kTW * elem_bytes(ET);
  constexpr int per = ET == 3 ? 2 : 1;
  const long nw = (static_cast<long>(gridDim.x) * blockDim.x) >> 5;
  for (long t = (static_cast<long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
       t < static_cast<long>(kc) * ntile; t += nw) {
    const long k = k0 + t / ntile;
    const unsigned char* tile = A + (static_cast<size_t>(k) * ntile + t % ntile) * tb;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int i = ro; i < m; i += 4) {
      const int off = i * kTW + ((q ^ (i & 7)) << 2);
      float4 a;
      if constexpr (ET >= 2) {
        const size_t o = (static_cast<size_t>(k) * m + i) * per;
        const float s1 = rscale[o];
        a = static_cast<float4>(*reinterpret_cast<const __nv_fp8x4_e4m3*>(tile + off));
        a = make_float4(a.x * s1, a.y * s1, a.z * s1, a.w * s1);
        if constexpr (ET == 3) {
          const float s2 = rscale[o + 1];
          const float4 l = static_cast<float4>(
              *reinterpret_cast<const __nv_fp8x4_e4m3*>(tile + static_cast<size_t>(m) * kTW + off));
          a = make_float4(fmaf(l.x, s2, a.x), fmaf(l.y, s2, a.y), fmaf(l.z, s2, a.z), fmaf(l.w, s2, a.w));
        }
      } else {
        a = sweep::load4<ET>(tile, m, i, q, nullptr, nullptr);
      }
      acc.x = fmaf(a.x, a.x, acc.x);
      acc.y = fmaf(a.y, a.y, acc.y);
      acc.z = fmaf(a.z, a.z, acc.z);
      acc.w = fmaf(a.w, a.w, acc.w);
    }
#pragma unroll
    for (int o = 8; o <= 16; o <<= 1) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
      acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o);
      acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
    }
    int v = max(max(__float_as_int(fabsf(acc.x)), __float_as_int(fabsf(acc.y))),
                max(__float_as_int(fabsf(acc.z)), __float_as_int(fabsf(acc.w))));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) atomicMax(nmax2 + k, v);
  }
}
__global__ void norms_fin_kernel(int k0, int kc, float* nmax) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < kc) nmax[k0 + t] = sqrtf(nmax[k0 + t] + kTinySq);
}

}  // namespace

void stream_plan(StreamProblem& P, int R) {
  const int m = P.L.m, ntile = P.L.ns / kTW;
  P.wstride = (m * R + 3) & ~3;
  P.astride = (m + 3) & ~3;
  // Column chunks of the W units: eight of a column (finer units balance the
  // grid: n = 1000, q = 1000 gives 16.4 units per warp), four from 96 tiles on
  // (the chunks' partial W are then 2 R / tbw / 32 of A_k's bytes), and U of a
  // chunk within 40 KB of shared memory.
  const int cap = std::max(1, 40 * 1024 / (kTW * w_chunks4(R) * 16));
  const int want = (ntile + (ntile >= 96 ? 4 : 8) - 1) / (ntile >= 96 ? 4 : 8);
  P.tbw = std::max(1, std::min(cap, want));
  P.ncw = (ntile + P.tbw - 1) / P.tbw;
  P.nrb = (m + w_rows(R) - 1) / w_rows(R);
  // Column steps: 128 threads while four columns fit an SM with their support
  // staged, 256 threads for larger columns, the support's columns read from
  // memory when two staged columns do not fit.  The thread count (which fixes
  // the order of the sums) by the problem's own sizes, so that a batch runs
  // the same arithmetic.
  auto smem = [&](int v, bool next) {
    return step_carve(R, m, P.L.n, P.L.rho, P.astride, v, next).total;
  };
  const size_t two = 112 * 1024;
  const bool small = smem(0, true) <= 54 * 1024;
  P.fvar = small ? 0 : smem(1, false) <= two ? 1 : 2;
  P.nvar = small ? 0 : smem(1, true) <= two ? 1 : 2;
}

bool stream_shape(const StreamProblem* P, int nprob, int R, int et, int nsm, int grid_limit,
                  StreamShape* S, std::vector<StreamAssign>* asg) {
  *S = StreamShape{};
  S->R = R;
  S->et = et;
  const size_t two = 113 * 1024 - 256, one = static_cast<size_t>(smem_optin_limit()) - 1024;
  const int planes = et == 3 ? 2 : 1, eb = elem_bytes(et);
  int m_max = 0, ncols = 0;
  unsigned us = 0;
  double work = 0;
  for (int i = 0; i < nprob; ++i) {
    const StreamProblem& p = P[i];
    m_max = std::max(m_max, p.L.m);
    S->maxtile = std::max(S->maxtile, p.L.ns / kTW);
    S->te = std::max(S->te, p.te);
    us = std::max(us, static_cast<unsigned>(p.tbw * kTW * w_chunks4(R) * 16));
    ncols += p.L.q;
    work += static_cast<double>(p.L.q) * p.nrb * p.ncw * p.tbw;
    S->fsmem[p.fvar] = std::max<size_t>(
        S->fsmem[p.fvar], step_carve(R, p.L.m, p.L.n, p.L.rho, p.astride, p.fvar, false).total);
    S->nsmem[p.nvar] = std::max<size_t>(
        S->nsmem[p.nvar], step_carve(R, p.L.m, p.L.n, p.L.rho, p.astride, p.nvar, true).total);
    if (S->fsmem[p.fvar] > one || S->nsmem[p.nvar] > one) return false;
  }
  if (S->te > kStreamMaxRounds) return false;
  // W: pieces of about 4 KB, as many stages as two CTAs per SM allow
  S->us_bytes = (us + 127u) & ~127u;
  const unsigned sub = static_cast<unsigned>(w_rows(R) * kTW * eb);
  S->wtpp = std::max(1, std::min(32 / planes, static_cast<int>(4096 / sub)));
  const size_t wstage = static_cast<size_t>(sub) * S->wtpp;
  const size_t bars = static_cast<size_t>(kSW) * kMaxStage * 8;
  S->wS = static_cast<int>(std::min<size_t>(kMaxStage, (two - S->us_bytes - bars) / (kSW * wstage)));
  if (S->wS < 2) return false;
  S->wsmem = S->us_bytes + kSW * S->wS * wstage + bars;
  // A^T: pieces of about 4 KB spread evenly over the rows
  const int rmax = 4096 / (kTW * eb);
  const int np = (m_max + rmax - 1) / rmax;
  S->grp = ((m_max + np - 1) / np + 15) / 16 * 16;
  const size_t gstage = static_cast<size_t>(S->grp) * (kTW * eb + planes * 4);
  S->gS = static_cast<int>(std::min<size_t>(kMaxStage, (two - bars) / (kSW * gstage)));
  S->gsmem = kSW * S->gS * gstage + bars;
  S->grid = 2 * nsm;
  if (grid_limit > 0) S->grid = std::min(S->grid, grid_limit);
  // columns at once in the steps: what fits, scaled like the streaming grid
  auto step_grid = [&](size_t smem, int cap) {
    const int fit = static_cast<int>(std::max<size_t>(1, std::min<size_t>(cap, 227 * 1024 / (smem + 2048))));
    return std::max(1, std::min(ncols, static_cast<int>(static_cast<long>(fit) * S->grid / 2)));
  };
  for (int v = 0; v < 3; ++v) {
    S->fgrid[v] = S->fsmem[v] ? step_grid(S->fsmem[v], v == 0 ? 8 : 3) : 0;
    S->ngrid[v] = S->nsmem[v] ? step_grid(S->nsmem[v], v == 0 ? 6 : 3) : 0;
  }
  // W assignments: every (problem, chunk) gets CTAs by its share of the work
  // (at least one; CTAs take several assignments when there are more)
  asg->clear();
  for (int i = 0; i < nprob; ++i) {
    const StreamProblem& p = P[i];
    const double w = static_cast<double>(p.L.q) * p.nrb * p.tbw;  // one chunk
    const int units = (p.L.q * p.nrb + kSW - 1) / kSW;
    const int cnt = std::min(std::max(1, static_cast<int>(S->grid * (w / work))), units);
    for (int cc = 0; cc < p.ncw; ++cc)
      for (int x = 0; x < cnt; ++x) asg->push_back(StreamAssign{i, cc, x, cnt});
  }
  return true;
}

cudaError_t stream_prepare(int R, int et) {
  void* fs[] = {pick_w(R, et),        pick_g(et),           pick_step(R, 0, 0), pick_step(R, 0, 1),
                pick_step(R, 0, 2), pick_step(R, 1, 0), pick_step(R, 1, 1), pick_step(R, 1, 2)};
  for (void* f : fs) {
    // what a CTA may request beside the kernel's static shared memory
    cudaFuncAttributes at{};
    cudaError_t e = cudaFuncGetAttributes(&at, f);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem_optin_limit() - static_cast<int>(at.sharedSizeBytes));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int stream_launches(int te) { return 3 + 2 * te; }

cudaError_t stream_sweep(const StreamTable& T, const StreamShape& S, int mode,
                         const StreamAssign* asg, int nasg, cudaStream_t s) {
  StreamTable t = T;
  cudaError_t e = cudaSuccess;
  auto first = [&]() {
    int a_n = nasg, wS = S.wS, tpp = S.wtpp;
    unsigned us = S.us_bytes;
    void* wa[] = {&t, &asg, &a_n, &wS, &tpp, &us};
    cudaError_t x = cudaLaunchKernel(pick_w(S.R, S.et), dim3(std::min(S.grid, nasg)), dim3(kStreamNT),
                                     wa, S.wsmem, s);
    void* sa[] = {&t};
    for (int v = 0; v < 3; ++v)
      if (x == cudaSuccess && S.fgrid[v])
        x = cudaLaunchKernel(pick_step(S.R, 0, v), dim3(S.fgrid[v]), dim3(step_threads(v)), sa, S.fsmem[v], s);
    return x;
  };
  auto pass = [&](const int* list, const int* count, int final) {
    int mt = S.maxtile, gS = S.gS, rp = S.grp;
    void* ga[] = {&t, &list, &count, &final, &mt, &gS, &rp};
    return cudaLaunchKernel(pick_g(S.et), dim3(S.grid), dim3(kStreamNT), ga, S.gsmem, s);
  };
  auto next = [&](int round, int zero) {
    void* na[] = {&t, &round, &zero};
    cudaError_t x = cudaSuccess;
    for (int v = 0; v < 3; ++v)
      if (x == cudaSuccess && S.ngrid[v])
        x = cudaLaunchKernel(pick_step(S.R, 1, v), dim3(S.ngrid[v]), dim3(step_threads(v)), na, S.nsmem[v], s);
    return x;
  };
  if (mode == kModeInit) {
    init_vec_kernel<<<std::min(T.ncols, 1216), 128, 0, s>>>(t);
    e = cudaGetLastError();
  } else {
    e = first();
  }
  if (mode == kModeLS || e != cudaSuccess) return e;
  for (int rd = 0; rd < S.te && e == cudaSuccess; ++rd) {
    const int zero = mode == kModeInit && rd == 0;
    e = zero ? pass(nullptr, nullptr, 0)
             : pass(t.list + static_cast<size_t>(rd & 1) * t.ncols, t.cnt + rd, 0);
    if (e == cudaSuccess) e = next(rd, zero);
  }
  if (e == cudaSuccess) e = pass(nullptr, nullptr, 1);
  return e;
}

cudaError_t stream_norms(const GaussLayout& L, const void* A, const float* rscale, int k0, int kc,
                         float* nmax, cudaStream_t s) {
  const unsigned char* a = static_cast<const unsigned char*>(A);
  cudaError_t e = cudaMemsetAsync(nmax + k0, 0, sizeof(float) * kc, s);
  if (e != cudaSuccess) return e;
  int* n2 = reinterpret_cast<int*>(nmax);
  switch (L.et) {
    case 0: norms_kernel<0><<<1216, 256, 0, s>>>(L, a, rscale, k0, kc, n2); break;
    case 1: norms_kernel<1><<<1216, 256, 0, s>>>(L, a, rscale, k0, kc, n2); break;
    case 2: norms_kernel<2><<<1216, 256, 0, s>>>(L, a, rscale, k0, kc, n2); break;
    default: norms_kernel<3><<<1216, 256, 0, s>>>(L, a, rscale, k0, kc, n2); break;
  }
  norms_fin_kernel<<<(kc + 255) / 256, 256, 0, s>>>(k0, kc, nmax);
  return cudaGetLastError();
}

}  // namespace lrs
