// tcw_step.cu -- the exhaustive search as step functions over the sorted sky
// (tcw_step.cuh): Doppler rows, the search kernel, the map's range of powers.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "tcw_pair.cuh"
#include "tcw_step.cuh"

namespace tcw {
namespace {

constexpr int kStepThreads = 1024;
constexpr int kStepWarps = kStepThreads / 32;
// Segments between two normalisations of the difference cells: a cell's low
// word takes at most 8 bin differences of at most 2^16 per (segment, detector),
// 2 detectors, so 2^11 segments stay within 2^31 (and their rows within 12 bits).
constexpr int kStepCarry = 2048;
constexpr int kExactSpan = 8;    // boundaries either side of the track that the exact search goes to
constexpr int kStepTerms = 5;    // fp32 terms of the track beyond the quadratic one
constexpr int kStepTurn = 16;    // rows whose heads a warp holds (segments of a turn x detectors of a pass)
// Entries of a warp's list (global memory), and the most that one round of lookups adds: 2 detectors,
// 7 boundaries and the lookups themselves.
constexpr int kStepSlowMore = 2 * 8 * 32;
constexpr int kStepSlow = kStepSlowMore + 256;
constexpr int kStepLookup = 7;   // in place of a step's number: the whole lookup
// A threshold's or a sky's place within a bucket of the row's table: 2^-14 of a bucket, biased by a bucket.
constexpr int kFracBits = 14, kFracShift = 32 - kFracBits;
constexpr int kErrMax = 0x3ffe;               // largest error bound in these units: anything may be near
constexpr unsigned kWindowSlow = 1u << 11;    // in a window's first word: not for the fast placing

// Terms of the anchors' series by the size of the step d: the dropped ones,
// |C(r, K)| d^K with |C(r, K)| <= 1/16 for r <= 1, stay below 2^-56.
constexpr int kAnchorK0 = 7, kAnchorK1 = 9, kAnchorK2 = 14;
constexpr int kAnchorD0 = 0x3f700000, kAnchorD1 = 0x3f900000, kAnchorD2 = 0x3fb00000;   // 2^-8, 2^-6, 2^-4 (high words)

// Anchor time of tile ti, as tile_anchor_time of tcw_persist.cuh.
__device__ __forceinline__ double anchor_time(const double* t_mid, int n_seg, double T0, int shift, int ti) {
  const int j0 = ti << shift;
  return fmax(t_mid[j0 + (min(1 << shift, n_seg - j0) - 1) / 2], T0);
}

// ---------------------------------------------------------------------------
// Tile anchors (as anchor_chain_kernel / anchor_kernel in tcw_persist.cu) with
// the track constants of StepTile: one thread per (template, run of kAnchorRun
// tiles), FP64.  Bound by the FP64 pipe (19 cycles per warp instruction and SM,
// conversions and roundings included), so the binomial series takes only the
// terms that its step needs, reciprocals start from fp32, and nothing is
// converted: about 35 FP64 instructions per anchor (74 with full series,
// divisions and conversions); 2.6e5 templates x 10800 segments 23.3 -> 18.7 ms.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) step_tile_kernel(StepTileParams p) {
  const AnchorParams& a = p.a;
  const int runs = (a.n_tiles + kAnchorRun - 1) / kAnchorRun;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)a.Bpad * runs) return;
  const int b = (int)(i / runs), t0 = (int)(i % runs) * kAnchorRun;
  const int t1 = min(a.n_tiles, t0 + kAnchorRun);
  const double tau = a.tau[b], r = 1.0 / (a.nbr[b] - 1.0), inv_df = 1.0 / p.df, f0 = a.f0[b];
  const double ne2 = -0.5 * (r + 1.0);   // C(e, 2) / e = (e - 1) / 2, e = -r
  const double fb = p.f_min * inv_df;
  double c[kAnchorTerms];   // C(r, k); those from kAnchorK2 on when a step needs them
  bool all_terms = false;
  c[0] = 1.0;
#pragma unroll
  for (int k = 1; k < kAnchorK2; ++k) c[k] = c[k - 1] * fma(r, 1.0 / k, -(k - 1.0) / k);
  double h = 0.0, ta_prev = 0.0, y = 0.0;
  for (int ti = t0; ti < t1; ++ti) {
    const double ta = anchor_time(a.t_mid, a.n_seg, a.T0, a.tile_shift, ti);
    if (ti == t0 || !a.chain) {
      h = pow((ta - a.T0) / tau + 1.0, r) / f0;
    } else {
      // u'/u - 1 = (t_a' - t_a) / (tau u) = (t_a' - t_a) y
      const double d = (ta - ta_prev) * y;
      const int dh = r <= 1.0 ? __double2hiint(d) : INT_MAX;   // anchor times ascend: d >= 0
      double g = 0.0;   // u'^r / u^r - 1
      if (dh >= kAnchorD2) {
        if (!all_terms) {
#pragma unroll
          for (int k = kAnchorK2; k < kAnchorTerms; ++k) c[k] = c[k - 1] * fma(r, 1.0 / k, -(k - 1.0) / k);
          all_terms = true;
        }
#pragma unroll
        for (int k = kAnchorTerms - 1; k >= kAnchorK2; --k) g = fma(g, d, c[k]);
      }
      if (dh >= kAnchorD1) {
#pragma unroll
        for (int k = kAnchorK2 - 1; k >= kAnchorK1; --k) g = fma(g, d, c[k]);
      }
      if (dh >= kAnchorD0) {
#pragma unroll
        for (int k = kAnchorK1 - 1; k >= kAnchorK0; --k) g = fma(g, d, c[k]);
      }
#pragma unroll
      for (int k = kAnchorK0 - 1; k >= 1; --k) g = fma(g, d, c[k]);
      g *= d;
      h = fma(h, g, h);
    }
    y = reciprocal(tau + (ta - a.T0));
    const int64_t o = (int64_t)b * a.n_tiles + ti;
    reinterpret_cast<double2*>(a.anchors)[o] = make_double2(h, y);
    const double X = reciprocal(h * p.df);
    // nearest whole bin: the low word of xa + 1.5 2^52
    const double xa = X - fb, m = xa + 6755399441055744.0;
    const double A = -r * X * y, Q = A * y * ne2;
    StepTile t;
    // far outside any band: no lookups
    t.base = fabs(xa) < 1.0e9 ? __double2loint(m) : INT_MIN / 2;
    t.frac = near_float(xa - (m - 6755399441055744.0));
    split_float(A, t.A_hi, t.A_lo);
    split_float(Q, t.Q_hi, t.Q_lo);
    t.X = near_float(X);
    t.s = near_float(y);
    int4* w = reinterpret_cast<int4*>(p.tiles + o);
    const int4* v = reinterpret_cast<const int4*>(&t);
    w[0] = v[0];
    w[1] = v[1];
    ta_prev = ta;
  }
}

// ---------------------------------------------------------------------------
// Sky order of one (pass, chunk): positions sorted by the grid value at the
// pass's middle segment (ties by index), by counting; and each sky's position
// in the order of the pass before.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int doppler_q(const double* v, const double* n, double inv_q) {
  const double dD = (v[0] * n[0] + v[1] * n[1] + v[2] * n[2]) / kLightSpeed;   // Eq. 2
  return (int32_t)fmax(fmin(floor(dD * inv_q), 2147483647.0), -2147483648.0);
}

__global__ void __launch_bounds__(kStepMaxChunk) step_order_kernel(StepRowsParams p) {
  __shared__ int s_q[kStepMaxChunk];
  const int c = blockIdx.y, i = threadIdx.x;
  const int rows = min(p.chunk, p.S - c * p.chunk);
  auto rank_in = [&](int pass) {
    const int per = p.n_det / p.dets_per_pass;
    const int e = pass / per, d = p.dets_per_pass == 1 ? pass % per : 0;
    const int js = e * p.pass_seg, je = min(p.n_seg, js + p.pass_seg);
    const double* v = p.vel + ((int64_t)d * p.n_seg + (js + je - 1) / 2) * 3;
    __syncthreads();
    if (i < rows) s_q[i] = doppler_q(v, p.nhat + (int64_t)(c * p.chunk + i) * 3, p.inv_q);
    __syncthreads();
    int rank = 0;
    if (i < rows)
      for (int k = 0; k < rows; ++k) rank += s_q[k] < s_q[i] || (s_q[k] == s_q[i] && k < i);
    return rank;
  };
  const int pass = blockIdx.x;
  const int rank = rank_in(pass), before = pass > 0 ? rank_in(pass - 1) : 0;
  if (i >= rows) return;
  const int64_t o = ((int64_t)pass * p.n_chunks + c) * p.cpad;
  // positions past the last sky repeat it
  for (int k = rank; k < (rank == rows - 1 ? p.cpad : rank + 1); ++k) {
    p.order[o + k] = (int16_t)i;
    p.remap[o + k] = (int16_t)before;
  }
}

// Place of a threshold (or of a sky's grid value) in a row's table, in 2^-32 of
// a bucket: exact, so monotone in v.
__device__ __forceinline__ uint64_t step_place(int v, int qmin, int scale) {
  return (uint64_t)((unsigned)v - (unsigned)qmin) * (unsigned)scale;
}

__device__ __forceinline__ int step_bucket(uint64_t place, int n) {
  return (int)min((unsigned)(place >> 32), (unsigned)n - 1u);
}

// ---------------------------------------------------------------------------
// Doppler rows (Eq. 2): one CTA per (segment, detector, chunk), one thread per
// 8 skies.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) step_rows_kernel(StepRowsParams p) {
  __shared__ int s_max[4], s_min[4];
  __shared__ int s_q[kStepMaxChunk];
  __shared__ uint16_t s_from[step_buckets(kStepMaxChunk)], s_to[step_buckets(kStepMaxChunk)];
  const int d = blockIdx.x % p.n_det, j = blockIdx.x / p.n_det, c = blockIdx.y;
  const int nb = p.cpad / kStepBlock, nk = step_buckets(p.cpad);
  const int g = threadIdx.x, lane = g & 31, warp = g >> 5;
  const int64_t dj = (int64_t)d * p.n_seg + j;
  const double* v = p.vel + dj * 3;
  const int64_t row = ((int64_t)c * p.n_seg + j) * p.n_det + d;
  const int pass = j / p.pass_seg * (p.n_det / p.dets_per_pass) + (p.dets_per_pass == 1 ? d : 0);
  const int16_t* order = p.order ? p.order + ((int64_t)pass * p.n_chunks + c) * p.cpad : nullptr;
  int qv[kStepBlock];
  int mx = INT_MIN, mn = INT_MAX;
  if (g < nb) {
#pragma unroll
    for (int i = 0; i < kStepBlock; ++i) {
      const int k = g * kStepBlock + i;
      const int s = min(c * p.chunk + (order ? (int)order[k] : min(k, p.chunk - 1)), p.S - 1);
      qv[i] = doppler_q(v, p.nhat + (int64_t)s * 3, p.inv_q);
      mx = max(mx, qv[i]);
      mn = min(mn, qv[i]);
    }
    int4* o = reinterpret_cast<int4*>(p.q + row * p.cpad + g * kStepBlock);
    o[0] = make_int4(qv[0], qv[1], qv[2], qv[3]);
    o[1] = make_int4(qv[4], qv[5], qv[6], qv[7]);
  }
  // exclusive prefix maximum and suffix minimum over the threads
  int U = mx, L = mn;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, U, off), b = __shfl_down_sync(0xffffffffu, L, off);
    if (lane >= off) U = max(U, a);
    if (lane + off < 32) L = min(L, b);
  }
  if (lane == 31) s_max[warp] = U;
  if (lane == 0) s_min[warp] = L;
  int Ue = __shfl_up_sync(0xffffffffu, U, 1), Le = __shfl_down_sync(0xffffffffu, L, 1);
  if (lane == 0) Ue = INT_MIN;
  if (lane == 31) Le = INT_MAX;
  __syncthreads();
  int qmin = INT_MAX, qmax = INT_MIN;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    if (w < warp) Ue = max(Ue, s_max[w]);
    if (w > warp) Le = min(Le, s_min[w]);
    qmin = min(qmin, s_min[w]);
    qmax = max(qmax, s_max[w]);
  }
  const uint64_t span1 = (uint64_t)((unsigned)qmax - (unsigned)qmin) + 1;
  const int scale = (int)(unsigned)min(((uint64_t)nk << 32) / span1, (uint64_t)0xffffffffu);
  if (g < nb) {
    // Bucket k's window: from the first position whose prefix maximum falls into
    // bucket k or a later one, to the first position whose suffix minimum falls
    // into a later one, with a margin for the error of a threshold.  Position i
    // fills the buckets that it is the first for.
    auto up = [&](int v) {
      return step_bucket(step_place((int)min((long long)v + p.eps_max, (long long)INT_MAX), qmin, scale), nk);
    };
    auto down = [&](int v) {
      return step_bucket(step_place((int)max((long long)v - p.eps_max, (long long)qmin), qmin, scale), nk);
    };
#pragma unroll
    for (int i = 0; i < kStepBlock; ++i) s_q[g * kStepBlock + i] = qv[i];
    int u = Ue, ub = g > 0 ? up(Ue) : -1;
    int l[kStepBlock];
    int run = Le;
#pragma unroll
    for (int i = kStepBlock - 1; i >= 0; --i) {
      run = min(run, qv[i]);
      l[i] = run;
    }
#pragma unroll
    for (int i = 0; i < kStepBlock; ++i) {
      const int pos = g * kStepBlock + i;
      u = max(u, qv[i]);
      // the last position takes what is left: no threshold leads past the row
      const int nu = pos + 1 < p.cpad ? up(u) : nk - 1;
      for (int k = ub + 1; k <= nu; ++k) s_from[k] = (uint16_t)pos;
      ub = nu;
      // suffix minimum from pos on to that from pos + 1 on
      const int a = down(l[i]);
      const int next = i + 1 < kStepBlock ? l[i + 1] : Le;
      const int b = pos + 1 < p.cpad ? down(next) : nk;
      for (int k = a; k < b; ++k) s_to[k] = (uint16_t)(pos + 1);
    }
  }
  __syncthreads();
  uint32_t* tab = p.tab + row * nk;
  uint2* fast = p.fast + row * nk;
  for (int k = threadIdx.x; k < nk; k += blockDim.x) {
    const int from = s_from[k], to = s_to[k];
    tab[k] = (uint32_t)from | (uint32_t)to << 11;
    // the window's skies within the bucket
    unsigned o[3] = {0xffffu, 0xffffu, 0xffffu};
    bool slow = to > from + 3;
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (from + i < to) {
        slow = slow || (i > 0 && s_q[from + i] < s_q[from + i - 1]);
        const long long at = (long long)(step_place(s_q[from + i], qmin, scale) >> kFracShift) - ((long long)k << kFracBits);
        o[i] = (unsigned)max(min(at + (1 << kFracBits), 65000ll), 0ll);
      }
    fast[k] = make_uint2((unsigned)from | (slow ? kWindowSlow : 0u) | o[0] << 16, o[1] | o[2] << 16);
  }
  if (g == 0) {
    int4* m = p.head + row * kStepHead;
    const double ta = anchor_time(p.t_mid, p.n_seg, p.T0, p.tile_shift, j >> p.tile_shift);
    const double tj = p.t_mid[j], dt = tj - ta, d2 = dt * dt;
    const float dth = tj >= p.T0 ? (float)dt : NAN, d2h = (float)d2;
    const float w = p.weights[dj];
    m[0] = make_int4(qmin, qmax, scale, __float_as_int(w));
    m[1] = make_int4(__float_as_int(dth), __float_as_int((float)(dt - (double)(float)dt)), __float_as_int(d2h),
                     __float_as_int((float)(d2 - (double)d2h)));
    longlong2 wi;
    wi.x = __double2ll_rn((double)w * p.w1_scale);
    wi.y = __double2ll_rn((double)w * (double)w * p.w2_scale);
    if (c == 0) p.wfix[(int64_t)j * p.n_det + d] = wi;
    if (c == 0 && tj >= p.T0) {
      atomicAdd(p.wtot + 2 * (blockIdx.x % kStepSlots), (unsigned long long)wi.x);
      atomicAdd(p.wtot + 2 * (blockIdx.x % kStepSlots) + 1, (unsigned long long)wi.y);
    }
  }
}

// The largest |rho| of a map and its level (MapRange): one read of the map.  out[0]:
// bits of the largest; [1], [2]: infinity's bits minus those of the smallest maximum of
// a run of kLevelRun values at least half of which are nonzero, or fewer; [3], [4]:
// the number of such runs (zero at launch).  Bound by memory: four loads in flight per
// thread and one set of atomics per block (a load at a time and a set per warp: 60 us
// for 128 MB and 172 for 800 MB; 31 and 145 so; 31 and 118 for the maximum alone).
template <typename T>
__global__ void map_range_kernel(const T* x, int64_t n, unsigned* out) {
  constexpr unsigned kInf = 0x7f800000u, kAll = 0xffffffffu;
  constexpr int V = 16 / sizeof(T), R = kLevelRun / V;   // values of a load, lanes of a run
  __shared__ unsigned s_out[kMapWords];
  unsigned m = 0, low[2] = {0, 0}, runs[2] = {0, 0};
  const int lane = threadIdx.x & 31;
  const int64_t nv = n / V, stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  auto bits = [](T v) {
    float f;
    if constexpr (sizeof(T) == 2) f = __half2float(v);
    else f = v;
    return __float_as_uint(f) & 0x7fffffffu;
  };
  if (threadIdx.x < kMapWords) s_out[threadIdx.x] = 0;
  __syncthreads();
  // kLoads in flight per thread; lanes past the end take zeros
  constexpr int kLoads = 4;
  for (int64_t i = i0; i - lane < nv; i += kLoads * stride) {
    int4 v[kLoads];
#pragma unroll
    for (int q = 0; q < kLoads; ++q)
      v[q] = i + q * stride < nv ? __ldg(reinterpret_cast<const int4*>(x) + i + q * stride) : make_int4(0, 0, 0, 0);
#pragma unroll
    for (int q = 0; q < kLoads; ++q) {
      const T* e = reinterpret_cast<const T*>(&v[q]);
      unsigned r = 0, c = 0;
#pragma unroll
      for (int k = 0; k < V; ++k) {
        const unsigned b = bits(e[k]);
        r = max(r, b);
        c += b != 0;
      }
      m = max(m, r);
#pragma unroll
      for (int off = 1; off < R; off <<= 1) {
        r = max(r, __shfl_xor_sync(kAll, r, off));
        c += __shfl_xor_sync(kAll, c, off);
      }
      if ((lane & (R - 1)) == 0 && ((i + q * stride) | (R - 1)) < nv && r > 0 && r < kInf) {
        const int few = c < kLevelRun / 2;
        low[few] = max(low[few], kInf - r);
        ++runs[few];
      }
    }
  }
  for (int64_t i = nv * V + i0; i < n; i += stride) m = max(m, bits(x[i]));
  m = __reduce_max_sync(kAll, m);
  if (lane == 0) atomicMax(s_out, m);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const unsigned l = __reduce_max_sync(kAll, low[k]), c = __reduce_add_sync(kAll, runs[k]);
    if (lane == 0 && c) {
      atomicMax(s_out + 1 + k, l);
      atomicAdd(s_out + 3 + k, c);
    }
  }
  __syncthreads();
  if (threadIdx.x < 3) atomicMax(out + threadIdx.x, s_out[threadIdx.x]);
  else if (threadIdx.x < kMapWords) atomicAdd(out + threadIdx.x, s_out[threadIdx.x]);
}

// Shared memory of the search kernel for `cells` difference cells (templates x
// (row + 1)): two word planes, the heads of each warp's turn (and in their place
// the piece sums of a pass's end), FP64 and fp32 series coefficients, df / f0
// (amplitude weights), per-template sums.  What is left of the SM's memory is L1: a smaller layout
// shows (see step_kernel).
constexpr size_t kStepPart = 3 * kStepThreads * 8;
static_assert(kStepWarps * kStepTurn * kStepHead * 16 <= kStepPart, "the heads fit the piece sums' place");
struct StepLayout {
  size_t part, coef, fcoef, head, famp, tsum, total;
  __host__ __device__ constexpr explicit StepLayout(int cells)
      : part(((size_t)cells * 8 + 15) & ~(size_t)15),
        coef(part + kStepPart),
        fcoef(coef + (size_t)kMaxSeriesTerms * 8 * 32),
        head(part),
        famp(fcoef + (size_t)32 * 20),
        tsum(famp + (size_t)32 * 8),
        total(tsum + (size_t)32 * 4 * 8) {}
};
static_assert(StepLayout(kStepCells + 32).total <= 232448 - 1024, "one CTA's shared memory");

// Value kinds VK: fp32 or fp16 powers, or number count and / or two-bin sums; each
// without and with amplitude weights, whose code and registers the others are spared
// (number count 30.9 -> 31.7 ms, two-bin 13.7 -> 13.9 with them).
enum { kF32 = 0, kF16 = 1, kGen = 2, kWithAmp = 3 };
template <int VK>
constexpr bool kAmp = VK >= kWithAmp;
template <int VK>
constexpr bool kGeneral = VK % kWithAmp == kGen;

// A value of the lookup at bin K of row (the caller checks the band); of two bins,
// their sum and its rounding error.
template <int VK>
using StepValue = std::conditional_t<kGeneral<VK>, float2, float>;
template <int VK>
__device__ __forceinline__ StepValue<VK> step_value(const StepParams& p, const StepEvent& ev, int64_t row, int K) {
  if constexpr (VK % kWithAmp == kF32) {
    return __ldg(static_cast<const float*>(ev.rho) + (row + K));
  } else if constexpr (VK % kWithAmp == kF16) {
    return __half2float(__ldg(static_cast<const __half*>(ev.rho) + (row + K)));
  } else {
    const int more = p.track_bins == 2 ? 1 : 0;
    if (ev.bits) {
      const uint32_t* r = ev.bits + row;
      float v = 0.f;
      for (int i = 0; i <= more; ++i) v += (float)((__ldg(r + ((K + i) >> 5)) >> ((K + i) & 31)) & 1u);
      return make_float2(v, 0.f);
    }
    auto power = [&](int64_t o) {
      return p.map_half ? __half2float(__ldg(static_cast<const __half*>(ev.rho) + o))
                        : __ldg(static_cast<const float*>(ev.rho) + o);
    };
    const float a = power(row + K), b = more ? power(row + K + 1) : 0.f;
    const float v = a + b, bb = v - a;   // the error of a sum, Knuth's two-sum
    return make_float2(v, (a - (v - bb)) + (b - bb));
  }
}

// Read-only loads of the lanes that are on, without a branch (0 elsewhere).
__device__ __forceinline__ float load_if(const float* p, bool on) {
  float v;
  asm("{\n.reg .pred q;\nsetp.ne.s32 q, %2, 0;\nmov.f32 %0, 0f00000000;\n@q ld.global.nc.f32 %0, [%1];\n}"
      : "=&f"(v)
      : "l"(p), "r"((int)on));
  return v;
}
__device__ __forceinline__ float load_if(const __half* p, bool on) {
  unsigned short v;
  asm("{\n.reg .pred q;\nsetp.ne.s32 q, %2, 0;\nmov.u16 %0, 0;\n@q ld.global.nc.u16 %0, [%1];\n}"
      : "=&h"(v)
      : "l"(p), "r"((int)on));
  return __half2float(__ushort_as_half(v));
}
__device__ __forceinline__ uint2 load_if(const uint2* p, bool on) {
  uint2 v;
  asm("{\n.reg .pred q;\nsetp.ne.s32 q, %3, 0;\nmov.u32 %0, 0;\nmov.u32 %1, 0;\n@q ld.global.nc.v2.u32 {%0, %1}, [%2];\n}"
      : "=&r"(v.x), "=&r"(v.y)
      : "l"(p), "r"((int)on));
  return v;
}
// Adds hi and lo to two shared words OFF bytes apart on the lanes that are on.
template <int OFF>
__device__ __forceinline__ void add_if(uint32_t cell, int hi, int lo, bool on) {
  asm volatile("{\n.reg .pred q;\nsetp.ne.s32 q, %3, 0;\n@q red.shared.add.s32 [%0], %1;\n@q red.shared.add.s32 [%0+%4], %2;\n}"
               :
               : "r"(cell), "r"(hi), "r"(lo), "r"((int)on), "n"(OFF));
}

// v * s rounded to the fixed-point grid: hi + lo 2^-16 with |lo| <= 2^15
// (|v s| < 2^22), each word plus kMagicBits, which cancels in differences.  The
// product is never rounded before the grid.
__device__ __forceinline__ void to_fixed(float v, float s, int& hi, int& lo) {
  const float t = fmaf(v, s, kMagic);
  const float r = fmaf(v, s, -(t - kMagic));
  hi = __float_as_int(t);
  lo = __float_as_int(fmaf(r, 65536.0f, kMagic));
}
// v s + more, |more| < 2^-22 |v s|
__device__ __forceinline__ void to_fixed(float v, float s, float more, int& hi, int& lo) {
  const float t = fmaf(v, s, kMagic);
  const float r = fmaf(v, s, -(t - kMagic)) + more;
  hi = __float_as_int(t);
  lo = __float_as_int(fmaf(r, 65536.0f, kMagic));
}
// The same on a grid of 2^-22 as one 64-bit word: the sums of weights are 64 bits.
constexpr int kWordBits = 22;
__device__ __forceinline__ long long fixed_word(float v, float s, float more) {
  constexpr float kUnit = (float)(1 << kWordBits);
  const float t = fmaf(v, s, kMagic);
  const float r = fmaf(v, s, -(t - kMagic)) + more;
  const int hi = __float_as_int(t) - kMagicBits, lo = __float_as_int(fmaf(r, kUnit, kMagic)) - kMagicBits;
  return (long long)hi * (1 << kWordBits) + lo;
}
// A value times the weight s + sl (sl with amplitude weights only).
template <int VK>
__device__ __forceinline__ void to_fixed(StepValue<VK> v, float s, float sl, int& hi, int& lo) {
  if constexpr (kGeneral<VK>) to_fixed(v.x, s, kAmp<VK> ? fmaf(v.y, s, v.x * sl) : v.y * s, hi, lo);
  else if constexpr (kAmp<VK>) to_fixed(v, s, v * sl, hi, lo);
  else to_fixed(v, s, hi, lo);
}

// (h + l)^n, 1 <= n and |l| < |h|, as an fp32 pair x + y with x the nearest float:
// products of pairs whose rounding errors are recovered by fma.
__device__ __forceinline__ float2 pair_power(float h, float l, int n) {
  const float s = h + l;
  l -= s - h;
  h = s;
  float x = h, y = l;
  for (int k = 1; k < n; ++k) {
    const float t = x * h;
    y = fmaf(x, h, -t) + fmaf(x, l, y * h);
    x = t;
  }
  const float t = x + y;
  return make_float2(t, y - (t - x));
}

// A lookup's weight w (f/f0)^p as an fp32 pair h + l: what the per-lookup kernel
// has in FP64.  Its words in the sums W1 and W2.
struct PairWeight {
  float h, l;
  __device__ __forceinline__ PairWeight(float w, float2 amp) {
    h = w * amp.x;
    l = fmaf(w, amp.x, -h) + w * amp.y;
  }
  __device__ __forceinline__ long long w1(const StepEvent& ev) const {
    return fixed_word(h, ev.w1_scale, l * ev.w1_scale);
  }
  __device__ __forceinline__ long long w2(const StepEvent& ev) const {
    return fixed_word(h, h * ev.w2_scale, 2.0f * h * l * ev.w2_scale);
  }
};

// The exact thresholds of (template b, segment j) on the q grid, as the group
// kernel takes them: theta_n = (V + n V2) >> 8 between the bins base + n and
// base + n + 1 (Eq. 1 in FP64 from the tile anchor; two-bin lookups: bin
// centres in place of edges).
struct StepExact {
  long long V, V2;
  double h;   // 1/f
  int base;
};
__device__ __forceinline__ StepExact step_exact(const StepParams& p, const StepEvent& ev, const double* coef, int b,
                                                int j, bool two) {
  const int ti = j >> p.tile_shift;
  const double2 an = reinterpret_cast<const double2*>(ev.anchors)[(int64_t)b * ev.n_tiles + ti];
  const double delta = (ev.t_mid[j] - anchor_time(ev.t_mid, ev.n_seg, ev.T0, p.tile_shift, ti)) * an.y;
  double R = coef[(p.nterms - 1) * 32];
  for (int k = p.nterms - 2; k >= 0; --k) R = fma(R, delta, coef[k * 32]);
  const double h = an.x * R;
  StepExact x;
  x.base = __float2int_rn((__frcp_rn((float)h) - (float)p.f_min) * (float)(1.0 / p.df));
  const double Q = p.df * h;
  const double A0 = fma((double)x.base + (two ? 1.0 : 0.5), Q, fma(p.f_min, h, -1.0));
  x.V = __double2ll_rn(A0 * (p.inv_q * 256.0)) + 128;
  x.V2 = __double2ll_rn(Q * (p.inv_q * 256.0));
  x.h = h;
  return x;
}

// v >> 8, saturated to 32 bits
__device__ __forceinline__ int saturate(long long v) {
  const int hi = (int)(v >> 32);
  const int r = (int)__funnelshift_r((unsigned)v, (unsigned)hi, 8);
  return hi >> 7 == r >> 31 ? r : (hi < 0 ? -2147483647 : 2147483647);
}

// Places one step with an exact threshold: calls place(position, up) where the
// state of the sorted skies changes.
template <typename F>
__device__ __forceinline__ void place_exact(const int32_t* q, uint32_t window, int th, const F& place) {
  const int to = (int)(window >> 11);
  bool above = false;
  for (int p = (int)(window & 0x7ff); p < to; ++p) {
    const bool m = __ldg(q + p) >= th;
    if (m != above) place(p, m);
    above = m;
  }
  if (!above) place(to, true);
}

// What the rare lookups of a block need (shared memory).
struct StepBlockCtx {
  const StepEvent* ev;
  int* chi;
  const double* coef;
  unsigned long long* tsum;
  longlong2* edge;
  int b0, cpad, nk, chunk;
  unsigned edge_mask;   // templates with band-edge weight steps (bit per template)
  unsigned n_edge;      // lookups at a band edge
};

// A lookup (template lt of the block; segment j, detector d) by the exact
// thresholds: all of it with its weights at a band edge (only < 0), or only its
// step `only`, whose fp32 threshold came too close to a sky.
template <int VK, int LT>
__device__ __forceinline__ void step_rare(const StepParams& p, StepBlockCtx& c, int lt, int j, int d, int only) {
  const StepEvent& ev = *c.ev;
  const bool two = kGeneral<VK> && p.track_bins == 2;
  const unsigned k_end = (unsigned)max(0, (int)p.n_bin - (two ? 1 : 0));
  const int64_t row = ((int64_t)c.chunk * ev.n_seg + j) * p.n_det + d;
  const int4 m0 = ev.head[row * kStepHead];
  const float dth = __int_as_float(ev.head[row * kStepHead + 1].x);
  if (!(dth == dth)) return;   // before T0
  const StepExact x = step_exact(p, ev, c.coef + lt, c.b0 + lt, j, two);
  float2 amp = make_float2(1.0f, 0.0f);
  if (kAmp<VK>) {
    // (f0/f)^p, and its reciprocal by a Newton step from fp32's
    const double rr = x.h * ev.f0[c.b0 + lt];
    const float rh = (float)rr;
    const float2 rp = pair_power(rh, (float)(rr - (double)rh), p.amp_power);
    const float u = __frcp_rn(rp.x);
    amp = make_float2(u, u * (fmaf(-rp.x, u, 1.0f) - rp.y * u));
  }
  const PairWeight w(__int_as_float(m0.w), amp);
  const float ws = w.h * ev.x_scale, wsl = w.l * ev.x_scale;
  const int64_t vrow =
      ((int64_t)d * ev.n_seg + j) * (kGeneral<VK> && ev.bits ? (int64_t)ev.bit_pitch : p.n_bin);
  const int qmin = m0.x, qmax = m0.y;
  auto value = [&](int K, int& h, int& l) {
    StepValue<VK> v{};
    if ((unsigned)K < k_end) v = step_value<VK>(p, ev, vrow, K);
    to_fixed<VK>(v, ws, wsl, h, l);
  };
  auto step = [&](int t, int K, long long e1, long long e2) {   // from bin K to K + 1
    int h0, l0, h1, l1;
    value(K, h0, l0);
    value(K + 1, h1, l1);
    const int dh = h1 - h0, dl = l1 - l0;
    const uint32_t win = __ldg(ev.tab + row * c.nk + step_bucket(step_place(t, qmin, m0.z), c.nk));
    place_exact(ev.q + row * c.cpad, win, t, [&](int pos, bool up) {
      int* const cell = c.chi + (pos << (LT + 1)) + lt;
      atomicAdd(cell, up ? dh : -dh);
      atomicAdd(cell + (1 << LT), up ? dl : -dl);
      if (e1 | e2) {
        unsigned long long* ec = reinterpret_cast<unsigned long long*>(c.edge + (int64_t)lt * (c.cpad + 1) + pos);
        atomicAdd(ec, (unsigned long long)(up ? e1 : -e1));
        atomicAdd(ec + 1, (unsigned long long)(up ? e2 : -e2));
      }
    });
  };
  // first boundary above the lowest sky
  int n = -kExactSpan;
  long long v = x.V + n * x.V2;
  while (n < kExactSpan && saturate(v) <= qmin) {
    v += x.V2;
    ++n;
  }
  const int K0 = x.base + n;   // the lowest sky's bin
  if (only >= 0) {
    step(saturate(v + only * x.V2), K0 + only, 0, 0);
    return;
  }
  int nb = 0;
  for (long long u = v; nb < kNThr && saturate(u) <= qmax; u += x.V2) ++nb;
  long long u1, u2;   // the lookup's weights
  if (kAmp<VK>) {
    u1 = w.w1(ev);
    u2 = w.w2(ev);
  } else {
    const longlong2 wi = ev.wfix[(int64_t)j * p.n_det + d];
    u1 = wi.x;
    u2 = wi.y;
  }
  const bool first = (unsigned)K0 < k_end;
  if (K0 < 0 || (unsigned)(K0 + nb) >= k_end) {
    atomicAdd(&c.n_edge, 1u);
    atomicOr(&c.edge_mask, 1u << lt);
  }
  int h0, l0;
  value(K0, h0, l0);
  atomicAdd(c.tsum + lt, (unsigned long long)((long long)(h0 - kMagicBits) * 65536 + (l0 - kMagicBits)));
  // W1, W2 start from every segment's weights, amplitude weights from 0
  if (first == kAmp<VK>) {
    atomicAdd(c.tsum + 32 + lt, (unsigned long long)(first ? u1 : -u1));
    atomicAdd(c.tsum + 64 + lt, (unsigned long long)(first ? u2 : -u2));
  }
  for (int i = 0; i < nb; ++i) {
    const bool ok0 = (unsigned)(K0 + i) < k_end, ok1 = (unsigned)(K0 + i + 1) < k_end;
    step(saturate(v + i * x.V2), K0 + i, ok1 == ok0 ? 0 : (ok1 ? u1 : -u1), ok1 == ok0 ? 0 : (ok1 ? u2 : -u2));
  }
}

// The end of a pass: prefix sums of the cells over the sky positions; after the
// last pass Psi (Eq. 4), before it the sums move to the next pass's sky order.
// All threads of the CTA; a call, so that its registers do not weigh on the
// search loop.
template <int VK, int LT>
__device__ __noinline__ void step_fold(const StepParams& p, StepBlockCtx& s_ctx, unsigned char* smem, long long* part,
                                       int pass, bool last) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int T = 1 << LT, pieces = kStepThreads >> LT;
  const StepEvent& ev = *s_ctx.ev;
  int* const chi = reinterpret_cast<int*>(smem);
  int* const clo = chi + T;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t = tid & (T - 1), pc = tid >> LT, cpad = s_ctx.cpad;
  const int len = (cpad + pieces - 1) / pieces;
  const int p0 = min(cpad, pc * len), p1 = min(cpad, p0 + len);
  const unsigned long long* const tsum = s_ctx.tsum;
  longlong2* const edge_acc = s_ctx.edge + kStepCells + 32;
  longlong2* const ecol = s_ctx.edge + (int64_t)t * (cpad + 1);
  const bool two = kGeneral<VK> && p.track_bins == 2;
  const int chunk = s_ctx.chunk, b0 = s_ctx.b0;
  const bool te = (s_ctx.edge_mask >> t) & 1u;
  {
    long long sx = 0, s1 = 0, s2 = 0;
    for (int q = p0; q < p1; ++q) {
      const int c = (q << (LT + 1)) + t;
      sx += (long long)chi[c] * 65536 + clo[c];
      if (te) {
        const longlong2 v = __ldcg(ecol + q);
        s1 += v.x;
        s2 += v.y;
      }
    }
    part[tid] = sx;
    part[kStepThreads + tid] = s1;
    part[2 * kStepThreads + tid] = s2;
  }
  __syncthreads();
  // exclusive scans over a template's pieces (32, 64 or 256), one warp per template
  for (int tt = warp; tt < T; tt += kStepWarps) {
    const int ks = s_ctx.edge_mask >> tt & 1u ? 3 : 1;
    for (int k = 0; k < ks; ++k) {
      long long run = 0;
      for (int i0 = 0; i0 < pieces; i0 += 32) {
        long long* const q = part + k * kStepThreads + ((i0 + lane) << LT) + tt;
        const long long v = i0 + lane < pieces ? *q : 0;
        long long sum = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const long long u = __shfl_up_sync(kAll, sum, off);
          if (lane >= off) sum += u;
        }
        if (i0 + lane < pieces) *q = run + sum - v;
        run += __shfl_sync(kAll, sum, 31);
      }
    }
  }
  __syncthreads();
  if (!last) {
    // the sums move to the next pass's order of the skies: prefix sums in place, then their
    // differences along the new order (exact integers modulo 2^48)
    long long X = part[tid], w1 = part[kStepThreads + tid], w2 = part[2 * kStepThreads + tid];
    for (int q = p0; q < p1; ++q) {
      const int c = (q << (LT + 1)) + t;
      X += (long long)chi[c] * 65536 + clo[c];
      chi[c] = (int)(X >> 16);
      clo[c] = (int)(X & 0xffff);
      if (te) {
        const longlong2 v = __ldcg(ecol + q);
        w1 += v.x;
        w2 += v.y;
        __stcg(edge_acc + (int64_t)t * cpad + q, make_longlong2(w1, w2));
      }
    }
    __syncthreads();
    const int16_t* map = ev.remap + ((int64_t)(pass + 1) * ev.n_chunks + chunk) * cpad;
    long long prev = 0;
    longlong2 eprev = make_longlong2(0, 0);
    if (p0 > 0 && p0 < p1) {
      const int m = map[p0 - 1], c = (m << (LT + 1)) + t;
      prev = (long long)chi[c] * 65536 + clo[c];
      if (te) eprev = __ldcg(edge_acc + (int64_t)t * cpad + m);
    }
    constexpr int kLen = kStepMaxChunk * 16 / kStepThreads;   // positions of a piece
    int dh[kLen], dl[kLen];
#pragma unroll
    for (int i = 0; i < kLen; ++i) {
      if (p0 + i < p1) {
        const int m = map[p0 + i], c = (m << (LT + 1)) + t;
        const long long v = (long long)chi[c] * 65536 + clo[c], u = v - prev;
        prev = v;
        dh[i] = (int)(u >> 16);
        dl[i] = (int)(u & 0xffff);
        if (te) {
          const longlong2 w = __ldcg(edge_acc + (int64_t)t * cpad + m);
          __stcg(ecol + p0 + i, make_longlong2(w.x - eprev.x, w.y - eprev.y));
          eprev = w;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kLen; ++i) {
      if (p0 + i < p1) {
        const int c = ((p0 + i) << (LT + 1)) + t;
        chi[c] = dh[i];
        clo[c] = dl[i];
      }
    }
  } else {
    // Eq. 4: <s> = mq W1, sigma^2 = vq W2 (power: 1, 1; number count: q, q(1-q)),
    // both doubled for two-bin lookups
    const double nbins = two ? 2.0 : 1.0;
    const bool count = kGeneral<VK> && p.nc_q > 0.0;
    const double mq = nbins * (count ? p.nc_q : 1.0);
    const double vq = nbins * (count ? p.nc_q * (1.0 - p.nc_q) : 1.0);
    const double m_units = mq * ev.w1_unit / ev.x_unit;   // mean of one W1 unit, in units of X
    const int64_t sky0 = (int64_t)chunk * ev.chunk;
    const int rows = min(ev.chunk, ev.S - (int)sky0);
    long long X = part[tid] + (long long)tsum[t];
    long long w1 = (long long)tsum[32 + t], w2 = (long long)tsum[64 + t];
    if (te) {
      w1 += part[kStepThreads + tid];
      w2 += part[2 * kStepThreads + tid];
    }
    // skies without band-edge steps share W1, W2 and the mean
    long long mean = 0;
    float W2f = 0.f, Rh = 0.f, Rl = 0.f;   // Rh + Rl: 2^24 units of X in sigma
    auto moments = [&]() {
      mean = __double2ll_rn((double)w1 * m_units);
      W2f = (float)((double)w2 * ev.w2_unit);
      // 1 / sqrt(vq w2) as an fp32 pair: rsqrtf and one Newton step, r + r (1 - v r^2) / 2,
      // with v r^2 - 1 in fp32 pairs; what it drops is below 2^-42
      const double v = vq * (double)w2;
      const float vh = (float)v, vl = (float)(v - (double)vh);
      const float r = rsqrtf(vh), p2 = r * r;
      const float e = fmaf(vh, p2, -1.0f) + fmaf(vh, fmaf(r, r, -p2), vl * p2);
      Rh = r * ev.r_unit;
      Rl = -0.5f * Rh * e;
    };
    moments();
    const int16_t* order = ev.order ? ev.order + ((int64_t)pass * ev.n_chunks + chunk) * cpad : nullptr;
    for (int q = p0; q < p1; ++q) {
      const int c = (q << (LT + 1)) + t;
      X += (long long)chi[c] * 65536 + clo[c];
      chi[c] = clo[c] = 0;
      if (te) {
        const longlong2 v = __ldcg(ecol + q);
        __stcg(ecol + q, make_longlong2(0, 0));
        w1 += v.x;
        w2 += v.y;
        if (v.x | v.y) moments();
      }
      if (q >= rows) continue;
      // the cells' high words wrap at 2^31, so X is known modulo 2^48
      const long long x = (long long)((unsigned long long)X << 16) >> 16;
      const int64_t o = (sky0 + (order ? (int)order[q] : q)) * ev.Bpad + b0 + t;
      // x - mean as a 2^24 + b, both exact in fp32, so that Psi is rounded once
      const long long u = x - mean;
      const int a = (int)((u + (1 << 23)) >> 24);
      const float af = (float)a, bf = (float)(int)(u - ((long long)a << 24)) * (1.0f / 16777216.0f);
      ev.psi[o] = W2f > 0.f ? fmaf(af, Rh, fmaf(af, Rl, bf * Rh)) : -INFINITY;
      if (ev.S_out) {
        ev.S_out[o] = (float)((double)x * ev.x_unit);
        ev.W1_out[o] = (float)((double)w1 * ev.w1_unit);
        ev.W2_out[o] = W2f;
      }
    }
  }
}

// The search kernel: one CTA per SM takes (sky chunk, template block) items from
// a counter; the difference cells of a block (4, 16 or 32 templates x up to 1024
// skies, two words each) live in shared memory, one column per template.  A
// lane owns one (template, segment) of its warp's turn: the fp32 track, the
// first sky's bin, and for each bin boundary inside the chunk's Doppler range a
// step, placed by one 8-byte table entry of the threshold's bucket.  What fp32
// cannot decide (a sky within the threshold's error, about 2 in 1000 steps),
// skies out of order, crowded buckets and lookups at a band edge go on a list
// that the warp works through with the exact FP64 thresholds once it is full or
// the pass moves on, with all its lanes, so that the search loop has no FP64 and
// no calls and few spills.
// It is bound by the latency of its scattered reads (values and table entries,
// one per lane): about 150 instructions per 32 (template, segment) and 100 more
// for each round of steps, 0.66 issued per scheduler and cycle with one sky and
// 0.45 with 1024, nothing saturated; hence 32 warps (24: 3-10 % slower), and a
// shared layout that leaves 92 KB of L1 (28 KB: 1.5 times the time).
// 2e5 templates x 1024 skies x 2 detectors x 1e4 segments: 655 ms by the group
// kernel, 276 with the track in fp32 pairs and every step searched where it
// arises, 160 with steps queued per warp and compared with skies read from the
// rows, 146 with the list worked through turn by turn, 139 with it worked through
// full, 133 with tiles of 64 segments and sums that round Psi once; one sky and one
// detector: 205, 50, 24, 22.8, 22.6, 18.6 ms; 8 events of 100-800 skies and 1.2e4
// templates: 121 ms by the group kernel, 19.2 turn by turn, 16.9 full, 15.2.
template <int VK, int DP, int LT>
__global__ void __launch_bounds__(kStepThreads, 1) step_kernel(StepParams p, int cells) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  __shared__ unsigned long long s_wtot[2];
  __shared__ int s_turn;
  __shared__ StepBlockCtx s_ctx;
  __shared__ StepEvent s_ev;   // the item's event: read in the loops without a trip to global memory
  const StepLayout L(cells);
  int* const chi = reinterpret_cast<int*>(smem);
  constexpr int T = 1 << LT;      // templates of a block
  int* const clo = chi + T;       // cell (position, template) at [position][word][template]
  long long* const part = reinterpret_cast<long long*>(smem + L.part);
  double* const coef = reinterpret_cast<double*>(smem + L.coef);
  float4* const fcoef = reinterpret_cast<float4*>(smem + L.fcoef);   // [32]: C(e, 3) .. C(e, 6)
  float* const fcoef7 = reinterpret_cast<float*>(fcoef + 32);        // [32]: C(e, 7)
  float2* const famp = reinterpret_cast<float2*>(smem + L.famp);     // [32]: df / f0 as an fp32 pair
  int4* const slow_list = p.slow + ((int64_t)blockIdx.x * kStepWarps + (threadIdx.x >> 5)) * kStepSlow;
  int4* const heads = reinterpret_cast<int4*>(smem + L.head) + (threadIdx.x >> 5) * kStepTurn * kStepHead;
  unsigned long long* const tsum = reinterpret_cast<unsigned long long*>(smem + L.tsum);   // X0, W1, W2 [32]
  const int tid = threadIdx.x, lane = tid & 31;
  const bool two = kGeneral<VK> && p.track_bins == 2;
  constexpr unsigned kAll = 0xffffffffu;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int n_bin = (int)p.n_bin;
  const float hb = two ? 1.0f : 0.5f;   // boundary n lies at base + n + hb
  longlong2* const edge = p.edge + (int64_t)blockIdx.x * (2 * kStepCells + 32);

  for (int i = tid; i < 2 * cells; i += kStepThreads) chi[i] = 0;
  if (tid == 0) s_ctx.n_edge = 0;

  while (true) {
    __syncthreads();
    if (tid == 0) {
      s_item = (int)atomicAdd(p.next, 1u);
    }
    __syncthreads();
    if (s_item >= p.n_items) break;
    int4 item;
    if (p.items) {
      item = p.items[s_item];
    } else {
      const int blocks = p.events[0].Bpad >> LT, g0 = s_item / p.n_chunks * p.bank_chunk;
      item = make_int4(0, s_item % p.n_chunks, g0 << LT, min(p.bank_chunk, blocks - g0));
    }
    for (int i = tid; i < (int)(sizeof(StepEvent) / 4); i += kStepThreads)
      reinterpret_cast<int*>(&s_ev)[i] = reinterpret_cast<const int*>(p.events + item.x)[i];
    __syncthreads();
    const StepEvent& ev = s_ev;
    const int cpad = ev.cpad;
    const int n_seg = ev.n_seg, sub = min(ev.sub_shift, DP == 1 ? 4 : 3);
    const int lt = lane & (T - 1), ls = lane >> LT;
    constexpr int lps = 32 >> LT;
    const unsigned t_mask = T == 32 ? kAll : (1u << T) - 1u;
    const int nk = step_buckets(cpad);
    const int vpitch = kGeneral<VK> && ev.bits ? ev.bit_pitch : n_bin;
    const int64_t row0 = (int64_t)item.y * n_seg * p.n_det;
    const float xs = ev.x_scale;

    // W1, W2 of every segment from T0 on (unit and per-segment weights: lookups
    // outside the band are taken off; amplitude weights are summed per lookup)
    if (tid < 2) {
      long long sum = 0;
      if (!kAmp<VK>)
        for (int i = 0; i < kStepSlots; ++i) sum += __ldg(ev.wtot + 2 * i + tid);
      s_wtot[tid] = (unsigned long long)sum;
    }
    __syncthreads();
    if (tid < 32 * 3) tsum[tid] = tid < 32 ? 0 : s_wtot[tid / 32 - 1];

    for (int tb = 0; tb < item.w; ++tb) {
      const int b0 = item.z + tb * T, b = b0 + lt;
      if (tid == 0) {
        s_ctx.ev = &ev;
        s_ctx.chi = chi;
        s_ctx.coef = coef;
        s_ctx.tsum = tsum;
        s_ctx.edge = edge;
        s_ctx.b0 = b0;
        s_ctx.cpad = cpad;
        s_ctx.nk = nk;
        s_ctx.chunk = item.y;
        s_ctx.edge_mask = 0;
      }
      if (tid < T) {
        // binomial coefficients C(r, k) of 1/f and C(e, k) of f, r = 1/(n - 1) = -e
        const double r = 1.0 / (ev.nbr[b0 + tid] - 1.0);
        double c = 1.0;
        for (int k = 0; k < p.nterms; ++k) {
          coef[k * 32 + tid] = c;
          c = c * (r - k) / (k + 1);
        }
        float cf[kStepTerms];
        c = 0.5 * r * (r + 1.0);
#pragma unroll
        for (int k = 0; k < kStepTerms; ++k) {
          c = c * (-r - (k + 2)) / (k + 3);
          cf[k] = (float)c;
        }
        fcoef[tid] = make_float4(cf[0], cf[1], cf[2], cf[3]);
        fcoef7[tid] = cf[4];
        if (kAmp<VK>) {
          const double u = p.df / ev.f0[b0 + tid];
          famp[tid] = make_float2((float)u, (float)(u - (double)(float)u));
        }
      }
      __syncthreads();
      long long X0 = 0;
      for (int pass = 0; pass < ev.passes; ++pass) {
        const int per = p.n_det / DP;
        const int d0 = DP == 1 ? pass % per : 0;
        const int js = pass / per * ev.pass_seg, je = min(n_seg, js + ev.pass_seg);
        for (int jc = js; jc < je; jc += kStepCarry) {
          const int jce = min(je, jc + kStepCarry);
          // The warps take the turns as they come: their lengths in time differ.  The last turn's worth of
          // each warp goes in quarters (a full round of segments at least), so that the warps end a pass
          // closer together.
          const int small = min(sub, max(sub - 2, max(2, 5 - LT))), big = max(0, ((jce - jc) >> sub) - kStepWarps);
          if (tid == 0) s_turn = 0;
          __syncthreads();
          int j0 = 0, jn = 0;   // the warp's turn: segments left to it
          int nslow = 0;        // steps and lookups in the warp's list
          while (true) {
            if (j0 >= jn) {
              int turn = 0;
              if (lane == 0) turn = atomicAdd(&s_turn, 1);
              turn = __shfl_sync(kAll, turn, 0);
              j0 = jc + (turn < big ? turn << sub : (big << sub) + ((turn - big) << small));
              jn = min(jce, j0 + (1 << (turn < big ? sub : small)));
            }
            const bool end = j0 >= jce;
            if (nslow > kStepSlow - kStepSlowMore || (end && nslow > 0)) {
              // the list, when it fills up and before the pass moves on
              __syncwarp();
              const int64_t row1 = row0 + (int64_t)jc * p.n_det + d0;
              for (int i = lane; i < nslow; i += 32) {
                const int4 e = __ldcg(slow_list + i);
                const int rr = e.w >> 17, le = e.z & 31, dl = e.z >> 5;
                int only = e.w >> 14 & 7;
                if (only != kStepLookup) {
                  const int64_t row = row1 + (int64_t)(rr / DP) * p.n_det + rr % DP;
                  const int32_t* const q = ev.q + row * cpad;
                  const int4 m = ev.head[row * kStepHead];
                  const uint64_t pl = step_place(e.x, m.x, m.z);
                  const uint32_t win = __ldg(ev.tab + (row * nk + step_bucket(pl, nk)));
                  const int er = e.w & 0x3fff;
                  bool near = er == kErrMax;
                  for (int k = (int)(win & 0x7ffu); k < (int)(win >> 11); ++k) {
                    const long long off = (long long)(step_place(__ldg(q + k), m.x, m.z) >> kFracShift) -
                                          (long long)(pl >> kFracShift);
                    near = near || llabs(off) <= er;
                  }
                  if (!near) {
                    place_exact(q, win, e.x, [&](int pos, bool up) {
                      int* const cell = chi + ((pos << (LT + 1)) + le);
                      atomicAdd(cell, up ? e.y : -e.y);
                      atomicAdd(cell + T, up ? dl : -dl);
                    });
                    continue;
                  }
                } else {
                  only = -1;
                }
                step_rare<VK, LT>(p, s_ctx, le, jc + rr / DP, d0 + rr % DP, only);
              }
              nslow = 0;
              __syncwarp();
            }
            if (end) break;
            const int64_t rbase = row0 + (int64_t)j0 * p.n_det + d0;   // first row of the turn
            const int64_t vbase = ((int64_t)d0 * n_seg + j0) * vpitch;
            unsigned scale = 0;   // the finest buckets of the turn's rows
            {
              // heads of the turn's rows
              __syncwarp();
              const int nr = (jn - j0) * DP;
              if (lane < nr) {
                const int4* h = ev.head + (rbase + (int64_t)(lane / DP) * p.n_det + lane % DP) * kStepHead;
                const int4 m = __ldg(h);
                heads[lane * kStepHead] = m;
                scale = (unsigned)m.z;
                heads[lane * kStepHead + 1] = __ldg(h + 1);
              }
              scale = __reduce_max_sync(kAll, scale);
              __syncwarp();
            }
            // dt at the ends of the turn; NaN before T0
            const float dt_first = __int_as_float(heads[1].x);
            const float dt_last = __int_as_float(heads[((jn - j0) * DP - 1) * kStepHead + 1].x);
            if (!(dt_last == dt_last)) {
              j0 = jn;
              continue;
            }
            const int4* tp =
                reinterpret_cast<const int4*>(ev.tiles + ((int64_t)b * ev.n_tiles + (j0 >> p.tile_shift)));
            const int4 t0 = __ldg(tp), t1 = __ldg(tp + 1);
            const int base_a = t0.x;
            const float frac_a = __int_as_float(t0.y), A_hi = __int_as_float(t0.z), A_lo = __int_as_float(t0.w);
            const float Q_hi = __int_as_float(t1.x), Q_lo = __int_as_float(t1.y), Xf = __int_as_float(t1.z),
                        sg = __int_as_float(t1.w);
            // The template's bins over the turn (tracks fall, Doppler shifts below 3 bins): wholly in the
            // band, wholly out of it, or at an edge (or T0): every lookup goes on the list
            bool edge;
            unsigned outside;
            // the thresholds' error bound at the turn's lowest frequency in fractions of its finest
            // buckets
            int eps;
            {
              const float x0 = fmaf(A_hi, dt_first, fmaf(Q_hi, dt_first * dt_first, (float)base_a));
              const float x1 = fmaf(A_hi, dt_last, fmaf(Q_hi, dt_last * dt_last, (float)base_a));
              const bool whole = dt_first == dt_first;
              const bool in = whole && fminf(x0, x1) >= 8.0f && fmaxf(x0, x1) <= (float)n_bin - 10.0f;
              const bool out = whole && (fmaxf(x0, x1) < -8.0f || fminf(x0, x1) > (float)n_bin + 8.0f);
              outside = __ballot_sync(kAll, out);
              edge = !out && !in;
              const float F1 = Xf + (fminf(x0, x1) - (float)base_a);
              const float e = fmaf(rcp_approx(F1) * p.inv_q_f, p.eps, 1.5f) * (float)scale;
              eps = (int)fminf(fmaf(e, 1.0f / (1 << kFracShift), 3.0f), (float)kErrMax);
            }
            const bool mine = !((outside >> lane) & 1u);
            // a row's number within the segments from jc on, in place
            const int rr0 = (j0 - jc) * DP;
            const uint32_t cells0 = (uint32_t)__cvta_generic_to_shared(chi + lt);
            // Places step i of a lookup, one per lane that is on: at the sky at which the threshold lies
            // among the bucket's.  The others go on the list: longer windows, skies out of order, a sky
            // within the threshold's error.
            auto place = [&](bool on, int i, int th, uint32_t at, uint2 w, int dh, int dl, int rr) {
              const int low = (int)at - eps;
              const int o0 = (int)(w.x >> 16) - low, o1 = (int)(w.y & 0xffffu) - low, o2 = (int)(w.y >> 16) - low;
              const unsigned wide = 2u * (unsigned)eps;
              const bool slow = on && ((unsigned)o0 <= wide || (unsigned)o1 <= wide || (unsigned)o2 <= wide ||
                                       (w.x & kWindowSlow) || eps == kErrMax);
              const int pos = (int)(w.x & 0x7ffu) + (o0 < eps) + (o1 < eps) + (o2 < eps);
              add_if<T * 4>(cells0 + (uint32_t)(pos << (LT + 3)), dh, dl, on && !slow);
              if (const unsigned vote = __ballot_sync(kAll, slow)) {
                // threshold; difference words, template; row, step, error
                if (slow)
                  slow_list[nslow + __popc(vote & lt_mask)] = make_int4(th, dh, dl * 32 | lt, rr << 17 | i << 14 | eps);
                nslow += __popc(vote);
              }
            };
            const int ns = jn - j0;
            int jb = outside == kAll ? ns : 0;
            // the turn's first-sky powers, each with kMagicBits, and their number: sums modulo 2^32
            unsigned xh = 0, xl = 0, nx = 0;
            for (; jb < ns && nslow <= kStepSlow - kStepSlowMore; jb += lps) {
              const int jr = min(jb + ls, ns - 1);
              const bool here = mine && jb + ls < ns;
              const int4* head = heads + jr * DP * kStepHead;
              const float4 dt = *reinterpret_cast<const float4*>(head + 1);
              // the unshifted track's position base + frac and F = f/df (see StepTile): the linear and
              // quadratic terms as products of fp32 pairs whose rounding errors are recovered by fma and
              // whose integer parts are split off exactly, the rest an fp32 series
              const float pl = A_hi * dt.x, plr = rintf(pl);
              const float pq = Q_hi * dt.z, pqr = rintf(pq);
              const float dl3 = dt.x * sg;
              const float4 cf = fcoef[lt];
              float hs = fmaf(fcoef7[lt], dl3, cf.w);
              hs = fmaf(hs, dl3, cf.z);
              hs = fmaf(hs, dl3, cf.y);
              hs = fmaf(hs, dl3, cf.x);
              const float p3 = Xf * (dl3 * dl3 * dl3 * hs);
              const float small = (fmaf(A_hi, dt.x, -pl) + fmaf(A_hi, dt.y, A_lo * dt.x)) +
                                  (fmaf(Q_hi, dt.z, -pq) + fmaf(Q_hi, dt.w, Q_lo * dt.z)) + p3;
              const float F = (Xf + pl) + (pq + p3);
              const float Fq = F * p.q, R = rcp_approx(F) * p.inv_q_f;
              const float y0 = ((frac_a + (pl - plr)) + ((pq - pqr) + small)) - hb;
              float2 amp = make_float2(1.0f, 0.0f);
              if (kAmp<VK> && here && !edge) {
                // f/f0 as an fp32 pair, from the whole bins and the fraction of f/df apart
                const float2 u = famp[lt];
                const float fi = ((float)base_a + p.x_min_i) + (plr + pqr), ff = (y0 + hb) + p.x_min_f;
                const float rh = fi * u.x;
                amp = pair_power(rh, fmaf(fi, u.x, -rh) + fmaf(fi, u.y, ff * u.x), p.amp_power);
              }
#pragma unroll 1
              for (int dd = 0; dd < DP; ++dd) {
                const int4 m0 = head[dd * kStepHead];
                // the lowest and the highest sky's distance from boundary 0, in bins: boundaries in between
                const float zl = fmaf(Fq, (float)m0.x, y0), zh = fmaf(Fq, (float)m0.y, y0);
                const float fl = floorf(zl), fh = floorf(zh);
                const bool close = here && (edge || fabsf((zl - fl) - 0.5f) > 0.5f - p.eps ||
                                            fabsf((zh - fh) - 0.5f) > 0.5f - p.eps);
                const bool on = here && !close;
                const int rl = jr * p.n_det + dd, rr = rr0 + jr * DP + dd;
                if (const unsigned vote = __ballot_sync(kAll, close)) {
                  if (close)
                    slow_list[nslow + __popc(vote & lt_mask)] = make_int4(0, 0, lt, rr << 17 | kStepLookup << 14);
                  nslow += __popc(vote);
                }
                const int nb = on ? min((int)(fh - fl), kNThr - 1) : 0;
                const int K = base_a + 1 + (int)(plr + pqr + fl);   // the lowest sky's bin
                const int64_t vrow = vbase + (int64_t)(dd * n_seg + jr) * vpitch;
                // the loads of the lookup and its first two steps at once
                const PairWeight w(__int_as_float(m0.w), amp);
                const float ws = w.h * xs, wsl = w.l * xs;
                auto value = [&](int o, bool c) {   // of bin K + o
                  if constexpr (VK % kWithAmp == kF32) return load_if(static_cast<const float*>(ev.rho) + (vrow + K) + o, c);
                  else if constexpr (VK % kWithAmp == kF16) return load_if(static_cast<const __half*>(ev.rho) + (vrow + K) + o, c);
                  else return c ? step_value<VK>(p, ev, vrow, K + o) : make_float2(0.f, 0.f);
                };
                const StepValue<VK> v0 = value(0, on);
                const unsigned some = __ballot_sync(kAll, nb > 0);
                const uint2* const tr = ev.fast + (rbase + rl) * nk;
                const float y1 = fl + 1.0f - y0;
                auto window = [&](int t, uint32_t& at, bool c) {
                  const uint64_t pl = step_place(t, m0.x, m0.z);
                  at = ((uint32_t)pl >> kFracShift) + (1u << kFracBits);
                  return load_if(tr + step_bucket(pl, nk), c);
                };
                StepValue<VK> v1{}, vn{};
                int th0 = 0, th = 0;
                uint2 win0 = make_uint2(0, 0), win = win0;
                uint32_t at0 = 0, at = 0;
                if (some) {
                  th0 = __float2int_rn(y1 * R);
                  th = __float2int_rn((y1 + 1.0f) * R);
                  v1 = value(1, nb > 0);
                  win0 = window(th0, at0, nb > 0);
                  vn = value(2, nb > 1);
                  win = window(th, at, nb > 1);
                }
                int h0, l0, h1, l1;
                to_fixed<VK>(v0, ws, wsl, h0, l0);
                xh += (unsigned)h0;
                xl += (unsigned)l0;
                ++nx;
                if (some) {
                  to_fixed<VK>(v1, ws, wsl, h1, l1);
                  place(nb > 0, 0, th0, at0, win0, h1 - h0, l1 - l0, rr);
                  for (int i = 1; __any_sync(kAll, nb > i); ++i) {
                    h0 = h1;
                    l0 = l1;
                    to_fixed<VK>(vn, ws, wsl, h1, l1);
                    // the next step's loads before this one's placing
                    const int th_i = th;
                    const uint32_t at_i = at;
                    const uint2 win_i = win;
                    vn = value(i + 2, nb > i + 1);
                    th = __float2int_rn((y1 + (float)(i + 1)) * R);
                    win = window(th, at, nb > i + 1);
                    place(nb > i, i, th_i, at_i, win_i, h1 - h0, l1 - l0, rr);
                  }
                }
                if (kAmp<VK> && on) {
                  atomicAdd(tsum + 32 + lt, (unsigned long long)w.w1(ev));
                  atomicAdd(tsum + 64 + lt, (unsigned long long)w.w2(ev));
                }
              }
            }
            X0 += (long long)(int)(xh - nx * kMagicBits) * 65536 + (int)(xl - nx * kMagicBits);
            {
              const int nr = min(jb, ns) * DP;
              if (!kAmp<VK> && (outside & t_mask)) {
                // out of the band: the turn's weights come off
                longlong2 wi = make_longlong2(0, 0);
                if (lane < nr) {
                  const float dth = __int_as_float(heads[lane * kStepHead + 1].x);
                  if (dth == dth) wi = ev.wfix[(int64_t)(j0 + lane / DP) * p.n_det + d0 + lane % DP];
                }
                for (int off = 16; off > 0; off >>= 1) {
                  wi.x += __shfl_xor_sync(kAll, wi.x, off);
                  wi.y += __shfl_xor_sync(kAll, wi.y, off);
                }
                if (ls == 0 && ((outside >> lane) & 1u)) {
                  atomicAdd(tsum + 32 + lt, (unsigned long long)-wi.x);
                  atomicAdd(tsum + 64 + lt, (unsigned long long)-wi.y);
                }
              }
              __syncwarp();
            }
            j0 += min(jb, ns);   // less than the turn when the list is full
          }
          if (jce < je) {
            // carry the low words over before they can overflow
            __syncthreads();
            for (int i = tid; i < (cpad + 1) << LT; i += kStepThreads) {
              const int c = i + (i >> LT << LT), l = clo[c];
              chi[c] += l >> 16;
              clo[c] = l & 0xffff;
            }
            __syncthreads();
          }
        }
        const bool last = pass == ev.passes - 1;
        if (last) {
          for (int off = T; off < 32; off <<= 1) X0 += __shfl_xor_sync(0xffffffffu, X0, off);
          if (ls == 0) atomicAdd(tsum + lt, (unsigned long long)X0);
        }
        __syncthreads();

        step_fold<VK, LT>(p, s_ctx, smem, part, pass, last);
        // the cells past the last sky
        if (tid < T) {
          const int c = (cpad << (LT + 1)) + tid;
          chi[c] = clo[c] = 0;
          if ((s_ctx.edge_mask >> tid) & 1u) __stcg(edge + (int64_t)tid * (cpad + 1) + cpad, make_longlong2(0, 0));
        }
        __syncthreads();
      }
      if (tid < 32 * 3) tsum[tid] = tid < 32 ? 0 : s_wtot[tid / 32 - 1];
      __syncthreads();
    }
  }
  __syncthreads();
  if (tid == 0 && s_ctx.n_edge) atomicAdd(p.n_general, (unsigned long long)s_ctx.n_edge);
}

template <int VK, int DP, int LT>
cudaError_t set_smem() {
  constexpr int kDevices = 64;
  static bool done[kDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < kDevices && done[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(step_kernel<VK, DP, LT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)StepLayout(kStepCells + 32).total);
  if (e == cudaSuccess && dev >= 0 && dev < kDevices) done[dev] = true;
  return e;
}

struct Prepare {
  template <int VK, int DP, int LT>
  cudaError_t run() const { return set_smem<VK, DP, LT>(); }
};

struct Launch {
  const StepParams& p;
  int cells, grid;
  cudaStream_t st;
  template <int VK, int DP, int LT>
  cudaError_t run() const {
    cudaError_t e = set_smem<VK, DP, LT>();
    if (e != cudaSuccess) return e;
    step_kernel<VK, DP, LT><<<grid, kStepThreads, StepLayout(cells).total, st>>>(p, cells);
    return cudaGetLastError();
  }
};

template <int DP, int LT, int AMP, typename F>
cudaError_t pick_value(const StepForm& v, const F& f) {
  if (v.general) return f.template run<AMP + kGen, DP, LT>();
  return v.half ? f.template run<AMP + kF16, DP, LT>() : f.template run<AMP + kF32, DP, LT>();
}
template <int DP, int LT, typename F>
cudaError_t pick_amp(const StepForm& v, const F& f) {
  return v.amp ? pick_value<DP, LT, kWithAmp>(v, f) : pick_value<DP, LT, 0>(v, f);
}
template <typename F>
cudaError_t pick(const StepForm& v, const F& f) {
  const int dp = v.dets_per_pass;
  if (dp == 1 && v.log_t == 2) return pick_amp<1, 2>(v, f);
  if (dp == 1 && v.log_t == 4) return pick_amp<1, 4>(v, f);
  if (dp == 1 && v.log_t == 5) return pick_amp<1, 5>(v, f);
  if (dp == 2 && v.log_t == 2) return pick_amp<2, 2>(v, f);
  if (dp == 2 && v.log_t == 4) return pick_amp<2, 4>(v, f);
  if (dp == 2 && v.log_t == 5) return pick_amp<2, 5>(v, f);
  return cudaErrorInvalidValue;
}

}  // namespace

size_t step_slow_bytes(int grid) { return (size_t)grid * kStepWarps * kStepSlow * sizeof(int4); }

MapRange map_range(const unsigned* out) {
  MapRange r;
  // runs with few nonzero powers are the edges of zeroed stretches, unless they are many
  const unsigned low = out[4] > out[3] / 16 ? std::max(out[1], out[2]) : out[1];
  const unsigned level = out[3] + out[4] ? 0x7f800000u - low : out[0];
  std::memcpy(&r.max, &out[0], 4);
  std::memcpy(&r.level, &level, 4);
  return r;
}

StepScales step_scales(const MapRange& map, int bins, const WeightRange& w, bool amp, double a_ref) {
  StepScales s;
  const double vmax = (double)map.max * bins;
  if (!(vmax >= 0.0) || !(vmax < 1e30) || !(w.max > 0.0)) return s;
  auto lg = [](double v) { return (int)std::ceil(std::log2(v)); };   // v <= 2^lg
  // the sums of a (template, sky), of powers and of their means, within 2^46 units and
  // one value within 2^21 2^16 units
  const double v = std::max(vmax, (double)bins);
  s.x = std::min(46 - lg(v * w.sum), 37 - lg(v * w.max));
  // sums of weights and of their squares below 2^60; amplitude weights are made by the
  // kernel in words of 2^42 (PairWeight), the others here in FP64
  const double max2 = (double)w.max * w.max, sum2 = w.sum * w.max;
  s.w1 = std::min(60 - lg(w.sum), amp ? 42 - lg(w.max) : INT_MAX);
  s.w2 = std::min(60 - lg(sum2), amp ? 42 - lg(max2) : INT_MAX) & ~1;   // even: the root of its unit is a power of 2
  // one unit at most 2^-22 of the smallest weighted power, the noise's mean or, where
  // the map lies lower, twice its level: a sum of m rounded values is then off by about
  // 0.3 sqrt(m) 2^-22 of it, 7e-8 of the standard deviation sqrt(m) that Eq. 4 divides
  // by and less of S
  const double p = map.level > 0 ? std::min(1.0, 2.0 * (double)map.level) : 1.0;
  const int need = 22 - (int)std::floor(std::log2((double)w.min * a_ref * p));
  // W1 and W2 of the smallest weights alone to 2^-25, as fp32 has each of them; squares
  // of amplitude weights, no two of which are alike, to 2^-21 each
  const double a = std::log2((double)w.min * a_ref);
  const bool weights = s.w1 >= 24 - std::floor(a) && s.w2 >= (amp ? 20 : 24) - std::floor(2 * a);
  // exponents that fp32 scales hold (the plain weights' W2 words are made in FP64)
  s.ok = weights && s.x >= need && std::abs(s.x) < 100 && std::abs(s.w1) < 100 && std::abs(s.w2) < (amp ? 130 : 150) &&
         need < 100;
  return s;
}

StepTrack step_track(const double* t_mid, int64_t n_seg, double T0, int most, double tau_min, double r_max,
                     double x_max, double x_top, double db, double f_min, double df, double inv_q) {
  StepTrack r;
  // Bins are compared with the band's edges in fp32, 8 bins and more inside it, and the
  // exact thresholds are looked for 8 boundaries either side of an fp32 estimate of the
  // track's bin.  Up to 2^23 bins that estimate is off by at most 3 (five roundings of
  // 2^-24 in f, f_min and their difference) and a comparison by 1; beyond, neither holds.
  if (!(x_top <= 8388608.0)) return r;
  auto cbound = [&](int k) {   // |C(e, k)| for |e| <= r_max
    double c = 1.0;
    for (int i = 0; i < k; ++i) c *= (r_max + i) / (i + 1);
    return c;
  };
  for (int shift = ilog2(most); shift >= 2; --shift) {
    const int tile = 1 << shift;
    double dmax = 0;   // |t - t_a| / (tau + t_a - T0)
    for (int64_t j0 = 0; j0 < n_seg; j0 += tile) {
      const int64_t jn = std::min<int64_t>(tile, n_seg - j0);
      const double ta = std::max(t_mid[j0 + (jn - 1) / 2], T0), te = t_mid[j0 + jn - 1];
      if (te < T0) continue;
      dmax = std::max(dmax, std::max(te - ta, ta - std::max(t_mid[j0], T0)) / (tau_min + (ta - T0)));
    }
    // the series' dropped terms and the fp32 rounding of its cubic part, in bins
    if (!(dmax <= 0.1) || x_max * cbound(3) * std::pow(dmax, 3) > 0.25 ||
        x_max * cbound(kStepTerms + 3) * std::pow(dmax, kStepTerms + 3) > 2e-8 || x_max * r_max * dmax > 2.0e6)
      continue;
    r.nterms = series_terms_for(t_mid, n_seg, T0, tile, tau_min, r_max);
    if (r.nterms < 1) continue;
    r.shift = shift;
    // Error of an fp32 threshold: the position's sums (values up to 2) and the
    // cubic part 4e-7, the difference to the boundary 1.2e-7 (1 + y), and four
    // roundings of 6e-8 of y (F, 1/F, their products) for y = db + 1 bins
    // at most; emulated worst cases stay below 0.7 of it.
    r.eps = (float)(4.0e-7 + 1.2e-7 * (2.0 + db) + 2.4e-7 * (1.0 + db));
    // in grid units, most at the lowest frequency
    const double f_low = std::max(f_min / df - 8.0, 0.0);
    if (!(f_low >= 64.0)) return r;
    const double worst = r.eps * inv_q / f_low;
    if (!(worst < 120.0 * (1 << 20))) return r;
    r.eps_max = (int)std::ceil(worst) + 2;
    r.ok = true;
    return r;
  }
  return r;
}

int step_block(const StepGeometry& g, int Bpad, int bank_chunk, int grid, double rows) {
  int best = g.log_t;
  double least = 0;
  for (int lt : {5, 4, 2}) {
    if (lt > g.log_t) continue;
    const int64_t blocks = Bpad >> lt, items = g.n_chunks * ((blocks + bank_chunk - 1) / bank_chunk);
    const double ns = lt == 5 ? 2.8 : lt == 4 ? 3.9 : 5.6;
    const double per = (double)std::min<int64_t>(bank_chunk, blocks);   // blocks of an item
    const double us = (double)((items + grid - 1) / grid) * per * (rows * (1 << lt) * ns * 1e-3 + g.passes * 20.0);
    if (lt == g.log_t || us < 0.95 * least) {
      best = lt;
      least = us;
    }
  }
  return best;
}

StepGeometry step_geometry(int64_t S, int D, int64_t n_seg, int tile, const double* v, bool split) {
  StepGeometry g{};
  g.n_chunks = (int)((S + kStepMaxChunk - 1) / kStepMaxChunk);
  g.chunk = (int)(((S + g.n_chunks - 1) / g.n_chunks + 15) / 16 * 16);
  g.n_chunks = (int)((S + g.chunk - 1) / g.chunk);
  const int most = (int)(S < g.chunk ? S : g.chunk);
  g.cpad = (most + kStepBlock - 1) / kStepBlock * kStepBlock;
  g.log_t = (g.cpad + 1) * 32 <= kStepCells + 32 ? 5 : 4;
  // Drift of the detectors' direction of motion (rad) away from a pass's
  // middle: it displaces a sky by up to drift / 2 of a whole-sky list sorted at
  // the middle.  Places out of order cost difference steps of their own (1.2 per
  // boundary at a displacement of 3, 4.5 at 10: emulated on Fibonacci and random
  // lists), a pass costs one fold of the cells.  The places are those of a list
  // of one chunk's length: in a longer list the skies lie closer and the chunks
  // see n_chunks times as many (over 11 h 3 % of the windows are longer than 3
  // skies at 1024 skies, 40 % at 4000 and 69 % at 16000, emulated).
  auto drift = [&](int64_t j0, int64_t j1, int d0, int d1) {
    const double* m = v + ((int64_t)d0 * n_seg + (j0 + j1 - 1) / 2) * 3;
    const double mn = std::sqrt(m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
    double worst = 0;
    for (int d = d0; d < d1; ++d)
      for (int64_t j : {j0, (j0 + j1) / 2, j1 - 1}) {
        const double* x = v + ((int64_t)d * n_seg + j) * 3;
        const double n = std::sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
        if (!(n > 0) || !(mn > 0)) continue;
        double s = 0;
        for (int a = 0; a < 3; ++a) s += (x[a] / n - m[a] / mn) * (x[a] / n - m[a] / mn);
        worst = std::max(worst, std::sqrt(s));
      }
    return worst;
  };
  constexpr double kPlaces = 3.0;
  const double half = 0.5 * (double)most;
  g.dets_per_pass = D;
  int64_t runs = 1;
  if (D > 1 && (split || half * drift(0, n_seg, 0, D) > kPlaces)) g.dets_per_pass = 1;
  if (g.dets_per_pass == 1) {
    // passes of equal length, short enough for the places at both ends
    for (; runs < 64; ++runs) {
      const int64_t L = (n_seg + runs - 1) / runs;
      if (L < 8 * tile) break;
      double worst = 0;
      for (int64_t e = 0; e < runs; ++e)
        for (int d = 0; d < D; ++d)
          if (e * L < n_seg) worst = std::max(worst, drift(e * L, std::min(n_seg, (e + 1) * L), d, d + 1));
      if (half * worst <= kPlaces) break;
    }
  }
  // whole rounds of the 32 warps' turns of 16 segments where a pass is long enough
  const int unit = n_seg / runs >= 512 ? 512 : tile;
  const int64_t L = std::max<int64_t>(1, ((n_seg + runs - 1) / runs + unit / 2) / unit) * unit;
  g.pass_seg = (int)std::min<int64_t>(L, INT32_MAX / 2);
  g.passes = (int)((n_seg + g.pass_seg - 1) / g.pass_seg) * (D / g.dets_per_pass);
  return g;
}

cudaError_t launch_step_rows(const StepRowsParams& p, cudaStream_t st) {
  if (p.order) {
    step_order_kernel<<<dim3((unsigned)p.passes, (unsigned)p.n_chunks), kStepMaxChunk, 0, st>>>(p);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const int nb = p.cpad / kStepBlock;
  const int threads = (nb + 31) / 32 * 32;
  step_rows_kernel<<<dim3((unsigned)(p.n_seg * p.n_det), (unsigned)p.n_chunks), threads, 0, st>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_map_range(const void* rho, bool half, int64_t n, unsigned* out, cudaStream_t st) {
  const int64_t blocks = std::min<int64_t>((n + 8191) / 8192, 152 * 8);
  if (half)
    map_range_kernel<__half><<<(unsigned)blocks, 256, 0, st>>>(static_cast<const __half*>(rho), n, out);
  else
    map_range_kernel<float><<<(unsigned)blocks, 256, 0, st>>>(static_cast<const float*>(rho), n, out);
  return cudaGetLastError();
}

cudaError_t step_prepare(const StepForm& v) { return pick(v, Prepare{}); }

cudaError_t launch_step(const StepParams& p, const StepForm& v, int cells, int grid, cudaStream_t st) {
  if (p.n_det < 1 || p.n_det % v.dets_per_pass || cells > kStepCells + 32 || p.nterms < 1 ||
      (p.amp_power > 0) != v.amp)
    return cudaErrorInvalidValue;
  if (grid <= 0) return cudaSuccess;
  return pick(v, Launch{p, cells, grid, st});
}

cudaError_t launch_step_tiles(const StepTileParams& p, cudaStream_t st) {
  const int threads = 128;
  const int64_t total = (int64_t)p.a.Bpad * ((p.a.n_tiles + kAnchorRun - 1) / kAnchorRun);
  if (total == 0) return cudaSuccess;
  step_tile_kernel<<<(unsigned)((total + threads - 1) / threads), threads, 0, st>>>(p);
  return cudaGetLastError();
}

}  // namespace tcw
