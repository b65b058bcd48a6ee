// tcw_step.cu -- the exhaustive search as step functions over the sorted sky
// (tcw_step.cuh): Doppler rows, the search kernel, the map's largest value.
#include <algorithm>
#include <climits>
#include <cmath>

#include "tcw_step.cuh"

namespace tcw {
namespace {

constexpr int kStepThreads = 1024;
constexpr int kStepWarps = kStepThreads / 32;
// Segments between two normalisations of the difference cells: a cell's low
// word takes at most 8 bin differences of at most 2^16 per (segment, detector),
// 2 detectors, so 2^11 segments stay within 2^31.
constexpr int kStepCarry = 2048;
// fp32-pair track series: coefficients 1..4 as pairs, 5..kFastTerms as fp32
constexpr int kFastTerms = 9;
constexpr int kFastWords = 8 + (kFastTerms - 4);   // fp32 words of a template's coefficients
constexpr int kCoefBytes = kMaxSeriesTerms * 8;    // per template, either form
static_assert(kFastWords * 4 <= kCoefBytes, "coefficients fit");

// ---------------------------------------------------------------------------
// Sky order of one (pass, chunk): positions sorted by the grid value at the
// pass's middle segment (ties by index), by counting.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int doppler_q(const double* v, const double* n, double inv_q) {
  const double dD = (v[0] * n[0] + v[1] * n[1] + v[2] * n[2]) / kLightSpeed;   // Eq. 2
  return (int32_t)fmax(fmin(floor(dD * inv_q), 2147483647.0), -2147483648.0);
}

__global__ void __launch_bounds__(kStepMaxChunk) step_order_kernel(StepRowsParams p) {
  __shared__ int s_q[kStepMaxChunk];
  const int pass = blockIdx.x, c = blockIdx.y, i = threadIdx.x;
  const int per = p.n_det / p.dets_per_pass;
  const int e = pass / per, d = p.dets_per_pass == 1 ? pass % per : 0;
  const int js = e * p.pass_seg, je = min(p.n_seg, js + p.pass_seg);
  const double* v = p.vel + ((int64_t)d * p.n_seg + (js + je - 1) / 2) * 3;
  const int rows = min(p.chunk, p.S - c * p.chunk);
  if (i < rows) s_q[i] = doppler_q(v, p.nhat + (int64_t)(c * p.chunk + i) * 3, p.inv_q);
  __syncthreads();
  if (i >= rows) return;
  const int q = s_q[i];
  int rank = 0;
  for (int k = 0; k < rows; ++k) rank += s_q[k] < q || (s_q[k] == q && k < i);
  int16_t* o = p.order + ((int64_t)pass * p.n_chunks + c) * p.cpad;
  o[rank] = (int16_t)i;
  if (rank == rows - 1)
    for (int k = rows; k < p.cpad; ++k) o[k] = (int16_t)i;
}

// ---------------------------------------------------------------------------
// Doppler rows (Eq. 2): one CTA per (segment, detector, chunk), one thread per
// block of 8 skies.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) step_rows_kernel(StepRowsParams p) {
  __shared__ int s_max[4], s_min[4];
  const int d = blockIdx.x % p.n_det, j = blockIdx.x / p.n_det, c = blockIdx.y;
  const int nb = p.cpad / kStepBlock;
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
  // inclusive prefix maximum, exclusive suffix minimum over the blocks
  int U = mx, L = mn;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, U, off), b = __shfl_down_sync(0xffffffffu, L, off);
    if (lane >= off) U = max(U, a);
    if (lane + off < 32) L = min(L, b);
  }
  if (lane == 31) s_max[warp] = U;
  if (lane == 0) s_min[warp] = L;
  int Ln = __shfl_down_sync(0xffffffffu, L, 1);
  if (lane == 31) Ln = INT_MAX;
  __syncthreads();
  int qmin = INT_MAX, qmax = INT_MIN;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    if (w < warp) U = max(U, s_max[w]);
    if (w > warp) Ln = min(Ln, s_min[w]);
    qmin = min(qmin, s_min[w]);
    qmax = max(qmax, s_max[w]);
  }
  int4* m = p.meta + row * step_meta(p.cpad);
  if (g < nb) reinterpret_cast<int2*>(m + kStepHead)[g] = make_int2(U, Ln);
  if (g == 0) {
    // t_j - t_a from the anchor time of the tile (tile_anchor_time of tcw_persist.cuh)
    const int t0 = j >> p.tile_shift << p.tile_shift;
    const double ta = fmax(p.t_mid[t0 + (min(1 << p.tile_shift, p.n_seg - t0) - 1) / 2], p.T0);
    const double tj = p.t_mid[j], dt = tj - ta;
    const float dth = tj >= p.T0 ? (float)dt : NAN;
    m[0] = make_int4(qmin, qmax, __float_as_int(dth), __float_as_int((float)(dt - (double)dth)));
    const float w = p.weights[dj];
    const float span = (float)((double)qmax - (double)qmin);
    m[1] = make_int4(__float_as_int(span > 0.f ? (float)nb / span : 0.f), __float_as_int(w), 0, 0);
    longlong2 wi;
    wi.x = __double2ll_rn((double)w * p.w1_scale);
    wi.y = __double2ll_rn((double)w * (double)w * p.w2_scale);
    *reinterpret_cast<longlong2*>(m + 2) = wi;
  }
}

template <typename T>
__global__ void absmax_kernel(const T* x, int64_t n, unsigned* out) {
  unsigned m = 0;
  constexpr int V = 16 / sizeof(T);
  const int64_t nv = n / V, stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  auto take = [&](T v) {
    float f;
    if constexpr (sizeof(T) == 2) f = __half2float(v);
    else f = v;
    m = max(m, __float_as_uint(f) & 0x7fffffffu);
  };
  for (int64_t i = i0; i < nv; i += stride) {
    const int4 v = reinterpret_cast<const int4*>(x)[i];
    const T* e = reinterpret_cast<const T*>(&v);
#pragma unroll
    for (int k = 0; k < V; ++k) take(e[k]);
  }
  for (int64_t i = nv * V + i0; i < n; i += stride) take(x[i]);
  for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

// Shared memory of the search kernel for `cells` difference cells (templates x
// (row + 1)): two word planes, piece sums of the epilogue, track series
// coefficients, per-template sums.
struct StepLayout {
  size_t lo, part, coef, tsum, total;
  __host__ __device__ constexpr explicit StepLayout(int cells)
      : lo((size_t)cells * 4),
        part(((size_t)cells * 8 + 15) & ~(size_t)15),
        coef(part + (size_t)3 * kStepThreads * 8),
        tsum(coef + (size_t)kCoefBytes * 32),
        total(tsum + (size_t)32 * 4 * 8) {}
};

// A value of the lookup at bin K (the caller checks the band).
// VK 0: fp32 power, 1: fp16 power, 2: number count and / or two-bin sums.
template <int VK>
__device__ __forceinline__ float step_value(const StepParams& p, const StepEvent& ev, int64_t row, int K) {
  if constexpr (VK == 0) {
    return __ldg(static_cast<const float*>(ev.rho) + row * p.n_bin + K);
  } else if constexpr (VK == 1) {
    return __half2float(__ldg(static_cast<const __half*>(ev.rho) + row * p.n_bin + K));
  } else {
    const int more = p.track_bins == 2 ? 1 : 0;
    float v = 0.f;
    if (ev.bits) {
      const uint32_t* r = ev.bits + row * ev.bit_pitch;
      for (int i = 0; i <= more; ++i) v += (float)((__ldg(r + ((K + i) >> 5)) >> ((K + i) & 31)) & 1u);
    } else {
      for (int i = 0; i <= more; ++i) {
        const int64_t o = row * p.n_bin + K + i;
        v += p.map_half ? __half2float(__ldg(static_cast<const __half*>(ev.rho) + o))
                        : __ldg(static_cast<const float*>(ev.rho) + o);
      }
    }
    return v;
  }
}

// v * s rounded to the fixed-point grid: hi + lo 2^-16 with |lo| <= 2^15
// (|v s| < 2^22).  The product is never rounded before the grid.
__device__ __forceinline__ void to_fixed(float v, float s, int& hi, int& lo) {
  const float t = fmaf(v, s, kMagic);
  const float r = fmaf(v, s, -(t - kMagic));
  hi = __float_as_int(t) - kMagicBits;
  lo = __float_as_int(fmaf(r, 65536.0f, kMagic)) - kMagicBits;
}

// An fp32 pair hi + lo.
struct Pair {
  float h, l;
};
__device__ __forceinline__ Pair pair_of(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ Pair pair_mul(Pair a, Pair b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  return {p, fmaf(a.l, b.h, e)};
}
// c + a b for |c| >= |a b|
__device__ __forceinline__ Pair pair_fma(Pair a, Pair b, Pair c) {
  const Pair m = pair_mul(a, b);
  const float h = c.h + m.h;
  return {h, (m.h - (h - c.h)) + (c.l + m.l)};
}
// round((h + l) 2^e) with s1 = 2^(e - 22), s2 = 2^e
__device__ __forceinline__ long long pair_fixed(Pair a, float s1, float s2) {
  const int hi = __float2int_rn(a.h * s1);
  const float r = fmaf(a.h, s1, -(float)hi);
  return (long long)hi * 4194304 + __float2int_rn(fmaf(r, 4194304.0f, a.l * s2));
}

// The search kernel: one CTA per SM takes (sky chunk, template block) items from
// a counter; the difference cells of a block (16 or 32 templates x up to 1024
// skies, two words each) live in shared memory, one column per template.  A
// lane owns one (template, segment) of its warp's turn: the track, the first
// sky's bin, and for each bin boundary inside the chunk's Doppler range one
// search in the row and one difference.  It is bound by the latency and the
// number of its instructions (nothing is saturated), so as many warps as fit
// (32; 24 and 16 measured slower).  2e5 templates x 1024 skies x 2 detectors x
// 1e4 segments: 644 ms by the group kernel -> 276 ms; one sky: 204 -> 50 ms.
template <int VK, int DP, bool FAST>
__global__ void __launch_bounds__(kStepThreads, 1) step_kernel(StepParams p, int cells) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  __shared__ unsigned s_edge;   // templates with band-edge weight steps (bit per template)
  const StepLayout L(cells);
  int* const chi = reinterpret_cast<int*>(smem);
  int* const clo = reinterpret_cast<int*>(smem + L.lo);
  long long* const part = reinterpret_cast<long long*>(smem + L.part);
  double* const coef = reinterpret_cast<double*>(smem + L.coef);
  float* const fcoef = reinterpret_cast<float*>(smem + L.coef);   // [word][32]: c1 hi lo .. c4 hi lo, c5 ..
  unsigned long long* const tsum = reinterpret_cast<unsigned long long*>(smem + L.tsum);   // X0, W1, W2 [32]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float fmin_f = (float)p.f_min, inv_df_f = (float)(1.0 / p.df);
  const bool two = VK == 2 && p.track_bins == 2;
  const int more_bins = two ? 1 : 0;
  const int n_bin = (int)p.n_bin;
  longlong2* const edge = p.edge + (int64_t)blockIdx.x * (2 * kStepCells + 32);
  longlong2* const edge_acc = edge + kStepCells + 32;
  long long* const acc = p.acc + (int64_t)blockIdx.x * kStepCells;
  unsigned long long ngen = 0;

  for (int i = tid; i < cells; i += kStepThreads) chi[i] = clo[i] = 0;

  while (true) {
    __syncthreads();
    if (tid == 0) {
      s_item = (int)atomicAdd(p.next, 1u);
      s_edge = 0;
    }
    if (tid < 32 * 4) tsum[tid] = 0;
    __syncthreads();
    if (s_item >= p.n_items) break;
    int4 item;
    if (p.items) {
      item = p.items[s_item];
    } else {
      const int blocks = p.events[0].Bpad >> p.events[0].log_t, g0 = s_item / p.n_chunks * p.bank_chunk;
      item = make_int4(0, s_item % p.n_chunks, g0 << p.events[0].log_t, min(p.bank_chunk, blocks - g0));
    }
    const StepEvent& ev = p.events[item.x];
    const int log_t = ev.log_t, T = 1 << log_t, cpad = ev.cpad;
    const int n_seg = ev.n_seg;
    const int lt = lane & (T - 1), ls = lane >> log_t, lps = 32 >> log_t;
    const int meta_n = step_meta(cpad);
    const int64_t row0 = (int64_t)item.y * n_seg * p.n_det;
    const float xs = ev.x_scale;
    // epilogue roles: template t, piece pc of the positions
    const int t = tid & (T - 1), pc = tid >> log_t, pieces = kStepThreads >> log_t;
    const int len = (cpad + pieces - 1) / pieces;
    const int p0 = min(cpad, pc * len), p1 = min(cpad, p0 + len);
    longlong2* const ecol = edge + (int64_t)t * (cpad + 1);

    for (int tb = 0; tb < item.w; ++tb) {
      const int b0 = item.z + tb * T, b = b0 + lt;
      if (tid < T) {
        // binomial coefficients C(r, k) of (1 + delta)^r, r = 1/(n - 1)
        const double r = 1.0 / (ev.nbr[b0 + tid] - 1.0);
        double c = 1.0;
        if constexpr (FAST) {
          for (int k = 1; k <= kFastTerms; ++k) {
            c = c * (r - (k - 1)) / k;
            if (k <= 4) {
              const Pair q = pair_of(c);
              fcoef[(2 * k - 2) * 32 + tid] = q.h;
              fcoef[(2 * k - 1) * 32 + tid] = q.l;
            } else {
              fcoef[(k + 3) * 32 + tid] = (float)c;
            }
          }
        } else {
          for (int k = 0; k < p.nterms; ++k) {
            coef[k * 32 + tid] = c;
            c = c * (r - k) / (k + 1);
          }
        }
      }
      __syncthreads();
      long long X0 = 0, W1 = 0, W2 = 0;
      for (int pass = 0; pass < ev.passes; ++pass) {
        const int per = p.n_det / DP;
        const int d0 = DP == 1 ? pass % per : 0;
        const int js = pass / per * ev.pass_seg, je = min(n_seg, js + ev.pass_seg);
        for (int jc = js; jc < je; jc += kStepCarry) {
          const int jce = min(je, jc + kStepCarry);
          for (int j0 = jc + (warp << p.sub_shift); j0 < jce; j0 += kStepWarps << p.sub_shift) {
            const int ti = j0 >> p.tile_shift;
            const double2 an = reinterpret_cast<const double2*>(ev.anchors)[(int64_t)b * ev.n_tiles + ti];
            // constants of (template, tile)
            Pair io, io1, qa;
            float fa = 0.f;
            int Ba = 0;
            long long E11 = 0, Q10 = 0;
            double ta = 0.0;
            if constexpr (FAST) {
              // h = 1/f = h_a (1 + g); c_K h - 1 = E_a + (1 + E_a) g + (K - K_a) df h_a (1 + g)
              // with c_a the bin centre nearest to f_a and E_a = c_a h_a - 1
              fa = __frcp_rn((float)an.x);
              Ba = __float2int_rn((fa - fmin_f) * inv_df_f);
              const double Qd = p.df * an.x;
              const double Ea = fma((double)Ba, Qd, fma(p.f_min, an.x, -1.0));
              io = pair_of(an.y);
              io1 = pair_of(fma(an.y, Ea, an.y));
              qa = pair_of(Qd);
              E11 = __double2ll_rn(ldexp(Ea, 19) * p.inv_q);
              Q10 = __double2ll_rn(ldexp(Qd, 18) * p.inv_q);
            } else {
              const int t0 = ti << p.tile_shift;
              ta = fmax(ev.t_mid[t0 + (min(1 << p.tile_shift, n_seg - t0) - 1) / 2], ev.T0);
            }
            const int jn = min(jce, j0 + (1 << p.sub_shift));
            for (int j = j0 + ls; j < jn; j += lps) {
              const int4* meta = ev.meta + (row0 + (int64_t)j * p.n_det + d0) * meta_n;
              int4 m0 = __ldg(meta);
              const float dth = __int_as_float(m0.z);
              if (!(dth == dth)) continue;   // before T0
              // track (Eq. 1): f, the nearest bin `base` of the unshifted track, and the thresholds
              // theta_n = c_K / f - 1 between the bins K = base + n and K + 1 (two-bin lookups: the
              // bin centres f_min + (K + 1) df in place of the edges)
              float f, h_f0 = 1.f;
              int base;
              long long A, B;   // FAST: theta_n = (A + B (2 n + 1 or 2)) >> 11 >> 8; else (A + n B) >> 8
              long long G = 0;
              if constexpr (FAST) {
                const Pair dt{dth, __int_as_float(m0.w)};
                const Pair dl = pair_mul(dt, io), dl1 = pair_mul(dt, io1);
                float s = fcoef[(kFastTerms + 3) * 32 + lt];
#pragma unroll
                for (int k = kFastTerms - 1; k >= 5; --k) s = fmaf(dl.h, s, fcoef[(k + 3) * 32 + lt]);
                Pair sp{fcoef[6 * 32 + lt], fmaf(dl.h, s, fcoef[7 * 32 + lt])};
#pragma unroll
                for (int k = 3; k >= 1; --k)
                  sp = pair_fma(dl, sp, {fcoef[(2 * k - 2) * 32 + lt], fcoef[(2 * k - 1) * 32 + lt]});
                const Pair g = pair_mul(dl, sp);
                const Pair gq = pair_mul(qa, g);
                f = fa * __frcp_rn(1.0f + g.h);
                h_f0 = 1.0f + g.h;
                const float sg = __int_as_float((p.q_exp + 8 + 127) << 23);   // 2^(q_exp + 8)
                G = pair_fixed(pair_mul(dl1, sp), sg * (1.0f / 4194304.0f), sg);
                B = Q10 + pair_fixed(gq, sg * (1.0f / 4096.0f), sg * 1024.0f);
                const float x = (f - fmin_f) * inv_df_f;
                base = __float2int_rn(x);
                A = E11 + 1024 + (long long)(2 * (base - Ba) + (two ? 2 : 1)) * B;
                G += 128;
              } else {
                const double delta = (ev.t_mid[j] - ta) * an.y;
                double R = coef[(p.nterms - 1) * 32 + lt];
#pragma unroll 4
                for (int k = p.nterms - 2; k >= 0; --k) R = fma(R, delta, coef[k * 32 + lt]);
                const double h = an.x * R;
                f = __frcp_rn((float)h);
                base = __float2int_rn((f - fmin_f) * inv_df_f);
                const double Q = p.df * h;
                const double A0 = fma((double)base + (two ? 1.0 : 0.5), Q, fma(p.f_min, h, -1.0));
                A = __double2ll_rn(A0 * (p.inv_q * 256.0)) + 128;
                B = __double2ll_rn(Q * (p.inv_q * 256.0));
                h_f0 = (float)(h * ev.f0[b]);
              }
              auto threshold = [&](int n) {
                long long v = FAST ? (((A + (long long)(2 * n) * B) >> 11) + G) >> 8 : (A + (long long)n * B) >> 8;
                v = v > 2147483647LL ? 2147483647LL : (v < -2147483647LL ? -2147483647LL : v);
                return (int)v;
              };
              float amp = 1.0f;
              if (p.amp_power > 0) {
                if constexpr (FAST) h_f0 *= (float)(an.x * ev.f0[b]);
                float rp = h_f0;
                for (int k = 1; k < p.amp_power; ++k) rp *= h_f0;
                amp = __frcp_rn(rp);
              }
              const float F = f * inv_df_f;
              const float x = (f - fmin_f) * inv_df_f;
              if (!(base >= -kMHi && base < n_bin - kMLo)) continue;
              const float y0 = x - (float)base - (two ? 1.0f : 0.5f), Fq = F * p.q;
#pragma unroll
              for (int dd = 0; dd < DP; ++dd) {
                if (dd > 0) {
                  meta += meta_n;
                  m0 = __ldg(meta);
                }
                const int qmin = m0.x, qmax = m0.y;
                const int4 m1 = __ldg(meta + 1);
                const float w = __int_as_float(m1.y) * amp;
                const float ws = w * xs;
                const int64_t rrow = (int64_t)(d0 + dd) * n_seg + j;
                // first threshold above the lowest sky: an estimate good to 1e-2 bins, then exact
                int n = (int)floorf(fmaf(Fq, (float)qmin, y0)) + 1;
                int th = threshold(n);
                if (th <= qmin) {
                  th = threshold(++n);
                } else {
                  const int tl = threshold(n - 1);
                  if (tl > qmin) {
                    --n;
                    th = tl;
                  }
                }
                int K = base + n;   // the lowest sky's bin
                const bool okK = K >= 0 && K + more_bins < n_bin;
                bool step = th <= qmax;
                bool okN = step && K + 1 >= 0 && K + 1 + more_bins < n_bin;
                const float v0 = okK ? step_value<VK>(p, ev, rrow, K) : 0.f;
                float vn = okN ? step_value<VK>(p, ev, rrow, K + 1) : 0.f;
                int h0 = 0, l0 = 0;
                to_fixed(v0, ws, h0, l0);
                X0 += (long long)h0 * 65536 + l0;
                if (okK) {
                  if (p.amp_power > 0) {
                    int wh, wl;
                    to_fixed(w, ev.w1_scale, wh, wl);
                    W1 += (long long)wh * 65536 + wl;
                    to_fixed(w, w * ev.w2_scale, wh, wl);
                    W2 += (long long)wh * 65536 + wl;
                  } else {
                    const longlong2 wi = *reinterpret_cast<const longlong2*>(meta + 2);
                    W1 += wi.x;
                    W2 += wi.y;
                  }
                }
                bool ok0 = okK, any_edge = !okK;
                for (int it = 0; it < kNThr && step; ++it) {
                  // the step from bin K to K + 1 at threshold th; the next one's power is fetched ahead
                  ++K;
                  const int th1 = threshold(++n);
                  const bool step1 = th1 <= qmax;
                  const bool okN1 = step1 && K + 1 >= 0 && K + 1 + more_bins < n_bin;
                  const float vn1 = okN1 ? step_value<VK>(p, ev, rrow, K + 1) : 0.f;
                  const bool ok1 = okN;
                  int h1, l1;
                  to_fixed(vn, ws, h1, l1);
                  const int dh = h1 - h0, dl = l1 - l0;
                  const int we = (int)ok1 - (int)ok0;   // weight step at a band edge
                  long long e1w = 0, e2w = 0;
                  if (we) {
                    any_edge = true;
                    if (p.amp_power > 0) {
                      int wh, wl;
                      to_fixed(w, ev.w1_scale, wh, wl);
                      e1w = we * ((long long)wh * 65536 + wl);
                      to_fixed(w, w * ev.w2_scale, wh, wl);
                      e2w = we * ((long long)wh * 65536 + wl);
                    } else {
                      const longlong2 wi = *reinterpret_cast<const longlong2*>(meta + 2);
                      e1w = we * wi.x;
                      e2w = we * wi.y;
                    }
                  }
                  auto place = [&](int pos, bool plus) {
                    const int cell = (pos << log_t) + lt;
                    atomicAdd(chi + cell, plus ? dh : -dh);
                    atomicAdd(clo + cell, plus ? dl : -dl);
                    if (we) {
                      unsigned long long* ec =
                          reinterpret_cast<unsigned long long*>(edge + (int64_t)lt * (cpad + 1) + pos);
                      atomicAdd(ec, (unsigned long long)(plus ? e1w : -e1w));
                      atomicAdd(ec + 1, (unsigned long long)(plus ? e2w : -e2w));
                    }
                  };
                  // the first block that reaches th, then every block until all later skies do
                  const int2* const blk = reinterpret_cast<const int2*>(meta + kStepHead);
                  int g = min((int)((float)((unsigned)th - (unsigned)qmin) * __int_as_float(m1.x)),
                              cpad / kStepBlock - 1);
                  int2 bk = __ldg(blk + g);
                  if (bk.x < th) {
                    do bk = __ldg(blk + ++g);
                    while (bk.x < th);
                  } else {
                    while (g > 0) {
                      const int2 pb = __ldg(blk + g - 1);
                      if (pb.x < th) break;
                      bk = pb;
                      --g;
                    }
                  }
                  const int4* qr = reinterpret_cast<const int4*>(
                      ev.q + (row0 + (int64_t)j * p.n_det + d0 + dd) * cpad);
                  unsigned below = 1;   // the sky before this block is below th
                  while (true) {
                    const int4 ua = __ldg(qr + 2 * g), ub = __ldg(qr + 2 * g + 1);
                    const unsigned m = (unsigned)(ua.x >= th) | (unsigned)(ua.y >= th) << 1 |
                                       (unsigned)(ua.z >= th) << 2 | (unsigned)(ua.w >= th) << 3 |
                                       (unsigned)(ub.x >= th) << 4 | (unsigned)(ub.y >= th) << 5 |
                                       (unsigned)(ub.z >= th) << 6 | (unsigned)(ub.w >= th) << 7;
                    unsigned tr = (m ^ (m << 1 | (below ^ 1u))) & 0xffu;
                    while (tr) {
                      const int bit = __ffs(tr) - 1;
                      place(kStepBlock * g + bit, (m >> bit) & 1u);
                      tr &= tr - 1;
                    }
                    below = (m >> 7) ^ 1u;
                    if (bk.y >= th) break;
                    bk = __ldg(blk + ++g);
                  }
                  if (below) place(kStepBlock * (g + 1), true);
                  h0 = h1;
                  l0 = l1;
                  ok0 = ok1;
                  th = th1;
                  step = step1;
                  okN = okN1;
                  vn = vn1;
                }
                if (any_edge) {
                  ++ngen;
                  atomicOr(&s_edge, 1u << lt);
                }
              }
            }
          }
          if (jce < je) {
            // carry the low words over before they can overflow
            __syncthreads();
            for (int i = tid; i < cells; i += kStepThreads) {
              const int l = clo[i];
              chi[i] += l >> 16;
              clo[i] = l & 0xffff;
            }
            __syncthreads();
          }
        }
        const bool last = pass == ev.passes - 1;
        if (last) {
          for (int off = T; off < 32; off <<= 1) {
            X0 += __shfl_xor_sync(0xffffffffu, X0, off);
            W1 += __shfl_xor_sync(0xffffffffu, W1, off);
            W2 += __shfl_xor_sync(0xffffffffu, W2, off);
          }
          if (ls == 0) {
            atomicAdd(tsum + lt, (unsigned long long)X0);
            atomicAdd(tsum + 32 + lt, (unsigned long long)W1);
            atomicAdd(tsum + 64 + lt, (unsigned long long)W2);
          }
        }
        __syncthreads();

        // ---- prefix sums of the pass over its positions ----
        const bool te = (s_edge >> t) & 1u;
        {
          long long sx = 0, s1 = 0, s2 = 0;
          for (int q = p0; q < p1; ++q) {
            const int c = (q << log_t) + t;
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
        if (tid < 3 * 32) {
          // exclusive scan over the pieces, one thread per (sum, template)
          const int k = tid >> 5, tt = tid & 31;
          if (tt < T) {
            long long run = last ? (long long)tsum[k * 32 + tt] : 0;
            for (int i = 0; i < pieces; ++i) {
              long long* const q = part + k * kStepThreads + (i << log_t) + tt;
              const long long v = *q;
              *q = run;
              run += v;
            }
          }
        }
        __syncthreads();
        {
          // Eq. 4: <s> = mq W1, sigma^2 = vq W2 (power: 1, 1; number count: q, q(1-q)),
          // both doubled for two-bin lookups
          const double nbins = two ? 2.0 : 1.0;
          const bool count = VK == 2 && p.nc_q > 0.0;
          const double mq = nbins * (count ? p.nc_q : 1.0);
          const float vq = (float)(nbins * (count ? p.nc_q * (1.0 - p.nc_q) : 1.0));
          const double m_units = mq * ev.w1_unit / ev.x_unit;   // mean of one W1 unit, in units of X
          const float x_unit = (float)ev.x_unit;
          const int64_t sky0 = (int64_t)item.y * ev.chunk;
          const int rows = min(ev.chunk, ev.S - (int)sky0);
          long long X = part[tid], w1 = part[kStepThreads + tid], w2 = part[2 * kStepThreads + tid];
          // skies without band-edge steps share W1, W2 and the mean
          long long mean = 0;
          float W2f = 0.f, rs = 0.f;
          auto moments = [&](long long a1, long long a2) {
            mean = __double2ll_rn((double)a1 * m_units);
            W2f = (float)((double)a2 * ev.w2_unit);
            rs = W2f > 0.f ? rsqrtf(vq * W2f) : 0.f;
          };
          if (last) moments(w1, w2);
          auto finish = [&](int sky, long long x, long long a1) {
            // the cells' high words wrap at 2^31, so x is known modulo 2^48
            const long long xs48 = (long long)((unsigned long long)x << 16) >> 16;
            const int64_t o = (sky0 + sky) * ev.Bpad + b0 + t;
            ev.psi[o] = W2f > 0.f ? (float)(xs48 - mean) * x_unit * rs : -INFINITY;
            if (ev.S_out) {
              ev.S_out[o] = (float)((double)xs48 * ev.x_unit);
              ev.W1_out[o] = (float)((double)a1 * ev.w1_unit);
              ev.W2_out[o] = W2f;
            }
          };
          const int16_t* order = ev.order ? ev.order + ((int64_t)pass * ev.n_chunks + item.y) * cpad : nullptr;
          for (int q = p0; q < p1; ++q) {
            const int c = (q << log_t) + t;
            X += (long long)chi[c] * 65536 + clo[c];
            chi[c] = clo[c] = 0;
            if (te) {
              const longlong2 v = __ldcg(ecol + q);
              __stcg(ecol + q, make_longlong2(0, 0));
              w1 += v.x;
              w2 += v.y;
            }
            if (q >= rows) continue;
            if (!order) {
              if (te) moments(w1, w2);
              finish(q, X, w1);
              continue;
            }
            // several passes: the sky's sums so far, kept by the sky's own index
            const int sky = order[q];
            const int a = (sky << log_t) + t;
            long long x = X;
            if (pass > 0) x += __ldcg(acc + a);
            if (te) {
              longlong2 v = __ldcg(edge_acc + a);
              v.x += w1;
              v.y += w2;
              if (last) {
                __stcg(edge_acc + a, make_longlong2(0, 0));
                moments(v.x, v.y);
                finish(sky, x, v.x);
              } else {
                __stcg(edge_acc + a, v);
                __stcg(acc + a, x);
              }
            } else if (last) {
              finish(sky, x, w1);
            } else {
              __stcg(acc + a, x);
            }
          }
        }
        // the cells past the last sky
        if (tid < T) {
          const int c = (cpad << log_t) + tid;
          chi[c] = clo[c] = 0;
          if ((s_edge >> tid) & 1u) __stcg(edge + (int64_t)tid * (cpad + 1) + cpad, make_longlong2(0, 0));
        }
        __syncthreads();
      }
      if (tid == 0) s_edge = 0;
      if (tid < 32 * 4) tsum[tid] = 0;
      __syncthreads();
    }
  }
  if (ngen) atomicAdd(p.n_general, ngen);
}

template <int VK, int DP, bool FAST>
cudaError_t set_smem() {
  constexpr int kDevices = 64;
  static bool done[kDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < kDevices && done[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(step_kernel<VK, DP, FAST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)StepLayout(kStepCells + 32).total);
  if (e == cudaSuccess && dev >= 0 && dev < kDevices) done[dev] = true;
  return e;
}

struct Prepare {
  template <int VK, int DP, bool FAST>
  cudaError_t run() const { return set_smem<VK, DP, FAST>(); }
};

struct Launch {
  const StepParams& p;
  int cells, grid;
  cudaStream_t st;
  template <int VK, int DP, bool FAST>
  cudaError_t run() const {
    cudaError_t e = set_smem<VK, DP, FAST>();
    if (e != cudaSuccess) return e;
    step_kernel<VK, DP, FAST><<<grid, kStepThreads, StepLayout(cells).total, st>>>(p, cells);
    return cudaGetLastError();
  }
};

template <int VK, int DP, typename F>
cudaError_t pick_fast(bool fast, const F& f) {
  return fast ? f.template run<VK, DP, true>() : f.template run<VK, DP, false>();
}
template <int DP, typename F>
cudaError_t pick_value(bool half, bool general, bool fast, const F& f) {
  if (general) return pick_fast<2, DP>(fast, f);
  return half ? pick_fast<1, DP>(fast, f) : pick_fast<0, DP>(fast, f);
}
template <typename F>
cudaError_t pick(int dp, bool half, bool general, bool fast, const F& f) {
  if (dp == 1) return pick_value<1>(half, general, fast, f);
  if (dp == 2) return pick_value<2>(half, general, fast, f);
  return cudaErrorInvalidValue;
}

}  // namespace

StepScales step_scales(double vmax, double w_min, double w_max, double a_ref, int64_t n) {
  StepScales s;
  if (!(vmax >= 0.0) || !(vmax < 1e30) || !(w_max > 0.0) || !(w_min > 0.0) || n < 1) return s;
  auto lg = [](double v) { return (int)std::ceil(std::log2(v)) + 1; };   // v < 2^lg, with a margin
  const int lm = lg(std::max(vmax, 1.0) * w_max), lw = lg(w_max), lw2 = lg(w_max * w_max), ln = lg((double)n);
  // the sum of a (template, sky) below 2^47 units and one value below 2^21 2^16 units
  s.x = std::min(46 - ln - lm, 36 - lm);
  s.w1 = std::min(36 - lw, 60 - ln - lw);
  s.w2 = std::min(36 - lw2, 60 - ln - lw2);
  // one unit at most 2^-20 of the smallest weighted unit power: a sum of n
  // rounded values is then off by about 0.3 sqrt(n) 2^-20 of it, 3e-7 of the
  // standard deviation sqrt(n) that Eq. 4 divides by
  const int need = 20 - (int)std::floor(std::log2(w_min * a_ref));
  s.ok = s.x >= need && std::abs(s.x) < 100 && std::abs(s.w1) < 100 && std::abs(s.w2) < 100 && need < 100;
  return s;
}

int step_fast_track(const double* t_mid, int64_t n_seg, double T0, int tile, double tau_min, double r_max,
                    double f_min, double df, int q_exp) {
  // fixed-point words: thresholds in units of 2^-(q_exp + 8), 2^-(q_exp + 18) for the bin spacing
  // df/f (f >= 64 bins for every lookup in the band)
  if (!(f_min >= 72.0 * df) || q_exp > 45 || q_exp < 20) return 0;
  double dmax = 0;
  for (int64_t j0 = 0; j0 < n_seg; j0 += tile) {
    const int64_t jn = std::min<int64_t>(tile, n_seg - j0);
    const double ta = std::max(t_mid[j0 + (jn - 1) / 2], T0);
    if (t_mid[j0 + jn - 1] < T0) continue;
    dmax = std::max(dmax, std::max(std::fabs(t_mid[j0 + jn - 1] - ta), std::fabs(std::max(t_mid[j0], T0) - ta)) /
                              (tau_min + (ta - T0)));
  }
  if (!(dmax <= 0.04) || !(r_max <= 1.0)) return 0;
  auto term = [&](int k) {   // |C(r, k)| delta^k
    double c = 1.0;
    for (int i = 0; i < k; ++i) c *= (r_max + i) / (i + 1) * dmax;
    return c;
  };
  // the fp32 terms' rounding and the first dropped term below a quarter unit of 2^-52
  return term(5) < std::ldexp(1.0, -30) && term(kFastTerms + 1) < std::ldexp(1.0, -54) ? 1 : 0;
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
  // middle: it displaces a sky by up to S drift / 2 places of a whole-sky list
  // sorted at the middle.  Places out of order cost difference steps of their
  // own (1.2 per boundary at a displacement of 3, 4.5 at 10: emulated on
  // Fibonacci and random lists), a pass costs one fold of the cells.
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
  const int64_t L = ((n_seg + runs - 1) / runs + tile - 1) / tile * tile;
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

cudaError_t launch_absmax(const void* rho, bool half, int64_t n, unsigned* out, cudaStream_t st) {
  const int64_t blocks = std::min<int64_t>((n + 8191) / 8192, 152 * 16);
  if (half)
    absmax_kernel<__half><<<(unsigned)blocks, 256, 0, st>>>(static_cast<const __half*>(rho), n, out);
  else
    absmax_kernel<float><<<(unsigned)blocks, 256, 0, st>>>(static_cast<const float*>(rho), n, out);
  return cudaGetLastError();
}

cudaError_t step_prepare(int dets_per_pass, bool half, bool general, bool fast) {
  return pick(dets_per_pass, half, general, fast, Prepare{});
}

cudaError_t launch_step(const StepParams& p, int dets_per_pass, bool half, bool general, bool fast, int cells,
                        int grid, cudaStream_t st) {
  if (p.n_det < 1 || p.n_det % dets_per_pass || cells > kStepCells + 32 || (!fast && p.nterms < 1))
    return cudaErrorInvalidValue;
  if (grid <= 0) return cudaSuccess;
  return pick(dets_per_pass, half, general, fast, Launch{p, cells, grid, st});
}

}  // namespace tcw
