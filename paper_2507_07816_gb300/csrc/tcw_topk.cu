// tcw_topk.cu -- exact per-sky top-k of Psi (the selection step after Eq. 4).
//
// Order: Psi descending, then caller template index ascending.  Each candidate
// is a unique 64-bit key (order-preserving Psi bits << 32 | ~caller index).  A
// radix select narrows a row down to at most kTopkCand candidates that hold the
// k best, most often by Psi alone; those are gathered and bitonic-sorted in
// shared memory.  One CTA per sky row.
#include "tcw_internal.cuh"

namespace tcw {
namespace {

constexpr int kTopkThreads = 1024;
constexpr int kTopkCand = 2048;   // candidates sorted at the end (k <= 1024)
constexpr int kTopkBits = 11, kTopkBins = 1 << kTopkBits;
static_assert(kTopkBins == 2 * kTopkThreads, "two bins per thread");

__device__ __forceinline__ uint32_t ord_bits(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unord_bits(uint32_t o) {
  const uint32_t u = (o & 0x80000000u) ? (o & 0x7fffffffu) : ~o;
  return __uint_as_float(u);
}

// Bound by latency (a row's reads come from L2) and, where many values share a
// digit, by shared-memory atomics on one word: a warp's lanes with the first
// lane's digit are counted by one addition.  A pass over the row costs more than
// sorting 2048 candidates, so the passes stop there, and the caller indices are
// read for the candidates only (8 passes over both before): 64 rows of 2.6e5
// templates 750 -> 185 us.
__global__ void __launch_bounds__(kTopkThreads) topk_kernel(const float* psi, int Bpad, int B, int k,
                                                            const int32_t* bank_perm,
                                                            const int32_t* sky_perm, float* psi_out,
                                                            int64_t* idx_out) {
  __shared__ unsigned hist[kTopkBins];
  __shared__ unsigned long long sel[kTopkCand];
  __shared__ unsigned s_warp[kTopkThreads / 32];
  __shared__ unsigned s_digit, s_above, s_in, s_count;
  const int row = blockIdx.x;
  const float* x = psi + (int64_t)row * Bpad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr unsigned kAll = 0xffffffffu;
  auto key_of = [&](int b) {
    return (unsigned long long)ord_bits(x[b]) << 32 | (uint32_t)(~(uint32_t)bank_perm[b]);
  };

  // keys >= prefix under mask: `above` of them beyond the prefix, `in` with it
  unsigned long long prefix = 0, mask = 0;
  unsigned above = 0, in = (unsigned)B;
  for (int pass = 0; pass < 6 && above + in > (unsigned)kTopkCand; ++pass) {
    // digits of 11, 11 and 10 bits of Psi, then of the caller index
    const bool low = pass >= 3;
    const int p3 = low ? pass - 3 : pass;
    const int shift = p3 == 0 ? 21 : p3 == 1 ? 10 : 0;
    const unsigned width = p3 == 2 ? (1u << 10) - 1u : (1u << kTopkBits) - 1u;
    hist[tid] = 0;
    hist[tid + kTopkThreads] = 0;
    __syncthreads();
    const uint32_t hi = (uint32_t)(prefix >> 32), hi_mask = (uint32_t)(mask >> 32);
#pragma unroll 4
    for (int b0 = warp * 32; b0 < B; b0 += kTopkThreads) {
      const int b = b0 + lane;
      const uint32_t u = b < B ? ord_bits(x[b]) : 0u;
      bool on = b < B && (u & hi_mask) == hi;
      uint32_t v = u;
      if (low && on) {
        v = ~(uint32_t)bank_perm[b];
        on = (v & (uint32_t)mask) == (uint32_t)prefix;
      }
      const unsigned digit = (v >> shift) & width;
      const unsigned active = __ballot_sync(kAll, on);
      if (!active) continue;
      const int first = __ffs(active) - 1;
      const unsigned d0 = __shfl_sync(kAll, digit, first);
      const unsigned same = __ballot_sync(kAll, on && digit == d0);
      if (lane == first)
        atomicAdd(&hist[d0], (unsigned)__popc(same));
      else if (on && digit != d0)
        atomicAdd(&hist[digit], 1u);
    }
    __syncthreads();
    // the digit at which the count from the top reaches k - above
    const unsigned rem = (unsigned)k - above;
    const int top = kTopkBins - 1 - 2 * tid;   // this thread's bins: top, top - 1
    const unsigned c0 = hist[top], c1 = hist[top - 1];
    unsigned sum = c0 + c1;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned o = __shfl_up_sync(kAll, sum, off);
      if (lane >= off) sum += o;
    }
    if (lane == 31) s_warp[warp] = sum;
    __syncthreads();
    unsigned before = lane < warp ? s_warp[lane] : 0u;
    before = __reduce_add_sync(kAll, before) + sum - c0 - c1;
    if (before < rem && before + c0 >= rem) {
      s_digit = (unsigned)top;
      s_above = before;
      s_in = c0;
    } else if (before + c0 < rem && before + c0 + c1 >= rem) {
      s_digit = (unsigned)top - 1u;
      s_above = before + c0;
      s_in = c1;
    }
    __syncthreads();
    prefix |= (unsigned long long)s_digit << (shift + (low ? 0 : 32));
    mask |= (unsigned long long)width << (shift + (low ? 0 : 32));
    above += s_above;
    in = s_in;
    if (in == (unsigned)k - above) break;   // exactly k keys from the prefix on
  }
  if (tid == 0) s_count = 0;
  const int found = (int)(above + in);   // k <= found <= kTopkCand
  int room = 2;
  while (room < found) room <<= 1;
  for (int i = tid; i < room; i += kTopkThreads) sel[i] = 0ull;
  __syncthreads();
  const uint32_t hi = (uint32_t)(prefix >> 32), hi_mask = (uint32_t)(mask >> 32);
#pragma unroll 4
  for (int b = tid; b < B; b += kTopkThreads) {
    if ((ord_bits(x[b]) & hi_mask) < hi) continue;
    const unsigned long long key = key_of(b);
    if ((key & mask) >= prefix) {
      const unsigned pos = atomicAdd(&s_count, 1u);
      if (pos < (unsigned)kTopkCand) sel[pos] = key;
    }
  }
  __syncthreads();
  // bitonic sort, descending
  for (int size = 2; size <= room; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = tid; i < room / 2; i += kTopkThreads) {
        const int a = 2 * i - (i & (stride - 1)), c = a + stride;   // pairs (a, a ^ stride), a the lower
        const bool desc = (a & size) == 0;
        const unsigned long long va = sel[a], vc = sel[c];
        if (desc ? (va < vc) : (va > vc)) {
          sel[a] = vc;
          sel[c] = va;
        }
      }
      __syncthreads();
    }
  }
  const int64_t out_row = sky_perm[row];
  for (int i = tid; i < k; i += kTopkThreads) {
    const unsigned long long key = sel[i];
    psi_out[out_row * k + i] = unord_bits((uint32_t)(key >> 32));
    idx_out[out_row * k + i] = (int64_t)(~(uint32_t)(key & 0xffffffffull));
  }
}

}  // namespace

cudaError_t launch_topk(const float* psi, int Bpad, int B, int S, int k, const int32_t* bank_perm,
                        const int32_t* sky_perm, float* psi_out, int64_t* idx_out,
                        cudaStream_t st) {
  topk_kernel<<<S, kTopkThreads, 0, st>>>(psi, Bpad, B, k, bank_perm, sky_perm, psi_out, idx_out);
  return cudaGetLastError();
}

}  // namespace tcw
