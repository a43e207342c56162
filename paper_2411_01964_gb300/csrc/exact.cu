// exact.cu -- the exact squarefree test behind stragglers and point queries.
//
// Algorithm 2 (Sec. 3) only reads the sieve.  Where n - 2^k falls below a
// tile's look-back window (a "straggler"), or for a single point n, the flag
// is decided directly, exactly and without floating point:
//   s (odd, >= 1) is squarefree  <=>  no prime p with p^3 <= s has p^2 | s,
//   and the cofactor r = s / prod{p | s : p^3 <= s} is not a perfect square.
// (After removing every prime factor p with p^3 <= s, r <= s has only prime
// factors q with q^3 > s >= r, so r is 1, a prime, a product of two distinct
// primes, or q^2; only the last is not squarefree.)  Divisibility by p uses the
// Granlund-Montgomery (1994, Sec. 9) test with p^-1 mod 2^64, and the exact
// quotient s/p is s * p^-1 mod 2^64.  One warp tests one s, lanes striding the
// prime table; the warp stops at the first p with p^2 | s.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "strike.h"
#include "sv_internal.h"

namespace sv {

// Warp-cooperative: is the odd number s >= 1 squarefree?  All 32 lanes call
// it with the same s and get the same answer.
__device__ bool warp_squarefree(uint64_t s, const PrimeTab &pt) {
  const uint32_t lane = threadIdx.x & 31u;
  if (s < 9) return true;  // 1, 3, 5, 7
  uint64_t r = s;
  for (uint32_t base = 0; base < pt.n_div; base += 32) {
    const uint32_t i = base + lane;
    bool in = false, div = false, sq = false;
    uint64_t inv = 0;
    if (i < pt.n_div) {
      const uint64_t p = pt.p[i];
      in = p * p * p <= s;  // p < 2^21: no overflow
      if (in) {
        inv = pt.inv[i];
        const uint64_t lim = pt.lim[i];
        const uint64_t t = s * inv;  // s / p when p | s
        if (t <= lim) {
          div = true;
          sq = (t * inv) <= lim;  // p | s/p
        }
      }
    }
    if (__any_sync(0xFFFFFFFFu, sq)) return false;
    uint32_t m = __ballot_sync(0xFFFFFFFFu, div);
    while (m) {
      const int src = __ffs(m) - 1;
      m &= m - 1;
      r *= __shfl_sync(0xFFFFFFFFu, inv, src);  // exact division by that prime
    }
    if (!__any_sync(0xFFFFFFFFu, in)) break;  // primes ascend: no lane left with p^3 <= s
  }
  if (r == 1) return true;
  const uint64_t x = isqrt_u64(r);
  return x * x != r;
}

// mink continued from k0 for odd n (warp-cooperative); 255 if none.
__device__ uint32_t warp_min_k_from(uint64_t n, uint32_t k0, const PrimeTab &pt) {
  for (uint32_t k = k0; k < 63 && (1ull << k) < n; ++k)
    if (warp_squarefree(n - (1ull << k), pt)) return k;
  return kFailK;
}

__global__ void __launch_bounds__(256) straggler_kernel(StragArgs a) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t gw = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  unsigned long long cnt = a.hdr->strag_count;
  if (cnt > a.strag_cap) cnt = a.strag_cap;
  for (uint64_t e = gw; e < cnt; e += nw) {
    const Straggler st = a.strag[e];
    const uint32_t k = warp_min_k_from(st.n, st.k0, a.pt);
    if (lane == 0) {
      const ReqDesc &R = a.reqs[st.req];
      ResultSlot *slot = &a.slots[R.slot];
      if (k != kFailK) {
        atomicAdd(&slot->hist[k], 1ull);
        atomicMin(&slot->first_n[k], (unsigned long long)st.n);
        if (k >= a.rec_t) {
          if (a.stage_n) {
            // ordered lists: join the staged entries of the tile holding n
            const uint64_t t = tile_index((((st.n - 1) >> 1) >> 5) - (uint64_t)R.w0, a.tw, a.tw_inv);
            if (t < R.n_tiles) {
              const uint32_t gt = R.tile_base + (uint32_t)t;
              const uint32_t e = atomicAdd(&a.stage_cnt[gt], 1u);
              if (e < a.stage_cap) {
                a.stage_n[(size_t)gt * kStageCap + e] = st.n;
                a.stage_k[(size_t)gt * kStageCap + e] = (uint8_t)k;
              } else {
                atomicOr(&a.hdr->status, kStListStage);
              }
            } else {
              atomicOr(&a.hdr->status, kStBadTile);
            }
          } else {
            const unsigned long long idx = atomicAdd(&slot->list_count, 1ull);
            if (idx < R.list_cap) {
              a.list_n[R.list_off + idx] = st.n;
              a.list_k[R.list_off + idx] = (uint8_t)k;
            }
          }
        }
      } else {
        const unsigned long long idx = atomicAdd(&slot->fail_count, 1ull);
        if (idx < R.fail_cap) a.fail_n[R.fail_off + idx] = st.n;
      }
      if (R.per_n_k) R.per_n_k[(st.n - R.nlo) >> 1] = (uint8_t)k;
    }
  }
}

cudaError_t launch_stragglers(const StragArgs &a, uint32_t grid, cudaStream_t st) {
  straggler_kernel<<<grid, 256, 0, st>>>(a);
  return cudaGetLastError();
}

// ---- point queries -------------------------------------------------------------
// Both kernels rule a prime p out with 32-bit arithmetic.  With s = s1 2^32 + s0
// and r = 2^32 mod p, v = s1 r + s0 is s modulo p; if p divides it, v = p k with
// k <= s1 + (2^32 - 1)/p < 2^32, so that k is the low word of v times the low
// word of p^-1:
//   p | s  =>  (s1 r + s0) p^-1 mod 2^32 <= s1 + floor(2^32 / p) + 1,
// two multiplies, an addition and a compare.  Other primes pass with a chance
// of about 1/p + s1/2^32; who passes is decided by the whole 64-bit test.  From
// 2^52 on, where s1 lets too many pass, the high word of t = s p^-1 mod 2^64 is
// compared instead (p | s means t <= lim, hence t_hi <= lim_hi).
// Primes somewhat past the cube root of s may be tested too: dividing one out
// leaves r = 1, a prime, or (r = p^2) finds p^2 | s, so the test stays exact.
// The 32-bit test's constants lie side by side, one 16-byte load per prime
// (PrimeTab::word): its multiplies, at a quarter of the logic rate, are to be
// what bounds the kernels, not addresses and loads.
constexpr uint64_t kShortTest = 1ull << 52;
__device__ __forceinline__ bool maybe_divides_short(uint64_t s, const PrimeWord &w) {
  const uint32_t s0 = (uint32_t)s, s1 = (uint32_t)(s >> 32);
  return (s1 * w.r + s0) * w.inv <= s1 + (w.lim + 1u);
}
__device__ __forceinline__ bool maybe_divides_long(uint64_t s, uint64_t inv, uint32_t lim_hi) {
  const uint32_t s0 = (uint32_t)s, s1 = (uint32_t)(s >> 32), i0 = (uint32_t)inv, i1 = (uint32_t)(inv >> 32);
  return __umulhi(s0, i0) + s0 * i1 + s1 * i0 <= lim_hi;
}
// Which of the K values may be divisible by prime i (below the padded table's end).
template <bool SHORT, int K>
__device__ __forceinline__ bool any_may_divide(const PrimeTab &pt, uint32_t i, const PrimeWord &w, const uint64_t (&s)[K]) {
  bool any = false;
  if (SHORT) {
#pragma unroll
    for (int j = 0; j < K; ++j) any |= maybe_divides_short(s[j], w);
  } else {
    const uint64_t inv = i < pt.n_div ? pt.inv[i] : 1ull;
#pragma unroll
    for (int j = 0; j < K; ++j) any |= maybe_divides_long(s[j], inv, w.lim);
  }
  return any;
}

// The table of the 32-bit test, padded by words that divide next to nothing (p
// = 2^32 - 1 lies above every cube root).
__global__ void prime_words_kernel(const uint32_t *p, const uint64_t *inv, uint32_t n_div, uint32_t n_out, PrimeWord *out) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_out) return;
  PrimeWord w{0u, 1u, 0u, 0xFFFFFFFFu};
  if (i < n_div) {
    const uint32_t q = (uint32_t)((1ull << 32) / p[i]);
    w = PrimeWord{0u - p[i] * q, (uint32_t)inv[i], q, p[i]};
  }
  out[i] = w;
}
cudaError_t launch_prime_words(const uint32_t *p, const uint64_t *inv, uint32_t n_div, PrimeWord *out, cudaStream_t st) {
  const uint32_t n = prime_words(n_div);
  prime_words_kernel<<<(n + 255) / 256, 256, 0, st>>>(p, inv, n_div, n, out);
  return cudaGetLastError();
}

// p^3 <= x for a word's prime (p < 2^21: no overflow; the padding's is above)
__device__ __forceinline__ bool cube_le(uint32_t p, uint64_t x) { return p < (1u << 21) && (uint64_t)p * p * p <= x; }

// r = s less its prime divisors up to the cube root: squarefree unless r is a
// square above 1 (an odd square is 1 modulo 8)
__device__ __forceinline__ bool cofactor_squarefree(uint64_t r) {
  if (r == 1 || (r & 7u) != 1) return true;
  const uint64_t x = isqrt_u64(r);
  return x * x != r;
}

constexpr uint32_t kMaxDivisors = 16;  // a product of 16 odd primes exceeds 2^62

// A block per point, its threads striding the primes (U per thread and step,
// their loads in flight together), and K exponents at a time: with few points,
// so that one pass over the primes mostly suffices.  A point below `small`
// needs few primes, and the block's barriers would be most of its time: the
// warps of the first blocks take those, one each.
template <int K, int U>
__global__ void __launch_bounds__(1024) points_block_kernel(PrimeTab pt, const uint64_t *pts, uint64_t count,
                                                            uint64_t small, uint8_t *out) {
  __shared__ uint32_t bad, n_div[K];   // bad: bit j, p^2 divides the j-th value
  __shared__ uint64_t div_inv[K][kMaxDivisors];
  __shared__ uint32_t found;
  __shared__ uint64_t n_s;
  const uint32_t tid = threadIdx.x, T = blockDim.x;
  const uint64_t e = blockIdx.x;    // a block per point
  if (tid == 0) n_s = pts[e];       // (perhaps in host memory: read once)
  {
    const uint64_t ew = e * (T >> 5) + (tid >> 5);
    const uint64_t n = ew < count ? pts[ew] : ~0ull;
    if (n < small) {
      const uint32_t k = n >= 3 && (n & 1ull) ? warp_min_k_from(n, 1, pt) : 0u;
      if ((tid & 31u) == 0) out[ew] = (uint8_t)k;
    }
  }
  __syncthreads();
  const uint64_t n = n_s;
  if (n < small) return;
  uint32_t k = 0;
  {
    if (n & 1ull) {
      for (uint32_t k0 = 1;; k0 += K) {
        __syncthreads();  // the previous round's results have been read
        if (tid == 0) {
          bad = 0;
          found = k0 < 63 && (1ull << k0) < n ? 0u : (uint32_t)kFailK;
        }
        if (tid < K) n_div[tid] = 0;
        __syncthreads();
        if (found) break;  // no exponent left
        uint64_t s[K];
#pragma unroll
        for (int j = 0; j < K; ++j) {
          const uint32_t kj = k0 + (uint32_t)j;
          s[j] = kj < 63 && (1ull << kj) < n ? n - (1ull << kj) : 1ull;  // (1: never the answer, see below)
        }
        auto walk = [&](auto short_test) {
          constexpr bool kShort = decltype(short_test)::value;
          for (uint32_t base = tid; base < pt.n_div; base += U * T) {  // (the table is padded by a step)
            PrimeWord w[U];
#pragma unroll
            for (int u = 0; u < U; ++u) w[u] = pt.word[base + (uint32_t)u * T];
            if (!cube_le(w[0].p, n)) break;  // primes ascend
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const uint32_t i = base + (uint32_t)u * T;
              if (!any_may_divide<kShort>(pt, i, w[u], s) || i >= pt.n_div) continue;
              const uint64_t lim = pt.lim[i], inv = pt.inv[i];
#pragma unroll
              for (int j = 0; j < K; ++j) {
                const uint64_t t = s[j] * inv;
                if (t > lim) continue;
                if (t * inv <= lim) atomicOr(&bad, 1u << j);
                const uint32_t d = atomicAdd(&n_div[j], 1u);
                if (d < kMaxDivisors) div_inv[j][d] = inv;
              }
            }
          }
        };
        if (n < kShortTest) walk(std::true_type());
        else walk(std::false_type());
        __syncthreads();
        if (tid < 32) {  // lane j decides the j-th value
          bool ok = false;
          const uint32_t j = tid, kj = k0 + j;
          if (j < (uint32_t)K && kj < 63 && (1ull << kj) < n && !((bad >> j) & 1u)) {
            uint64_t r = n - (1ull << kj);
            for (uint32_t d = 0; d < min(n_div[j], kMaxDivisors); ++d) r *= div_inv[j][d];  // exact divisions
            ok = cofactor_squarefree(r);
          }
          const uint32_t bal = __ballot_sync(0xFFFFFFFFu, ok);
          if (tid == 0 && bal) found = k0 + (uint32_t)__ffs(bal) - 1u;
        }
        __syncthreads();
        if (found) break;
      }
      k = found;
    }
  }
  if (tid == 0) out[e] = (uint8_t)k;
}

// Many points: a warp takes kSlots points at a time and walks the primes once
// for all of them (one load per prime for kSlots tests).  The first 32 primes,
// which decide nearly every value that is not squarefree, come first and
// alone: each slot's exponent advances until its value passes them.
constexpr int kSlots = 4;
__global__ void __launch_bounds__(256) points_warp_kernel(PrimeTab pt, const uint64_t *pts, uint64_t count,
                                                          uint8_t *out) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t gw = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint64_t small_p = lane < pt.n_div ? pt.p[lane] : 0ull;
  const uint64_t small_inv = lane < pt.n_div ? pt.inv[lane] : 0ull, small_lim = lane < pt.n_div ? pt.lim[lane] : 0ull;
  // value n - 2^k, its cofactor so far, point index (~0: none left)
  uint64_t s[kSlots], r[kSlots], e[kSlots];
  uint32_t k[kSlots];  // exponent under test; 0: the slot takes a new point
  uint64_t next = gw;
  auto take = [&](int j) {
    k[j] = 1;
    e[j] = next < count ? next : ~0ull;
    s[j] = next < count ? pts[next] - 2u : 0ull;
    if (next < count) next += nw;
  };
#pragma unroll
  for (int j = 0; j < kSlots; ++j) k[j] = 0;
  for (;;) {
    bool live = false;
    // new points for the slots without one, their loads in flight together
#pragma unroll
    for (int j = 0; j < kSlots; ++j)
      if (k[j] == 0) take(j);
#pragma unroll
    for (int j = 0; j < kSlots; ++j) {
      // the next value of this slot that passes the first 32 primes
      for (;;) {
        if (e[j] == ~0ull) {  // the slot idles (s = 1 has no divisor)
          s[j] = r[j] = 1;
          break;
        }
        const uint64_t n = s[j] + (1ull << k[j]);
        if (n < 3 || !(n & 1ull)) {
          if (lane == 0) out[e[j]] = 0;
          take(j);
          continue;
        }
        if (k[j] >= 63 || (1ull << k[j]) >= n) {
          if (lane == 0) out[e[j]] = kFailK;
          take(j);
          continue;
        }
        const uint64_t t = s[j] * small_inv;
        const bool div = small_p && t <= small_lim;
        if (__any_sync(0xFFFFFFFFu, div && t * small_inv <= small_lim)) {
          s[j] -= 1ull << k[j]++;
          continue;
        }
        uint32_t m = __ballot_sync(0xFFFFFFFFu, div);
        r[j] = s[j];
        while (m) {
          const int src = __ffs(m) - 1;
          m &= m - 1;
          r[j] *= __shfl_sync(0xFFFFFFFFu, small_inv, src);
        }
        live = true;
        break;
      }
    }
    if (!live) return;
    uint64_t top = 0;
#pragma unroll
    for (int j = 0; j < kSlots; ++j) top = s[j] > top ? s[j] : top;
    uint32_t bad = 0;
    // the primes to walk: those with p^3 <= top, none if the last of the first
    // 32 is above; 32 probes a step, first 32 primes apart, then over the rest
    // of the table (at most five loads one behind the other; halving the table
    // took seventeen)
    uint32_t n_walk = 0;
    if (__all_sync(0xFFFFFFFFu, small_p && cube_le((uint32_t)small_p, top))) {
      n_walk = 32;
      bool near = true;
      for (uint32_t len = min(pt.n_div - 32u, 1024u); len;) {
        const uint32_t step = (len + 31u) >> 5, probe = lane * step;
        const bool in = probe < len && cube_le(pt.word[n_walk + probe].p, top);
        const uint32_t b = (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, in));  // (primes ascend)
        if (b == 0) break;
        n_walk += (b - 1u) * step + 1u;
        len = near && b == 32u ? pt.n_div - n_walk : min(step - 1u, len - (b - 1u) * step - 1u);
        near = false;
      }
    }
    auto walk = [&](auto short_test) {
      constexpr bool kShort = decltype(short_test)::value;
      for (uint32_t i0 = 32u + lane; i0 < n_walk + lane; i0 += 64) {  // (the table is padded by a step)
        PrimeWord w[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) w[u] = pt.word[i0 + 32u * u];
        bool any = false;
#pragma unroll
        for (int u = 0; u < 2; ++u) any |= any_may_divide<kShort>(pt, i0 + 32u * u, w[u], s);
        if (!__any_sync(0xFFFFFFFFu, any)) continue;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint32_t i = i0 + 32u * u;
          if (!__any_sync(0xFFFFFFFFu, any_may_divide<kShort>(pt, i, w[u], s))) continue;
          const uint64_t inv = i < pt.n_div ? pt.inv[i] : 0ull, lim = i < pt.n_div ? pt.lim[i] : 0ull;
#pragma unroll
          for (int j = 0; j < kSlots; ++j) {
            const uint64_t t = s[j] * inv;
            const bool div = i < pt.n_div && t <= lim;
            uint32_t m = __ballot_sync(0xFFFFFFFFu, div);
            if (!m) continue;
            if (__any_sync(0xFFFFFFFFu, div && t * inv <= lim)) bad |= 1u << j;
            while (m) {
              const int src = __ffs(m) - 1;
              m &= m - 1;
              r[j] *= __shfl_sync(0xFFFFFFFFu, inv, src);
            }
          }
        }
      }
    };
    if (top < kShortTest) walk(std::true_type());
    else walk(std::false_type());
#pragma unroll
    for (int j = 0; j < kSlots; ++j) {
      if (e[j] == ~0ull) continue;
      if (!((bad >> j) & 1u) && cofactor_squarefree(r[j])) {
        if (lane == 0) out[e[j]] = (uint8_t)k[j];
        k[j] = 0;
      } else {
        s[j] -= 1ull << k[j]++;
      }
    }
  }
}

// Bound: few points by the latency of one pass over the primes (about 10^4 for
// n near 2^50, ten per thread of a block), many by the multiplies (two per
// prime and value, a quarter of the logic rate).  One warp per point, with two
// 64-bit products, 64-bit compares and two votes per 32 primes, took 962 us on
// the device for 65536 points; the high word of the 64-bit product alone 372;
// the 32-bit test 193.
// The lines, with both sides measured, n near 2^50: a block of 1024 threads per
// point while two fit every SM (304 points: 13 us; blocks of 256 with two
// exponents 15); those (7296 points: 59 us, four points per warp 66; 2048: 23
// and 52) up to 48 points per SM; then a warp per four points (16384 points: 68
// us, blocks 138).
// What counts as a small point depends on how long the blocks queue: up to eight
// blocks per SM all are resident and a block is as fast as a warp from 2^20 on
// (1024 points below 2^30: 7 us either way); 2000 points below 2^30 take 8 us by
// warps and 10 in blocks, 5000 below 2^36 15 and 17, below 2^20 7 and 15.
cudaError_t launch_points(PrimeTab pt, const uint64_t *pts, uint64_t count, uint8_t *out, uint32_t num_sms,
                          cudaStream_t st) {
  if (count == 0) return cudaSuccess;
  const uint64_t sms = num_sms;
  const uint64_t small = 1ull << (count <= 8 * sms ? 20 : count <= 20 * sms ? 34 : 38);
  if (count <= 2 * sms)
    points_block_kernel<4, 2><<<(uint32_t)count, 1024, 0, st>>>(pt, pts, count, small, out);
  else if (count <= 48 * sms)
    points_block_kernel<2, 4><<<(uint32_t)count, 256, 0, st>>>(pt, pts, count, small, out);
  else
    points_warp_kernel<<<(uint32_t)std::min<uint64_t>((count + 8 * kSlots - 1) / (8 * kSlots), 4 * sms), 256, 0, st>>>(
        pt, pts, count, out);
  return cudaGetLastError();
}

}  // namespace sv
