// streams.cu -- the fused range path in the stream layout: Algorithms 1 and 2
// of Sec. 3 per shared-memory tile, for launches that want aggregates and
// ordered lists (mink >= T, T >= 6) and no per-n output.
//
// Layout.  A window of 32 M consecutive odd integers (bits) is cut into 32
// streams of M bits, and stream b is bit b of the M shared-memory words:
// window bit J sits in bit J div M of word J mod M.  The flags of n - 2^k,
// which lie 2^(k-1) bits below n, are then simply another word,
//     look(i, 2^(k-1)) = word i - 2^(k-1)
// (below word 0 a stream continues in the previous one: the last words moved
// up by one bit), so the word-parallel search needs no funnel shifts: a
// thread walks kRun consecutive words and keeps the previous eight in
// registers.  In the linear layout of tiles.cu the search takes 29
// instructions per word, here about 11 (see scan_run).
// A set bit means "struck" (not squarefree), so the search ANDs words.
//
// Words per thread: kRun = 36, four times an odd number, so that 16-byte
// loads at a lane stride of kRun words meet no bank conflict; M = kRun times
// the block's threads.
//
// Per tile: 1. stamp the multiples of 9, 25, 49 and 121 from two periodic
// tables; 2. strike the other primes (see phase 2); 3. search k = 1..5 in
// registers, finish the words that still hold an n (one in 4500) by whole-word
// look-back up to k = kwin and leave the rest to the exact test; 4. add the
// tile's counts to its range's slot and stage its listed n, as tiles.cu does.
//
// Bound: integer issue and the logic pipe (22 thousand warp instructions per
// tile of 585504 odd n, 0.65 issued per scheduler and cycle, the logic pipe half
// busy, over 70% in the search), then the barriers between the phases.
// [2^40, 2^40 + 2^34): 398 us, against 601 us of tile_kernel<0, 4> in the linear
// layout.  Blocks of 512 threads, two per SM: four of 256 took 4% longer, a tile
// queue in chunks of 6 or 12 tiles instead of 8 1% and 5%.  Counting the n left
// after k = 4 by their bits' columns, with a recount where two met, instead of
// word by word: 9% longer (they come in clusters).  Larger dense primes one per
// warp instead of eight: 2%.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "strike.h"
#include "sv_internal.h"

namespace sv {

namespace {

constexpr uint32_t kRun = kStreamRun;
constexpr uint32_t kWarpQueue = 8;      // pieces queued per warp and tile (one in four warps has any)
constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr uint32_t kMaxDense = kMaxDensePrimes;

// The stamped primes: word i's struck bits of a set of primes depend only on
// (window start + i) mod P, P the product of their squares.
constexpr uint32_t kPa = 9 * 121, kPb = 25 * 49;
constexpr uint32_t kStampStep = 192;    // words a warp stamps per step (it divides every window); the tables run
                                        // this far past their periods
constexpr uint32_t kOffB = kPa + kStampStep;
constexpr uint32_t kStampWords = kOffB + kPb + kStampStep;
static_assert(kStampWords <= kStreamStampStride, "the context's table slots hold a table");

// What the block needs to know of a tile, made by one thread while the
// previous tile is struck.
struct TileDesc {
  int64_t wbit;            // the window's first bit (may lie below 0 at a range near 0)
  uint32_t tile;           // global index; >= the launch's tiles: none left
  uint32_t slot, n_sparse, fresh;  // fresh: the primes' offsets are computed, not carried
  uint32_t search;         // the first occurrences of k <= 5 are searched
  uint32_t vlo, vhi;       // valid n: window bits [vlo, vhi)
  uint32_t M, magic, size; // the window's words; their stamp table if it is not the launch's
  uint32_t ea, eb;         // the window start modulo kPa, kPb
  uint32_t req_idx;
};

struct StreamShared {
  TileDesc desc[2];
  ReqDesc req;          // the range of the newest descriptor
  uint32_t chunk_end;
  uint32_t n_strag, lst_cnt;
  uint32_t u[5];          // n unresolved after k = 1 .. 5 (the runs' sums)
  uint32_t hist[kMaxK];   // counts of the n resolved outside the runs
  uint32_t first[kMaxK];  // window bit of the smallest n with mink = k (kNone: none)
  uint4 dense[kMaxDense];        // q = p^2, 32 q mod M in bytes, 32 q div M, a tile's bits mod q
  uint32_t dense_r[kMaxDense];   // window bit of its first strike, below q
  unsigned long long lst_n[kStageCap];
  uint8_t lst_k[kStageCap];
  uint32_t q_cnt[kMaxStrikeWarps];
  uint32_t q_word[kMaxStrikeWarps][kWarpQueue];  // the first word of a queued piece
};

// The window and what it needs to be read: words, their number, magic to
// divide a window bit by M (exact below 32 M for every M used, see
// stream_magic).
struct Win {
  uint32_t *w;
  uint32_t M, magic;
  __device__ __forceinline__ void split(uint32_t bit, uint32_t *word, uint32_t *b) const {
    *b = __umulhi(bit, magic);
    *word = bit - *b * M;
  }
  __device__ __forceinline__ void strike(uint32_t bit) const {
    uint32_t i, b;
    split(bit, &i, &b);
    atomicOr(&w[i], 1u << b);
  }
  // the struck flags d bits below the 32 n of word i; bits that would lie
  // below the window read as 0 (no n whose look-back is asked has any)
  __device__ __forceinline__ uint32_t look(uint32_t i, uint32_t d) const {
    int32_t x = (int32_t)i - (int32_t)d;
    uint32_t s = 0;
    while (x < 0) {
      x += (int32_t)M;
      ++s;
    }
    return s < 32 ? w[x] << s : 0u;
  }
};

// The hot loops address shared memory by 32-bit addresses: pointers would be
// stepped in 64 bits.
__device__ __forceinline__ void strike_at(uint32_t addr, uint32_t mask) {
  asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(addr), "r"(mask) : "memory");
}
__device__ __forceinline__ uint32_t lds(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void lds4(uint32_t addr, uint32_t *v) {
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void sts(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// Three-input logic, one instruction each: a ^ b ^ c, the majority, (a & b) | c.
__device__ __forceinline__ uint32_t xor3(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0x96;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0xE8;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ uint32_t and_or(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

__device__ __forceinline__ uint32_t bits_from(uint32_t b) { return b >= 32u ? 0u : 0xFFFFFFFFu << b; }

// Finish the n (bits u) of word i from exponent k on: k .. kwin by whole-word
// look-back, the rest to the exact test.  Called by single lanes.
__device__ __noinline__ void finish_word(const Win win, uint32_t i, uint32_t u, uint32_t k, const TileArgs &a,
                                         StreamShared &sh, int64_t wbit, uint32_t req) {
  const uint32_t kwin = a.g.kwin, rec_t = a.g.rec_t;
  for (; k <= kwin && u; ++k) {
    uint32_t h = u & ~win.look(i, 1u << (k - 1));
    u ^= h;
    if (h) {
      if (k > 1) atomicAdd(&sh.hist[k], (uint32_t)__popc(h));  // (k = 1 is what the others leave, see the flush)
      atomicMin(&sh.first[k], (uint32_t)(__ffs(h) - 1) * win.M + i);
      if (k >= rec_t) {
        while (h) {
          const uint32_t b = __ffs(h) - 1;
          h &= h - 1;
          const uint32_t e = atomicAdd(&sh.lst_cnt, 1u);
          if (e < kStageCap) {
            sh.lst_n[e] = (unsigned long long)(2 * (wbit + (int64_t)(b * win.M + i)) + 1);
            sh.lst_k[e] = (uint8_t)k;
          }
        }
      }
    }
  }
  if (u) atomicAdd(&sh.n_strag, (uint32_t)__popc(u));
  while (u) {
    const uint32_t b = __ffs(u) - 1;
    u &= u - 1;
    const unsigned long long idx = atomicAdd(&a.hdr->strag_count, 1ull);
    if (idx < a.strag_cap) {
      Straggler s;
      s.n = (uint64_t)(2 * (wbit + (int64_t)(b * win.M + i)) + 1);
      s.k0 = kwin + 1u;
      s.req = req;
      a.strag[idx] = s;
    } else {
      atomicOr(&a.hdr->status, kStStragOverflow);
    }
  }
}

// Sums of population counts.  The logic pipe bounds the search, the count
// pipe (an eighth of its rate) comes next, the multiply-add pipe is nearly
// idle: the sums are multiply-adds by a 1 that the compiler cannot see, and
// carry-save addition, one logic operation per word, halves the counts where
// that evens the two pipes out (k = 1, 2 and 3; the sets of k = 4 are counted word
// by word).
__device__ __forceinline__ uint32_t add_count(uint32_t x, uint32_t one, uint32_t sum) {
  uint32_t d;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(__popc(x)), "r"(one), "r"(sum));
  return d;
}
struct Counter {
  uint32_t ones = 0, twos = 0;  // ones: one bit per column still to be counted; twos: counted pairs
  __device__ __forceinline__ void add(const uint32_t (&u)[4], uint32_t one) {
    const uint32_t a = maj3(ones, u[0], u[1]);
    ones = xor3(ones, u[0], u[1]);
    const uint32_t b = maj3(ones, u[2], u[3]);
    ones = xor3(ones, u[2], u[3]);
    twos = add_count(b, one, add_count(a, one, twos));
  }
  __device__ __forceinline__ uint32_t total() const { return 2u * twos + __popc(ones); }
};

// The n of word i (bits vm) left after k = 4, word by word.
__device__ __forceinline__ uint32_t left_after_4(const Win win, uint32_t i, uint32_t vm) {
  return vm & win.look(i, 1) & win.look(i, 2) & win.look(i, 4) & win.look(i, 8);
}

// The search over one thread's run of words i0 .. i0 + kRun - 1, for the n of
// the bits vm.  With z the struck words, the n left after k = 1, 2, 3, 4, 5
// are z[i-1], & z[i-2], & z[i-4], & z[i-8], & z[i-16]: one logic operation per
// word and k.  The sets of k = 1..4 are counted (hist[k] = U_(k-1) - U_k).
// When a lane has an n left after k = 5 among kPiece words (one piece in
// 380), it queues the piece.  MASK false: vm is all ones.  FIRST5: the tile
// may hold the range's first n of k = 5.
constexpr uint32_t kPiece = 12;
static_assert(kRun % kPiece == 0 && kPiece % 4 == 0, "a run is whole pieces");
template <bool MASK, bool FIRST5>
__device__ __forceinline__ void scan_run(const Win win, uint32_t base, uint32_t i0, uint32_t vm, StreamShared &sh,
                                         uint32_t warp, uint32_t one, uint32_t (&U)[4]) {
  uint32_t z[kRun + 16];
  const uint32_t at = base + 4u * i0;
  {
    // the 16 words below the run; below word 0 the streams' continuations
    // (bit 0 of those words' n lies in the margin)
    const uint32_t below = i0 ? at : base + 4u * win.M, up = i0 ? 0u : 1u;
#pragma unroll
    for (uint32_t j = 0; j < 16; j += 4) lds4(below - 64u + 4u * j, z + j);
#pragma unroll
    for (uint32_t j = 0; j < 16; ++j) z[j] <<= up;
  }
  Counter c1, c2, c3;
  uint32_t n4 = 0;
#pragma unroll
  for (uint32_t h = 0; h < kRun; h += kPiece) {
    uint32_t left = 0;
#pragma unroll
    for (uint32_t g = h; g < h + kPiece; g += 4) {
      lds4(at + 4u * g, z + g + 16);
      uint32_t u1[4], u2[4], u3[4], u4[4];
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) {
        const uint32_t *p = z + 16 + g + j;
        u1[j] = MASK ? p[-1] & vm : p[-1];
        u2[j] = u1[j] & p[-2];
        u3[j] = u2[j] & p[-4];
        u4[j] = u3[j] & p[-8];
        left = and_or(u4[j], p[-16], left);
        if (FIRST5) {
          const uint32_t f = u4[j] & ~p[-16];
          if (f) atomicMin(&sh.first[5], (uint32_t)(__ffs(f) - 1) * win.M + i0 + g + j);
        }
      }
      c1.add(u1, one);
      c2.add(u2, one);
      c3.add(u3, one);
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) n4 = add_count(u4[j], one, n4);
    }
    if (__any_sync(0xFFFFFFFFu, left)) {
      if (left) {
        const uint32_t e = atomicAdd(&sh.q_cnt[warp], 1u);
        if (e < kWarpQueue) sh.q_word[warp][e] = i0 + h;  // (a full queue: the warp searches its words again)
      }
    }
  }
  U[0] = c1.total();
  U[1] = c2.total();
  U[2] = c3.total();
  U[3] = n4;
}

// One warp's piece of a dense prime, or of kGroup consecutive ones with kLanes
// lanes each (the larger primes, whose strikes would leave most lanes of a
// warp idle or each pay a warp's set-up): lane l of a prime's L lanes strikes
// the window bits r + q (l + L m), m = m0 .. m0 + n - 1.  q is odd and M a
// multiple of 32, so one prime's lanes lie on different banks.  A step of L q
// moves a lane dw words up and db streams on (one more when it runs past word
// M); past the last stream its mask is shifted out and it strikes nothing.
constexpr uint32_t kGroup = 8, kLanes = 32 / kGroup;
__device__ __forceinline__ bool grouped(uint32_t q, uint32_t M) { return 32u * M < 128u * q; }  // under 128 strikes
__device__ __forceinline__ void strike_task(const Win win, uint32_t base, const StreamShared &sh, const StrikeTask t,
                                            uint32_t lane, uint32_t nd) {
  const bool group = t.d & kStrikeGroup;
  const uint32_t d = group ? min((t.d & ~kStrikeGroup) + lane / kLanes, nd - 1u) : t.d;
  const uint32_t l = group ? lane % kLanes : lane + 32u * t.m0;
  const uint4 c = sh.dense[d];  // q, dw in bytes, db
  const uint32_t bit = sh.dense_r[d] + c.x * l;
  const uint32_t M4 = 4u * win.M;
  uint32_t x = 0, mask = 0;
  if (bit < 32u * win.M) {
    uint32_t b;
    win.split(bit, &x, &b);
    x *= 4u;
    mask = 1u << b;
  }
  x += base;
  const uint32_t end = base + M4;
  strike_at(x, mask);
  if (!group && c.z == 0) {  // q < M / 32
#pragma unroll 8
    for (uint32_t n = t.n - 1u; n; --n)
      asm volatile(
          "{\n.reg .pred p;\n"
          "add.u32 %0, %0, %2;\n"
          "setp.ge.u32 p, %0, %3;\n"
          "@p sub.u32 %0, %0, %4;\n"
          "@p shl.b32 %1, %1, 1;\n"
          "red.shared.or.b32 [%0], %1;\n}"
          : "+r"(x), "+r"(mask)
          : "r"(c.y), "r"(end), "r"(M4)
          : "memory");
  } else {
    for (uint32_t n = t.n - 1u; n; --n)  // (a shift by 32 or more leaves 0)
      asm volatile(
          "{\n.reg .pred p;\n"
          "add.u32 %0, %0, %2;\n"
          "setp.ge.u32 p, %0, %3;\n"
          "shl.b32 %1, %1, %5;\n"
          "@p sub.u32 %0, %0, %4;\n"
          "@p shl.b32 %1, %1, 1;\n"
          "red.shared.or.b32 [%0], %1;\n}"
          : "+r"(x), "+r"(mask)
          : "r"(c.y), "r"(end), "r"(M4), "r"(c.z)
          : "memory");
  }
}

// The tile queue: chunks of consecutive tiles, so that one CTA works a
// range's tiles in order and the primes' offsets carry from one window to the
// next; the last 4 tiles per CTA go one at a time, which evens out the CTAs'
// finishing times (the split of tiles.cu, where it was measured).
__device__ __forceinline__ void chunk_range(uint32_t j, uint32_t total, uint32_t ctas, uint32_t *s, uint32_t *e) {
  const uint32_t chunk = 8u, reserve = 4u * ctas;
  const uint32_t n_big = total > reserve ? (total - reserve) / chunk : 0u;
  uint64_t b, f;
  if (j < n_big) {
    b = (uint64_t)j * chunk;
    f = b + chunk;
  } else {
    b = (uint64_t)n_big * chunk + (j - n_big);
    f = b + 1;
  }
  *s = (uint32_t)min(b, (uint64_t)total);
  *e = (uint32_t)min(f, (uint64_t)total);
}

// x mod m for a window start, which may lie below bit 0
__device__ __forceinline__ uint32_t floor_mod(int64_t x, uint32_t m) {
  const uint32_t r = (uint32_t)((uint64_t)(x < 0 ? -x : x) % m);
  return x < 0 && r ? m - r : r;
}

// Window bit of the first strike of q at or above the window start A (in
// [0, q)); below bit 0 the pattern simply continues, those bits are struck anyway.
__device__ __forceinline__ uint64_t first_in_window(int64_t A, uint64_t q, uint64_t mu) {
  if (A >= 0) return first_strike((uint64_t)A, q, mu);
  return (((q - 1) >> 1) + (uint64_t)(-A)) % q;
}

// Describes tile t in D; `prev`: the tile before it in this block (kNone:
// none).  One thread.
__device__ __forceinline__ void describe(const StreamArgs &s, StreamShared &sh, TileDesc &D, const TileDesc &P,
                                         uint32_t t, uint32_t prev, uint32_t total, uint32_t n_reqs, uint32_t M) {
  const TileArgs &a = s.t;
  const Geometry &g = a.g;
  D.tile = t;
  if (t >= total) return;
  uint32_t fresh = prev == kNone || t != prev + 1u;  // not the previous tile's successor
  uint32_t r = prev == kNone ? kNone : P.req_idx;
  if (r == kNone || t - sh.req.tile_base >= sh.req.n_tiles) {
    // the range of tile t: the next one, else a search
    uint32_t lo;
    if (r != kNone && r + 1u < n_reqs && a.reqs[r + 1u].tile_base <= t &&
        t - a.reqs[r + 1u].tile_base < a.reqs[r + 1u].n_tiles) {
      lo = r + 1u;
    } else {
      uint32_t hi = n_reqs;
      lo = 0;
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a.reqs[mid].tile_base <= t) lo = mid; else hi = mid;
      }
    }
    r = lo;
    sh.req = a.reqs[lo];
    fresh = 1;
  }
  const ReqDesc &R = sh.req;
  if (t - R.tile_base >= R.n_tiles) {  // bounds check, never expected: the block stops
    atomicOr(&a.hdr->status, kStBadTile);
    D.tile = kNone;
    return;
  }
  const int64_t wbit = 32 * (R.w0 + (int64_t)(t - R.tile_base) * g.tw - (int64_t)g.mw);
  D.req_idx = r;
  D.slot = R.slot;
  D.fresh = fresh;
  // A range's first tile, if it is whole, holds its first n of every k <= 5
  // (k = 5 comes about 80 times in a tile of 2^19 odd n): the other tiles
  // are not searched.  The host sees a k that occurs without a first n and
  // repeats the launch with every tile searched.
  D.search = t == R.tile_base || s.search_all;
  D.n_sparse = min(g.i_large, max(R.n_primes, g.i_dense)) - g.i_dense;  // <= sparse_room (host guarantees)
  D.wbit = wbit;
  // (a planned tile holds at least one n)
  D.vlo = (uint32_t)(max((int64_t)R.jlo, wbit + 32 * (int64_t)g.mw) - wbit);
  D.vhi = (uint32_t)(min((int64_t)R.jhi, wbit + 32 * (int64_t)M) - wbit);
  if (fresh) {
    D.ea = floor_mod(wbit, kPa);
    D.eb = floor_mod(wbit, kPb);
  } else {
    D.ea = (P.ea + 32u * g.tw) % kPa;
    D.eb = (P.eb + 32u * g.tw) % kPb;
  }
  // A range's last tile may need far fewer bits: its window is then the
  // smallest of 32 x 36 x 2^j words that holds them (short ranges, 2^16
  // integers at most, take 1152 words).
  D.M = M;
  D.magic = s.magic;
  D.size = 0;
  if (D.vhi <= 16u * M) {
    D.M = kRun * kStreamMinThreads;
    while (32u * D.M < D.vhi) {
      D.M <<= 1;
      ++D.size;
    }
    D.magic = 0xFFFFFFFFu / D.M + 1u;
  }
}

// Stamps M words (a multiple of kStampStep): a warp takes kStampStep words per
// step from one position in each table.  From the block's own tables (shared
// address tab) or, for a smaller window, from its size's (global memory).
__device__ __forceinline__ void stamp(uint32_t base, uint32_t M, uint32_t tab, uint32_t ea, uint32_t eb,
                                      uint32_t warp, uint32_t nwarps, uint32_t lane) {
  ea = (ea + kStampStep * warp) % kPa;
  eb = (eb + kStampStep * warp) % kPb;
  const uint32_t da = 4u * ((kStampStep * nwarps) % kPa), db = 4u * ((kStampStep * nwarps) % kPb);
  // lane's addresses; a position that passes its period goes back by it
  uint32_t pa = tab + 4u * (ea + lane), pb = tab + 4u * (kOffB + eb + lane);
  const uint32_t ma = tab + 4u * (kPa + lane), mb = tab + 4u * (kOffB + kPb + lane);
  const uint32_t step = 4u * kStampStep * nwarps, end = base + 4u * M;
  for (uint32_t w = base + 4u * (kStampStep * warp + lane); w < end; w += step) {
    uint32_t x[kStampStep / 32], y[kStampStep / 32];
#pragma unroll
    for (uint32_t h = 0; h < kStampStep / 32; ++h) {
      x[h] = lds(pa + 128u * h);
      y[h] = lds(pb + 128u * h);
    }
#pragma unroll
    for (uint32_t h = 0; h < kStampStep / 32; ++h) sts(w + 128u * h, x[h] | y[h]);
    pa += da;
    if (pa >= ma) pa -= 4u * kPa;
    pb += db;
    if (pb >= mb) pb -= 4u * kPb;
  }
}
__device__ __noinline__ void stamp_small(uint32_t *w, uint32_t M, const uint32_t *tab, uint32_t ea, uint32_t eb) {
  for (uint32_t i = threadIdx.x; i < M; i += blockDim.x) w[i] = tab[(ea + i) % kPa] | tab[kOffB + (eb + i) % kPb];
}

__global__ void __launch_bounds__(512, 2) stream_kernel(const __grid_constant__ StreamArgs s) {
  extern __shared__ __align__(16) uint32_t dyn[];
  __shared__ StreamShared sh;
  __shared__ uint32_t stab[kStampWords];
  const TileArgs &a = s.t;
  const Geometry &g = a.g;
  const uint32_t tid = threadIdx.x, S = blockDim.x, lane = tid & 31u, warp = tid >> 5, nwarps = S >> 5;
  const uint32_t M = kRun * S;
  const uint32_t T = 32u * g.tw;  // a window starts T bits above the previous one
  uint32_t *sparse_off = dyn + M, *sparse_q = sparse_off + s.sparse_room;
  const uint32_t win_addr = (uint32_t)__cvta_generic_to_shared(dyn), tab_addr = (uint32_t)__cvta_generic_to_shared(stab);
  const uint32_t total = a.hdr->total_tiles, n_reqs = a.hdr->n_reqs;
  const uint32_t nd = g.i_dense - g.i_med;  // <= kMaxDense (host guarantees)
  {
    uint32_t j = 0;  // the table of this block size
    while ((kStreamMinThreads << j) < S) ++j;
    const uint32_t *tab = s.stamp + j * kStreamStampStride;
    for (uint32_t i = tid; i < kStampWords; i += S) stab[i] = tab[i];
  }
  for (uint32_t i = tid; i < (uint32_t)kMaxK; i += S) {
    sh.hist[i] = 0;
    sh.first[i] = kNone;
  }
  for (uint32_t d = tid; d < nd; d += S) {
    const uint32_t p = a.pt.p[g.i_med + d], q = p * p;  // q <= 32 M / kDenseMinHits
    const uint32_t L = grouped(q, M) ? kLanes : 32u;
    sh.dense[d] = make_uint4(q, 4u * ((L * q) % M), (L * q) / M, T % q);
  }
  if (tid < nwarps) sh.q_cnt[tid] = 0;
  if (tid == 0) {
    sh.n_strag = sh.lst_cnt = 0;
    for (uint32_t k = 0; k < 5; ++k) sh.u[k] = 0;
    uint32_t cs, ce;
    chunk_range((uint32_t)atomicAdd(&a.hdr->work_counter, 1ull), total, gridDim.x, &cs, &ce);
    sh.chunk_end = ce;
    describe(s, sh, sh.desc[0], sh.desc[0], cs, kNone, total, n_reqs, M);
  }
  __syncthreads();

  for (uint32_t buf = 0;; buf ^= 1u) {
    const TileDesc &D = sh.desc[buf];
    const uint32_t gt = D.tile;
    if (gt >= total) break;
    Win win;
    win.w = dyn;
    win.M = D.M;
    win.magic = D.magic;
    const bool full = win.M == M;
    const uint32_t nbits = 32u * win.M;
    ResultSlot *slot = &a.slots[D.slot];

    // ---- 1. stamp; the primes' first strikes; the bucket's entries ----------
    // (thread 0: the chunk after this one, used below, when it has arrived)
    uint32_t next = gt + 1u, next_chunk = kNone;
    if (tid == 0 && next >= sh.chunk_end) next_chunk = (uint32_t)atomicAdd(&a.hdr->work_counter, 1ull);
    const uint32_t *bd = a.bucket_data + (size_t)gt * g.bucket_cap;
    const uint32_t nb = min(a.bucket_count[gt], g.bucket_cap);
    const uint32_t bv0 = tid < g.bucket_cap ? bd[tid] : 0u;  // (the first nb entries are written)
    const uint32_t n_sparse = D.n_sparse;
    if (D.fresh) {
      for (uint32_t j = tid; j < nd + n_sparse; j += S) {
        const uint64_t p = a.pt.p[g.i_med + j], q = p * p;
        const uint32_t r = (uint32_t)first_in_window(D.wbit, q, a.pt.mu[g.i_med + j]);
        if (j < nd) {
          sh.dense_r[j] = r;
        } else {
          sparse_off[j - nd] = r;
          sparse_q[j - nd] = (uint32_t)q;
        }
      }
    } else {
      for (uint32_t d = tid; d < nd; d += S) {  // the previous window began T bits lower
        const uint4 c = sh.dense[d];
        const uint32_t r = sh.dense_r[d];
        sh.dense_r[d] = r >= c.w ? r - c.w : r + c.x - c.w;
      }
    }
    if (full) stamp(win_addr, M, tab_addr, D.ea, D.eb, warp, nwarps, lane);
    else stamp_small(dyn, win.M, s.stamp + D.size * kStreamStampStride, D.ea, D.eb);
    __syncthreads();

    // ---- 2. strikes ------------------------------------------------------------
    if (tid == 0) {
      if (next_chunk != kNone) {
        uint32_t ce;
        chunk_range(next_chunk, total, gridDim.x, &next, &ce);
        sh.chunk_end = ce;
      }
      describe(s, sh, sh.desc[buf ^ 1u], D, next, gt, total, n_reqs, M);
      a.bucket_count[gt] = 0;  // read by every thread above
    }
    // dense primes: the planned tasks of this warp; in a smaller window one
    // warp per prime, 32 consecutive strikes at a time
    if (full) {
      for (uint32_t x = s.plan.start[warp]; x < s.plan.start[warp + 1]; ++x)
        strike_task(win, win_addr, sh, s.plan.task[x], lane, nd);
    } else {
      for (uint32_t d = warp; d < nd; d += nwarps) {
        const uint32_t q = sh.dense[d].x;
        for (uint32_t bit = sh.dense_r[d] + lane * q; bit < nbits; bit += 32u * q) win.strike(bit);
      }
    }
    // sparse primes, one thread each; their offsets carry to the next window
    for (uint32_t j = S - 1u - tid; j < n_sparse; j += S) {
      const uint32_t q = sparse_q[j];
      uint32_t b = sparse_off[j];
      for (; b < nbits; b += q) win.strike(b);
      if (full) {
        b -= T;
        while (b >= q) b -= q;
        sparse_off[j] = b;
      }
    }
    for (uint32_t e = tid; e < nb; e += S) {
      const uint32_t b = e < S ? bv0 : bd[e];
      if (b < nbits) win.strike(b);
      else atomicOr(&a.hdr->status, kStBadTile);
    }
    // integers below 1 are not squarefree (only a range's first window, near 0)
    if (D.wbit < 0)
      for (uint32_t b = tid; b < (uint32_t)min((int64_t)nbits, -D.wbit); b += S) win.strike(b);
    __syncthreads();

    // ---- 3. the search -----------------------------------------------------------
    // The valid bits of one thread's run are the same for all its words
    // except where the run holds word vlo mod M or vhi mod M: there the runs
    // take the bits valid throughout, and the few other n (at most kRun - 1
    // at either end) are looked at one by one.
    const uint32_t vlo = D.vlo, vhi = D.vhi;
    const bool search = D.search != 0;
    uint32_t il, bl, ih, bh;
    win.split(vlo, &il, &bl);
    win.split(vhi, &ih, &bh);  // vhi = nbits: stream 32, word 0
    if (!full) {
      // a small window: its words one by one, so that every warp has some (a
      // range of 23457 integers 45 to 42 us a call; one warp's runs would be
      // the latency of the tile)
      uint32_t U[5] = {0, 0, 0, 0, 0};
      for (uint32_t i = tid; i < win.M; i += S) {
        uint32_t u = bits_from(i >= il ? bl : bl + 1u) & ~bits_from(i < ih ? bh + 1u : bh);
        if (!u) continue;
#pragma unroll
        for (uint32_t k = 1; k <= 5; ++k) {
          const uint32_t z = win.look(i, 1u << (k - 1));
          if (k == 5 && search && (u & ~z)) atomicMin(&sh.first[5], (uint32_t)(__ffs(u & ~z) - 1) * win.M + i);
          u &= z;
          U[k - 1] += __popc(u);
        }
        if (u) finish_word(win, i, u, 6, a, sh, D.wbit, D.req_idx);
      }
      __syncwarp();
#pragma unroll
      for (uint32_t k = 0; k < 5; ++k) {
        const uint32_t x = __reduce_add_sync(0xFFFFFFFFu, U[k]);
        if (lane == 0 && x) atomicAdd(&sh.u[k], x);
      }
    } else {
      const uint32_t i0 = kRun * tid;
      const uint32_t vm = bits_from(i0 >= il ? bl : bl + 1u) & ~bits_from(i0 + kRun <= ih ? bh + 1u : bh);
      uint32_t U[4];
      if (search) scan_run<true, true>(win, win_addr, i0, vm, sh, warp, s.one, U);
      else if (__all_sync(0xFFFFFFFFu, vm == 0xFFFFFFFFu)) scan_run<false, false>(win, win_addr, i0, vm, sh, warp, s.one, U);
      else scan_run<true, false>(win, win_addr, i0, vm, sh, warp, s.one, U);
#pragma unroll
      for (uint32_t k = 0; k < 4; ++k) {
        const uint32_t x = __reduce_add_sync(0xFFFFFFFFu, U[k]);
        if (lane == 0) atomicAdd(&sh.u[k], x);
      }
      // the queued pieces (a queue that overflowed is left aside and every
      // word of the warp searched again)
      __syncwarp();
      const uint32_t nq = *(volatile uint32_t *)&sh.q_cnt[warp];
      if (nq) {
        const bool again = nq > kWarpQueue;
        uint32_t left = 0;
        for (uint32_t e = lane; e < (again ? 32u * kRun : nq * kPiece); e += 32u) {
          const uint32_t i = again ? kRun * 32u * warp + e : sh.q_word[warp][e / kPiece] + e % kPiece;
          const uint32_t r0 = i / kRun * kRun;  // its run's valid bits, as above
          uint32_t u = bits_from(r0 >= il ? bl : bl + 1u) & ~bits_from(r0 + kRun <= ih ? bh + 1u : bh);
          u = left_after_4(win, i, u) & win.look(i, 16);
          left += __popc(u);
          if (u) finish_word(win, i, u, 6, a, sh, D.wbit, D.req_idx);
        }
        __syncwarp();
        left = __reduce_add_sync(0xFFFFFFFFu, left);
        if (lane == 0) {
          atomicAdd(&sh.u[4], left);
          sh.q_cnt[warp] = 0;
        }
      }
    }
    if (full && (il % kRun || ih % kRun)) {  // (not inside a range: the margin is a multiple of kRun)
      const uint32_t run_l = il / kRun, run_h = ih / kRun;
      // [e0, e1): the start of the range inside its run; [f0, f1): its end
      uint32_t e0 = vlo, e1 = vlo, f0 = vhi, f1 = vhi;
      if (il % kRun) e1 = min(bl * win.M + (run_l + 1u) * kRun, vhi);
      if (ih % kRun && !(bl == bh && run_l == run_h && il % kRun)) f0 = max(bh * win.M + run_h * kRun, vlo);
      const uint32_t ne = e1 - e0, nf = f1 - f0;
      for (uint32_t x = tid; x < ne + nf; x += S) {
        uint32_t i, b;
        win.split(x < ne ? e0 + x : f0 + (x - ne), &i, &b);
        finish_word(win, i, 1u << b, 1, a, sh, D.wbit, D.req_idx);
      }
    }
    // first occurrences of k = 1..4: the tile's n one by one from the first
    // on, 32 per warp, until none can lie above (k = 4 comes once in about
    // 500 n)
    if (search) {
      for (uint32_t b0 = vlo + 32u * warp; b0 < vhi; b0 += 32u * nwarps) {
        uint32_t open = 0;
        for (uint32_t k = 1; k <= 4; ++k)
          if (*(volatile uint32_t *)&sh.first[k] >= b0) open |= 1u << k;
        open = __reduce_or_sync(0xFFFFFFFFu, open);
        if (!open) break;
        const uint32_t bit = b0 + lane;
        uint32_t kk = 0;
        if (bit < vhi) {
          uint32_t i, b;
          win.split(bit, &i, &b);
          for (uint32_t k = 4; k >= 1; --k)
            if (!((win.look(i, 1u << (k - 1)) >> b) & 1u)) kk = k;
        }
        for (uint32_t k = 1; k <= 4; ++k) {
          const uint32_t bal = __ballot_sync(0xFFFFFFFFu, kk == k);
          if (((open >> k) & 1u) && bal && lane == (uint32_t)(__ffs(bal) - 1)) atomicMin(&sh.first[k], bit);
        }
        __syncwarp();
      }
    }
    __syncthreads();

    // ---- 4. tile aggregates into the range's slot (the last warp, while the
    //         others start on the next tile) ------------------------------------
    if (warp == nwarps - 1u) {
      unsigned long long h0 = sh.hist[lane], h1 = sh.hist[lane + 32];
      if (lane >= 2 && lane <= 5) h0 += sh.u[lane - 2] - sh.u[lane - 1];
      // k = 1 was not counted: every other valid n of the tile is accounted for
      unsigned long long rest = (lane >= 2 ? h0 : 0ull) + h1;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) rest += __shfl_xor_sync(0xFFFFFFFFu, rest, o);
      rest += sh.n_strag;
      if (lane == 1) h0 = (unsigned long long)(vhi - vlo) - rest;
      // (in a tile that was not searched, k <= 5 has only the few n looked at one by one)
      const uint32_t f0 = search || lane > 5 ? sh.first[lane] : kNone, f1 = sh.first[lane + 32];
      if (h0) atomicAdd(&slot->hist[lane], h0);
      if (h1) atomicAdd(&slot->hist[lane + 32], h1);
      if (f0 != kNone) atomicMin(&slot->first_n[lane], 2ull * (unsigned long long)(D.wbit + (int64_t)f0) + 1ull);
      if (f1 != kNone) atomicMin(&slot->first_n[lane + 32], 2ull * (unsigned long long)(D.wbit + (int64_t)f1) + 1ull);
      // the tile's list entries to its staging slot (ordered later)
      const uint32_t m = sh.lst_cnt, ms = min(m, g.stage_cap);
      for (uint32_t e = lane; e < ms; e += 32u) {
        a.stage_n[(size_t)gt * kStageCap + e] = sh.lst_n[e];
        a.stage_k[(size_t)gt * kStageCap + e] = sh.lst_k[e];
      }
      __syncwarp();  // everything above is read before it is reset
      sh.hist[lane] = 0;
      sh.hist[lane + 32] = 0;
      sh.first[lane] = kNone;
      sh.first[lane + 32] = kNone;
      if (lane < 5) sh.u[lane] = 0;
      if (lane == 0) {
        a.stage_cnt[gt] = ms;
        if (m > ms) atomicOr(&a.hdr->status, kStListStage);
        sh.n_strag = sh.lst_cnt = 0;
      }
    }
  }
}

// The stamp tables of windows of M words: entry e of table A (B) holds the
// bits b for which (e + b M) lies on an odd multiple of one of its primes'
// squares, i.e. is (q - 1) / 2 modulo q.
__global__ void stamp_table_kernel(uint32_t *out, uint32_t M) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kStampWords) return;
  const bool second = i >= kOffB;
  const uint32_t e = second ? i - kOffB : i;
  uint32_t v = 0;
#pragma unroll
  for (uint32_t h = 0; h < 2; ++h) {
    const uint32_t q = second ? (h ? 49u : 25u) : (h ? 121u : 9u);
    for (uint32_t b = 0; b < 32; ++b)
      if ((e + b * M) % q == (q - 1) / 2) v |= 1u << b;
  }
  out[i] = v;
}

}  // namespace

cudaError_t launch_stamp_tables(uint32_t *d_tables, cudaStream_t st) {
  for (uint32_t j = 0; j < kStreamSizes; ++j) {
    stamp_table_kernel<<<(kStampWords + 255) / 256, 256, 0, st>>>(d_tables + j * kStreamStampStride,
                                                                 kRun * (kStreamMinThreads << j));
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// ceil(2^32 / M): with M = 36 S, S a power of two up to 512, umulhi(x, magic)
// is x div M for every x <= 32 M (the excess magic M - 2^32 times 32 stays
// below 2^32 / M).
uint32_t stream_magic(uint32_t M) { return (uint32_t)(((1ull << 32) + M - 1) / M); }

// Deals the dense primes' strikes to the block's warps in pieces of at most
// half a warp's fair share.  The longest pieces go first, each to the warp with
// the least work so far, its threads' sparse primes and warp 0's next tile
// included.  Costs are in instructions.
void plan_strikes(const uint32_t *primes, uint32_t nd, uint32_t n_sparse, uint32_t threads, StrikePlan *plan) {
  struct Job {
    uint32_t cost;
    StrikeTask t;
  };
  std::memset(plan, 0, sizeof(*plan));
  const uint32_t M = kRun * threads, nw = threads / 32;
  constexpr uint32_t kSetup = 24, kStep = 6, kSparseSetup = 30, kSparseStrike = 30, kDescribe = 250;
  uint32_t load[kMaxStrikeWarps] = {0};
  load[0] = kDescribe;
  uint32_t sum = kDescribe;
  for (uint32_t j0 = 0; j0 < n_sparse; j0 += 32) {  // 32 sparse primes per warp, from the last warp down
    const uint64_t q = (uint64_t)primes[nd + j0] * primes[nd + j0];
    const uint32_t c = kSparseSetup + kSparseStrike * (uint32_t)(32ull * M / q + 1);
    load[nw - 1 - (j0 / 32) % nw] += c;
    sum += c;
  }
  // steps of L strikes r + q (l + L m) below 32 M, r < q
  auto steps_of = [&](uint32_t d, uint32_t L) { return (32 * M - 1) / (L * primes[d] * primes[d]) + 1; };
  uint32_t n_single = 0;  // the first primes have a warp each (see grouped())
  while (n_single < nd && 32ull * M >= 128ull * primes[n_single] * primes[n_single]) ++n_single;
  for (uint32_t d = 0; d < n_single; ++d) sum += kSetup + kStep * steps_of(d, 32);
  for (uint32_t d = n_single; d < nd; d += kGroup) sum += kSetup + kStep * steps_of(d, kLanes);
  const uint32_t share = std::max(sum / nw, 1u);
  Job jobs[kMaxStrikeTasks];
  uint32_t nj = 0;
  for (uint32_t d = n_single; d < nd; d += kGroup) {  // (the last group's spare lanes repeat prime nd - 1: harmless)
    const uint32_t steps = steps_of(d, kLanes);
    jobs[nj++] = {kSetup + kStep * steps, {0, (uint8_t)(d | kStrikeGroup), (uint8_t)steps}};
  }
  for (uint32_t d = 0; d < n_single; ++d) {
    const uint32_t steps = steps_of(d, 32);
    // as many pieces as the task table can still hold
    uint32_t pieces = std::max(1u, (2 * kStep * steps + share - 1) / share);
    pieces = std::min(std::min(pieces, steps), kMaxStrikeTasks - nj - (n_single - 1 - d));
    for (uint32_t h = 0; h < pieces; ++h) {
      const uint32_t m0 = steps * h / pieces, m1 = steps * (h + 1) / pieces;
      jobs[nj++] = {kSetup + kStep * (m1 - m0), {(uint16_t)m0, (uint8_t)d, (uint8_t)(m1 - m0)}};
    }
  }
  std::stable_sort(jobs, jobs + nj, [](const Job &x, const Job &y) { return x.cost > y.cost; });
  uint8_t of[kMaxStrikeTasks];
  for (uint32_t j = 0; j < nj; ++j) {
    uint32_t w = 0;
    for (uint32_t x = 1; x < nw; ++x)
      if (load[x] < load[w]) w = x;
    of[j] = (uint8_t)w;
    load[w] += jobs[j].cost;
  }
  uint32_t at = 0;
  for (uint32_t w = 0; w < nw; ++w) {
    plan->start[w] = (uint8_t)at;
    for (uint32_t j = 0; j < nj; ++j)
      if (of[j] == w) plan->task[at++] = jobs[j].t;
  }
  for (uint32_t w = nw; w <= kMaxStrikeWarps; ++w) plan->start[w] = (uint8_t)at;
}

size_t stream_smem(uint32_t threads, uint32_t sparse_room) {
  return 4ull * (kRun * threads + 2ull * sparse_room);
}

size_t stream_static_smem() { return sizeof(StreamShared) + 4 * kStampWords + 64; }

cudaError_t stream_kernel_setup(int optin) {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, stream_kernel);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

cudaError_t launch_stream_tiles(const StreamArgs &s, uint32_t grid, cudaStream_t st) {
  if (grid == 0) return cudaSuccess;
  stream_kernel<<<grid, s.t.g.threads, stream_smem(s.t.g.threads, s.sparse_room), st>>>(s);
  return cudaGetLastError();
}

}  // namespace sv
