// align.cu -- Dynamic Token Warping between draft and proxy target tokens
// (§4.1, Alg. 1) with the byte-level Levenshtein token distance (App. H).
//
// One pair (request) is aligned by one warp, or by a CTA of several warps when
// the batch holds so few or so long pairs that warps would be missing. Per pair:
//  1. stage the tokens' byte strings in shared memory: draft tokens transposed,
//     four rows to a word, target tokens as codes of the pair's distinct bytes;
//  2. per distinct byte and four rows, the words that say where the byte
//     occurs in each row's token (the edit distance's match vectors);
//  3. the banded local-cost tile d(i,j), a byte per cell: a lane takes eight
//     rows at once, one byte of two words each, through the bit-parallel edit
//     distance (tokens of more than 8 bytes by the plain recurrence);
//  4. sweep the anti-diagonals i + j = s in registers: a lane owns pairs of
//     consecutive rows, packed in the halves of a word, so that a cell's
//     neighbours are its own registers and, for its first row, one shuffle;
//     each cell's choice of predecessor (diagonal, then (i-1,j), then (i,j-1)
//     on ties) is two bits of a word stored every 8 diagonals;
//  5. backtrack from (k, m) on one lane, then write path, C*, the map
//     i*(j) = max{i : (i,j) on the path} and the needed-draft-row flags.
#include <algorithm>
#include <cstdint>

#include "tt_device.cuh"
#include "tt_launch.h"
#include "tt_f2.cuh"

namespace tt {

namespace {

// Edit distance by the textbook row recurrence, for tokens longer than 8
// bytes (bytes read from the global tables; ns, nt <= TT_MAX_TOKEN_BYTES).
__device__ __noinline__ int lev_rows(const uint8_t* s, int ns, const uint8_t* t, int nt) {
  if (ns > nt) {  // keep the row short
    const uint8_t* u = s; s = t; t = u;
    int n = ns; ns = nt; nt = n;
  }
  uint16_t row[TT_MAX_TOKEN_BYTES + 1];
  for (int i = 0; i <= ns; ++i) row[i] = uint16_t(i);
  for (int j = 1; j <= nt; ++j) {
    uint8_t tj = t[j - 1];
    int diag = row[0];
    row[0] = uint16_t(j);
    for (int i = 1; i <= ns; ++i) {
      int up = row[i];
      int v = min(min(up + 1, int(row[i - 1]) + 1), diag + (s[i - 1] == tj ? 0 : 1));
      diag = up;
      row[i] = uint16_t(v);
    }
  }
  return row[ns];
}

template <int N>
struct Int {
  static constexpr int value = N;
};

constexpr int kSymCap = 48;  // distinct target bytes of a pair with match vectors kept
constexpr int kLongFlag = 1 << 16;  // some token of the pair is longer than 8 bytes
constexpr uint32_t kOut4 = 0x80808080u;   // cost bytes of cells outside the band
constexpr uint32_t kInf2 = 0xff80ff80u;   // infinite accumulated cost, two 16-bit halves
constexpr int kMaxCost = 127;             // larger costs are stored as this and recomputed
// The packed sweep holds accumulated costs times four in 16 bits: they must
// stay below kInf2's 0xff80 (65408) with 4 (k + m) (longest token) to spare.
constexpr int kPackedMax = 16000;

// Storage of the cost tile. Rows are taken in pairs p (rows 2p + 1 and 2p + 2)
// and stored by diagonal: cell (i, j) of pair p is byte r = (i - 1) & 1 of the
// 16-bit entry sigma = i + j - 2, entries counted from the pair's first band
// diagonal rounded down to a multiple of 8 (first_block(p)). A block of 8
// diagonals is 16 bytes; a pair has row_blocks(m, W0) of them (an odd count,
// so that neighbouring lanes' 16-byte loads fall into different banks), and as
// many 32-bit words of predecessor choices.
__host__ __device__ __forceinline__ int row_blocks(int m, int W0) {
  const int n = 2 * W0 + 2;  // band columns of the two rows; one diagonal more than that
  return (((n < m ? n : m) + 15) >> 3) | 1;
}
__device__ __forceinline__ int first_block(int p, int W0) {
  return (2 * p + max(0, 2 * p - W0)) >> 3;
}

// Shared memory of one pair, for sequences of at most K and M tokens.
struct PairSmem {
  uint64_t* tok;    // [M] target tokens: 8 bytes, then the codes of those bytes
  uint8_t* tile;    // [16 * tile_blocks] local costs
  uint32_t* path;   // [K + M] backtracked cells (i << 16 | j), reverse order (over tile)
  uint32_t* trans;  // [G][8] byte p of four draft tokens: row 4 g + r in byte r; G is the
                    // groups of four rows, an even count
  uint32_t* peq;    // [kSymCap][G] match vectors of a byte with four rows' tokens
  uint32_t* dirs;   // [tile_blocks] predecessor choices: per pair and 8 diagonals a word,
                    // row r in half r, the first diagonal's two bits on top (over peq)
  uint32_t* pmask;  // [G] one bit per byte of each of four rows' tokens
  uint32_t* seen;   // [8] which byte values occur in the target tokens
  uint8_t* symch;   // [kSymCap] the byte of each code
  uint16_t* len_d;  // [K] token byte lengths
  uint16_t* len_t;  // [M]
  size_t bytes;
};

__host__ __device__ __forceinline__ PairSmem carve(char* base, int K, int M, int tile_blocks) {
  PairSmem s;
  size_t off = 0;
  auto take = [&](size_t n) {
    char* r = base ? base + off : nullptr;
    off = (off + n + 15) & ~size_t(15);
    return r;
  };
  const int G = (K + 7) / 8 * 2;
  const int path_bytes = 4 * (K + M), peq_words = kSymCap * G;
  s.tok = reinterpret_cast<uint64_t*>(take(8 * size_t(M)));
  s.tile = reinterpret_cast<uint8_t*>(
      take(size_t(16 * tile_blocks > path_bytes ? 16 * tile_blocks : path_bytes)));
  s.path = reinterpret_cast<uint32_t*>(s.tile);
  s.trans = reinterpret_cast<uint32_t*>(take(32 * size_t(G)));
  s.peq = reinterpret_cast<uint32_t*>(
      take(4 * size_t(peq_words > tile_blocks ? peq_words : tile_blocks)));
  s.dirs = s.peq;
  s.pmask = reinterpret_cast<uint32_t*>(take(4 * size_t(G)));
  s.seen = reinterpret_cast<uint32_t*>(take(32));
  s.symch = reinterpret_cast<uint8_t*>(take(kSymCap));
  s.len_d = reinterpret_cast<uint16_t*>(take(2 * size_t(K)));
  s.len_t = reinterpret_cast<uint16_t*>(take(2 * size_t(M)));
  s.bytes = off;
  return s;
}

// The n <= 8 bytes at v.bytes + o, packed little-endian: two aligned 8-byte
// loads where both lie inside the table, else byte by byte.
__device__ __forceinline__ uint64_t load_packed8(const tt_vocab& v, int64_t o, int n) {
  if (n == 0) return 0;
  const uint8_t* p = v.bytes + o;
  const uintptr_t a = reinterpret_cast<uintptr_t>(p) & ~uintptr_t(7);
  const int sh = int(reinterpret_cast<uintptr_t>(p) & 7);
  const bool two = sh + n > 8;
  uint64_t w;
  if (a >= reinterpret_cast<uintptr_t>(v.bytes) &&
      a + (two ? 16 : 8) <= reinterpret_cast<uintptr_t>(v.bytes) + uint64_t(v.n_bytes)) {
    const uint64_t* q = reinterpret_cast<const uint64_t*>(a);
    const uint64_t lo = __ldg(q), hi = two ? __ldg(q + 1) : 0;
    w = lo >> (8 * sh);
    if (sh) w |= hi << (64 - 8 * sh);
  } else {
    uint8_t by[8];
#pragma unroll
    for (int y = 0; y < 8; ++y) by[y] = y < n ? p[y] : uint8_t(0);
    w = 0;
#pragma unroll
    for (int y = 0; y < 8; ++y) w |= uint64_t(by[y]) << (8 * y);
  }
  return n < 8 ? w & ((1ull << (8 * n)) - 1) : w;
}

// Match vectors of byte c with four rows' tokens (8 bytes each, transposed):
// bit p of byte r is set iff byte p of row r equals c. A byte of t is zero iff
// the high bit of its byte of ~(((t & 0x7f..) + 0x7f..) | t | 0x7f..) is set.
// Past a token's end the bytes are zero and may match c = 0; those bits lie
// above the token's last one, and nothing in the recurrence moves down.
__device__ __forceinline__ uint32_t match4(const uint4& w0, const uint4& w1, uint32_t c) {
  const uint32_t cc = c * 0x01010101u;
  const uint32_t ww[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
  uint32_t eq = 0;
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const uint32_t t = ww[p] ^ cc;
    const uint32_t z = ~(((t & 0x7f7f7f7fu) + 0x7f7f7f7fu) | t | 0x7f7f7f7fu);
    eq |= z >> (7 - p);
  }
  return eq;
}

// Bit counts of the four bytes of x.
__device__ __forceinline__ uint32_t popc4(uint32_t x) {
  x = x - ((x >> 1) & 0x55555555u);
  x = (x & 0x33333333u) + ((x >> 2) & 0x33333333u);
  return (x + (x >> 4)) & 0x0f0f0f0fu;
}

// One column of the bit-parallel edit distance (Myers 1999, in Hyyro's global
// form) for four 8-bit vectors held in the bytes of a word. The one addition,
// of a subset of Pv's bits to Pv, is kept from carrying between bytes.
__device__ __forceinline__ void lev_step4(uint32_t Eq, uint32_t& Pv, uint32_t& Mv) {
  const uint32_t sum = (Eq & Pv & 0x7f7f7f7fu) + (Pv & 0x7f7f7f7fu);
  // (Eq & Pv) + Pv per byte is sum ^ ((Pv & ~Eq) & 0x80..): the top bits of
  // the two terms differ exactly where Pv is set and Eq is not
  const uint32_t Xh = ((sum ^ (Pv & ~Eq & 0x80808080u)) ^ Pv) | Eq;
  const uint32_t Xv = Eq | Mv;
  uint32_t Ph = Mv | ~(Xh | Pv);
  uint32_t Mh = Pv & Xh;
  Ph = ((Ph << 1) & 0xfefefefeu) | 0x01010101u;  // row 0 grows by one per column
  Mh = (Mh << 1) & 0xfefefefeu;
  Pv = Mh | ~(Xv | Ph);
  Mv = Ph & Xv;
}

// Barrier of the pair's WPP warps (a CTA holds one pair when WPP > 1).
template <int WPP>
__device__ __forceinline__ void pair_sync() {
  if constexpr (WPP == 1) __syncwarp();
  else __syncthreads();
}

// The OR of a few flag bits over the pair's threads, and a barrier.
template <int WPP>
__device__ __forceinline__ int pair_or(int flag) {
  if constexpr (WPP == 1) {
    flag = __reduce_or_sync(0xffffffffu, flag);
    __syncwarp();
    return flag;
  } else {
    int all = 0;
    for (int bit : {TT_REQ_ID_OUT_OF_RANGE, TT_REQ_TOO_LONG, kLongFlag})
      if (__syncthreads_or(flag & bit)) all |= bit;
    return all;
  }
}

// The maximum over the pair's threads (`word` holds 0 on entry and exit).
template <int WPP>
__device__ __forceinline__ int pair_max(int v, uint32_t* word) {
  v = int(__reduce_max_sync(0xffffffffu, unsigned(v)));
  if constexpr (WPP > 1) {
    if ((threadIdx.x & 31) == 0) atomicMax(word, unsigned(v));
    __syncthreads();
    v = int(*word);
    __syncthreads();
    if (threadIdx.x == 0) *word = 0;
    __syncthreads();
  }
  return v;
}

struct PairDims {
  int k, m, W0, nb;  // lengths, band half-width, blocks stored per row pair
};

// Two cost bytes of a word (the lower or the upper two) as halves, each byte's
// sign spread over its half's upper byte. (__byte_perm has no sign mode.)
template <int ODD>
__device__ __forceinline__ uint32_t cost_halves(uint32_t w) {
  uint32_t r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(w), "n"(ODD ? 0xb3a2 : 0x9180));
  return r;
}

// Local cost d(i, j) (1-based) by the plain recurrence.
__device__ __forceinline__ int long_cost(const AlignArgs& a, const PairSmem& sm, int d0, int t0,
                                         int i, int j) {
  const int di = a.draft_ids[d0 + i - 1], ti = a.target_ids[t0 + j - 1];
  return lev_rows(a.vd.bytes + a.vd.offsets[di], sm.len_d[i - 1],
                  a.vt.bytes + a.vt.offsets[ti], sm.len_t[j - 1]);
}

// The band's cells with a token of more than 8 bytes; a cost above kMaxCost is
// stored as that and recomputed in the sweep. The cells lie scattered (a long
// token's row and column), and the recurrence takes thousands of cycles: a warp
// looks 32 cells over at a time and queues those it finds, one per lane, until
// every lane has one. (With each cell computed where it was found, one or two
// lanes worked at a time: 1024 pairs of 16 x 20 tokens, one in fifty long, took
// 86 us; 40 now.)
__device__ __noinline__ void long_costs(const AlignArgs& a, int d0, int t0, PairSmem sm,
                                        PairDims d, int t, int nt) {
  const int lane = t & 31;
  int held = 0, cell = 0;  // lanes below `held` have a cell queued
  auto compute = [&]() {
    const int i = cell / d.m + 1, j = cell - (i - 1) * d.m + 1, p = (i - 1) >> 1;
    sm.tile[16 * (p * d.nb - first_block(p, d.W0)) + 2 * (i + j - 2) + ((i - 1) & 1)] =
        uint8_t(min(long_cost(a, sm, d0, t0, i, j), kMaxCost));
  };
  for (int q0 = t - lane; q0 < d.k * d.m; q0 += nt) {
    const int q = q0 + lane;
    bool mine = q < d.k * d.m;
    if (mine) {
      const int i = q / d.m + 1, j = q - (i - 1) * d.m + 1;
      mine = abs(i - j) <= d.W0 && (sm.len_d[i - 1] > 8 || sm.len_t[j - 1] > 8);
    }
    for (unsigned found = __ballot_sync(0xffffffffu, mine); found;) {
      // lane held + x takes the x-th cell found
      const int x = lane - held, n = __popc(found), take = min(32 - held, n);
      const int src = x >= 0 && x < take ? int(__fns(found, 0, x + 1)) : 0;
      const int c = __shfl_sync(0xffffffffu, q, src);
      if (x >= 0 && x < take) cell = c;
      held += take;
      found = take == n ? 0u : found & ~((2u << __fns(found, 0, take)) - 1u);
      if (held == 32) {
        compute();
        __syncwarp();
        held = 0;
      }
    }
  }
  if (lane < held) compute();
}

// One anti-diagonal of NP row pairs of a lane. cost: the pairs' entries of
// this diagonal as halves (a byte with its sign spread, so a cell outside the
// band is 0xff80 and the maximum below makes its value infinite). Values are
// kept times four: with 1 added for (i-1, j) and 2 for (i, j-1), one minimum
// gives the smallest predecessor, ties in the order diagonal, (i-1, j),
// (i, j-1), and its two low bits are the choice.
template <int NP>
__device__ __forceinline__ void sweep_step(uint32_t x, uint32_t (&cur)[NP], uint32_t (&diag)[NP],
                                           uint32_t (&acc)[NP], const uint32_t (&cost)[NP]) {
#pragma unroll
  for (int q = NP - 1; q >= 0; --q) {
    // the cells above: the pair above's second row, then this pair's first
    const uint32_t up = __byte_perm(q > 0 ? cur[q > 0 ? q - 1 : 0] : x, cur[q], 0x5432);
    const uint32_t best =
        __viaddmin_u16x2(up, 0x00010001u, __viaddmin_u16x2(cur[q], 0x00020002u, diag[q]));
    diag[q] = up;  // the diagonal neighbours of the next step
    acc[q] = acc[q] * 4 + (best & 0x00030003u);
    const uint32_t v = (best & 0xfffcfffcu) + ((cost[q] & 0x007f007fu) << 2);
    cur[q] = __vmaxu2(v, cost[q]);
  }
}

// The anti-diagonal sweep by one warp, in 16-bit halves. Pairs of rows are
// taken in blocks of NP; block b belongs to lane b mod 32, which moves on to
// block b + 32 when the band has left it (never while all rows fit on the 32
// lanes): k <= 64 NP or W0 <= 56 NP, so that a lane has left its block, at a
// multiple of 8 diagonals, before the next one or its upper neighbour's next
// one enters the band. A step waits for one shuffle and six dependent
// instructions. Returns C(k, m).
template <int NP>
__device__ int sweep(const PairSmem& sm, const PairDims& d, int lane) {
  const int k = d.k, m = d.m, W0 = d.W0;
  const int n_pairs = (k + 1) >> 1, last = k + m - 2;  // the last diagonal
  int p0 = lane * NP;                                  // first pair of the lane's block
  uint32_t cur[NP], diag[NP], acc[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    cur[q] = diag[q] = kInf2;
    acc[q] = 0;
  }
  if (lane == 0) diag[0] = kInf2 & 0xffff0000u;  // C(0, 0) = 0
  for (int s8 = 0; s8 <= last; s8 += 8) {
    uint4 cw[NP];
    int at[NP];  // the pairs' entry of this block, or -1
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const int p = p0 + q, e = (s8 >> 3) - first_block(p, W0);
      at[q] = p < n_pairs && unsigned(e) < unsigned(d.nb) ? p * d.nb + e : -1;
      cw[q] = at[q] >= 0 ? reinterpret_cast<const uint4*>(sm.tile)[at[q]]
                         : make_uint4(kOut4, kOut4, kOut4, kOut4);
    }
    const int n = min(8, last + 1 - s8);
    if (n == 8) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        uint32_t x = __shfl_sync(0xffffffffu, cur[NP - 1], (lane + 31) & 31);
        if (p0 == 0) x = kInf2;  // row 0
        uint32_t cost[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          const uint32_t w = (e >> 1) == 0 ? cw[q].x : (e >> 1) == 1 ? cw[q].y
                             : (e >> 1) == 2 ? cw[q].z : cw[q].w;
          cost[q] = (e & 1) ? cost_halves<1>(w) : cost_halves<0>(w);
        }
        sweep_step<NP>(x, cur, diag, acc, cost);
      }
    } else {  // the last few diagonals, one at a time
#pragma unroll 1
      for (int e = 0; e < n; ++e) {
        uint32_t x = __shfl_sync(0xffffffffu, cur[NP - 1], (lane + 31) & 31);
        if (p0 == 0) x = kInf2;
        uint32_t cost[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          cost[q] = cost_halves<0>(cw[q].x);
          const bool odd = e & 1;  // two entries to a word
          cw[q].x = odd ? cw[q].y : cw[q].x >> 16;
          cw[q].y = odd ? cw[q].z : cw[q].y;
          cw[q].z = odd ? cw[q].w : cw[q].z;
        }
        sweep_step<NP>(x, cur, diag, acc, cost);
      }
#pragma unroll
      for (int q = 0; q < NP; ++q) acc[q] <<= 2 * (8 - n);
    }
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      if (at[q] >= 0) sm.dirs[at[q]] = acc[q];
      acc[q] = 0;
    }
    // the band has left the block, and the row below has read its last cell
    const int il = 2 * (p0 + NP);  // its last row
    if (p0 + 32 * NP < n_pairs && s8 + 6 >= il + min(m, il + W0) - 2) {
      p0 += 32 * NP;
#pragma unroll
      for (int q = 0; q < NP; ++q) cur[q] = kInf2;
    }
  }
  const int p = (k - 1) >> 1;
  uint32_t v = 0;
#pragma unroll
  for (int q = 0; q < NP; ++q)
    if (q == p % NP) v = cur[q];
  v = __shfl_sync(0xffffffffu, v, (p / NP) & 31);
  return int((k & 1) ? v & 0xffffu : v >> 16) >> 2;
}

// The same in 32 bits, for pairs whose costs may pass 16 bits or kMaxCost
// (very long tokens): a lane holds pairs p = lane * 4 .. + 3 of at most 128.
__device__ __noinline__ int sweep_wide(const AlignArgs& a, int d0, int t0, PairSmem sm, PairDims d,
                                       int lane) {
  constexpr int R = TT_MAX_K / 32;
  constexpr int kInf4 = 0x3ffffffc;  // grows by at most 4 x 256 on each of 768 diagonals
  const int k = d.k, m = d.m, W0 = d.W0, last = k + m - 2;
  int cur[R], prev[R];
  uint32_t acc[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    cur[r] = prev[r] = kInf4;
    acc[r] = 0;
  }
  int up_prev = lane == 0 ? 0 : kInf4;
#pragma unroll 1
  for (int s = 0; s <= last; ++s) {
    int up = __shfl_up_sync(0xffffffffu, cur[R - 1], 1);
    if (lane == 0) up = kInf4;
#pragma unroll
    for (int r = R - 1; r >= 0; --r) {
      const int i = lane * R + r + 1, j = s + 2 - i, p = (i - 1) >> 1;
      const int u = r > 0 ? cur[r > 0 ? r - 1 : 0] : up;
      const int dg = r > 0 ? prev[r > 0 ? r - 1 : 0] : up_prev;
      const int best = min(min(dg, u + 1), cur[r] + 2);
      acc[r] = acc[r] * 4 + (best & 3);
      int v = kInf4;
      if (i <= k && j >= max(1, i - W0) && j <= min(m, i + W0)) {
        const int e = s - 8 * first_block(p, W0);
        int cost = sm.tile[16 * p * d.nb + 2 * e + ((i - 1) & 1)];
        if (cost == kMaxCost) cost = long_cost(a, sm, d0, t0, i, j);
        v = (best & ~3) + 4 * cost;
      }
      if ((s & 7) == 7 || s == last) {
        const int e = (s >> 3) - first_block(p, W0);
        if (i <= k && unsigned(e) < unsigned(d.nb))
          reinterpret_cast<uint16_t*>(sm.dirs)[2 * (p * d.nb + e) + ((i - 1) & 1)] =
              uint16_t(acc[r] << (2 * (7 - (s & 7))));
        acc[r] = 0;
      }
      prev[r] = cur[r];
      cur[r] = v;
    }
    up_prev = up;
  }
  int v = 0;
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (r == (k - 1) % R) v = cur[r];
  return __shfl_sync(0xffffffffu, v, (k - 1) / R) >> 2;
}

// The WPP warps of a pair (thread t of them) align pair b in its own
// shared-memory region.
template <int WPP>
__device__ __forceinline__ void align_pair(const AlignArgs& a, int b, char* region, int t) {
  constexpr int NT = 32 * WPP;
  const int K = a.max_k, M = a.max_m, lane = t & 31;
  const PairSmem sm = carve(region, K, M, a.tile_blocks);

  if (!csr_ok(a.draft_off, b, a.n_draft) || !csr_ok(a.target_off, b, a.n_target)) {
    if (t == 0) {
      a.status[b] = TT_REQ_BAD_OFFSETS;
      if (a.path_len) a.path_len[b] = 0;
      if (a.cost) a.cost[b] = -1;
    }
    return;
  }
  const int d0 = a.draft_off[b], k = a.draft_off[b + 1] - d0;
  const int t0 = a.target_off[b], m = a.target_off[b + 1] - t0;
  if (a.excl)  // the row pass leaves these columns out of its sums
    for (int j = t; j <= m; j += NT)
      a.excl[int64_t(t0) + b + j] = j < m ? a.target_cols[t0 + j] : -1;
  int st = 0;
  if (k == 0 || m == 0) st |= TT_REQ_EMPTY;
  if (k > K || m > M || k > TT_MAX_K || m > TT_MAX_M) st |= TT_REQ_TOO_LONG;
  const int k8 = (k + 7) & ~7;  // rows of whole groups
  PairDims dm;
  dm.k = k;
  dm.m = m;
  dm.W0 = a.window < 0 ? k + m : max(a.window, abs(k - m));
  dm.nb = row_blocks(m, dm.W0);
  bool has_long = false;
  int longest = 8;  // bound on the pair's token lengths
  if (st == 0) {
    // every cell starts outside the band
    for (int q = t; q < ((k + 1) >> 1) * dm.nb; q += NT)
      reinterpret_cast<uint4*>(sm.tile)[q] = make_uint4(kOut4, kOut4, kOut4, kOut4);
    // stage every token: length and (if <= 8 bytes) its bytes
    int flag = 0;
    // U tokens in flight per thread, three dependent loads each
    auto stage = [&](int xb, auto unroll) {
      constexpr int U = decltype(unroll)::value;
      int id[U];
      int64_t o0[U], o1[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int x = xb + u * NT;
        id[u] = x < k                       ? a.draft_ids[d0 + x]
                : (x >= k8 && x < k8 + m) ? a.target_ids[t0 + x - k8]
                                            : 0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int x = xb + u * NT;
        const tt_vocab& v = x < k8 ? a.vd : a.vt;
        o0[u] = o1[u] = 0;
        if (x < k || (x >= k8 && x < k8 + m)) {
          if (id[u] < 0 || id[u] >= v.n_tokens) {
            flag |= TT_REQ_ID_OUT_OF_RANGE;
          } else {
            o0[u] = v.offsets[id[u]];
            o1[u] = v.offsets[id[u] + 1];
          }
        }
      }
      uint64_t packed[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const tt_vocab& v = xb + u * NT < k8 ? a.vd : a.vt;
        const int64_t n = o1[u] - o0[u];
        packed[u] = 0;
        if (o0[u] < 0 || o1[u] > v.n_bytes || n < 0) {
          flag |= TT_REQ_ID_OUT_OF_RANGE;
        } else if (n > TT_MAX_TOKEN_BYTES) {
          flag |= TT_REQ_TOO_LONG;
        } else if (n > 8) {
          flag |= kLongFlag;
          longest = max(longest, int(n));
        } else {
          packed[u] = load_packed8(v, o0[u], int(n));
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int x = xb + u * NT;
        const uint16_t ln = uint16_t(o1[u] - o0[u]);
        if (x < k8) {
          uint8_t* tr = reinterpret_cast<uint8_t*>(sm.trans) + (x >> 2) * 32 + (x & 3);
#pragma unroll
          for (int y = 0; y < 8; ++y) tr[4 * y] = uint8_t(packed[u] >> (8 * y));
          reinterpret_cast<uint8_t*>(sm.pmask)[x] = uint8_t((1u << min(int(ln), 8)) - 1u);
          if (x < k) sm.len_d[x] = ln;
        } else if (x < k8 + m) {
          sm.tok[x - k8] = packed[u];
          sm.len_t[x - k8] = ln;
        }
      }
    };
    if (k8 + m <= NT) {
      stage(t, Int<1>());
    } else {
      for (int xb = t; xb < k8 + m; xb += 4 * NT) stage(xb, Int<4>());
    }
    if (t < 8) sm.seen[t] = 0;
    flag = pair_or<WPP>(flag);  // (and the barrier after the staging stores)
    has_long = (flag & kLongFlag) != 0;
    if (has_long) longest = pair_max<WPP>(longest, sm.seen + 7);
    st = flag & ~kLongFlag;
  }
  if (st != 0) {
    for (int j = t; j < m; j += NT)
      if (a.map) a.map[t0 + j] = -1;
    for (int i = t; i < k; i += NT)
      if (a.need) a.need[d0 + i] = 0;
    if (t == 0) {
      a.status[b] = st;
      if (a.path_len) a.path_len[b] = 0;
      if (a.cost) a.cost[b] = -1;
    }
    return;
  }

  const int W0 = dm.W0, G = k8 >> 2;

  // 1. the distinct bytes of the target tokens, unless the pair is so small
  // that forming the match vectors where they are used costs less (at most
  // four columns x rows / 4 per lane). Byte c has the code of the number of
  // distinct bytes below it.
  bool coded = G * m > 128;
  if (coded) {
    for (int j = t; j < m; j += NT) {
      const int n = sm.len_t[j];
      uint64_t w = sm.tok[j];
      for (int y = 0; y < (n <= 8 ? n : 0); ++y, w >>= 8)
        atomicOr(&sm.seen[uint32_t(w & 255) >> 5], 1u << (uint32_t(w) & 31));
    }
    pair_sync<WPP>();
    int n_sym = 0;      // (the same on every thread)
    uint64_t rank = 0;  // distinct bytes below each word of `seen`, a byte each
#pragma unroll
    for (int y = 0; y < 8; ++y) {
      rank |= uint64_t(min(n_sym, 255)) << (8 * y);
      n_sym += __popc(sm.seen[y]);
    }
    coded = n_sym <= kSymCap;
    if (coded) {
      auto code_of = [&](uint32_t c) -> uint32_t {
        return (uint32_t(rank >> (8 * (c >> 5))) & 255u) +
               __popc(sm.seen[c >> 5] & ((1u << (c & 31)) - 1u));
      };
      for (int c = t; c < 256; c += NT)
        if (sm.seen[c >> 5] >> (c & 31) & 1u) sm.symch[code_of(c)] = uint8_t(c);
      for (int j = t; j < m; j += NT) {
        const int n = sm.len_t[j];
        uint64_t w = sm.tok[j], o = 0;
        for (int y = 0; y < (n <= 8 ? n : 0); ++y, w >>= 8)
          o |= uint64_t(code_of(uint32_t(w) & 255u)) << (8 * y);
        sm.tok[j] = o;
      }
      pair_sync<WPP>();
      // 2. match vectors of every code with every four rows
      for (int q = t; q < n_sym * G; q += NT) {
        const int sy = q / G, g = q - sy * G;
        const uint4* tr = reinterpret_cast<const uint4*>(sm.trans + 8 * g);
        sm.peq[q] = match4(tr[0], tr[1], sm.symch[sy]);
      }
    }
    pair_sync<WPP>();
  }

  // 3. banded local costs: a lane takes the rows of GR groups of four (two, or
  // one where the match vectors are formed on the spot) of one column, four
  // neighbouring lanes four columns. Lanes that share columns run equally long
  // (a column's loop is as long as its token), so a block of four columns' row
  // groups come one after the other. (Cells of longer tokens are set after.)
  auto fill = [&](auto groups, auto&& match) {
    constexpr int GR = decltype(groups)::value, NR = 4 * GR;
    // row groups that the band may touch; x / ng = x * inv >> 20 for x < 8192
    const int ng = min((k + NR - 1) / NR, (min(k, 2 * W0 + 4) + NR - 1) / NR + 1);
    const int n_task = ((m + 3) >> 2) * ng * 4;
    const uint32_t inv = ((1u << 20) + ng - 1) / ng;
    for (int q = t; q < n_task; q += NT) {
      const int cb = int((uint32_t(q >> 2) * inv) >> 20);
      const int g = (max(1, 4 * cb + 1 - W0) - 1) / NR + (q >> 2) - cb * ng;
      const int c = 4 * cb + (q & 3);  // column (0-based)
      const int r0 = max(0, c - W0 - NR * g), r1 = min(min(k, c + 1 + W0) - NR * g, NR);
      if (c >= m || r0 >= r1) continue;  // no row of the group is in the band
      const int lt = sm.len_t[c], n = min(lt, 8);
      const uint64_t w8 = sm.tok[c];
      uint32_t P[GR], M[GR], d[GR];
#pragma unroll
      for (int h = 0; h < GR; ++h) {
        P[h] = 0xffffffffu;
        M[h] = 0;
      }
      uint32_t w = uint32_t(w8);
#pragma unroll 1
      for (int y = 0; y < n; ++y) {
        uint32_t eq[GR];
        match(w & 255u, g, eq);
#pragma unroll
        for (int h = 0; h < GR; ++h) lev_step4(eq[h], P[h], M[h]);
        w = y == 3 ? uint32_t(w8 >> 32) : w >> 8;
      }
#pragma unroll
      for (int h = 0; h < GR; ++h) {
        // D(lp, lt) = lt + the vertical steps up to the token's last byte
        const uint32_t pm = sm.pmask[GR * g + h];
        d[h] = popc4(P[h] & pm) + uint32_t(n) * 0x01010101u - popc4(M[h] & pm);
      }
      // rows NR g + 2 h and the next one (0-based) are a pair; sigma = row + column
#pragma unroll
      for (int h = 0; h < 2 * GR; ++h) {
        const int p = 2 * GR * g + h;
        const uint32_t v = d[h >> 1] >> (16 * (h & 1));
        uint8_t* e = sm.tile + 16 * (p * dm.nb - first_block(p, W0)) + 2 * (2 * p + c);
        if (r0 <= 2 * h && 2 * h < r1) e[0] = uint8_t(v);
        if (r0 <= 2 * h + 1 && 2 * h + 1 < r1) e[3] = uint8_t(v >> 8);
      }
    }
  };
  if (coded) {
    fill(Int<2>(), [&](uint32_t code, int g, uint32_t (&eq)[2]) {
      const uint2 e = reinterpret_cast<const uint2*>(sm.peq)[code * (G >> 1) + g];
      eq[0] = e.x;
      eq[1] = e.y;
    });
  } else {
    fill(Int<1>(), [&](uint32_t c, int g, uint32_t (&eq)[1]) {
      const uint4* tr = reinterpret_cast<const uint4*>(sm.trans + 8 * g);
      eq[0] = match4(tr[0], tr[1], c);
    });
  }
  pair_sync<WPP>();
  if (has_long) {
    long_costs(a, d0, t0, sm, dm, t, NT);
    pair_sync<WPP>();
  }

  if (WPP > 1 && t >= 32) return;  // (the CTA meets again before the region is reused)

  // 4. the anti-diagonal sweep: the fewest row pairs per lane that fit
  int cstar;
  auto fits = [&](int np) { return k <= 64 * np || W0 <= 56 * np; };
  if (has_long && (longest > kMaxCost || (k + m) * longest > kPackedMax))
    cstar = sweep_wide(a, d0, t0, sm, dm, lane);
  else if (fits(1)) cstar = sweep<1>(sm, dm, lane);
  else if (WPP == 1 || fits(2)) cstar = sweep<2>(sm, dm, lane);  // (one warp: k <= 128)
  else cstar = sweep<4>(sm, dm, lane);
  __syncwarp();

  // 5. backtrack on lane 0, from (k, m) to (1, 1)
  int L = 0;
  if (lane == 0) {
    // The next cell's word is at one of three places that do not depend on this
    // cell's choice; only the selection waits for it. `row` is the place of
    // the row's pair at diagonal 0; sg = i + j - 2.
    int i = k, sg = k + m - 2;
    int row = ((k - 1) >> 1) * dm.nb - first_block((k - 1) >> 1, W0);
    int at = row + (sg >> 3);
    do {
      const uint32_t w = sm.dirs[at];
      // row i is half (i - 1) & 1; the block's first diagonal has the top bits
      const int sh = ((i - 1) & 1) * 16 + 14 - 2 * (sg & 7);
      const int q = (i - 1) >> 1;  // leaving the pair's first row: pair q - 1
      const int up = row + ((i & 1) ? first_block(q, W0) - first_block(q - 1, W0) - dm.nb : 0);
      const int a0 = up + ((sg - 2) >> 3), a1 = up + ((sg - 1) >> 3), a2 = row + ((sg - 1) >> 3);
      sm.path[L++] = (uint32_t(i) << 16) | uint32_t(sg + 2 - i);
      const int dir = (w >> sh) & 3;  // 0 diagonal, 1 (i-1, j), 2 (i, j-1)
      at = dir == 0 ? a0 : (dir == 1 ? a1 : a2);
      row = dir == 2 ? row : up;
      i -= dir == 2 ? 0 : 1;
      sg -= dir == 0 ? 2 : 1;
    } while (i >= 1 && sg + 2 - i >= 1 && L < k + m);
  }
  L = __shfl_sync(0xffffffffu, L, 0);
  for (int i = lane; i < k; i += 32)
    if (a.need) a.need[d0 + i] = 0;
  __syncwarp();

  // 6. outputs in forward order
  int32_t* pout = a.path ? a.path + 2 * (size_t(d0) + t0) : nullptr;
  for (int x = lane; x < L; x += 32) {
    const uint32_t cell = sm.path[L - 1 - x];
    const int i = int(cell >> 16), j = int(cell & 0xffffu);
    if (pout) {
      pout[2 * x] = i - 1;
      pout[2 * x + 1] = j - 1;
    }
    // last cell of column j on the path carries the largest i
    const bool last_in_col = x == L - 1 || int(sm.path[L - 2 - x] & 0xffffu) != j;
    if (last_in_col) {
      if (a.map) a.map[t0 + j - 1] = i - 1;
      if (a.need) a.need[d0 + i - 1] = 1;
    }
  }
  if (lane == 0) {
    a.status[b] = 0;
    if (a.path_len) a.path_len[b] = L;
    if (a.cost) a.cost[b] = cstar;
  }
}

// Forms of the kernel for large pairs, a CTA each (128 blocks of the cost tile,
// about 2048 cells, and more). Staging, match vectors and costs run on all
// warps, sweep and backtrack on one. 4096 pairs of 64 x 81 tokens without a
// band: 118 us with 4 warps per pair, 135 with 2, 176 with 1 (shared memory
// holds 16 pairs per SM, so more warps per pair mean more warps); 32 pairs of
// 256 x 325: 76 us with 16 warps, 80 with 8. One cell at a time on one warp per
// pair took 460 us and 1040 us.
constexpr int kAlignMid = 4;
constexpr int kAlignWide = 16;
// Shared memory per SM given to them in a step. The row pass keeps 30 MB in
// flight and an access takes over 6 us beside it, so few pairs at a time are
// slow: a step of 4096 pairs took 1.47 ms with 100 KB, 1.51 with 50, 1.73 with 30.
constexpr int kAlignRoom = 100 * 1024;

__host__ __device__ constexpr int align_threads(int wpp) {
  return wpp == 1 ? kAlignWarpsMax * 32 : wpp * 32;
}

// WPP warps per pair. With one, a CTA holds several pairs; before the row pass
// at most one such CTA per SM, whose warps loop over the pairs (the row pass's
// CTAs fit beside it and stream target rows while the pairs are aligned). With
// several, a CTA holds one pair at a time.
template <int WPP>
__global__ void __launch_bounds__(align_threads(WPP), 1024 / align_threads(WPP))
    align_kernel(const __grid_constant__ AlignArgs a) {
  extern __shared__ __align__(16) char smem_raw[];
  // the row pass may start streaming target rows now; it waits for this grid
  // before it reads the needed-draft-row flags
  if (a.after_grid) grid_dependency_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (a.work && blockIdx.x == 0 && threadIdx.x < kWorkShards)
    a.work[threadIdx.x * kWorkStride] = a.work[threadIdx.x * kWorkStride + kNucWork] =
        0ull;  // read after this grid ends
  if constexpr (WPP == 1) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    char* region = smem_raw + size_t(warp) * a.smem_per_pair;
    for (int b = blockIdx.x * a.pairs_per_block + warp; b < a.B;
         b += int(gridDim.x) * a.pairs_per_block) {
      align_pair<1>(a, b, region, lane);
      __syncwarp();  // the region is reused by the warp's next pair
    }
  } else {
    for (int b = blockIdx.x; b < a.B; b += int(gridDim.x)) {
      align_pair<WPP>(a, b, smem_raw, threadIdx.x);
      __syncthreads();  // the region is reused by the next pair
    }
  }
}

}  // namespace

// The band's half-width as the kernel takes it. |i - j| of a pair is below
// TT_MAX_K + TT_MAX_M, so wider bands (any w >= 0 is allowed) are that band, and
// the kernel's and the tile's arithmetic on twice the width fits an int.
int align_window(int window) { return min(window, TT_MAX_K + TT_MAX_M); }

// Blocks of the cost tile that a pair of k <= max_k and m <= max_m tokens can
// need: (k + 1) / 2 row pairs of row_blocks(m, W0), W0 = max(window, |k - m|).
// For a given k, the row grows with m while m >= k (so m = max_m is the
// longest there); for m < k, 2 (k - m) + 2 falls while m grows, so a row has
// at most max(2 window, 2 k / 3) + 4 band columns, and never more than k.
int align_tile_blocks(int max_k, int max_m, int window) {
  window = align_window(window);
  int most = 0;
  for (int k = 1; k <= max_k; ++k) {
    int w;
    if (window < 0) {
      w = row_blocks(max_m, k + max_m);
    } else {
      w = max_m >= k ? row_blocks(max_m, max(window, max_m - k)) : 0;
      w = max(w, ((min(min(k, max_m), max(2 * window, 2 * k / 3) + 4) + 15) >> 3) | 1);
    }
    most = max(most, (k + 1) / 2 * w);
  }
  return most;
}

size_t align_smem_per_pair(int max_k, int max_m, int tile_blocks) {
  return carve(nullptr, max_k, max_m, tile_blocks).bytes;
}

cudaError_t preload_align() {
  const void* const kernels[] = {reinterpret_cast<const void*>(align_kernel<1>),
                                 reinterpret_cast<const void*>(align_kernel<kAlignMid>),
                                 reinterpret_cast<const void*>(align_kernel<kAlignWide>)};
  for (const void* f : kernels) {
    const cudaError_t e =
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kAlignSmemMax);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int WPP>
static cudaError_t launch_align_t(const AlignArgs& a, int blocks, int warps, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(blocks));
  cfg.blockDim = dim3(unsigned(warps * 32));
  cfg.dynamicSmemBytes = a.smem_per_pair * size_t(a.pairs_per_block);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = a.after_grid;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, align_kernel<WPP>, a);
}

cudaError_t launch_align(const AlignArgs& args, cudaStream_t stream) {
  static int n_sm[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (n_sm[dev] == 0 &&
      cudaDeviceGetAttribute(&n_sm[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    n_sm[dev] = 148;
  AlignArgs a = args;
  const int64_t sms = n_sm[dev];
  // Large pairs: a CTA per pair, of kAlignMid warps, or of kAlignWide warps
  // where one such CTA per pair would leave the chip idle (at most two pairs
  // per SM) and for drafts whose sweep needs four row pairs per lane. Before
  // the row pass as many CTAs as kAlignRoom holds per SM, which
  // loop over the pairs.
  if (a.tile_blocks >= 128) {
    a.pairs_per_block = 1;
    const int64_t in_step = sms * std::max<int64_t>(1, kAlignRoom / int64_t(a.smem_per_pair));
    const int blocks = int(a.work ? std::min<int64_t>(a.B, in_step) : a.B);
    return a.max_k > 128 || a.B <= 2 * sms
               ? launch_align_t<kAlignWide>(a, blocks, kAlignWide, stream)
               : launch_align_t<kAlignMid>(a, blocks, kAlignMid, stream);
  }
  // Small pairs: a warp each, spread over the SMs while the batch is small.
  // Before the row pass at most one CTA of kAlignWarpsStep warps per SM, whose
  // warps loop over the pairs, so that the row pass's CTAs fit beside it and
  // stream target rows while it runs; an alignment on its own takes as many
  // CTAs as fit.
  const int spread = int((a.B + sms - 1) / sms);
  const int most = std::min(a.work ? kAlignWarpsStep : kAlignWarpsMax, spread);
  a.pairs_per_block =
      std::max(1, std::min(most, int((a.work ? 30 * 1024 : kAlignRoom) / a.smem_per_pair)));
  const int per_pair = (a.B + a.pairs_per_block - 1) / a.pairs_per_block;
  const int blocks = a.work ? int(std::min<int64_t>(per_pair, sms)) : per_pair;
  return launch_align_t<1>(a, blocks, a.pairs_per_block, stream);
}

}  // namespace tt
