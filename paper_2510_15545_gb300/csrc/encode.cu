// encode.cu -- re-encoding of the draft string into target tokens (§4.2,
// App. A.1), the Lemma-1 byte check (App. A.1) and the delta-pos histogram of
// the DTW paths (§4.1, App. K).
//
// Re-encoding is greedy longest match over the target vocabulary, through an
// index of every prefix of every token: an open-addressing table whose slot
// holds the prefix's key, its length and the token it spells exactly (if any).
// A match at position p ends before the first prefix of the text that no token
// starts with. One CTA per request decodes the draft and matches a position per
// thread; a second kernel turns the per-request counts into CSR offsets and
// compacts the tokens.
//
// Both are bound by dependent accesses, not by bytes: a position's prefixes of
// up to eight bytes, whose keys are the bytes themselves, are therefore probed
// all at once. 256 requests of 16 draft tokens: encode 11 us and finish 4.7 us
// with cold caches; a warp per request probing one prefix after another, with a
// scan and a compaction kernel behind it, took 35, 3.5 and 3.2 us.
#include <cstdint>
#include <cstring>
#include <vector>

#include "tt_device.cuh"
#include "tt_f2.cuh"
#include "tt_launch.h"

namespace tt {

namespace {

// ------------------------------------------------------------- the index

struct IndexHeader {
  uint32_t magic;
  int32_t n_slots;   // power of two
  int32_t max_len;   // longest token in bytes
  int32_t n_tokens;
  int64_t reserved[6];
};

struct Slot {
  uint64_t key;  // the prefix's bytes (up to 8) or its fingerprint (longer)
  int32_t len;   // prefix length in bytes; 0 = empty slot
  int32_t id;    // token spelled by exactly this prefix, -1 = none
};

static_assert(sizeof(IndexHeader) == 64 && sizeof(Slot) == 16, "index layout");
constexpr uint32_t kIndexMagic = 0x58495454u;
constexpr int kMaxIndexTokens = 1 << 22;  // ids fit 22 bits beside a 9-bit length

// MurmurHash3's 64-bit finaliser (A. Appleby, public domain).
__host__ __device__ __forceinline__ uint64_t fmix64(uint64_t x) {
  x ^= x >> 33;
  x *= 0xff51afd7ed558ccdull;
  x ^= x >> 33;
  x *= 0xc4ceb9fe1a85ec53ull;
  x ^= x >> 33;
  return x;
}

// Key of a prefix of length L from the key of its first L-1 bytes: the bytes
// themselves (little-endian) up to 8, then a chained fingerprint.
__host__ __device__ __forceinline__ uint64_t key_step(uint64_t key, uint8_t byte, int L) {
  if (L <= 8) return key | (uint64_t(byte) << (8 * (L - 1)));
  return fmix64(key + uint64_t(byte) * 0x9e3779b97f4a7c15ull + uint64_t(L));
}

__host__ __device__ __forceinline__ uint32_t home_slot(uint64_t key, int L, int n_slots) {
  return uint32_t(fmix64(key ^ (uint64_t(L) * 0xc2b2ae3d27d4eb4full))) & uint32_t(n_slots - 1);
}

size_t slots_for(int64_t n_bytes) {
  const size_t need = size_t(2 * (n_bytes > 0 ? n_bytes : 1));
  size_t s = 16;
  while (s < need) s <<= 1;
  return s;
}

// ------------------------------------------------------------- re-encoding

constexpr int kEncThreads = 128;

struct EncArgs {
  int B, n_draft, max_m;
  const int32_t* draft_off;
  const int32_t* draft_ids;
  tt_vocab vd, vt;
  const IndexHeader* hdr;
  const Slot* slots;
  int32_t* pad_ids;  // [B * max_m]
  int32_t* counts;   // [B]
  int32_t* status;   // [B]
};

__device__ __forceinline__ bool token_ok(const tt_vocab& v, int id) {
  if (id < 0 || id >= v.n_tokens) return false;
  const int64_t o0 = v.offsets[id], o1 = v.offsets[id + 1];
  return o0 >= 0 && o1 >= o0 && o1 <= v.n_bytes;
}

// Token `id` of vt spells s[0..L).
__device__ bool spells(const tt_vocab& vt, int id, const uint8_t* s, int L) {
  const int64_t o0 = vt.offsets[id];
  if (vt.offsets[id + 1] - o0 != L) return false;
  for (int x = 0; x < L; ++x)
    if (vt.bytes[o0 + x] != s[x]) return false;
  return true;
}

// Copies len bytes, eight loads in flight at a time, as far as they lie before dst_end.
__device__ __forceinline__ void copy_token(uint8_t* dst, const uint8_t* dst_end,
                                           const uint8_t* src, int len) {
  for (int x0 = 0; x0 < len; x0 += 8) {
    uint8_t v[8];
#pragma unroll
    for (int x = 0; x < 8; ++x) v[x] = x0 + x < len ? src[x0 + x] : uint8_t(0);
#pragma unroll
    for (int x = 0; x < 8; ++x)
      if (x0 + x < len && dst + x0 + x < dst_end) dst[x0 + x] = v[x];
  }
}

// Longest match of the text at s with at most lim bytes: (token id << 9) |
// length, 0 = none. Prefixes of up to eight bytes are probed together, one slot
// of each per round, until each is found or reaches an empty slot; a prefix that
// no token starts with ends the longer ones too. Longer prefixes are walked.
__device__ int longest_match(const EncArgs& a, const uint8_t* s, int lim, int n_slots) {
  constexpr int kKeys = 8;
  const uint32_t mask = uint32_t(n_slots - 1);
  uint64_t text = 0;
#pragma unroll
  for (int x = 0; x < kKeys; ++x)
    if (x < lim) text |= uint64_t(s[x]) << (8 * x);
  auto key_of = [&](int L) { return text & (~0ull >> (64 - 8 * L)); };
  uint32_t at[kKeys];
  int id[kKeys];  // token of each prefix found (-1: none)
#pragma unroll
  for (int x = 0; x < kKeys; ++x) {
    at[x] = home_slot(key_of(x + 1), x + 1, n_slots);
    id[x] = -1;
  }
  int open_to = max(0, min(kKeys, lim));       // prefixes that may still be found
  uint32_t open = (1u << open_to) - 1;         // bit L - 1: not settled yet
  for (int probe = 0; open && probe < n_slots; ++probe) {  // the table is at most half full
    uint4 sl[kKeys];
#pragma unroll
    for (int x = 0; x < kKeys; ++x)
      if ((open >> x) & 1u) sl[x] = *reinterpret_cast<const uint4*>(a.slots + at[x]);
#pragma unroll
    for (int x = 0; x < kKeys; ++x) {
      if (!((open >> x) & 1u)) continue;
      const uint64_t key = uint64_t(sl[x].x) | (uint64_t(sl[x].y) << 32);
      if (int(sl[x].z) == 0) {
        open_to = min(open_to, x);
        open &= (1u << x) - 1;
      } else if (int(sl[x].z) == x + 1 && key == key_of(x + 1)) {
        id[x] = int(sl[x].w);
        open &= ~(1u << x);
      } else {
        at[x] = (at[x] + 1) & mask;
      }
    }
  }
  if (open) open_to = min(open_to, __ffs(open) - 1);  // (no empty slot: never a built table)
  int best = 0;
#pragma unroll
  for (int x = 0; x < kKeys; ++x)
    // (an id past vt's table means the index belongs to another vocabulary)
    if (x < open_to && id[x] >= 0 && id[x] < a.vt.n_tokens) best = (id[x] << 9) | (x + 1);
  if (open_to < kKeys) return best;
  uint64_t key = text;
  for (int L = kKeys + 1; L <= lim; ++L) {
    key = key_step(key, s[L - 1], L);
    uint32_t h = home_slot(key, L, n_slots);
    int found = -2;  // -2: no token starts with these L bytes
    for (int probe = 0; probe < n_slots; ++probe) {
      const Slot sl = a.slots[h];
      if (sl.len == 0) break;
      if (sl.len == L && sl.key == key) {
        found = sl.id;
        break;
      }
      h = (h + 1) & mask;
    }
    if (found == -2) break;
    if (found >= 0 && found < a.vt.n_tokens && spells(a.vt, found, s, L)) best = (found << 9) | L;
  }
  return best;
}

__global__ void __launch_bounds__(kEncThreads) encode_kernel(EncArgs a) {
  constexpr int kWarps = kEncThreads / 32;
  __shared__ uint8_t text[TT_MAX_ENCODE_BYTES];
  // longest match at each position: (token id << 9) | length, 0 = none
  __shared__ int32_t match[TT_MAX_ENCODE_BYTES];
  __shared__ int s_wsum[kWarps];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int b = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  int st = 0, k = 0, d0 = 0, m = 0;
  const bool index_ok = a.hdr->magic == kIndexMagic && a.hdr->n_slots >= 16 &&
                        (a.hdr->n_slots & (a.hdr->n_slots - 1)) == 0;
  const int max_len = a.hdr->max_len, n_slots = a.hdr->n_slots;
  if (!csr_ok(a.draft_off, b, a.n_draft)) {
    st = TT_REQ_BAD_OFFSETS;
  } else {
    d0 = a.draft_off[b];
    k = a.draft_off[b + 1] - d0;
    if (k == 0) st |= TT_REQ_EMPTY;
  }
  int n = 0;
  if (st == 0) {
    // decode_d: the draft tokens' bytes, a token per thread and round
    int bad = 0;
    int64_t base = 0;
    for (int r = 0; r < k; r += kEncThreads) {
      const int i = r + tid;
      int64_t o0 = 0, len64 = 0;
      if (i < k) {
        const int id = a.draft_ids[d0 + i];
        if (token_ok(a.vd, id)) {
          o0 = a.vd.offsets[id];
          len64 = a.vd.offsets[id + 1] - o0;
        } else {
          bad = 1;
        }
      }
      // (a longer token makes the request too long all the same)
      const int len = int(min(len64, int64_t(TT_MAX_ENCODE_BYTES + 1)));
      int incl = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      if (lane == 31) s_wsum[warp] = incl;
      __syncthreads();
      int before = 0, all = 0;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        if (w < warp) before += s_wsum[w];
        all += s_wsum[w];
      }
      __syncthreads();
      const int64_t start = base + before + incl - len;
      if (start < TT_MAX_ENCODE_BYTES)
        copy_token(text + start, text + TT_MAX_ENCODE_BYTES, a.vd.bytes + o0, len);
      base += all;
    }
    if (__syncthreads_or(bad)) st |= TT_REQ_ID_OUT_OF_RANGE;
    else if (base > TT_MAX_ENCODE_BYTES) st |= TT_REQ_TOO_LONG;
    n = int(min(base, int64_t(TT_MAX_ENCODE_BYTES)));
  }
  if (st == 0 && !index_ok) st = TT_REQ_INTERNAL;
  if (st == 0) {
    // the longest target token at every position
    for (int p = tid; p < n; p += kEncThreads)
      match[p] = longest_match(a, text + p, min(max_len, n - p), n_slots);
    __syncthreads();
    // encode_t: greedy walk over the matches
    if (tid == 0) {
      int p = 0;
      while (p < n) {
        const int mt = match[p];
        if (mt == 0) {
          st |= TT_REQ_NO_MATCH;
          break;
        }
        if (m >= a.max_m) {
          st |= TT_REQ_TOO_LONG;
          break;
        }
        a.pad_ids[int64_t(b) * a.max_m + m] = mt >> 9;
        ++m;
        p += mt & 511;
      }
    }
  }
  if (tid == 0) {
    a.counts[b] = st == 0 ? m : 0;
    a.status[b] = st;
  }
}

struct FinArgs {
  int B, max_m, capacity;
  const int32_t* pad_ids;
  const int32_t* counts;
  int32_t* status;
  int32_t* target_off;
  int32_t* target_ids;
};

constexpr int kFinThreads = 256;
constexpr int kFinCtas = 152;  // one per SM of a GB300 (any number gives the same result)

// Inclusive block scan of one int64 per thread; returns the block total in *total.
__device__ int64_t block_scan(int64_t v, int64_t* s_warp, int64_t* total) {
  constexpr int kWarps = kFinThreads / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t n = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += n;
  }
  if (lane == 31) s_warp[warp] = v;
  __syncthreads();
  int64_t before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    if (w < warp) before += s_warp[w];
    all += s_warp[w];
  }
  __syncthreads();
  *total = all;
  return v + before;
}

// CSR offsets with the capacity rule, and the compaction of the padded tokens.
// Each CTA takes a block of requests and adds up the counts of all before it
// (they lie in L2; a grid of one CTA per SM reads them 152 times at most),
// which saves a scan kernel between the two. A request is written while the
// running count, its own included, is within the capacity.
__global__ void __launch_bounds__(kFinThreads) encode_finish_kernel(FinArgs a) {
  __shared__ int64_t s_warp[kFinThreads / 32];
  __shared__ int32_t s_to[kFinThreads], s_n[kFinThreads];
  __shared__ int s_written;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b0 = int(int64_t(a.B) * blockIdx.x / gridDim.x);
  const int b1 = int(int64_t(a.B) * (blockIdx.x + 1) / gridDim.x);
  grid_dependency_wait();
  if (blockIdx.x == 0 && tid == 0) a.target_off[0] = 0;
  int64_t sum = 0, base, tot;
#pragma unroll 8
  for (int b = tid; b < b0; b += kFinThreads) sum += a.counts[b];
  block_scan(sum, s_warp, &base);
  // entries written before this block: all, or up to the last request that fits
  int written = int(min(base, int64_t(a.capacity)));
  if (base > a.capacity) {
    if (tid == 0) s_written = 0;
    int64_t run = 0;
    for (int c = 0; c < b0; c += kFinThreads) {
      const int b = c + tid;
      const int64_t end = run + block_scan(b < b0 ? a.counts[b] : 0, s_warp, &tot);
      if (end <= a.capacity) atomicMax(&s_written, int(end));
      run += tot;
      if (run > a.capacity) break;
    }
    __syncthreads();
    written = s_written;
  }
  for (int c = b0; c < b1; c += kFinThreads) {
    const int b = c + tid;
    const int cnt = b < b1 ? a.counts[b] : 0;
    if (tid == 0) s_written = written;
    const int64_t end = base + block_scan(cnt, s_warp, &tot);
    base += tot;
    const bool fits = end <= a.capacity;
    if (fits) atomicMax(&s_written, int(end));
    s_to[tid] = int(end) - cnt;
    s_n[tid] = fits ? cnt : 0;
    __syncthreads();
    written = s_written;  // (running counts never fall: later ends are at least these)
    if (b < b1) {
      const int st = a.status[b];
      if (st == 0 && !fits) a.status[b] = st | TT_REQ_TOO_LONG;
      a.target_off[b + 1] = fits ? int(end) : written;
    }
    for (int q = warp; q < min(kFinThreads, b1 - c); q += kFinThreads / 32)
      for (int j = lane; j < s_n[q]; j += 32)
        a.target_ids[s_to[q] + j] = a.pad_ids[int64_t(c + q) * a.max_m + j];
    __syncthreads();
  }
}

// ------------------------------------------------------- Lemma-1 byte check

constexpr int kConsThreads = 128;

struct ConsArgs {
  int B, n_draft, n_target, max_k, max_m;
  const int32_t* draft_off;
  const int32_t* draft_ids;
  const int32_t* target_off;
  const int32_t* target_ids;
  tt_vocab vd, vt;
  int32_t* status;
};

// One warp: the tokens' starts in the table (at) and the inclusive prefix sums
// of their byte lengths in pre[1..n] (pre[0] = 0), for n <= cap tokens; whether
// all ids are good.
__device__ bool byte_prefix(const tt_vocab& v, const int32_t* ids, int n, int cap, int32_t* pre,
                            int64_t* at, int lane) {
  int base = 0, bad = 0;
  if (lane == 0) pre[0] = 0;
  for (int r = 0; r < n; r += 32) {
    const int i = r + lane;
    int64_t o0 = 0;
    int len = 0;
    if (i < n) {
      const int id = ids[i];
      if (token_ok(v, id)) {
        o0 = v.offsets[id];
        len = int(v.offsets[id + 1] - o0);
      } else {
        bad = 1;
      }
    }
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    if (i < min(n, cap)) {
      pre[i + 1] = base + incl;
      at[i] = o0;
    }
    base += __shfl_sync(0xffffffffu, incl, 31);
  }
  return !__any_sync(0xffffffffu, bad);
}

// Byte at position p of the concatenation (pre: prefix sums of n tokens).
__device__ __forceinline__ uint8_t byte_at(const tt_vocab& v, const int64_t* at,
                                           const int32_t* pre, int n, int p) {
  int lo = 0, hi = n - 1;  // last token whose start is <= p
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= p) lo = mid;
    else hi = mid - 1;
  }
  return v.bytes[at[lo] + (p - pre[lo])];
}

// One CTA per request: a warp for each side's prefix sums, then a byte per
// thread, found through tables in shared memory so that each costs one access
// (13 us for 256 requests with a warp per request and three dependent accesses
// per byte, 6 us now, cold).
__global__ void __launch_bounds__(kConsThreads) consistency_kernel(ConsArgs a) {
  __shared__ int32_t s_pd[TT_MAX_K + 1], s_pt[TT_MAX_M + 1];
  __shared__ int64_t s_ad[TT_MAX_K], s_at[TT_MAX_M];
  const int b = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int st = 0;
  if (!csr_ok(a.draft_off, b, a.n_draft) || !csr_ok(a.target_off, b, a.n_target)) {
    if (tid == 0) a.status[b] = TT_REQ_BAD_OFFSETS;
    return;
  }
  const int d0 = a.draft_off[b], k = a.draft_off[b + 1] - d0;
  const int t0 = a.target_off[b], m = a.target_off[b + 1] - t0;
  if (k > a.max_k || m > a.max_m) st |= TT_REQ_TOO_LONG;
  bool good = true;
  if (warp == 0) good = byte_prefix(a.vd, a.draft_ids + d0, k, TT_MAX_K, s_pd, s_ad, lane);
  if (warp == 1) good = byte_prefix(a.vt, a.target_ids + t0, m, TT_MAX_M, s_pt, s_at, lane);
  if (__syncthreads_or(!good)) st |= TT_REQ_ID_OUT_OF_RANGE;
  if (st == 0) {
    const int nd = s_pd[k], nt = s_pt[m];
    int diff = nd != nt;
    for (int p = tid; !diff && p < nd; p += kConsThreads)
      diff = byte_at(a.vd, s_ad, s_pd, k, p) != byte_at(a.vt, s_at, s_pt, m, p);
    if (__syncthreads_or(diff)) st |= TT_REQ_INCONSISTENT;
  }
  if (tid == 0) a.status[b] = st;
}

// --------------------------------------------------- delta-pos histogram

// Two CTAs per SM at most, as each adds its bins to the global ones; a request
// is a chain of three dependent accesses, so a CTA has sixteen warps where four
// would have to take several requests in turn (4096 requests of 64 tokens: 10.6
// us with four warps, 5.0 with sixteen; 32 requests: 6.0 with either, and 0.6 us
// less around it with four).
constexpr int kDposWarps = 4, kDposWarpsMany = 16;
constexpr int kDposFly = 4;  // entries in flight per lane

struct DposArgs {
  int B, n_draft, n_target, mode, n_bins;
  const int32_t* draft_off;
  const int32_t* target_off;
  const int32_t* path;
  const int32_t* path_len;
  const int32_t* map;
  unsigned long long* hist;
};

__global__ void __launch_bounds__(32 * kDposWarpsMany) dpos_kernel(DposArgs a) {
  __shared__ unsigned int s_hist[TT_MAX_DPOS_BINS];
  for (int x = threadIdx.x; x < a.n_bins; x += blockDim.x) s_hist[x] = 0;
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const int top = a.n_bins - 1;
  for (int b = blockIdx.x * warps + warp; b < a.B; b += gridDim.x * warps) {
    if (!csr_ok(a.draft_off, b, a.n_draft) || !csr_ok(a.target_off, b, a.n_target)) continue;
    const int d0 = a.draft_off[b], k = a.draft_off[b + 1] - d0;
    const int t0 = a.target_off[b], m = a.target_off[b + 1] - t0;
    const int len = min(a.path_len[b], k + m);  // the request's path capacity
    if (len <= 0) continue;
    if (a.mode == 0) {
      const int32_t* pp = a.path + 2 * (int64_t(d0) + t0);
      for (int x0 = lane; x0 < len; x0 += 32 * kDposFly) {
        int d[kDposFly];
#pragma unroll
        for (int q = 0; q < kDposFly; ++q) {
          const int x = x0 + 32 * q;
          d[q] = x < len ? abs(pp[2 * x] - pp[2 * x + 1]) : -1;
        }
#pragma unroll
        for (int q = 0; q < kDposFly; ++q)
          if (x0 + 32 * q < len) atomicAdd(&s_hist[min(d[q], top)], 1u);
      }
    } else {
      for (int j = lane; j < m; j += 32) {
        const int d = abs(a.map[t0 + j] - j);
        atomicAdd(&s_hist[min(d, top)], 1u);
      }
    }
  }
  __syncthreads();
  for (int x = threadIdx.x; x < a.n_bins; x += blockDim.x)
    if (s_hist[x]) atomicAdd(&a.hist[x], (unsigned long long)s_hist[x]);
}

bool batch_ok_lite(const tt_batch* b) {
  if (!b || b->B < 0 || b->n_draft < 0 || b->n_target < 0) return false;
  if (b->B == 0) return true;
  return b->draft_off && b->target_off && b->max_k >= 1 && b->max_k <= TT_MAX_K &&
         b->max_m >= 1 && b->max_m <= TT_MAX_M;
}

bool vocab_ok_lite(const tt_vocab* v) {
  return v && v->bytes && v->offsets && v->n_tokens >= 1 && v->n_bytes >= 0;
}

}  // namespace
}  // namespace tt

using namespace tt;

extern "C" size_t tt_vocab_index_bytes(int32_t n_tokens, int64_t n_bytes) {
  (void)n_tokens;
  return sizeof(IndexHeader) + slots_for(n_bytes) * sizeof(Slot);
}

extern "C" tt_status tt_vocab_index_build(const uint8_t* bytes, const int64_t* offsets,
                                          int32_t n_tokens, void* index, size_t index_bytes) {
  if (!offsets || !index || n_tokens < 1 || n_tokens > kMaxIndexTokens) return TT_ERR_INVALID_ARG;
  int64_t total = 0, max_len = 0;
  for (int32_t v = 0; v < n_tokens; ++v) {
    const int64_t len = offsets[v + 1] - offsets[v];
    if (offsets[v] < 0 || len < 0) return TT_ERR_INVALID_ARG;
    if (len > TT_MAX_TOKEN_BYTES) return TT_ERR_UNSUPPORTED;
    total += len;
    if (len > max_len) max_len = len;
  }
  if (total > 0 && !bytes) return TT_ERR_INVALID_ARG;
  if (index_bytes < sizeof(IndexHeader) + 16 * sizeof(Slot)) return TT_ERR_INVALID_ARG;
  size_t n_slots = 16;
  while (n_slots * 2 * sizeof(Slot) + sizeof(IndexHeader) <= index_bytes) n_slots *= 2;
  if (n_slots < size_t(2 * total) || n_slots > (size_t(1) << 30)) return TT_ERR_INVALID_ARG;

  IndexHeader* hdr = static_cast<IndexHeader*>(index);
  Slot* slots = reinterpret_cast<Slot*>(static_cast<char*>(index) + sizeof(IndexHeader));
  std::memset(index, 0, sizeof(IndexHeader) + n_slots * sizeof(Slot));
  std::vector<int32_t> owner(n_slots, -1);  // a token whose prefix created the slot
  const uint32_t mask = uint32_t(n_slots - 1);
  for (int32_t v = 0; v < n_tokens; ++v) {  // in id order: the smallest id keeps a string
    const uint8_t* s = bytes + offsets[v];
    const int len = int(offsets[v + 1] - offsets[v]);
    uint64_t key = 0;
    for (int L = 1; L <= len; ++L) {
      key = key_step(key, s[L - 1], L);
      uint32_t h = home_slot(key, L, int(n_slots));
      for (;;) {
        Slot& sl = slots[h];
        if (sl.len == 0) {
          sl.key = key;
          sl.len = L;
          sl.id = L == len ? v : -1;
          owner[h] = v;
          break;
        }
        if (sl.len == L && sl.key == key) {
          if (L > 8 && std::memcmp(bytes + offsets[owner[h]], s, size_t(L)) != 0)
            return TT_ERR_UNSUPPORTED;  // two different prefixes share a fingerprint
          if (L == len && sl.id < 0) sl.id = v;
          break;
        }
        h = (h + 1) & mask;
      }
    }
  }
  hdr->magic = kIndexMagic;
  hdr->n_slots = int32_t(n_slots);
  hdr->max_len = int32_t(max_len);
  hdr->n_tokens = n_tokens;
  return TT_OK;
}

extern "C" size_t tt_encode_workspace_bytes(int32_t B, int32_t max_m) {
  if (B < 0 || max_m < 0) return 0;
  return align256(sizeof(int32_t) * size_t(B) * size_t(max_m)) +
         align256(sizeof(int32_t) * size_t(B > 0 ? B : 1));
}

extern "C" tt_status tt_encode(int32_t B, int32_t n_draft, const int32_t* draft_off,
                               const int32_t* draft_ids,
                               const tt_vocab* vd, const tt_vocab* vt, const void* vt_index,
                               int32_t max_m, int32_t capacity, int32_t* target_off,
                               int32_t* target_ids, int32_t* status, void* workspace,
                               size_t workspace_bytes, void* stream) {
  if (B < 0 || n_draft < 0 || !target_off || max_m < 1 || max_m > TT_MAX_M || capacity < 0)
    return TT_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (B == 0) {
    const cudaError_t e = cudaMemsetAsync(target_off, 0, sizeof(int32_t), s);
    return e == cudaSuccess ? TT_OK : record_cuda_error(e);
  }
  if (!draft_off || (n_draft > 0 && !draft_ids) || !status || !vt_index ||
      (capacity > 0 && !target_ids) ||
      !vocab_ok_lite(vd) || !vocab_ok_lite(vt))
    return TT_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(vt_index) & 15) != 0) return TT_ERR_INVALID_ARG;
  if (!workspace || workspace_bytes < tt_encode_workspace_bytes(B, max_m) ||
      (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
    return TT_ERR_INVALID_ARG;
  EncArgs a;
  a.B = B;
  a.n_draft = n_draft;
  a.max_m = max_m;
  a.draft_off = draft_off;
  a.draft_ids = draft_ids;
  a.vd = *vd;
  a.vt = *vt;
  a.hdr = static_cast<const IndexHeader*>(vt_index);
  a.slots = reinterpret_cast<const Slot*>(static_cast<const char*>(vt_index) + sizeof(IndexHeader));
  a.pad_ids = static_cast<int32_t*>(workspace);
  a.counts = reinterpret_cast<int32_t*>(static_cast<char*>(workspace) +
                                        align256(sizeof(int32_t) * size_t(B) * size_t(max_m)));
  a.status = status;
  encode_kernel<<<B, kEncThreads, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return record_cuda_error(e);
  FinArgs f;
  f.B = B;
  f.max_m = max_m;
  f.capacity = capacity;
  f.pad_ids = a.pad_ids;
  f.counts = a.counts;
  f.status = status;
  f.target_off = target_off;
  f.target_ids = target_ids;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(B < kFinCtas ? B : kFinCtas));
  cfg.blockDim = dim3(kFinThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, encode_finish_kernel, f);
  return e == cudaSuccess ? TT_OK : record_cuda_error(e);
}

extern "C" tt_status tt_consistency(const tt_batch* batch, const tt_vocab* vd, const tt_vocab* vt,
                                    int32_t* status, void* stream) {
  if (!batch_ok_lite(batch)) return TT_ERR_INVALID_ARG;
  if (batch->B == 0) return TT_OK;
  if (!status || !vocab_ok_lite(vd) || !vocab_ok_lite(vt) ||
      (batch->n_draft > 0 && !batch->draft_ids) || (batch->n_target > 0 && !batch->target_ids))
    return TT_ERR_INVALID_ARG;
  ConsArgs a;
  a.B = batch->B;
  a.n_draft = batch->n_draft;
  a.n_target = batch->n_target;
  a.max_k = batch->max_k;
  a.max_m = batch->max_m;
  a.draft_off = batch->draft_off;
  a.draft_ids = batch->draft_ids;
  a.target_off = batch->target_off;
  a.target_ids = batch->target_ids;
  a.vd = *vd;
  a.vt = *vt;
  a.status = status;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  consistency_kernel<<<a.B, kConsThreads, 0, s>>>(a);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? TT_OK : record_cuda_error(e);
}

extern "C" tt_status tt_dpos_hist(const tt_batch* batch, const int32_t* path,
                                  const int32_t* path_len, const int32_t* map, int32_t mode,
                                  int32_t n_bins, int64_t* hist, void* stream) {
  if (!batch_ok_lite(batch) || (mode != 0 && mode != 1) || n_bins < 1 ||
      n_bins > TT_MAX_DPOS_BINS || !hist)
    return TT_ERR_INVALID_ARG;
  if (batch->B == 0) return TT_OK;
  if (!path_len || (mode == 0 && !path) || (mode == 1 && batch->n_target > 0 && !map))
    return TT_ERR_INVALID_ARG;
  DposArgs a;
  a.B = batch->B;
  a.n_draft = batch->n_draft;
  a.n_target = batch->n_target;
  a.mode = mode;
  a.n_bins = n_bins;
  a.draft_off = batch->draft_off;
  a.target_off = batch->target_off;
  a.path = path;
  a.path_len = path_len;
  a.map = map;
  a.hist = reinterpret_cast<unsigned long long*>(hist);
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess)
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int warps = a.B > 2 * sms * kDposWarps ? kDposWarpsMany : kDposWarps;
  const int want = (a.B + warps - 1) / warps;
  const int grid = want < 2 * sms ? want : 2 * sms;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  dpos_kernel<<<grid, 32 * warps, 0, s>>>(a);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? TT_OK : record_cuda_error(e);
}
