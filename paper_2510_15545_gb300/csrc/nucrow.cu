// nucrow.cu -- nucleus rows (top-p without top-k, App. F) of more than
// kNucRowUnits units of 8 KB: every row streamed from HBM once and its kept set
// found from what the CTA holds of it.
//
// One CTA per SM, three roles:
//  - a scheduling lane names the CTA's rows, up to kQueue ahead;
//  - kSW streaming warps, each with a stage of its own into which it copies its
//    next 8 KB unit (a 1-D bulk copy) as soon as it has worked through one: the
//    row's maximum so far, the chunks' partials (compensated sums), and the
//    candidates -- the logits within kCandDelta = 14 log2 units of the largest
//    seen so far, a superset of those within that of the row's maximum -- into
//    the warp's region of a buffer;
//  - kCW cut warps: when the row is through, its cut from the candidates, in
//    the other of two buffers while the next row streams. The candidates'
//    masses in 40-bit fixed point (sums the same in any order) are binned by
//    delta at 1/32 log2 unit, the bucket where the running mass reaches top_p
//    of the row's total is ranked, and the kept ones are added to their
//    chunks' masses.
// A warp's region that fills up first drops what a larger maximum has put
// below the bar, then raises the bar. A row whose cut lies below its bar, or
// whose crossing bucket holds more than kCross, gets head n = -1 (with its
// maximum and total) and is left to nucleus_kernel.
//
// The two kernels that did this before (a row pass for the maximum and the
// total, then a CTA per row that read the row again and worked through its
// candidates while its share of the SM streamed nothing) moved every row twice:
// 1133 + 1920 us for a step of 1024 requests (19,000 bf16 rows of 151,936 and
// 201,088 columns, 7.0 GB; top-p 0.9), 78 + 131 us for 64 (fp32, 0.5 GB). This
// one takes 1436 and 109 us. A unit costs about 1500 warp instructions, 1050 of
// them for maxima and sums, at 68 % of the issue slots: it is bound by those
// and by the dependent chain of a unit's candidates (without candidates it
// streams at 6.2 TB/s).
#include <algorithm>
#include <cstdint>

#include "tt_device.cuh"
#include "tt_launch.h"
#include "tt_f2.cuh"
#include "tt_ring.cuh"

namespace tt {

namespace {

constexpr int kSW = 20;         // streaming warps, one ring stage each
constexpr int kCW = 8;          // cut warps
constexpr int kCT = kCW * 32;
constexpr int kThreads = (kSW + kCW + 1) * 32;
constexpr int kStage = 8192;    // bytes of a unit
constexpr int kRegion = 160;    // candidates a streaming warp keeps of one row
constexpr float kCandDelta = 14.f;
// The maximum expected of a row (see stream_unit; log2 units): the lowest of
// the CTA's last rows of the family, rising by kPredRise a row.
constexpr float kPredNear = 12.f, kPredSlack = 3.f, kPredRise = 0.5f;
constexpr float kBucketsPerUnit = 32.f;
// (the fp32 delta of a candidate may round up to kCandDelta)
constexpr int kBuckets = int(kCandDelta) * 32 + 32;
constexpr int kCross = 128;     // candidates of the crossing bucket
constexpr float kFix = kFixScale;  // of the masses
static_assert(kBuckets >= kNucWideMax / kChunk, "chunk masses share the buckets' memory");
static_assert(kBuckets <= 2 * kCT, "two buckets per cut thread");

constexpr int kQueue = 4;       // rows named ahead

// A row of the CTA: a streaming warp's units of it are first, first + kSW, ...
struct NrTask {
  int64_t row;   // < 0: no more rows
  int32_t set;   // 0 draft rows, 1 target rows
  int32_t rot;   // the streaming warp that takes unit 0
};

struct NrDesc {  // one unit
  int64_t row;
  int32_t col0;    // its first column
  int32_t n;       // its columns
  int32_t n_smem;  // leading columns delivered by the bulk copy (rest read directly)
};

// What a streaming warp leaves of a row.
struct NrWarp {
  float zmax;  // its largest logit
  float bar;   // its region holds every logit above this
  int n;       // candidates
};

// A streaming warp's list of vectors that may hold candidates.
constexpr int kListed = 60;
struct NrList {
  int n;
  uint16_t v[kListed];
};

struct NrRow {  // one of the two rows in flight
  Cand cand[kSW][kRegion];
  NrWarp w[kSW];
  Partial part[kNucWideMax / kChunk];  // of its chunks
  int64_t row;  // < 0: the end
  int32_t set;
  uint32_t best;  // key of the largest logit seen so far
};

// Sums of masses (whole numbers up to 2^40), each held as the sums of its lower 20
// bits and of the others: kSW * kRegion terms do not overflow 32 bits, and 32-bit
// adds to shared memory are one instruction where 64-bit ones are a loop around
// compare-and-swap, whose lanes all meet at one chunk (a region's candidates are
// neighbours). With those the cuts held rows of many candidates up: 64 requests
// of 24,515 fp32 columns (Gaussian, sigma 2, top-p 0.9) took 117 us a step, 81
// now, and 1024 of Zipf logits 1572 and 1495.
struct MassSum {
  uint32_t lo[kBuckets], hi[kBuckets];
  __device__ __forceinline__ void clear(int i) { lo[i] = hi[i] = 0u; }
  __device__ __forceinline__ void add(int i, unsigned long long m) {
    atomicAdd(&lo[i], uint32_t(m) & 0xfffffu);
    atomicAdd(&hi[i], uint32_t(m >> 20));
  }
  __device__ __forceinline__ unsigned long long get(int i) const {
    return (static_cast<unsigned long long>(hi[i]) << 20) + lo[i];
  }
};
static_assert(kSW * kRegion <= 4000, "the sums of a row fit 32 bits");

struct NrSmem {
  char stage[kSW][kStage];
  NrRow r[2];
  union {  // the cut's phases, one after the other
    MassSum mass;  // of the buckets
    struct {
      Cand gc[kCross];
      unsigned long long gm[kCross];
    } x;
    MassSum cacc;  // of the chunks
  } u;
  uint64_t full[kSW];          // the warp's unit has arrived
  uint64_t named[kQueue], taken[kQueue];  // the queue's entry is there / read by every warp
  uint64_t done[2], freed[2];  // the row is through / its buffer is free again
  NrTask queue[kQueue];
  NrList list[kSW];
  unsigned long long wsum[kCW];
  F2 wf2[kCW];
  unsigned long long best, before, thr;
  float pred[2];  // largest logit expected of a draft / target row
  float tau_v;
  int tau_c, cross, n_gc, ok;
};
static_assert(sizeof(NrSmem) <= 227 * 1024, "one CTA per SM");

// Order-preserving key of a float (0 lies below every number's), and back.
__device__ __forceinline__ uint32_t float_key(float x) {
  const uint32_t u = __float_as_uint(x);
  return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k) {
  return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xffffffffu));
}

// Units of 8 KB of a row.
__device__ __forceinline__ int row_units(const RowSet& S, int dt) {
  const int per = dt == TT_F32 ? kStage / 4 : kStage / 2;
  return (S.V + per - 1) / per;
}

// -------------------------------------------------------------- the schedule
template <int DTD, int DTT>
__device__ void schedule(const NucRowArgs& a, NrSmem& sm) {
  const int64_t G = gridDim.x, g = blockIdx.x;
  int seq = 0, rot = 0;
  // Names the CTA's next row (row < 0: the end); false once a wait has run out.
  auto name = [&](bool tgt, int64_t row) -> bool {
    if (row >= 0 && !tgt && a.d.need && a.d.need[row] == 0) return true;  // not mapped to
    // every warp has read the entry's last row
    if (!mbar_wait(&sm.taken[seq % kQueue], ((seq / kQueue) & 1) ^ 1, a.wait_ns)) {
      report_error(a.err, a.epoch, TT_REQ_TIMEOUT);
      return false;
    }
    sm.queue[seq % kQueue] = NrTask{row, tgt ? 1 : 0, rot};
    mbar_arrive(&sm.named[seq % kQueue]);
    ++seq;
    // (short last rounds fall to other warps from row to row)
    if (row >= 0) rot = (rot + row_units(tgt ? a.t : a.d, tgt ? DTT : DTD)) % kSW;
    return true;
  };
  // Target rows do not depend on the grid before this one: a share of them (at
  // most half, at least one row per CTA) streams before the wait. The others,
  // then the draft rows, are drawn one by one from a counter.
  const int64_t per = a.work ? max(int64_t(1), a.rows_t / (2 * G)) : (a.rows_t + G - 1) / G;
  const int64_t fixed = min(a.rows_t, per * G);
  for (int64_t i = g; i < fixed; i += G)
    if (!name(true, i)) return;
  grid_dependency_wait();  // the counter and the needed-row flags are ready
  grid_launch_dependents();
  if (!a.work) {
    for (int64_t i = g; i < a.rows_d; i += G)
      if (!name(false, i)) return;
  } else {
    const int64_t rest = a.rows_t - fixed, pool = rest + a.rows_d;
    for (;;) {
      const int64_t i = int64_t(atomicAdd(a.work + kNucWork, 1ull));
      if (i >= pool) break;
      if (!(i < rest ? name(true, fixed + i) : name(false, i - rest))) return;
    }
  }
  name(true, -1);
}

// ------------------------------------------------------ the streaming warps

// A streaming warp's running state of one row.
struct NrState {
  float zmax, zc;  // largest logit; the region holds every logit above zc
  int n;
};

// Keeps the region's entries above zc; returns how many.
__device__ __forceinline__ int prune(Cand* region, int n, float zc, int lane) {
  int kept = 0;
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane;
    const Cand c = i < n ? region[i] : Cand{-INFINITY, 0};
    const bool k = i < n && c.v > zc;
    const unsigned m = __ballot_sync(0xffffffffu, k);
    if (k) region[kept + __popc(m & ((1u << lane) - 1u))] = c;  // (never past i)
    kept += __popc(m);
    __syncwarp();
  }
  return kept;
}

// Two fp32 values in one register pair (each half rounds as the scalar operation does).
__device__ __forceinline__ uint64_t pack2(float x, float y) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// x added to the compensated sum hs + ls (TwoSum); the same on register pairs.
__device__ __forceinline__ void comp_add(float& hs, float& ls, float x) {
  const float sx = __fadd_rn(hs, x), bb = __fsub_rn(sx, hs);
  ls = __fadd_rn(ls, __fadd_rn(__fsub_rn(hs, __fsub_rn(sx, bb)), __fsub_rn(x, bb)));
  hs = sx;
}
__device__ __forceinline__ void comp_add2(uint64_t& hs, uint64_t& ls, uint64_t x) {
  const uint64_t sx = add2(hs, x), bb = sub2(sx, hs);
  ls = add2(ls, add2(sub2(hs, sub2(sx, bb)), sub2(x, bb)));
  hs = sx;
}

// Sum over the warp of each lane's compensated sum, as one float.
__device__ __forceinline__ float comp_reduce(float hs, float ls) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, hs, o);
    const float ol = __shfl_xor_sync(0xffffffffu, ls, o);
    ls = __fadd_rn(ls, ol);
    comp_add(hs, ls, oh);
  }
  return __fadd_rn(hs, ls);
}

// Sum of 2^(z * scale - m) over one chunk of NV vectors per lane (sv[lane],
// sv[lane + 32], ..., those below nvec), each vector's terms added plainly and
// the vectors' sums in compensated pairs, then the lane's column of the ragged
// tail (zt, -inf: none).
template <int DT, int NV>
__device__ __forceinline__ float chunk_sum(const uint4* sv, int nvec, float zt, float m,
                                           float scale, int lane) {
  constexpr int VEC = DT == TT_F32 ? 4 : 8;
  float hs = 0.f, ls = 0.f;
#pragma unroll 4
  for (int v = 0; v < NV; ++v) {
    if (v * 32 + lane >= nvec) continue;
    const uint4 w = sv[v * 32 + lane];
    float b = 0.f;
#pragma unroll
    for (int q = 0; q < VEC; ++q) b += ex2_approx(fmaf(lane_elem<DT>(w, q), scale, -m));
    comp_add(hs, ls, b);
  }
  if (zt > -INFINITY) comp_add(hs, ls, ex2_approx(fmaf(zt, scale, -m)));
  return comp_reduce(hs, ls);
}

// The same for both chunks of a whole bf16 unit at once, one in each half of
// the register pairs (bit for bit the two sums taken apart).
__device__ __forceinline__ void chunk_sum2(const uint4* sv, float m0, float m1, float scale,
                                           int lane, float& s0, float& s1) {
  const uint64_t scale2 = pack2(scale, scale), nm2 = pack2(-m0, -m1);
  uint64_t hs = 0, ls = 0;
#pragma unroll 2
  for (int v = 0; v < 8; ++v) {
    const uint4 wa = sv[v * 32 + lane], wb = sv[(v + 8) * 32 + lane];
    uint64_t b = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      float x, y;
      unpack2(fma2(pack2(lane_elem<TT_BF16>(wa, q), lane_elem<TT_BF16>(wb, q)), scale2, nm2), x, y);
      b = add2(b, pack2(ex2_approx(x), ex2_approx(y)));
    }
    comp_add2(hs, ls, b);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t oh = __shfl_xor_sync(0xffffffffu, hs, o);
    const uint64_t ol = __shfl_xor_sync(0xffffffffu, ls, o);
    ls = add2(ls, ol);
    comp_add2(hs, ls, oh);
  }
  unpack2(add2(hs, ls), s0, s1);
}

// Largest of the 8 bf16 logits of a vector, in both halves of a word.
__device__ __forceinline__ uint32_t vec_max_bf16(const uint4& w) {
  const uint32_t m = max_bf16x2(max_bf16x2(w.x, w.y), max_bf16x2(w.z, w.w));
  return max_bf16x2(m, __byte_perm(m, 0, 0x1032));
}

// Raises the bar of a region that has no room for a unit's candidates, from
// where it stands and by whole log2 units, until the unit's vectors that reach it
// (a candidate each, at least) leave room. From 14 down in each unit, with a
// gathering after each step, it held flat rows up: 64 requests of Gaussian
// logits (sigma 1.5, fp32, 151,936 columns, top-p 0.9) took 2281 us, so 2061
// (1663 with the sums by 32-bit adds; the two kernels that this one replaced
// took 1950).
struct NrBar {
  float bar, zc;
  uint32_t flags;  // the vectors that reach it
  int n;           // entries left in the region
};
template <int DT>
__device__ __noinline__ NrBar raise_bar(const uint4* sv, int nvl, float base, float scale,
                                        Cand* region, int lane, NrBar b) {
  b.bar = fminf(b.bar, ceilf(__fsub_rn(base, __fmul_rn(b.zc, scale))));  // as it stands
  int most;
  do {
    b.bar -= 1.f;
    b.zc = b.bar > 0.f ? fmaxf(b.zc, __fdiv_rn(__fsub_rn(base, b.bar), scale)) : INFINITY;
    b.n = prune(region, b.n, b.zc, lane);
    b.flags = 0;
#pragma unroll 4
    for (int v = 0; v < nvl; ++v)
      if (vec_max<DT>(sv[v * 32 + lane]) > b.zc) b.flags |= 1u << v;
    most = kRegion - int(__reduce_add_sync(0xffffffffu, unsigned(__popc(b.flags))));
  } while (b.n > most && b.zc < INFINITY);
  return b;
}

// One unit: the partials of its chunks -- the largest z * scale and the sum of
// 2^(z * scale - that), as the row pass forms them for narrow nucleus rows --
// and its candidates. The vectors' maxima are kept, two to a word (bf16 as they
// are, fp32 as the upper halves of their keys), to tell which vectors to look
// at element by element.
template <int DT>
__device__ __forceinline__ void stream_unit(const char* stage, const NrDesc& d, const RowSet& S,
                                            int lane, NrState& st, Cand* region, NrList* list,
                                            NrRow& R, float pred) {
  constexpr int VEC = DT == TT_F32 ? 4 : 8;
  constexpr int NC = DT == TT_F32 ? 1 : 2;  // chunks per unit
  const uint4* sv = reinterpret_cast<const uint4*>(stage);
  const float scale = S.scale;
  const int nvec = d.n_smem / VEC;  // whole vectors held in shared memory
  float zt = -INFINITY;  // the ragged tail: one column per lane, in chunk n_smem / kChunk
  if (lane < d.n - d.n_smem)
    zt = load_logit<DT>(S.data + d.row * S.stride_bytes, int64_t(d.col0) + d.n_smem + lane);
  const int ct = d.n_smem / kChunk;
  const int nvl = max(0, min(16, (nvec - lane + 31) >> 5));  // the lane's vectors of the unit
  uint32_t key[NC];  // of the chunks' largest logits
  uint32_t vm[8];    // bf16: vectors v and v + 8; fp32: 2 v and 2 v + 1
  if constexpr (DT == TT_F32) {
    float zm = ct == 0 ? zt : -INFINITY;
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const float x = 2 * v < nvl ? vec_max<DT>(sv[2 * v * 32 + lane]) : -INFINITY;
      const float y = 2 * v + 1 < nvl ? vec_max<DT>(sv[(2 * v + 1) * 32 + lane]) : -INFINITY;
      zm = fmaxf(zm, fmaxf(x, y));
      vm[v] = __byte_perm(float_key(x), float_key(y), 0x7632);
    }
    key[0] = __reduce_max_sync(0xffffffffu, float_key(zm));
  } else {
    constexpr uint32_t kNone = 0xff80ff80u;  // two bf16 -inf
    uint32_t m2 = kNone;
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const uint32_t x = v < nvl ? vec_max_bf16(sv[v * 32 + lane]) : kNone;
      const uint32_t y = v + 8 < nvl ? vec_max_bf16(sv[(v + 8) * 32 + lane]) : kNone;
      vm[v] = __byte_perm(x, y, 0x5410);
      m2 = max_bf16x2(m2, vm[v]);
    }
    key[0] = __reduce_max_sync(
        0xffffffffu, float_key(fmaxf(__uint_as_float(m2 << 16), ct == 0 ? zt : -INFINITY)));
    key[NC - 1] = __reduce_max_sync(
        0xffffffffu,
        float_key(fmaxf(__uint_as_float(m2 & 0xffff0000u), ct == 1 ? zt : -INFINITY)));
  }
  const uint32_t ukey = NC == 2 ? max(key[0], key[NC - 1]) : key[0];
  const float um = key_float(ukey);
  // the row's largest logit so far
  const bool first = st.zmax == -INFINITY;
  if (um > st.zmax) {
    st.zmax = um;
    if (lane == 0) atomicMax(&R.best, ukey);
  }
  const float m0 = __fmul_rn(key_float(key[0]), scale);
  const float m1 = __fmul_rn(key_float(key[NC - 1]), scale);
  float s0 = 0.f, s1 = 0.f;
  if constexpr (NC == 2) {
    if (nvec == kStage / 16 && m0 > -INFINITY && m1 > -INFINITY) {
      chunk_sum2(sv, m0, m1, scale, lane, s0, s1);
    } else {  // a ragged unit: the chunks apart
      if (m0 > -INFINITY)
        s0 = chunk_sum<DT, 8>(sv, nvec, ct == 0 ? zt : -INFINITY, m0, scale, lane);
      if (m1 > -INFINITY)
        s1 = chunk_sum<DT, 8>(sv + 256, nvec - 256, ct == 1 ? zt : -INFINITY, m1, scale, lane);
    }
  } else {
    if (m0 > -INFINITY)
      s0 = chunk_sum<DT, 16>(sv, nvec, ct == 0 ? zt : -INFINITY, m0, scale, lane);
  }
  // The bar, from the row's largest logit as it stands now. On a row's first
  // units that is far below the row's (8 log2 units, with 30 times the
  // candidates), so a maximum near those of the CTA's last rows of the family is
  // taken for granted, unless what is seen of the row is far from it. (Where that
  // was too high, the row's bar is, too, and a cut below it leaves the row to
  // nucleus_kernel.)
  const uint32_t top =
      max(ukey, __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(&R.best), 0));
  float base = __fmul_rn(key_float(top), scale);
  if (first) {
    const float near = __fmul_rn(pred, scale);
    if (near - base <= kPredNear) base = fmaxf(base, near - kPredSlack);
  }
  auto bar_at = [&](float bar) { return __fdiv_rn(__fsub_rn(base, bar), scale); };
  float zc = fmaxf(st.zc, bar_at(kCandDelta));
  uint32_t flags = 0;  // the vectors that may hold a logit above zc
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    if constexpr (DT == TT_F32) {
      const uint32_t kc = float_key(zc) >> 16;
      flags |= (vm[v] & 0xffffu) >= kc ? 1u << (2 * v) : 0u;
      flags |= (vm[v] >> 16) >= kc ? 1u << (2 * v + 1) : 0u;
    } else {
      flags |= __uint_as_float(vm[v] << 16) > zc ? 1u << v : 0u;
      flags |= __uint_as_float(vm[v] & 0xffff0000u) > zc ? 1u << (v + 8) : 0u;
    }
  }
  flags &= (1u << nvl) - 1u;
  if (lane == 0) {
    Partial* part = R.part + d.col0 / kChunk;
    part[0] = Partial{m0, s0};
    if (NC == 2 && d.n > kChunk) part[1] = Partial{m1, s1};
  }
  // The candidates, appended to the warp's region: the flagged vectors are
  // listed, then their elements tested one per lane.
  for (float bar = kCandDelta;;) {
    // (each flagged vector holds one at least: what cannot fit is not gathered)
    int n = st.n + int(__reduce_add_sync(0xffffffffu, unsigned(__popc(flags))));
    if (n <= kRegion) {
      n = st.n;
      const bool tail = zt > zc;
      const unsigned mt = __ballot_sync(0xffffffffu, tail);
      if (tail && n + __popc(mt & ((1u << lane) - 1u)) < kRegion)
        region[n + __popc(mt & ((1u << lane) - 1u))] = Cand{zt, d.col0 + d.n_smem + lane};
      n += __popc(mt);
      for (uint32_t f = flags; n <= kRegion && __any_sync(0xffffffffu, f != 0u);) {
        if (lane == 0) list->n = 0;
        __syncwarp();
        int i = f ? atomicAdd(&list->n, __popc(f)) : kListed;
        for (; f && i < kListed; f &= f - 1, ++i)
          list->v[i] = uint16_t((__ffs(f) - 1) * 32 + lane);
        __syncwarp();
        const int nv = min(list->n, kListed);
        constexpr int kBatch = 4;  // elements in flight per lane
        for (int k = 0; k < nv; k += kBatch * 32 / VEC) {
          int x[kBatch];
          float z[kBatch];
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            const int e = k + q * (32 / VEC) + lane / VEC;
            x[q] = e < nv ? list->v[e] * VEC + lane % VEC : -1;
          }
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            const int y = max(x[q], 0);
            z[q] = DT == TT_F32 ? reinterpret_cast<const float*>(stage)[y]
                                : bf16_to_f32(reinterpret_cast<const uint16_t*>(stage)[y]);
          }
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            const bool take = x[q] >= 0 && z[q] > zc;
            const unsigned m = __ballot_sync(0xffffffffu, take);
            const int at = n + __popc(m & ((1u << lane) - 1u));
            if (take && at < kRegion) region[at] = Cand{z[q], d.col0 + x[q]};
            n += __popc(m);
          }
        }
        __syncwarp();
      }
    }
    if (n <= kRegion) {
      st.n = n;
      break;
    }
    // no room: drop what now lies below the bar, else raise the bar (for this
    // unit: the region is complete above the highest bar that it has seen)
    const int kept = prune(region, st.n, zc, lane);
    if (kept == st.n) {
      const NrBar b =
          raise_bar<DT>(sv, nvl, base, scale, region, lane, NrBar{bar, zc, flags, kept});
      bar = b.bar;
      zc = b.zc;
      flags = b.flags;
      st.n = b.n;
    } else {
      st.n = kept;
    }
  }
  st.zc = zc;
}

template <int DTD, int DTT>
__device__ void stream_rows(const NucRowArgs& a, NrSmem& sm, int warp, int lane) {
  char* stage = sm.stage[warp];
  int step = 0;  // units copied by this warp
  NrTask t = {-1, 0, 0};
  int u = 0, nu = 0;  // the warp's current unit of the row, and the row's units
  NrDesc d = {-1, 0, 0, 0};
  bool in_flight = false;  // a copy into the stage that has not been waited for
  auto timed_out = [&]() {
    if (lane == 0) report_error(a.err, a.epoch, TT_REQ_TIMEOUT);
    if (in_flight) mbar_wait(&sm.full[warp], (step - 1) & 1, a.wait_ns);
  };
  // Copies unit u of row t into the stage (whose last unit is worked through).
  auto copy = [&]() {
    const RowSet& S = t.set ? a.t : a.d;
    const int esz = (t.set ? DTT : DTD) == TT_F32 ? 4 : 2;
    d.row = t.row;
    d.col0 = u * (kStage / esz);
    d.n = min(kStage / esz, S.V - d.col0);
    const uint32_t bytes = uint32_t(d.n * esz) & ~15u;  // bulk copies move 16-byte units
    d.n_smem = int(bytes) / esz;
    __syncwarp();
    if (lane == 0) {
      // every bulk copy lies inside its row and starts on 16 bytes
      const char* src = S.data + t.row * S.stride_bytes + size_t(d.col0) * esz;
      const bool ok = t.row < S.n_rows && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
      if (!ok) report_error(a.err, a.epoch, TT_REQ_INTERNAL);
      // (test hook: in CTA 0 one of the copies is never made)
      if (blockIdx.x == 0 && step * kSW + warp == a.stall_stage) {
      } else if (ok && bytes > 0) {
        mbar_arrive_expect_tx(&sm.full[warp], bytes);
        bulk_copy_g2s(stage, src, bytes, &sm.full[warp]);
      } else {
        mbar_arrive(&sm.full[warp]);
      }
      if (!ok) d.row = -1;
    }
    d.row = __shfl_sync(0xffffffffu, d.row, 0);
    in_flight = !(blockIdx.x == 0 && step * kSW + warp == a.stall_stage);
    ++step;
  };
  // Takes up row `seq`: its entry of the queue, and the copy of the warp's first unit.
  auto take_up = [&](int seq) -> bool {
    if (!mbar_wait(&sm.named[seq % kQueue], (seq / kQueue) & 1, a.wait_ns)) return false;
    t = sm.queue[seq % kQueue];
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm.taken[seq % kQueue]);
    if (t.row < 0) return true;
    nu = row_units(t.set ? a.t : a.d, t.set ? DTT : DTD);
    u = warp >= t.rot ? warp - t.rot : warp + kSW - t.rot;
    if (u < nu) copy();
    return true;
  };
  if (!take_up(0)) return timed_out();
  for (int seq = 0;; ++seq) {
    NrRow& R = sm.r[seq & 1];
    // the row before last, in the same buffer, has been cut
    if (!mbar_wait(&sm.freed[seq & 1], ((seq >> 1) & 1) ^ 1, a.wait_ns)) return timed_out();
    if (warp == 0 && lane == 0) {
      R.row = t.row;
      R.set = t.set;
    }
    if (t.row < 0) {
      if (lane == 0) mbar_arrive(&sm.done[seq & 1]);
      return;
    }
    const RowSet& S = t.set ? a.t : a.d;
    const bool f32 = (t.set ? DTT : DTD) == TT_F32;
    NrState st;
    st.zmax = st.zc = -INFINITY;
    st.n = 0;
    const float pred = __shfl_sync(
        0xffffffffu, *reinterpret_cast<volatile float*>(&sm.pred[t.set]), 0);
    while (u < nu) {
      if (!mbar_wait(&sm.full[warp], (step - 1) & 1, a.wait_ns)) return timed_out();
      in_flight = false;
      if (d.row >= 0) {
        if (f32) stream_unit<TT_F32>(stage, d, S, lane, st, R.cand[warp], &sm.list[warp], R, pred);
        else stream_unit<TT_BF16>(stage, d, S, lane, st, R.cand[warp], &sm.list[warp], R, pred);
      }
      u += kSW;
      if (u < nu) copy();
    }
    __syncwarp();
    if (lane == 0) {
      R.w[warp] = NrWarp{st.zmax, st.zc, st.n};
      mbar_arrive(&sm.done[seq & 1]);
    }
    if (!take_up(seq + 1)) return timed_out();
  }
}

// ------------------------------------------------------------ the cut warps

__device__ __forceinline__ void cut_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kCT) : "memory");
}

__device__ void cut_rows(const NucRowArgs& a, NrSmem& sm, int tid) {
  const int lane = tid & 31, warp = tid >> 5;
  for (int seq = 0;; ++seq) {
    NrRow& R = sm.r[seq & 1];
    if (tid == 0) {
      sm.ok = mbar_wait(&sm.done[seq & 1], (seq >> 1) & 1, a.wait_ns) ? 1 : 0;
      if (!sm.ok) report_error(a.err, a.epoch, TT_REQ_TIMEOUT);
      sm.cross = -1;
      sm.n_gc = 0;
      sm.best = 0ull;
    }
    for (int i = tid; i < kBuckets; i += kCT) sm.u.mass.clear(i);
    cut_sync();
    if (!sm.ok || R.row < 0) return;
    const bool tgt = R.set != 0;
    const int64_t r = R.row;
    const RowSet& S = tgt ? a.t : a.d;
    KeptHead* head = (tgt ? a.head_t : a.head_d) + r;
    float* um = (tgt ? a.um_t : a.um_d) + r * S.nch;
    const int nch = S.nch;
    const float scale = S.scale;
    // every warp: the row's maximum and its largest bar
    const NrWarp mine = lane < kSW ? R.w[lane] : NrWarp{-INFINITY, -INFINITY, 0};
    const float M =
        __fmul_rn(key_float(__reduce_max_sync(0xffffffffu, float_key(mine.zmax))), scale);
    // candidates: z > zlim
    const float zlim = fmaxf(key_float(__reduce_max_sync(0xffffffffu, float_key(mine.bar))),
                             __fdiv_rn(__fsub_rn(M, kCandDelta), scale));
    // its total relative to 2^M
    F2 T = {0.f, 0.f};
    if (isfinite(M))
      for (int c = tid; c < nch; c += kCT) {
        const Partial q = R.part[c];
        if (q.m > -INFINITY) T = f2_add(T, F2{__fmul_rn(q.s, ex2_approx(q.m - M)), 0.f});
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      T = f2_add(T, F2{__shfl_xor_sync(0xffffffffu, T.hi, o),
                       __shfl_xor_sync(0xffffffffu, T.lo, o)});
    if (lane == 0) sm.wf2[warp] = T;
    cut_sync();
    T = {0.f, 0.f};
#pragma unroll
    for (int x = 0; x < kCW; ++x) T = f2_add(T, sm.wf2[x]);
    const bool sound =
        isfinite(M) && T.hi > 0.f && isfinite(T.hi) && isfinite(T.lo) && zlim < INFINITY;
    if (tid == 0 && sound) {
      // a sum of masses (whole numbers) is below top_p T exactly when below thr
      const double top_p = tgt ? a.top_p_t : a.top_p_d;
      sm.thr = (unsigned long long)ceil(top_p * (double(T.hi) + double(T.lo)) * double(kFix));
    }
    auto fixm = [&](float z) {
      return (unsigned long long)__float2ull_rn(exp2_scaled(z, scale, M) * kFix);
    };
    auto bucket = [&](float z) {  // non-increasing in z
      const float f = __fsub_rn(M, __fmul_rn(z, scale)) * kBucketsPerUnit;
      return f > 0.f ? min(kBuckets - 1, int(f)) : 0;
    };
    // every candidate of the row, a warp per region
    auto for_cands = [&](auto&& fn) {
      for (int x = warp; x < kSW; x += kCW) {
        const int n = R.w[x].n;
        for (int i = lane; i < n; i += 32) {
          const Cand c = R.cand[x][i];
          if (c.v > zlim) fn(c.v, c.c);
        }
      }
    };
    bool settled = false;
    if (sound) {
      for_cands([&](float z, int) { sm.u.mass.add(bucket(z), fixm(z)); });
      cut_sync();
      const unsigned long long thr = sm.thr;
      // the bucket whose inclusive running mass reaches thr, and the mass before it
      unsigned long long m0 = 2 * tid < kBuckets ? sm.u.mass.get(2 * tid) : 0ull;
      unsigned long long m1 = 2 * tid + 1 < kBuckets ? sm.u.mass.get(2 * tid + 1) : 0ull;
      unsigned long long incl = m0 + m1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) sm.wsum[warp] = incl;
      cut_sync();
      unsigned long long run = incl - m0 - m1;
      for (int x = 0; x < warp; ++x) run += sm.wsum[x];
      if (run < thr && run + m0 + m1 >= thr) {  // one thread at most
        const bool second = run + m0 < thr;
        sm.cross = 2 * tid + (second ? 1 : 0);
        sm.before = second ? run + m0 : run;
      }
      cut_sync();
      const int cb = sm.cross;
      if (cb >= 0) {
        const unsigned long long before = sm.before;
        // the crossing bucket's candidates, ranked: one is kept when the mass
        // ranked before it (larger logit, then smaller column) is below thr; the
        // last kept one has the most mass before it (every mass is positive)
        for_cands([&](float z, int x) {
          if (bucket(z) == cb) {
            const int j = atomicAdd(&sm.n_gc, 1);
            if (j < kCross) {
              sm.u.x.gc[j] = Cand{z, x};
              sm.u.x.gm[j] = fixm(z);
            }
          }
        });
        cut_sync();
        const int nc = sm.n_gc;
        if (nc <= kCross) {
          unsigned long long key = 0ull;
          if (tid < nc) {
            const Cand e = sm.u.x.gc[tid];
            unsigned long long pm = before;
#pragma unroll 4
            for (int j = 0; j < nc; ++j) {
              const Cand f = sm.u.x.gc[j];
              if (f.v > e.v || (f.v == e.v && f.c < e.c)) pm += sm.u.x.gm[j];
            }
            if (pm < thr) {
              key = pm + 1ull;
              atomicMax(&sm.best, key);
            }
          }
          cut_sync();
          if (key != 0ull && key == sm.best) {  // one candidate
            sm.tau_v = sm.u.x.gc[tid].v;
            sm.tau_c = sm.u.x.gc[tid].c;
          }
          cut_sync();
          const float tau = sm.tau_v;
          const int tau_col = sm.tau_c;
          // the kept candidates join their chunks; the header
          for (int c = tid; c < nch; c += kCT) sm.u.cacc.clear(c);
          cut_sync();
          for_cands([&](float z, int x) {
            if (z > tau || (z == tau && x <= tau_col)) sm.u.cacc.add(x / kChunk, fixm(z));
          });
          cut_sync();
          unsigned long long tot = 0ull;  // whole numbers: the same in any order
          for (int c = lane; c < nch; c += 32) tot += sm.u.cacc.get(c);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
          const KeptNorm kn = kept_norm(tot);
          for (int c = tid; c < nch; c += kCT) um[c] = kept_share(sm.u.cacc.get(c), kn);
          if (tid == 0) {
            const KeptScale ks = kept_scale(kn, M);
            *head = KeptHead{ks.lse, 1, tau, tau_col, M, ks.inv_s};
          }
          settled = true;
        }
      }
    }
    if (!settled && tid == 0)  // not finite; or left to nucleus_kernel, with the row's total
      *head = !isfinite(M) ? KeptHead{NAN, 0, NAN, -1, M, 0.f}
                           : KeptHead{T.lo, -1, 0.f, 0, M, T.hi};
    if (tid == 0) {
      R.best = 0u;
      const float zm = M / scale, low = sm.pred[tgt] + kPredRise / scale;
      sm.pred[tgt] = low > -INFINITY ? fminf(zm, low) : zm;
    }
    cut_sync();
    if (tid == 0) mbar_arrive(&sm.freed[seq & 1]);
  }
}

template <int DTD, int DTT>
__global__ void __launch_bounds__(kThreads, 1)
    nucleus_row_kernel(const __grid_constant__ NucRowArgs a) {
  extern __shared__ __align__(128) char raw[];
  NrSmem& sm = *reinterpret_cast<NrSmem*>(raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSW; ++s) mbar_init(&sm.full[s], 1);
    for (int s = 0; s < kQueue; ++s) {
      mbar_init(&sm.named[s], 1);
      mbar_init(&sm.taken[s], kSW);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sm.done[s], kSW);
      mbar_init(&sm.freed[s], 1);
      sm.r[s].best = 0u;
      sm.pred[s] = -INFINITY;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (warp < kSW) stream_rows<DTD, DTT>(a, sm, warp, lane);
  else if (warp < kSW + kCW) cut_rows(a, sm, threadIdx.x - kSW * 32);
  else if (lane == 0) schedule<DTD, DTT>(a, sm);
}

template <int DTD, int DTT>
cudaError_t preload_nr() {
  return cudaFuncSetAttribute(nucleus_row_kernel<DTD, DTT>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(NrSmem)));
}

template <int DTD, int DTT>
cudaError_t launch_nr(const NucRowArgs& a, cudaStream_t stream, int sm_count, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(std::min<int64_t>(a.rows_d + a.rows_t, sm_count)));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = sizeof(NrSmem);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, nucleus_row_kernel<DTD, DTT>, a);
}

}  // namespace

cudaError_t preload_nucleus_rows() {
  cudaError_t e;
  if ((e = preload_nr<TT_F32, TT_F32>()) != cudaSuccess) return e;
  if ((e = preload_nr<TT_F32, TT_BF16>()) != cudaSuccess) return e;
  if ((e = preload_nr<TT_BF16, TT_F32>()) != cudaSuccess) return e;
  return preload_nr<TT_BF16, TT_BF16>();
}

cudaError_t launch_nucleus_rows(const NucRowArgs& args, int dt_d, int dt_t, cudaStream_t stream,
                                int sm_count, bool pdl) {
  if (args.rows_d + args.rows_t == 0) return cudaSuccess;
  NucRowArgs a = args;
  next_launch_stall(&a.stall_stage, &a.wait_ns);
  if (dt_d == TT_F32 && dt_t == TT_F32) return launch_nr<TT_F32, TT_F32>(a, stream, sm_count, pdl);
  if (dt_d == TT_F32) return launch_nr<TT_F32, TT_BF16>(a, stream, sm_count, pdl);
  if (dt_t == TT_F32) return launch_nr<TT_BF16, TT_F32>(a, stream, sm_count, pdl);
  return launch_nr<TT_BF16, TT_BF16>(a, stream, sm_count, pdl);
}

}  // namespace tt
