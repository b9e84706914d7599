// pen.cu -- the per-request sets of the repetition penalty (the generation
// hyperparameter table, App. F: 1.1 for the Qwen2.5-0.5B model).
//
// A row's penalized columns are its request's history and the sequence tokens
// before the row's position (target row j: t_1..t_j; draft row i: d_1..d_i).
// pen_prep_kernel (one CTA per request, half of it per family) keeps one entry
// per column with the first sequence position holding it (-1 when the history
// does), so that row j penalizes the entry when first < j, and groups the
// entries by row unit. The row pass then gives these columns the row's own
// values in place (fp32 rows), or leaves them out of its unit lists and the
// kept-set kernel adds them back (bf16 rows).
//
// The entries go through a hash table in shared memory and are then counted,
// placed and written by unit (their order within a unit has no effect): a few
// passes of independent accesses over at most 3584 columns. 64 requests with
// 64 to 1024 history tokens: 14 us; a sort of each family's columns in turn
// (66 barrier-separated steps) took 40 us.
#include <cstdint>

#include "tt_device.cuh"
#include "tt_launch.h"
#include "tt_f2.cuh"

namespace tt {

namespace {

constexpr int kPT = 256;          // threads per family
constexpr int kSlots = 4096;      // hash table; a power of two
constexpr unsigned long long kEmpty = ~0ull;
static_assert(TT_MAX_HISTORY + TT_MAX_M < kSlots, "a request's entries leave slots free");

struct PenSmem {
  unsigned long long slot[kSlots];  // (column, first position + 1), kEmpty
  int32_t count[kMaxChunksPerRow];  // entries per unit, then the next place of each unit
  int32_t wsum[kPT / 32];
  int32_t bad;
};

// [lo, hi) = off[b] .. off[b + 1], empty when they are no range of [0, n).
__device__ __forceinline__ bool csr_range(const int32_t* off, int b, int n, int& lo, int& hi) {
  lo = hi = 0;
  if (!off) return true;
  const int a0 = off[b], a1 = off[b + 1];
  if (a0 < 0 || a1 < a0 || a1 > n) return false;
  lo = a0;
  hi = a1;
  return true;
}

// Barrier of one family's threads.
__device__ __forceinline__ void family_sync(int fam) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + fam), "n"(kPT) : "memory");
}

// The same, and whether any of them passed true.
__device__ __forceinline__ bool family_or(int fam, bool p) {
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.s32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred q, %2, %3, p;\n\t"
      "selp.s32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(int(p)), "r"(1 + fam), "n"(kPT)
      : "memory");
  return r != 0;
}

// Whether a family's offsets fall anywhere (fell[0]: draft, fell[1]: target).
// Batches of at most kPenSelfCheck requests go without: each CTA looks over the
// offsets before its own, which costs nothing there (64 to 1024 requests: the
// same time with and without the look) where a launch would cost 2 us; 4096
// requests (16 draft tokens, 2048 columns) take 428 us without any look, 482 with
// a look by each CTA and 427 with this kernel.
constexpr int kPenSelfCheck = 1024;
constexpr int kCheckThreads = 1024;
__global__ void __launch_bounds__(kCheckThreads) pen_check_kernel(PenArgs a, int32_t* fell) {
  for (int fam = 0; fam < 2; ++fam) {
    bool f = false;
    if (fam ? a.on_t : a.on_d) {
      const int32_t* hoff = fam ? a.hist_off_t : a.hist_off_d;
      const int32_t* soff = fam ? a.target_off : a.draft_off;
#pragma unroll 4
      for (int x = threadIdx.x; x < a.B; x += kCheckThreads)
        f |= (hoff && hoff[x] > hoff[x + 1]) || soff[x] > soff[x + 1];
    }
    f = __syncthreads_or(f);
    if (threadIdx.x == 0) fell[fam] = f;
  }
}

__global__ void __launch_bounds__(2 * kPT) pen_prep_kernel(PenArgs a) {
  extern __shared__ __align__(16) char raw[];
  __shared__ int s_status;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int b = blockIdx.x, fam = threadIdx.x / kPT, tid = threadIdx.x % kPT;
  const int lane = tid & 31, warp = tid >> 5;
  PenSmem& sm = reinterpret_cast<PenSmem*>(raw)[a.on_d && a.on_t ? fam : 0];
  const bool tgt = fam == 1;
  if (threadIdx.x == 0) s_status = 0;
  __syncthreads();
  if (tgt ? a.on_t : a.on_d) {
    const int V = tgt ? a.V_t : a.V_d;
    const int nlist = tgt ? a.nlist_t : a.nlist_d;
    const int lg = 31 - __clz(tgt ? a.unit_t : a.unit_d);  // a unit's columns: a power of two
    const int nch = tgt ? a.nch_t : a.nch_d;
    const int32_t* hoff = tgt ? a.hist_off_t : a.hist_off_d;
    const int32_t* soff = tgt ? a.target_off : a.draft_off;
    const int n_hist = tgt ? a.n_hist_t : a.n_hist_d, n_seq = tgt ? a.n_target : a.n_draft;
    int st = 0, h0, h1, s0, s1;
    const bool h_ok = csr_range(hoff, b, n_hist, h0, h1), s_ok = csr_range(soff, b, n_seq, s0, s1);
    if (!h_ok) st |= TT_REQ_BAD_OFFSETS;
    // without both ranges the request has no segment to write entries to (a bad
    // sequence range is reported by the other kernels)
    if (!h_ok || !s_ok) h1 = h0, s1 = s0;
    if (h1 - h0 > TT_MAX_HISTORY) {
      st |= TT_REQ_TOO_LONG;
      h1 = h0;
    }
    if (s1 - s0 > TT_MAX_M) s1 = s0;  // (too long: reported by the other kernels)
    int nh = h1 - h0, n = nh + (s1 - s0);
    // Offsets that fall somewhere before this request (which one of them is bad)
    // may put its segment over that of an earlier one.
    bool fell = a.fell && a.fell[fam] != 0;
    if (!a.fell) {
#pragma unroll 4
      for (int x = tid; x < b; x += kPT) fell |= (hoff && hoff[x] > h0) || soff[x] > s0;
    }
    const int32_t* hcols = (tgt ? a.hist_cols_t : a.hist_cols_d) + h0;
    const int32_t* scols = (tgt ? a.target_cols : a.draft_cols) + s0;
    int slots = 64;  // at least twice the entries where the table allows
    while (slots < 2 * n && slots < kSlots) slots <<= 1;
    for (int i = tid; i < slots; i += kPT) sm.slot[i] = kEmpty;
    for (int u = tid; u < nlist; u += kPT) sm.count[u] = 0;
    if (tid == 0) sm.bad = 0;
    if (family_or(fam, fell && n > 0)) {
      bool over = false;
      for (int x = tid; x < b; x += kPT) {
        int x0, x1, y0, y1;
        if (csr_range(hoff, x, n_hist, x0, x1) && csr_range(soff, x, n_seq, y0, y1))
          over |= max(x0 + y0, h0 + s0) < min(x1 + y1, h1 + s1);
      }
      if (family_or(fam, over)) {  // the earlier one keeps it
        st |= TT_REQ_BAD_OFFSETS;
        nh = n = 0;
      }
    }
    // one slot per column, holding the smallest first position (history: -1)
    constexpr int kFly = 4;  // columns in flight per thread
    for (int i0 = tid; i0 < n; i0 += kFly * kPT) {
      int c[kFly];
#pragma unroll
      for (int q = 0; q < kFly; ++q) {
        const int i = i0 + q * kPT;
        c[q] = i < nh ? hcols[i] : (i < n ? scols[i - nh] : -1);
      }
#pragma unroll
      for (int q = 0; q < kFly; ++q) {
        const int i = i0 + q * kPT;
        if (i >= n) break;
        if (c[q] < 0 || c[q] >= V) {
          if (i < nh) sm.bad = 1;  // (a sequence column: reported by the other kernels)
          continue;
        }
        const unsigned long long k = (static_cast<unsigned long long>(c[q]) << 32) |
                                     unsigned(i < nh ? 0 : i - nh + 1);
        unsigned h = (uint32_t(c[q]) * 2654435761u >> 16) & (slots - 1);
        for (;;) {  // (the table always has a free slot)
          const unsigned long long old = atomicCAS(&sm.slot[h], kEmpty, k);
          if (old == kEmpty) {
            atomicAdd(&sm.count[c[q] >> lg], 1);
            break;
          }
          if ((old >> 32) == (k >> 32)) {
            atomicMin(&sm.slot[h], k);
            break;
          }
          h = (h + 1) & (slots - 1);
        }
      }
    }
    family_sync(fam);
    // where each unit's entries start
    const int base = h0 + s0;  // the request's segment (capacity n; no other request's)
    int32_t* start = (tgt ? a.pstart_t : a.pstart_d) + int64_t(b) * (nch + 1);
    constexpr int kPer = kMaxChunksPerRow / kPT;
    int cnt[kPer], sum = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int u = tid * kPer + q;
      cnt[q] = u < nlist ? sm.count[u] : 0;
      sum += cnt[q];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) sm.wsum[warp] = incl;
    family_sync(fam);
    int at = incl - sum, total = 0;
#pragma unroll
    for (int w = 0; w < kPT / 32; ++w) {
      if (w < warp) at += sm.wsum[w];
      total += sm.wsum[w];
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int u = tid * kPer + q;
      if (u < nlist) {
        start[u] = at;
        sm.count[u] = at;
      }
      at += cnt[q];
    }
    family_sync(fam);
    PenEntry* out = (tgt ? a.pen_t : a.pen_d) + base;
    for (int i = tid; i < slots; i += kPT) {
      const unsigned long long k = sm.slot[i];
      if (k == kEmpty) continue;
      const int c = int(k >> 32);
      out[atomicAdd(&sm.count[c >> lg], 1)] = PenEntry{c, int(uint32_t(k)) - 1};
    }
    if (tid == 0) {
      start[nlist] = total;
      (tgt ? a.pbase_t : a.pbase_d)[b] = base;
      (tgt ? a.pcnt_t : a.pcnt_d)[b] = total;
      if (sm.bad) st |= TT_REQ_ID_OUT_OF_RANGE;
      if (st) atomicOr(&s_status, st);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) a.pstatus[b] = s_status;
}

}  // namespace

cudaError_t preload_pen() {
  cudaFuncAttributes fa;
  const cudaError_t e = cudaFuncGetAttributes(&fa, pen_check_kernel);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(pen_prep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              2 * int(sizeof(PenSmem)));
}

cudaError_t launch_pen_prep(const PenArgs& args, cudaStream_t stream) {
  if (args.B == 0 || !(args.on_d || args.on_t)) return cudaSuccess;
  const int families = (args.on_d ? 1 : 0) + (args.on_t ? 1 : 0);
  PenArgs a = args;
  if (args.B > kPenSelfCheck) {
    pen_check_kernel<<<1, kCheckThreads, 0, stream>>>(args, args.fell);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  } else {
    a.fell = nullptr;
  }
  pen_prep_kernel<<<args.B, 2 * kPT, families * sizeof(PenSmem), stream>>>(a);
  return cudaGetLastError();
}

}  // namespace tt
