// Selection of one unit (sequence, KV group) by the worker warps of the
// persistent kernels: pooling, top-k by pooled score, window, K/V gather
// (CompressKV Sec. 3.3 and 4).  256 threads that share named barrier kBarC.
#pragma once

#include "ckv_device.cuh"
#include "select_common.cuh"
#include "tile_math.cuh"

namespace ckv {
namespace {

constexpr int kCThreads = 256;     // worker threads of a CTA
constexpr int kBarC = 3;           // their named barrier
constexpr int kSelSamples = 1024;  // samples of a unit's pooled scores for the select threshold

constexpr int kSelWhole = 2 * kFusedCandCap;  // prefix keys of a unit whose keys all fit
constexpr int kSelGroups = 2048;  // groups of consecutive keys whose largest score is kept
struct SelShared {
  uint32_t key[kFusedCandCap];   // (all the keys of a unit of at most kSelWhole: with pos)
  int pos[kFusedCandCap];        // (while choosing a bound: samples)
  uint32_t gmax[kSelGroups];     // (of a unit of at most kSelWhole, and
  float stage_end[64];           // stage_end, while pooling: raw scores of a slice)
  RadixShared rs;
  int wcnt[8], wbase[8];
  int wcnt_ge[8];  // per-warp counts at the best threshold with at least k keys above
  alignas(16) uint32_t cnt[2][2][8];  // per-warp results of a bisection step
  uint32_t* rowmax;                   // the unit's row maxima, if it was pooled in pieces
};
static_assert(sizeof(SelShared) <= kSelRegion, "select scratch");
static_assert(kSelSamples <= kFusedCandCap, "samples live in the position array");
constexpr int kPoolStrip = 192;  // keys a warp pools at a time
constexpr int kPoolBuf = 256;    // ... with up to 62 neighbours, padded
static_assert(kPoolStrip + 62 <= kPoolBuf && kPoolStrip % 32 == 0, "a strip and its halo");
static_assert(8 * kPoolBuf <= kFusedCandCap && 8 * kPoolBuf <= kSelGroups + 64,
              "the warps' strips fit the position array and the group maxima's place");


// The call's parameters that the selection needs (in shared memory: read
// through a reference to the kernel's parameters they would come through L1).
struct SelCall {
  int* status;
  int num_kv_heads, pool_width, raw_scratch;
  const uint4* k;
  const uint4* v;
  uint4* k_out;
  uint4* v_out;
  long long tok_stride_v16, head_stride_v16;
};

__device__ __forceinline__ void cbar() { named_bar_sync(kBarC, kCThreads); }

// Zero the radix state (the workers' form of radix_init).
__device__ __forceinline__ void radix_init_grp(RadixShared& sh, int ct) {
  for (int i = ct; i < 2 * 256; i += kCThreads) sh.hist[i >> 8][i & 255] = 0u;
  if (ct < 2) {
    sh.key_or[ct] = 0u;
    sh.key_and[ct] = 0xFFFFFFFFu;
  }
}

// The workers' form of cta_kth_largest (256 threads, named barrier): the
// r-th largest of min(keys[j] - sub, clamp), j < count, of keys in global
// memory; *rem = how many of the keys equal to it are among the r largest.
__device__ __noinline__ uint32_t grp_kth_largest(const uint32_t* keys, int count, uint32_t sub,
                                                 uint32_t clamp, int r, RadixShared& sh, int slot,
                                                 int& pc, int* rem, int ct) {
  assume_shared(&sh);
  const int lane = ct & 31;
  const int iters = (count + 255) >> 8;
  auto key_at = [&](int j) -> uint32_t {
    return min(__ldcg(keys + j) - sub, clamp);
  };
  uint32_t ko = 0u, ka = 0xFFFFFFFFu;
#pragma unroll 2
  for (int i = 0; i < iters; ++i) {
    const int j = (i << 8) + ct;
    if (j < count) {
      const uint32_t key = key_at(j);
      ko |= key;
      ka &= key;
    }
  }
  ko = __reduce_or_sync(0xffffffffu, ko);
  ka = __reduce_and_sync(0xffffffffu, ka);
  if (lane == 0) {
    atomicOr(&sh.key_or[slot], ko);
    atomicAnd(&sh.key_and[slot], ka);
  }
  cbar();
  const uint32_t diff = sh.key_or[slot] ^ sh.key_and[slot];
  const uint32_t kand = sh.key_and[slot];
  int remaining = r;
  if (diff == 0u) {
    *rem = remaining;
    return kand;
  }
  int hb = 31 - __clz(diff);
  uint32_t pmask = hb == 31 ? 0u : ~((2u << hb) - 1u);
  uint32_t prefix = kand & pmask;
#pragma unroll 1
  while (hb >= 0) {
    const int width = min(8, hb + 1);
    const int shf = hb + 1 - width;
    const uint32_t fm = (1u << width) - 1u;
    uint32_t* hh = sh.hist[pc & 3];
    constexpr int kB = 4;  // keys per thread loaded before they are counted
#pragma unroll 1
    for (int i0 = 0; i0 < iters; i0 += kB) {
      uint32_t bin[kB];
      bool m[kB];
#pragma unroll
      for (int q = 0; q < kB; ++q) {
        const int j = ((i0 + q) << 8) + ct;
        const uint32_t key = j < count ? key_at(j) : 0u;
        m[q] = j < count && (key & pmask) == prefix;
        bin[q] = (key >> shf) & fm;
      }
#pragma unroll
      for (int q = 0; q < kB; ++q) {
        // one add per distinct bin of the warp (no same-address serialisation)
        const uint32_t act = __ballot_sync(0xffffffffu, m[q]);
        if (act == 0u) continue;
        const uint32_t lb = __shfl_sync(0xffffffffu, bin[q], __ffs(act) - 1);
        if (__all_sync(0xffffffffu, !m[q] || bin[q] == lb)) {
          if (lane == __ffs(act) - 1) atomicAdd(&hh[lb], static_cast<uint32_t>(__popc(act)));
        } else if (m[q]) {
          const uint32_t same = __match_any_sync(act, bin[q]);
          if (lane == __ffs(same) - 1)
            atomicAdd(&hh[bin[q]], static_cast<uint32_t>(__popc(same)));
        }
      }
    }
    sh.hist[(pc + 2) & 3][ct] = 0u;
    cbar();
    int bin, above;
    warp_pick_bin256(hh, remaining, lane, &bin, &above);
    remaining -= above;
    prefix |= static_cast<uint32_t>(bin) << shf;
    pmask |= fm << shf;
    hb = shf - 1;
    ++pc;
  }
  *rem = remaining;
  return prefix;
}

// select_common.cuh's bisection by the worker warps.
struct WorkerBarrier {
  __device__ __forceinline__ void operator()() const { cbar(); }
};
template <int kPer>
__device__ __noinline__ uint32_t bisect_kth(const uint32_t* keys, int count, int r, int slack,
                                            SelShared& sh, int* need_eq, int ct) {
  assume_shared(&sh);
  assume_shared(keys);
  return bisect_largest<kPer>(keys, count, r, slack, sh.cnt, need_eq, ct, WorkerBarrier{});
}
__device__ __forceinline__ uint32_t shared_kth(const uint32_t* keys, int count, int r, int slack,
                                               SelShared& sh, int* need_eq, int ct) {
  if (count <= 4 * kCThreads) return bisect_kth<4>(keys, count, r, slack, sh, need_eq, ct);
  if (count <= 12 * kCThreads) return bisect_kth<12>(keys, count, r, slack, sh, need_eq, ct);
  return bisect_kth<24>(keys, count, r, slack, sh, need_eq, ct);
}
static_assert(kSelWhole <= 24 * kCThreads && kSelGroups <= 12 * kCThreads, "bisected keys");

// Ordered emission of the selected entries of a key list in position order:
// entry j (key keys[j], position pos[j], or j without a list) is selected when
// its key is above tau, or equal to tau and fewer than need_eq equal keys
// precede it.  Selected entries go to out[0..k) in list order.  Each warp has
// a contiguous part of the list: it counts, then (one barrier later) emits.
__device__ __noinline__ void emit_selected(int count, uint32_t tau, int need_eq, int32_t* out, int k,
                                           SelShared& sh, int ct, const uint32_t* keys,
                                           const int* pos) {
  assume_shared(&sh);
  const int cw = ct >> 5;
  const int lane = ct & 31;
  const int seg = (count + 255) >> 8 << 5;  // entries per warp
  const int j0 = min(count, cw * seg);
  const int j1 = min(count, j0 + seg);
  int o = 0, eq_seen = 0;
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    int gt_n = 0, eq_n = 0;
#pragma unroll 2
    for (int jb = j0; jb < j1; jb += 32) {
      const int j = jb + lane;
      const uint32_t key = j < j1 ? keys[j] : 0u;
      const uint32_t mgt = __ballot_sync(0xffffffffu, j < j1 && key > tau);
      const uint32_t meq = __ballot_sync(0xffffffffu, j < j1 && key == tau);
      if (pass == 0) {
        gt_n += __popc(mgt);
        eq_n += __popc(meq);
      } else if ((mgt | meq) != 0u) {
        const uint32_t lt = lanemask_lt(lane);
        const bool take = (meq >> lane & 1u) && eq_seen + __popc(meq & lt) < need_eq;
        const uint32_t msel = mgt | __ballot_sync(0xffffffffu, take);
        const int slot = o + __popc(msel & lt);
        if ((msel >> lane & 1u) && slot < k) out[slot] = pos ? pos[j] : j;
        o += __popc(msel);
        eq_seen += __popc(meq);
      }
    }
    if (pass == 0) {
      if (lane == 0) {
        sh.wcnt[cw] = gt_n;
        sh.wbase[cw] = eq_n;
      }
      cbar();
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        const int g = sh.wcnt[w], q = sh.wbase[w];
        if (w < cw) {
          o += g + max(0, min(need_eq - eq_seen, q));
          eq_seen += q;
        }
      }
    }
  }
}

// Copy the K and V rows of out[0..count) (positions in the sequence) to the
// compressed cache rows out0 .. out0 + count - 1 of group g: a warp per row
// (lanes 0-15 its K, 16-31 its V, 16 bytes each), eight rows in flight.  A
// position outside the sequence (never, for a correct selection) is skipped
// and recorded.
__device__ __noinline__ void gather_rows(const SelCall& p, int seq0, int L, int g,
                                         const int32_t* out, int out0, int count, int ct) {
  assume_shared(&p);
  constexpr int kBatch = 8;
  constexpr int kRow16 = kHeadDim * 2 / 16;
  const int lane = ct & 31;
  const int part = lane & 15;
  const uint4* src = (lane < 16 ? p.k : p.v) + static_cast<long long>(seq0) * p.tok_stride_v16 +
                     static_cast<long long>(g) * p.head_stride_v16 + part;
  uint4* dst = (lane < 16 ? p.k_out : p.v_out) +
               (static_cast<long long>(out0) * p.num_kv_heads + g) * kRow16 + part;
  const long long stride = p.tok_stride_v16;
  const int dstride = p.num_kv_heads * kRow16;
  bool bad = false;
#pragma unroll 1
  for (int i0 = ct >> 5; i0 < count; i0 += kBatch * (kCThreads / 32)) {
    int tok[kBatch];
    uint4 v[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int i = i0 + k * (kCThreads / 32);
      tok[k] = i < count ? out[i] : 0;
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const bool ok = tok[k] >= 0 && tok[k] < L;
      bad |= !ok;
      tok[k] = ok ? tok[k] : -1;
      if (ok && i0 + k * (kCThreads / 32) < count) v[k] = __ldg(src + tok[k] * stride);
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int i = i0 + k * (kCThreads / 32);
      if (i < count && tok[k] >= 0) dst[static_cast<long long>(i) * dstride] = v[k];
    }
  }
  if (bad) atomicCAS(p.status, 0, CKV_DEV_ERR_INDEX);
}

// The keys >= lo of the 32-key rows [r0, r1) of a unit (one warp, eight rows
// in flight), skipping the rows of groups (2^e rows) whose largest key is
// below lo.  Counts from o on; with ckey, the keys and their positions go to
// slots o, o + 1, ... below cap, in position order.
__device__ __noinline__ int scan_rows(const uint32_t* keys, int n, int r0, int r1, int e,
                                      const uint32_t* gmax, uint32_t lo, int o, uint32_t* ckey,
                                      int* cpos, int cap, int lane) {
  assume_shared(gmax);
  constexpr int kU = 8;
#pragma unroll 1
  for (int r = r0; r < r1; r += 32) {
    uint32_t m = __ballot_sync(0xffffffffu, r + lane < r1 && gmax[(r + lane) >> e] >= lo);
#pragma unroll 1
    while (m != 0u) {
      uint32_t kv[kU];
      int at[kU];
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        at[q] = m != 0u ? (r + __ffs(m) - 1) * 32 + lane : n;
        m &= m - 1u;
        kv[q] = at[q] < n ? __ldcg(keys + at[q]) : 0u;
      }
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        const bool c = at[q] < n && kv[q] >= lo;
        const uint32_t mm = __ballot_sync(0xffffffffu, c);
        const int slot = o + __popc(mm & lanemask_lt(lane));
        if (ckey && c && slot < cap) {
          ckey[slot] = kv[q];
          cpos[slot] = at[q];
        }
        o += __popc(mm);
      }
    }
  }
  return o;
}

struct SelUnit {
  int g, seq0, L, W, out0, kept;
};

// Pools the unit's raw scores (sum from j - h to j + h, zeros outside [0, n),
// over P); writes them to `pooled` and, as keys, to `keys` when the unit is
// small enough for it (n <= kSelWhole), else keeps the largest of every group of
// 32 << e keys.  A warp takes every eighth strip of kPoolStrip keys, through
// its own part of shared memory and with the loads of its next two strips in
// flight.  Bound by instruction latency (two warps per scheduler): 22-27 us
// for 32736 keys with the seven taps of the usual width unrolled, 33-42 us
// with a loop over them.
// kRows: only the keys [j0, j1) of such a unit, the largest of every row of 32
// to rowmax.
template <bool kRows>
__device__ __forceinline__ void pool_strips(const float* raw, float* pooled, uint32_t* rowmax,
                                            int n, int j0, int j1, int e, int h, float fP,
                                            SelShared& sh, int ct) {
  constexpr int kPer = kPoolStrip / 32;          // keys per lane
  constexpr int kLoads = kPoolBuf / 32;  // with the halo
  assume_shared(&sh);
  const int lane = ct & 31;
  const bool keep = !kRows && n <= kSelWhole;
  float* const stage =
      (keep ? reinterpret_cast<float*>(sh.gmax) : reinterpret_cast<float*>(sh.pos)) +
      (ct >> 5) * kPoolBuf;
  float na[kLoads], nb[kLoads];
  auto load = [&](float (&nx)[kLoads], int base) {
#pragma unroll
    for (int q = 0; q < kLoads; ++q) {
      const int i = q * 32 + lane;
      const int j = base - h + i;
      nx[q] = i < kPoolStrip + 2 * h && j >= 0 && j < n ? __ldcg(raw + j) : 0.f;
    }
  };
  auto step = [&](float (&nx)[kLoads], int base) {
    __syncwarp();  // the strip before is read
#pragma unroll
    for (int q = 0; q < kLoads; ++q) stage[q * 32 + lane] = nx[q];
    __syncwarp();
    load(nx, base + 16 * kPoolStrip);
    float s[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) s[q] = 0.f;
    const float* a = stage + lane;
    if (h == 3) {  // the usual width, without a load's latency per tap
#pragma unroll
      for (int t = 0; t < 7; ++t)
#pragma unroll
        for (int q = 0; q < kPer; ++q) s[q] += a[q * 32 + t];
    } else {
#pragma unroll 4
      for (int t = 0; t <= 2 * h; ++t)
#pragma unroll
        for (int q = 0; q < kPer; ++q) s[q] += a[q * 32 + t];
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) s[q] = s[q] / fP;
    if (keep) {
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const int j = base + q * 32 + lane;
        if (j < n) pooled[j] = s[q];
        if (j < n) sh.key[j] = __float_as_uint(s[q]);
      }
    } else {
      uint32_t top = 0u;  // lane q: the largest of row q
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const int j = base + q * 32 + lane;
        const bool in = j < n;
        if (in) pooled[j] = s[q];
        const uint32_t m = __reduce_max_sync(0xffffffffu, in ? __float_as_uint(s[q]) : 0u);
        top = lane == q ? m : top;
      }
      if (lane < kPer && base + 32 * lane < n) {
        if constexpr (kRows) {
          rowmax[(base >> 5) + lane] = top;
        } else {
          atomicMax(&sh.gmax[(base + 32 * lane) >> (5 + e)], top);
        }
      }
    }
  };
  const int base0 = j0 + (ct >> 5) * kPoolStrip;
  load(na, base0);
  load(nb, base0 + 8 * kPoolStrip);
#pragma unroll 1
  for (int base = base0; base < j1; base += 16 * kPoolStrip) {
    step(na, base);
    if (base + 8 * kPoolStrip < j1) step(nb, base + 8 * kPoolStrip);
  }
}
__device__ __noinline__ void pool_unit(const float* raw, float* pooled, int n, int e, int h, float fP,
                                       SelShared& sh, int ct) {
  pool_strips<false>(raw, pooled, nullptr, n, 0, n, e, h, fP, sh, ct);
}

// Pooling in pieces: the units whose keys do not fit shared memory are pooled by
// all CTAs, a piece at a time, before one CTA selects (one 131072-token layer:
// 226 -> 163 us, 32768: 90 -> 82).  Where it gains nothing its code in the
// kernels costs 2-10% (32 layers of short prompts: 481 -> 536 us), so that they
// are instantiated with and without it.  A third instance is for calls whose
// layers take both kernels: it skips the other's sequences and pools in pieces
// or not (that code in the others costs 1-3%).
constexpr int kPlain = 0, kInPieces = 1, kMixed = 2;
constexpr int kPoolPiece = 32 * kPoolStrip;  // keys of a pooling task
__device__ __forceinline__ int pool_pieces(int n) {
  return n <= kSelWhole ? 0 : (n + kPoolPiece - 1) / kPoolPiece;
}
// One piece by the 256 threads, which then adds to *count.
__device__ __noinline__ void pool_piece(const float* raw, float* pooled, uint32_t* rowmax, int n,
                                        int piece, const SelCall& p, SelShared& sh, int* count,
                                        int add, int ct) {
  assume_shared(&p);
  const int j0 = piece * kPoolPiece;
  pool_strips<true>(raw, pooled, rowmax, n, j0, min(n, j0 + kPoolPiece), 0, (p.pool_width - 1) >> 1,
                    static_cast<float>(p.pool_width), sh, ct);
  __threadfence_block();
  cbar();
  if (ct == 0) {
    fence_acq_rel_gpu();  // (cumulative: the barrier's other writes too)
    atomicAdd(count, add);
  }
}

// The workers' tasks then, in one order that every CTA takes tickets of: of
// every unit its pieces, then its selection (pieces(s) -1: no tasks).  A ticket is taken before its
// task is ready: claims by compare-and-swap once a task is ready took 1 us
// apiece (152 CTAs at one counter).
struct TaskPos {
  int t;                    // the ticket; -1: none taken
  int s, off;               // a sequence at or before its own, the tickets before that
  int unit, piece, pieces;  // its task (unit -1: past the last); piece -1: the selection
};
template <class Pieces>
__device__ __forceinline__ void take_ticket(TaskPos& T, int* counter, int batch, int Hkv,
                                            Pieces pieces) {
  T.t = atomicAdd(counter, 1);
  T.unit = -1;
  for (; T.s < batch; ++T.s) {
    T.pieces = pieces(T.s);
    const int per = T.pieces + 1;
    const int r = T.t - T.off;
    if (r < Hkv * per) {
      const int g = r / per;
      T.unit = T.s * Hkv + g;
      T.piece = r - g * per;
      if (T.piece == T.pieces) T.piece = -1;
      return;
    }
    T.off += Hkv * per;
  }
}

// Selection of a unit.  Pooling (of a unit that was not pooled in pieces),
// then the top-k: a unit of at most
// kSelWhole prefix keys by bisection over its keys in shared
// memory; a longer one by a lower bound of the k-th largest score -- the k-th
// largest group maximum (k groups have a key at least that large) or, with
// fewer groups than k, a rank among samples -- then the candidates in position
// order and the bisection among them (a radix search among those in global
// memory, or all the unit's scores, when the bound keeps too few or too many); then the window and the K/V rows.  Pooled
// scores are >= 0: their bit patterns order like their values.
template <int kKind>
__device__ __noinline__ void select_unit(const SelCall& p, const SelUnit U, float* raw,
                                         float* pooled, int32_t* out, uint8_t* creg, int ct) {
  assume_shared(creg);
  assume_shared(&p);
  SelShared& sh = *reinterpret_cast<SelShared*>(creg);
  const int cw = ct >> 5;
  const int lane = ct & 31;
  const int L = U.L;
  const int W = U.W;
  const int n = max(L - W, 0);
  int e = 0;  // groups of 2^e rows of 32 keys
  while (((n + 31) >> 5) > (kSelGroups << e)) ++e;
  const int nr = (n + 31) >> 5;
  const int ng = (nr + (1 << e) - 1) >> e;
  if (kKind != kPlain && n > kSelWhole && (kKind == kInPieces || sh.rowmax)) {
    const uint32_t* const rowmax = sh.rowmax;
#pragma unroll 4
    for (int i = ct; i < ng; i += kCThreads) {
      uint32_t m = 0u;
      for (int r = i << e; r < min(nr, (i + 1) << e); ++r) m = max(m, __ldcg(rowmax + r));
      sh.gmax[i] = m;
    }
  } else {
    for (int i = ct; i < ng; i += kCThreads) sh.gmax[i] = 0u;
    cbar();
    pool_unit(raw, pooled, n, e, (p.pool_width - 1) >> 1, static_cast<float>(p.pool_width), sh, ct);
  }
  __threadfence_block();
  cbar();
  const int kept = U.kept;
  if (kept >= L) {  // keep everything
    for (int i = ct; i < L; i += kCThreads) out[i] = i;
    __threadfence_block();
    cbar();
    gather_rows(p, U.seq0, L, U.g, out, U.out0, L, ct);
    return;
  }
  const int k = kept - W;  // 0 <= k < n
  for (int w = ct; w < W; w += kCThreads) out[k + w] = n + w;
  if (k > 0) {
    const uint32_t* keys = reinterpret_cast<const uint32_t*>(pooled);
    uint32_t* samp = reinterpret_cast<uint32_t*>(sh.pos);
    const int seg = (nr + 7) >> 3;  // rows per warp
    const int r0 = min(nr, cw * seg);
    const int r1 = min(nr, r0 + seg);
    int pc = 0, need_eq = 0;
    uint32_t lo = 0, lo_ge = 0;
    int total = 0, tot_ge = -1;
    bool fast = false;
    const bool whole = n <= kSelWhole;  // every key is in shared memory
    bool by_group = ng >= k;
    const int ns = min(kSelSamples, n);
    const float mu = static_cast<float>(k) * static_cast<float>(ns) / static_cast<float>(n);
    int rs = min(ns, static_cast<int>(ceilf(mu + 3.f * sqrtf(mu))) + 2);
#pragma unroll 1
    for (int attempt = whole ? 2 : (by_group ? -1 : 0); attempt < 2; ++attempt) {
      if (attempt == 0)
        for (int i = ct; i < ns; i += kCThreads)
          samp[i] = __ldcg(keys + static_cast<int>((static_cast<long long>(i) * n) / ns));
      cbar();
      by_group = attempt < 0;
      lo = shared_kth(by_group ? sh.gmax : samp, by_group ? ng : ns, by_group ? k : rs,
                      by_group ? k >> 4 : 0, sh, &need_eq, ct);
      const int wc = scan_rows(keys, n, r0, r1, e, sh.gmax, lo, 0, nullptr, nullptr, 0, lane);
      if (lane == 0) sh.wcnt[cw] = wc;
      cbar();
      total = 0;
      for (int w = 0; w < 8; ++w) total += sh.wcnt[w];
      if (total >= k && (tot_ge < 0 || total < tot_ge)) {
        lo_ge = lo;
        tot_ge = total;
        if (ct < 8) sh.wcnt_ge[ct] = sh.wcnt[ct];
      }
      fast = total >= k && total <= kFusedCandCap;
      if (fast) break;
      cbar();  // every thread has read the counts
      if (by_group) continue;
      // aim at the middle of [k, capacity] from the density this attempt saw
      const float per = static_cast<float>(max(total, 1)) / static_cast<float>(rs);
      int want = static_cast<int>(ceilf(0.5f * static_cast<float>(k + kFusedCandCap) / per));
      want = total < k ? max(want, rs + 1) : min(want, rs - 1);
      if (want < 1 || want > ns || want == rs) break;
      rs = want;
    }
    // the candidates' radix starts afresh
    cbar();
    radix_init_grp(sh.rs, ct);
    pc = 0;
    need_eq = 0;
    // The candidates (keys >= lo) in position order: in shared memory when at
    // most kFusedCandCap, else -- when the raw scores are workspace, last read
    // above -- in the unit's raw-score row, keys in its first half and
    // positions in its second; else all of the unit's keys.
    const uint32_t* ckey = keys;
    const int* cpos = nullptr;
    int count = n;
    bool in_shared = true;
    if (whole) {
      ckey = sh.key;
    } else if (!fast && p.raw_scratch && tot_ge >= k && tot_ge <= n / 2) {
      lo = lo_ge;
      total = tot_ge;
      if (ct < 8) sh.wcnt[ct] = sh.wcnt_ge[ct];
      ckey = reinterpret_cast<uint32_t*>(raw);
      cpos = reinterpret_cast<int*>(raw + n / 2);
      count = total;
      in_shared = false;
    } else if (fast) {
      ckey = sh.key;
      cpos = sh.pos;
      count = total;
    } else {
      in_shared = false;
    }
    cbar();
    if (cpos) {
      int o = 0;
      for (int w = 0; w < cw; ++w) o += sh.wcnt[w];
      scan_rows(keys, n, r0, r1, e, sh.gmax, lo, o, const_cast<uint32_t*>(ckey),
                const_cast<int*>(cpos), total, lane);
      __threadfence_block();
      cbar();
    } else {
      lo = 0u;
    }
    uint32_t tau;
    if (in_shared) {
      tau = shared_kth(ckey, count, k, 0, sh, &need_eq, ct);
    } else {
      // offsets above the bound, clamped to 16 bits: at most two radix passes
      const uint32_t clamp = cpos ? 0xFFFFu : 0xFFFFFFFFu;
      const uint32_t td = grp_kth_largest(ckey, count, lo, clamp, k, sh.rs, 0, pc, &need_eq, ct);
      tau = lo + td;
      if (cpos && td == clamp)
        tau = grp_kth_largest(ckey, count, 0u, 0xFFFFFFFFu, k, sh.rs, 1, pc, &need_eq, ct);
    }
    emit_selected(count, tau, need_eq, out, k, sh, ct, ckey, cpos);
  }
  __threadfence_block();
  cbar();  // the indices written above are read back by the copy
  gather_rows(p, U.seq0, L, U.g, out, U.out0, kept, ct);
}

}  // namespace
}  // namespace ckv
