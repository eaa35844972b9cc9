// Persistent fused layer call (CompressKV Sec. 3.3 token selection with the
// SnapKV-style window of Sec. 4) for per-group selection: one launch scores
// every unit (sequence, KV group) of a call -- typically every layer of a
// model at the end of prefill -- pools the scores, takes the budgeted top-k,
// appends the window and gathers the retained K/V rows.
//
// For unit (s, g), with Q_S the N = |S_g| * W window-query rows of the
// group's SRH heads, z = <q, k> * scale and c = log2(e), query q (window
// position p_q) attends key j <= p_q with 2^(z_qj c) / D_q,
// D_q = sum_{j <= p_q} 2^(z_qj c).  The kernel makes two passes over the
// unit's K, both on tcgen05 tensor cores (logits in TMEM):
//   pass 1  per query row and epilogue warpgroup the pair (M, S) with
//           sum 2^(z c) = S 2^M over its tiles of a chunk of kChunkTiles K
//           tiles (each epilogue warp sums 2^(z c - R) against a reference R
//           per query row, its first scaled logit, raised when a sum passes
//           2^64); the workers merge a unit's pairs into log2 D_q once every
//           chunk of the unit is in;
//   pass 2  raw_j = sum_q 2^(z_qj c - log2 D_q) over the unit's prefix keys
//           j < n = L - W, straight from the logits in fp32; pass 2 of a
//           chunk is published only once its unit's denominators are merged
//           (it reads K again: in long calls pass 1 runs too far ahead for
//           L2 to keep it, so mostly from DRAM);
// then (unit_select.cuh) pooled_j = (sum_{t=-h..h} raw_{j+t}) / P with zeros
// outside [0, n), the k = kept - W largest pooled scores (ties to the lower
// position) in ascending position, the window, and the K/V rows.
// With the window queries' log-sum-exp given (given_lse) pass 1 is skipped
// and log2 D_q = LSE_q * log2(e).
//
// One CTA per SM runs for the whole call.  Its warps have fixed roles:
//   warp 3      claims chunks (a pass-2 chunk once its unit's denominators
//               are merged, else the next pass-1 chunk) and publishes them,
//               up to kDescs ahead, in a descriptor ring;
//   warp 0      loads each chunk's SRH query rows (one TMA box of W rows per
//               head and 64-column half) into one of two or three Q buffers
//               and streams its K tiles, by TMA, into a shared-memory ring;
//   warp 1      UMMA issue (M = 128 keys, N = query rows) in tile order, by
//               the whole warp with one lane issuing, and the TMEM
//               allocation.  (Two issuers, one per warpgroup, interleaved
//               their UMMAs, so that both warpgroups' tiles came late and at
//               the same time, and tensor-memory loads queued behind them.)
//   warps 4-11  two epilogue warpgroups; tile t of a chunk belongs to
//               warpgroup t % 2, each with its own TMEM buffers;
//   warps 12-19 workers: they merge a unit's pass-1 pairs into its
//               denominators once all its chunks are in, and select and
//               gather a unit once all its pass-2 chunks are in (one CTA per
//               unit).
// A pass-2 chunk is published once its claimer has seen (acquire) its unit's
// denominators merged; workers claim a merge only when it is ready, take
// tickets of the selections in order and merge while their own is not ready.
// Every wait therefore depends only on work claimed earlier by a running CTA
// that never waits on later work, so a
// call completes whatever the number of CTAs resident at once; every wait
// is bounded (FusedParams::wait_ns, kWaitTimeoutNs unless a test shortens it)
// and on expiry records CKV_ERR_DEVICE_TIMEOUT
// and stops the call.
// What bounds it: up to 64 query rows DRAM, both passes' reads (32 layers of
// 32768 tokens, 680 us); 128 and 192 rows the epilogue and, with few K stages
// beside the Q buffers, the loads' latency (16 layers of 32768 tokens: 433 and
// 649 us, 567 and 911 with one logit per register and key-per-lane sums and
// two UMMA issuers).
// References restart at every chunk and tile t of a chunk always goes to
// warpgroup t % 2, so the scores depend only on the chunk grid (fixed per
// unit), not on which CTA ran a chunk or what else the call holds.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cfloat>

#include "ckv_device.cuh"
#include "tile_math.cuh"
#include "unit_select.cuh"

namespace ckv {

namespace {

constexpr int kFWarps = 20;
constexpr int kFThreads = 32 * kFWarps;
constexpr int kProdWarp = 0;
constexpr int kMmaWarp = 1;
constexpr int kClaimWarp = 3;
constexpr int kEpiWarp0 = 4;  // warps 4..11: two warpgroups (TMEM lane quarter = warp % 4)
constexpr int kEpiWarps = 8;
constexpr int kCWarp0 = 12;   // warps 12..19
constexpr int kDescs = 2;     // chunk descriptors in flight (claimed ahead; 2 measured faster than 4)
constexpr int kNwg = kFusedPartsPerChunk;  // epilogue warpgroups (tile t of a chunk: t % kNwg)
constexpr int kPub = 6;       // chunks written, not yet published (publish ring)
constexpr float kShift = 7.0f;
constexpr float kRaiseSum = 18446744073709551616.0f;  // 2^64: fp32 column sums stay below it before R is raised
constexpr float kNegInf = -INFINITY;

// counters (ints at p.ctr)
constexpr int kCtrPass1 = 0;  // next pass-1 chunk
constexpr int kCtrPass2 = 1;  // next pass-2 chunk
constexpr int kCtrMerge = 2;  // next unit whose denominators to merge
constexpr int kCtrExit = 4;   // CTAs finished
constexpr int kCtrAbort = 5;  // set when any wait ran out
constexpr int kCtrTicket = 7; // the workers' next ticket
constexpr int kCtrNever = 6;  // never set: the test hook's stall waits for it

constexpr int kTaskEnd = 0;
constexpr int kTaskMerge = 1;
constexpr int kTaskSelect = 2;
constexpr int kTaskPool = 3;

struct ChunkDesc {
  int end, pass, s, g, t0, t1, chunk, n_rows;
};

static_assert(3 * kMaxQRows * 4 + 16 <= kSelRegion, "merge scratch");

constexpr int kWposBytes = kMaxQRows * 4;
constexpr int kBarBytes = 512;
static_assert((51 + 2 * kPub) * 8 <= kBarBytes, "mbarriers (the publish ring's last) fit their block");
constexpr int kMiscBytes = 256;  // TMEM address, abort flag, task, the selection's parameters
static_assert(64 + sizeof(SelCall) <= kMiscBytes, "misc block");
constexpr int kFixedBytes = kWposBytes + kBarBytes + kMiscBytes +
                            kDescs * static_cast<int>(sizeof(ChunkDesc));

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int ld_volatile(const int* p) {
  return *reinterpret_cast<const volatile int*>(p);
}

// Index of the i-th set bit of `bits` (i < popc(bits)).
__device__ __forceinline__ int nth_bit(uint32_t bits, int i) {
  for (int j = 0; j < i; ++j) bits &= bits - 1u;
  return __ffs(bits) - 1;
}

// Largest s in [0, n) with off[s] <= x (off ascending, off[n] > x).
__device__ __forceinline__ int find_seq(const int* off, int n, int x) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (off[mid] <= x) lo = mid; else hi = mid;
  }
  return lo;
}

struct Fused {
  const FusedParams& p;
  int* abort_cta;  // shared-memory abort flag of this CTA

  __device__ int len(int s) const { return p.cu_seqlens[s + 1] - p.cu_seqlens[s]; }
  __device__ int prefix(int s) const { return max(len(s) - p.window, 0); }
  __device__ int tiles(int s) const { return (len(s) + kTileTokens - 1) / kTileTokens; }
  __device__ int chunks_per_unit(int s) const {
    return (p.chunk_off[s + 1] - p.chunk_off[s]) / p.num_kv_heads;
  }
  // a sequence of a layer that the resident kernel takes
  __device__ bool not_here(int s) const {
    return p.chunk_off[s + 1] == p.chunk_off[s] && prefix(s) > 0;
  }
  // unit u, or the first unit after it whose sequence has chunks to merge
  __device__ int next_merge(int u) const {
    int s = u / p.num_kv_heads;
    if (s * p.num_kv_heads != u || s >= p.batch || chunks_per_unit(s) > 0) return u;
    do ++s; while (s < p.batch && chunks_per_unit(s) == 0);
    return s * p.num_kv_heads;
  }
  __device__ int list(int s, int g) const { return srh_group(s, g, p.seqs_per_mask, p.num_kv_heads); }
  __device__ int rows(int s, int g) const { return __popc(p.srh_bits[list(s, g)]) * p.window; }
  __device__ int* ticket(int u) const { return p.ctr + kFusedCtrHead + u; }
  __device__ int* p2done(int u) const { return p.ctr + kFusedCtrHead + p.n_units + u; }
  // 2 once the unit's denominators are merged, and 4 more per piece pooled
  __device__ int* bias_state(int u) const { return p.ctr + kFusedCtrHead + 2 * p.n_units + u; }
  __device__ bool aborted() const { return ld_volatile(p.ctr + kCtrAbort) != 0; }
  __device__ void raise_abort() const {
    atomicCAS(p.status, 0, CKV_DEV_ERR_TIMEOUT);
    atomicExch(p.ctr + kCtrAbort, 1);
    *reinterpret_cast<volatile int*>(abort_cta) = 1;
  }
  // Bounded wait (another CTA's progress) until *ptr >= target; false when
  // the call was aborted or the wait ran out.
  __device__ bool wait_counter(const int* ptr, int target) const {
    if (ld_acquire(ptr) >= target) return true;
    const uint64_t t0 = globaltimer_ns();
    for (;;) {
      __nanosleep(64);
      if (ld_acquire(ptr) >= target) return true;
      if (aborted() || *reinterpret_cast<volatile int*>(abort_cta)) return false;
      if (globaltimer_ns() - t0 > p.wait_ns) {
        raise_abort();
        return false;
      }
    }
  }
  // Bounded wait on one of this CTA's mbarriers; a timeout stops the call.
  __device__ bool wait_bar(uint32_t bar, uint32_t parity) const {
    if (mbar_test_wait(bar, parity)) return true;
    const bool ok = mbar_wait_bounded(bar, parity, abort_cta, p.status, p.wait_ns);
    if (!ok && !aborted()) atomicExch(p.ctr + kCtrAbort, 1);
    return ok;
  }
};

// ---------------------------------------------------------------- publishing
// The claimer thread publishes the chunks the epilogue has finished, in
// order: after the epilogue warps' arrivals (CTA-scope release/acquire) one
// GPU-scope fence covers a batch of finished chunks, then each chunk adds to
// its unit's counter (pass 1: the ticket the merge waits for; pass 2: the
// count the selection waits for).  The fence's wait for the writes thus
// stalls neither the epilogue nor the tile pipeline.
struct Publisher {
  const Fused& F;
  uint32_t full0, empty0;  // the publish ring's barriers
  int info[kPub];          // chunk i (slot i % kPub): unit * 2 + pass - 1
  int next, issued;        // first chunk not yet published; chunks issued

  __device__ uint32_t full(int i) const { return full0 + 8u * static_cast<uint32_t>(i % kPub); }
  __device__ uint32_t empty(int i) const { return empty0 + 8u * static_cast<uint32_t>(i % kPub); }
  __device__ void pump() {
    int k = next;
    while (k < issued && mbar_test_wait(full(k), static_cast<uint32_t>(k / kPub) & 1u)) ++k;
    if (k == next) return;
    fence_acq_rel_gpu();
    for (; next < k; ++next) {
      const int v = info[next % kPub];
      if (v & 1) {
        atomicAdd(F.p2done(v >> 1), kEpiWarps);
      } else {
        atomicAdd(F.ticket(v >> 1), kNwg);
      }
      mbar_arrive(empty(next));
    }
  }
  // Bounded wait on one of the CTA's mbarriers, publishing meanwhile.
  __device__ bool wait_bar(uint32_t bar, uint32_t parity) {
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t it = 1;; ++it) {
      if (mbar_try_wait(bar, parity)) return true;
      pump();
      if ((it & 63u) == 0 && !still_waiting(t0)) return false;
    }
  }
  // Bounded wait until at most `left` issued chunks are unpublished.
  __device__ bool wait_published(int left) {
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t it = 1; issued - next > left; ++it) {
      pump();
      __nanosleep(32);
      if ((it & 63u) == 0 && !still_waiting(t0)) return false;
    }
    return true;
  }
  __device__ bool still_waiting(uint64_t t0) const {
    if (F.aborted() || *reinterpret_cast<volatile int*>(F.abort_cta)) return false;
    if (globaltimer_ns() - t0 > F.p.wait_ns) {
      F.raise_abort();
      return false;
    }
    return true;
  }
};

// ---------------------------------------------------------------- claims
// The next chunk of this CTA.  Each claimer holds at most one pass-2 chunk it
// has claimed (*pending, taken with atomicAdd as soon as the previous one was
// published) and publishes it once its unit's denominators are merged (with
// the LSE given: at once); until then it claims pass-1 chunks.  Pass 1 keeps
// advancing while pass-2 chunks wait, and a pass-2 chunk never reaches the
// epilogue before its denominators.  When pass 1 is exhausted the claimer
// waits (bounded) for its pending chunk's unit, whose pass-1 chunks are then
// all claimed.  Returns false when both passes are exhausted (or aborted).
__device__ bool claim_chunk(const Fused& F, Publisher& pb, int* pending, int* pass, int* x) {
  const FusedParams& p = F.p;
  for (;;) {
    if (F.aborted() || *reinterpret_cast<volatile int*>(F.abort_cta)) return false;
    if (*pending < 0 && ld_volatile(p.ctr + kCtrPass2) < p.n_chunks) {
      const int y = atomicAdd(p.ctr + kCtrPass2, 1);
      if (y < p.n_chunks) *pending = y;
    }
    int u = -1;
    if (*pending >= 0) {
      const int s = find_seq(p.chunk_off, p.batch, *pending);
      u = s * p.num_kv_heads + (*pending - p.chunk_off[s]) / F.chunks_per_unit(s);
      if (p.given_lse || ld_acquire(F.bias_state(u)) >= 2) {
        *pass = 2;
        *x = *pending;
        *pending = -1;
        return true;
      }
    }
    if (!p.given_lse && ld_volatile(p.ctr + kCtrPass1) < p.n_chunks) {
      const int y = atomicAdd(p.ctr + kCtrPass1, 1);
      if (y < p.n_chunks) {
        *pass = 1;
        *x = y;
        return true;
      }
      continue;
    }
    if (*pending < 0) return false;  // both passes exhausted
    // pass 1 is exhausted: every pass-1 chunk of the pending chunk's unit is
    // claimed; wait (bounded) for its merge, publishing meanwhile (the merge
    // may wait for tickets this CTA holds)
    const uint64_t t0 = globaltimer_ns();
    while (ld_acquire(F.bias_state(u)) < 2) {
      pb.pump();
      __nanosleep(64);
      if (!pb.still_waiting(t0)) return false;
    }
  }
}

// ---------------------------------------------------------------- merge
// log2 D_q of unit u from its pass-1 pairs (one per chunk and warpgroup that
// takes tiles; one that got no tile of a chunk leaves (-inf, 0)), 256 worker
// threads: nm threads per query row, sixteen pairs in flight per thread.
__device__ __noinline__ void merge_unit(const Fused& F, int u, uint8_t* creg, int ct) {
  const FusedParams& p = F.p;
  const int s = u / p.num_kv_heads;
  const int g = u - s * p.num_kv_heads;
  const int N = F.rows(s, g);
  const int ncu = F.chunks_per_unit(s);
  float* s_mm = reinterpret_cast<float*>(creg);  // [256]
  float* s_mz = s_mm + kMaxQRows;                 // [256]
  if (ncu > 0 && N > 0) {
    constexpr int nwg = kNwg;
    const int nparts = nwg * ncu;  // the unit's chunks are consecutive
    const float2* parts = p.partials + static_cast<long long>(p.chunk_off[s] + g * ncu) *
                                           kFusedPartsPerChunk * p.part_stride;
    const int nm = kCThreads / N;
    const int q = ct % N;
    const int sub = ct / N;
    if (sub < nm) {
      float m = kNegInf, z = 0.f;
      for (int i0 = sub; i0 < nparts; i0 += 16 * nm) {
        float2 pr[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const int i = i0 + k * nm;  // pair i: chunk i / nwg, warpgroup i % nwg
          pr[k] = i < nparts
                      ? __ldcg(parts + (static_cast<long long>(i / nwg) * kFusedPartsPerChunk +
                                        i % nwg) * p.part_stride + q)
                      : make_float2(kNegInf, 0.f);
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          if (pr[k].x == kNegInf) continue;
          if (pr[k].x > m) {
            z = fmaf(z, ex2_approx(m - pr[k].x), pr[k].y);
            m = pr[k].x;
          } else {
            z = fmaf(pr[k].y, ex2_approx(pr[k].x - m), z);
          }
        }
      }
      s_mm[sub * N + q] = m;  // nm * N <= 256
      s_mz[sub * N + q] = z;
    }
    cbar();
    if (ct < N) {
      float m = kNegInf, z = 0.f;
      for (int j = 0; j < nm; ++j) {
        const float pm = s_mm[j * N + ct];
        const float pz = s_mz[j * N + ct];
        if (pm == kNegInf) continue;
        if (pm > m) {
          z = fmaf(z, ex2_approx(m - pm), pz);
          m = pm;
        } else {
          z = fmaf(pz, ex2_approx(pm - m), z);
        }
      }
      p.bias[static_cast<long long>(u) * p.part_stride + ct] = m + __log2f(z);
    }
  }
  fence_acq_rel_gpu();
  cbar();
  if (ct == 0) atomicExch(F.bias_state(u), 2);
}

// The workers' next task (one thread): the ticket's (a piece to pool once all
// the unit's pass-2 chunks are in, a selection then or once its pieces are
// pooled), or meanwhile the next unit to merge once all its pass-1 chunks are
// in; waits (bounded) while neither is ready.  (Claims by compare-and-swap of
// the next ready selection cost 1 us apiece: 48 layers of 12288 tokens of 128
// rows 720 -> 486 us with tickets, 60 layers of 4 prompts of 500 to 9000 of 64
// to 192 rows 3250 -> 1850.)
template <int kKind>
__device__ void claim_ticket(const Fused& F, TaskPos& T, int* task) {
  const FusedParams& p = F.p;
  if (T.t < 0)
    take_ticket(T, p.ctr + kCtrTicket, p.batch, p.num_kv_heads, [&](int s) {
      if (kKind == kMixed && F.not_here(s)) return -1;
      return kKind == kInPieces || (kKind == kMixed && p.in_pieces) ? pool_pieces(F.prefix(s)) : 0;
    });
  // what the task waits for; without one (every selection is ahead of the
  // first ticket past the last), the other units' merges
  const int* word = p.ctr + kCtrMerge;
  int target = p.given_lse ? 0 : (kKind == kMixed && F.next_merge(0) == p.n_units ? 0 : p.n_units);
  if (T.unit >= 0) {
    const bool pooled = kKind != kPlain && T.piece < 0 && T.pieces > 0;
    word = pooled ? F.bias_state(T.unit) : F.p2done(T.unit);
    target = pooled ? 4 * T.pieces : kEpiWarps * F.chunks_per_unit(T.s);
  }
  const int first = kKind == kMixed ? F.next_merge(0) : 0;
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    if (F.aborted() || *reinterpret_cast<volatile int*>(F.abort_cta)) break;
    if (ld_acquire(word) >= target) {
      if (T.unit < 0) break;
      task[0] = T.piece < 0 ? kTaskSelect : kTaskPool;
      task[1] = T.unit;
      task[2] = T.piece;
      if (kKind == kMixed) task[3] = T.pieces;
      T.t = -1;
      return;
    }
    if (!p.given_lse) {
      const int at = ld_volatile(p.ctr + kCtrMerge);
      const int m = kKind == kMixed ? max(at, first) : at;
      if (m < p.n_units &&
          ld_acquire(F.ticket(m)) >= kNwg * F.chunks_per_unit(m / p.num_kv_heads)) {
        if (atomicCAS(p.ctr + kCtrMerge, at, kKind == kMixed ? F.next_merge(m + 1) : m + 1) == at) {
          task[0] = kTaskMerge;
          task[1] = m;
          return;
        }
        continue;
      }
    }
    if (globaltimer_ns() - t0 > p.wait_ns) {
      F.raise_abort();
      break;
    }
    __nanosleep(128);
  }
  task[0] = kTaskEnd;
  task[1] = 0;
}

// Pass 1, rare: an exponent of this 32-column group passed 2^64 (or the
// references are still -inf): raise every query's R to kShift below its
// largest scaled logit among the warp's 32 keys, shrink the sums kept against
// the old R, and return this group's column sums against the new R (column
// lane).  The whole warp calls it; taddr is the group's first TMEM column.
__device__ __noinline__ float p1_raise_group(uint32_t taddr, float* rf, float* acc_c,
                                             const int* wpos, int lim, bool edge, bool key,
                                             int vis, float c, int lane) {
  uint32_t r[32];
  tmem_load32_async(taddr, r);
  tmem_wait_ld(r);
  uint32_t valid = 0u;
  float v[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const bool ok = j < lim && (!edge || (key && wpos[j] >= -vis));
    valid |= (ok ? 1u : 0u) << j;
    v[j] = ok ? __uint_as_float(r[j]) * c : kNegInf;
  }
  const float m = warp_transpose_max32(v, lane);  // column lane
  const float old = rf[lane];
  const float nw = fmaxf(old, m - kShift);
  acc_c[lane] *= (nw == old) ? 1.f : ((old == kNegInf) ? 0.f : ex2_approx(old - nw));
  __syncwarp();
  rf[lane] = nw;
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 32; ++j)
    v[j] = ((valid >> j) & 1u) ? ex2_approx(fmaf(__uint_as_float(r[j]), c, -rf[j])) : 0.f;
  return warp_transpose_sum32(v, lane);
}

__device__ __forceinline__ void wait_plain(uint32_t bar, uint32_t parity, uint64_t timeout_ns) {
  volatile int never = 0;
  mbar_wait_bounded(bar, parity, &never, nullptr, timeout_ns);
}

template <int kKind>
__global__ void __launch_bounds__(kFThreads, 1) fused_kernel(const __grid_constant__ FusedParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const int nst = p.stages;
  const int qh = p.q_half_bytes;
  const int rstride = p.row_stride;
  uint8_t* sK = base;
  const int nqb = p.q_bufs;
  uint8_t* sQ = base + nst * kTileBytes;  // nqb buffers of two 64-column halves
  const int nrow = 4 * kNwg;  // epilogue warps that take tiles
  float* sRef = reinterpret_cast<float*>(sQ + 2 * nqb * qh);  // [nrow][rstride]
  float* sAcc = sRef + nrow * rstride;                        // [nrow][rstride]
  int* sWpos = reinterpret_cast<int*>(sAcc + nrow * rstride);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sWpos + kMaxQRows);
  uint8_t* misc = reinterpret_cast<uint8_t*>(bars) + kBarBytes;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(misc);
  int* abort_cta = reinterpret_cast<int*>(misc + 4);
  int* s_task = reinterpret_cast<int*>(misc + 16);
  int* s_last = reinterpret_cast<int*>(misc + 32);
  SelCall& sel = *reinterpret_cast<SelCall*>(misc + 64);
  ChunkDesc* descs = reinterpret_cast<ChunkDesc*>(misc + kMiscBytes);
  uint8_t* creg = reinterpret_cast<uint8_t*>(descs + kDescs);

  const uint32_t bar0 = smem_u32(bars);
  auto full = [&](int i) { return bar0 + 8u * i; };             // K stage landed
  auto empty = [&](int i) { return bar0 + 8u * (8 + i); };      // K stage consumed
  auto tfull = [&](int b) { return bar0 + 8u * (16 + b); };     // TMEM buffer written
  auto tempty = [&](int b) { return bar0 + 8u * (24 + b); };    // TMEM buffer read
  auto dfull = [&](int i) { return bar0 + 8u * (32 + i); };     // descriptor written
  auto dempty = [&](int i) { return bar0 + 8u * (36 + i); };    // descriptor read by all
  auto qfull = [&](int i) { return bar0 + 8u * (40 + i); };     // Q buffer staged
  auto qempty = [&](int i) { return bar0 + 8u * (43 + i); };    // Q buffer's MMAs done
  auto wgbar = [&](int w) { return bar0 + 8u * (46 + w); };     // epilogue warpgroup sync
  auto pubfull = [&](int i) { return bar0 + 8u * (51 + i); };   // chunk's results written
  auto pubempty = [&](int i) { return bar0 + 8u * (51 + kPub + i); };  // chunk published

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int W = p.window;
  const int Hkv = p.num_kv_heads;
  const Fused F{p, abort_cta};

  if (threadIdx.x == 0) {
    for (int i = 0; i < nst; ++i) {
      mbar_init(full(i), 1);
      mbar_init(empty(i), 1);
    }
    for (int b = 0; b < p.nbuf; ++b) {
      mbar_init(tfull(b), 1);
      mbar_init(tempty(b), 4);  // the four warps of the owning warpgroup
    }
    for (int i = 0; i < kDescs; ++i) {
      mbar_init(dfull(i), 1);
      mbar_init(dempty(i), 2 + kEpiWarps);  // TMA producer, UMMA warp, epilogue warps
    }
    for (int i = 0; i < 3; ++i) {
      mbar_init(qfull(i), 1);
      mbar_init(qempty(i), 1);
    }
    for (int i = 0; i < kNwg; ++i) mbar_init(wgbar(i), 4);
    for (int i = 0; i < kPub; ++i) {
      mbar_init(pubfull(i), kEpiWarps);
      mbar_init(pubempty(i), 1);
    }
    *abort_cta = 0;
    sel = SelCall{p.status, Hkv, p.pool_width, p.raw_scratch, p.k, p.v, p.k_out, p.v_out,
                  p.tok_stride_v16, p.head_stride_v16};
    fence_mbar_init();
  }
  for (int q = threadIdx.x; q < kMaxQRows; q += kFThreads) sWpos[q] = q % W;
  if (warp == kMmaWarp) {
    tmem_alloc(smem_u32(tmem_holder), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = *tmem_holder;

  if (warp == kClaimWarp) {
    // ------------------------------------------------------------ chunk claims
    if (lane == 0) {
      Publisher pb{F, pubfull(0), pubempty(0), {}, 0, 0};
      int pending = -1;  // pass-2 chunk claimed, not yet published
      // test hook: a wait that cannot complete, before anything is issued;
      // it runs out after p.wait_ns and stops the call
      if (p.stall && blockIdx.x == 0) F.wait_counter(p.ctr + kCtrNever, 1);
      for (int c = 0;; ++c) {
        const int ds = c % kDescs;
        if (!pb.wait_bar(dempty(ds), ((c / kDescs) & 1) ^ 1)) break;
        ChunkDesc d;
        d.end = 1;
        int pass = 0, x = 0;
        if (claim_chunk(F, pb, &pending, &pass, &x)) {
          const int s = find_seq(p.chunk_off, p.batch, x);
          const int ncu = F.chunks_per_unit(s);
          const int local = x - p.chunk_off[s];
          const int g = local / ncu;
          const int cc = local - g * ncu;
          d.end = 0;
          d.pass = pass;
          d.s = s;
          d.g = g;
          d.t0 = cc * kChunkTiles;
          d.t1 = min(F.tiles(s), d.t0 + kChunkTiles);
          d.chunk = x;
          d.n_rows = F.rows(s, g);
          if (!pb.wait_published(kPub - 1)) break;  // a free slot in the publish ring
          pb.info[pb.issued % kPub] = (s * Hkv + g) * 2 + (pass - 1);
          ++pb.issued;
        }
        descs[ds] = d;
        mbar_arrive(dfull(ds));
        if (d.end) break;
      }
      pb.wait_published(0);  // every chunk this CTA processed
    }
    __syncwarp();
  } else if (warp == kProdWarp) {
    // ------------------------------------------------------------ TMA
    if (lane == 0) {
      // Pass 1 runs further ahead of pass 2 than L2 holds, so K marked
      // evict-last everywhere would evict itself in order and pass 2 would
      // miss all of it; marking a fixed 15% of its lines evict-last (the rest
      // evict-first) keeps that share in L2 until pass 2 reads it (measured:
      // 0.10-0.25 best, 2-3% faster than all evict-last, 4% slower with
      // none).  Pass 2 reads K for the last time; the query rows are reused
      // by every chunk of their unit.
      uint64_t pol1;
      asm volatile("createpolicy.fractional.L2::evict_last.L2::evict_first.b64 %0, 0.15;"
                   : "=l"(pol1));
      const uint64_t pol2 = l2_policy_evict_first();
      const uint64_t polq = l2_policy_evict_last();
      const int G = p.group_size;
      int st = 0;  // next K stage and its phase
      uint32_t ph = 0;
      uint32_t k_used = 0, k_phase = 0;  // per stage: filled, parity of its last fill
      int qb = 0;  // Q buffer of the next chunk and its phase
      uint32_t qph = 0;
      uint32_t q_issued = 0, q_phase = 0;  // per Q buffer: loads issued, phase of the last
      for (int c = 0;; ++c) {
        const int ds = c % kDescs;
        if (!F.wait_bar(dfull(ds), static_cast<uint32_t>(c / kDescs) & 1u)) break;
        const ChunkDesc d = descs[ds];
        mbar_arrive(dempty(ds));
        if (d.end) break;
        const uint64_t pol = d.pass == 1 ? pol1 : pol2;
        const int row0 = p.cu_seqlens[d.s];
        // the chunk's query rows: head block hi of the buffer holds the W
        // window rows of the group's hi-th SRH head
        if (!F.wait_bar(qempty(qb), qph ^ 1u)) break;
        {
          uint32_t bits = p.srh_bits[F.list(d.s, d.g)];
          mbar_arrive_expect_tx(qfull(qb), static_cast<uint32_t>(d.n_rows) * (kHeadDim * 2));
          const uint32_t qdst = smem_u32(sQ + qb * 2 * qh);
          for (int hi = 0; bits != 0u; ++hi, bits &= bits - 1u) {
            const int head = d.g * G + (__ffs(bits) - 1);
            const uint32_t dst = qdst + static_cast<uint32_t>(hi * W * 128);
            tma_load_4d(dst, &p.tmap_q, qfull(qb), 0, 0, head, d.s, polq);
            tma_load_4d(dst + qh, &p.tmap_q, qfull(qb), 64, 0, head, d.s, polq);
          }
          q_issued |= 1u << qb;
          q_phase = (q_phase & ~(1u << qb)) | (qph << qb);
          if (++qb == nqb) {
            qb = 0;
            qph ^= 1u;
          }
        }
        bool stop = false;
        for (int t = d.t0; t < d.t1; ++t) {
          if (!F.wait_bar(empty(st), ph ^ 1u)) {
            stop = true;
            break;
          }
          mbar_arrive_expect_tx(full(st), kTileBytes);
          const uint32_t dst = smem_u32(sK + st * kTileBytes);
          const int row = row0 + t * kTileTokens;
          tma_load_3d(dst, &p.tmap_k, full(st), 0, d.g, row, pol);
          tma_load_3d(dst + kHalfTileBytes, &p.tmap_k, full(st), 64, d.g, row, pol);
          k_used |= 1u << st;
          k_phase = (k_phase & ~(1u << st)) | (ph << st);
          if (++st == nst) {
            st = 0;
            ph ^= 1u;
          }
        }
        if (stop) break;
      }
      if (*reinterpret_cast<volatile int*>(abort_cta)) {
        // let the copies already issued land before the CTA can exit
        for (int i = 0; i < nst; ++i)
          if ((k_used >> i) & 1u) wait_plain(full(i), (k_phase >> i) & 1u, 100000000ull);
        for (int b = 0; b < nqb; ++b)
          if ((q_issued >> b) & 1u) wait_plain(qfull(b), (q_phase >> b) & 1u, 100000000ull);
      }
      // Tail: the UMMA warps release a stage (empty) and a Q buffer (qempty)
      // with tcgen05.commit arrivals that nobody else waits for at the end;
      // wait for the last ones, so that no asynchronous arrival can land in
      // this CTA's shared memory after it exits (bounded: after an abort some
      // never come).
      const uint64_t tail_ns = *reinterpret_cast<volatile int*>(abort_cta) ? 100000000ull
                                                                           : p.wait_ns;
      for (int i = 0; i < nst; ++i)
        if ((k_used >> i) & 1u) wait_plain(empty(i), (k_phase >> i) & 1u, tail_ns);
      for (int b = 0; b < nqb; ++b)
        if ((q_issued >> b) & 1u) wait_plain(qempty(b), (q_phase >> b) & 1u, tail_ns);
    }
    __syncwarp();
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------ UMMA issue
    auto wait_all = [&](uint32_t bar, uint32_t parity) {
      return __all_sync(0xffffffffu, F.wait_bar(bar, parity));
    };
    const uint64_t dk0 = smem_desc_sw128(smem_u32(sK));
    const int bpw = p.nbuf / kNwg;  // TMEM buffers per warpgroup (a power of two)
    const int lbpw = __ffs(bpw) - 1;
    int st = 0;  // next K stage and its phase
    uint32_t sph = 0;
    int qb = 0;  // Q buffer of the next chunk and its phase
    uint32_t qph = 0;
    int kw0 = 0, kw1 = 0;  // tiles issued per warpgroup
    int last_st = -1;
    uint32_t last_ph = 0;
    for (int c = 0;; ++c) {
      const int ds = c % kDescs;
      if (!wait_all(dfull(ds), static_cast<uint32_t>(c / kDescs) & 1u)) break;
      const int end = descs[ds].end, nt = descs[ds].t1 - descs[ds].t0, rows = descs[ds].n_rows;
      __syncwarp();
      if (lane == 0) mbar_arrive(dempty(ds));
      if (end) break;
      if (!wait_all(qfull(qb), qph)) break;
      const int Npad = (rows + 15) & ~15;
      const uint32_t idesc = umma_idesc_f16(kTileTokens, Npad, p.is_bf16 != 0);
      const uint64_t dq0 = smem_desc_sw128(smem_u32(sQ + qb * 2 * qh));
      const uint64_t qhalf = static_cast<uint64_t>(qh >> 4);
      bool stop = false;
#pragma unroll 1
      for (int t = 0; t < nt; ++t) {
        const int mw = t & 1;  // the warpgroup that takes the tile
        const int kk = mw ? kw1++ : kw0++;
        const int b = mw + kNwg * (kk & (bpw - 1));
        const uint32_t use = static_cast<uint32_t>(kk >> lbpw) & 1u;
        if (!wait_all(tempty(b), use ^ 1u) || !wait_all(full(st), sph)) {
          stop = true;
          break;
        }
        tc_fence_after();
        const uint32_t dt = tbase + static_cast<uint32_t>(b * p.tstride);
        const uint64_t dk = dk0 + static_cast<uint64_t>((st * kTileBytes) >> 4);
        if (elect_one()) {
#pragma unroll
          for (int k8 = 0; k8 < kHeadDim / 16; ++k8) {
            const uint64_t koff = ((k8 >> 2) * kHalfTileBytes + (k8 & 3) * 32) >> 4;
            const uint64_t qoff = (k8 >> 2) * qhalf + (((k8 & 3) * 32) >> 4);
            umma_f16(dt, dk + koff, dq0 + qoff, idesc, k8 > 0 ? 1u : 0u);
          }
          umma_commit(tfull(b));
          umma_commit(empty(st));
        }
        __syncwarp();
        last_st = st;
        last_ph = sph;
        if (++st == nst) {
          st = 0;
          sph ^= 1u;
        }
      }
      if (stop) break;
      if (elect_one()) umma_commit(qempty(qb));
      __syncwarp();
      if (++qb == nqb) {
        qb = 0;
        qph ^= 1u;
      }
    }
    if (lane == 0 && *reinterpret_cast<volatile int*>(abort_cta) && last_st >= 0)
      wait_plain(empty(last_st), last_ph, 100000000ull);  // MMAs done before TMEM is freed
    __syncwarp();
  } else if (warp >= kEpiWarp0 && warp < kEpiWarp0 + kEpiWarps) {
    // ------------------------------------------------------------ epilogue
    const int ew = warp - kEpiWarp0;
    const int wg = ew >> 2;
    const int qd = warp & 3;  // TMEM lane quarter of this warp
    const int tw = (ew & 3) * 32 + lane;
    constexpr int nwg = kNwg;
    float* ref = sRef + ew * rstride;
    float* acc_s = sAcc + ew * rstride;
    const float c = p.c;
    const uint64_t c2 = pack2(c, c);
    const int bcol = block_col(lane);
    const int bpw = p.nbuf / nwg;  // a power of two
    const int lbpw = __ffs(bpw) - 1;
    const int G = p.group_size;
    int kc = 0;       // tiles this warpgroup has taken
    int nsync = 0;    // warpgroup syncs so far (mbarrier phase)
    bool stop = false;
    // bounded barriers (a warp that stopped cannot hang the others)
    // the chunk's results are written: its claimer publishes it (fence, then
    // the unit's counter) off the epilogue's path
    auto publish = [&](int ci) -> bool {
      const int k = ci % kPub;
      bool ok = true;
      if (ci >= kPub && lane == 0) ok = F.wait_bar(pubempty(k), static_cast<uint32_t>(ci / kPub - 1) & 1u);
      __syncwarp();
      if (lane == 0 && ok) mbar_arrive(pubfull(k));
      return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
    };
    auto wg_sync = [&]() -> bool {
      __syncwarp();
      if (lane == 0) mbar_arrive(wgbar(wg));
      const bool ok = F.wait_bar(wgbar(wg), static_cast<uint32_t>(nsync) & 1u);
      ++nsync;
      return __all_sync(0xffffffffu, ok);
    };
    for (int ci = 0; !stop; ++ci) {
      const int ds = ci % kDescs;
      const bool got = F.wait_bar(dfull(ds), static_cast<uint32_t>(ci / kDescs) & 1u);
      if (!__all_sync(0xffffffffu, got)) break;
      const ChunkDesc d = descs[ds];
      __syncwarp();
      if (lane == 0) mbar_arrive(dempty(ds));
      if (d.end) break;
      const int s = d.s;
      const int g = d.g;
      const int N = d.n_rows;
      const int L = F.len(s);
      const int n = L - W;
      const int u = s * Hkv + g;
      const long long soff = static_cast<long long>(g) * p.p_total + p.cu_prefix[s];
      if (d.pass == 1) {
        // ---------------------------------------- pass 1: softmax statistics
        // Per query row q the warp keeps a reference R_q and sums
        // 2^(z c - R_q) over its keys, reduced across the lanes every tile.
        for (int q = lane; q < N; q += 32) {
          ref[q] = kNegInf;
          acc_s[q] = 0.f;
        }
        __syncwarp();
        bool first = true;  // no tile of this chunk accumulated yet
        for (int tile = d.t0 + wg; tile < d.t1; tile += nwg) {
          const int kk = kc++;
          const int b = wg + nwg * (kk & (bpw - 1));
          const uint32_t use = static_cast<uint32_t>(kk >> lbpw) & 1u;
          const bool ok = F.wait_bar(tfull(b), use);
          if (!__all_sync(0xffffffffu, ok)) {
            stop = true;
            break;
          }
          tc_fence_after();
          const int tok0 = tile * kTileTokens + qd * 32;  // the warp's first key
          const uint32_t taddr = tbase + (static_cast<uint32_t>(qd * 32) << 16) +
                                 static_cast<uint32_t>(b * p.tstride);
          const bool edge = (tile + 1) * kTileTokens > n;
#pragma unroll 1
          for (int c0 = 0; c0 < N; c0 += 32) {
            uint32_t r[32];  // the logits
            tmem_load_block(taddr + c0, r);
            const int lim = min(32, N - c0);  // 32 or 16
            float2* rf = reinterpret_cast<float2*>(ref + c0) + (lane & 3);  // columns 8 j + 2 (lane % 4)
            uint64_t nr[4];
            if (first && !edge) {
              // the warp's first tile of the chunk: its first key's scaled
              // logit is the reference of each query row (any reference
              // within 2^64 of the largest keeps the fp32 sums exact enough)
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const float r0 = __shfl_sync(0xffffffffu, __uint_as_float(r[4 * j]) * c, lane & 3);
                const float r1 =
                    __shfl_sync(0xffffffffu, __uint_as_float(r[4 * j + 1]) * c, lane & 3);
                nr[j] = pack2(-r0, -r1);
                if (lane < 4) rf[4 * j] = make_float2(r0, r1);
              }
              __syncwarp();
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const float2 x = rf[4 * j];
                nr[j] = pack2(-x.x, -x.y);
              }
            }
            float v[8];  // sums of 2^(z c - R) over the lane's keys
            if (edge) {
              const uint32_t ok = block_mask(c0, W, lim, tok0, n, L, lane);
#pragma unroll
              for (int i = 0; i < 8; ++i) v[i] = 0.f;
#pragma unroll
              for (int e = 0; e < 32; ++e) {
                const int j = (e >> 2) & 3;
                float n0, n1;
                unpack2(nr[j], n0, n1);
                const float x = ex2_approx(fmaf(__uint_as_float(r[e]), c, (e & 1) ? n1 : n0));
                v[2 * j + (e & 1)] += (ok >> e) & 1u ? x : 0.f;
              }
            } else {
              uint64_t s2[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
              for (int e = 0; e < 32; e += 2) {
                const int j = (e >> 2) & 3;
                const uint64_t z = pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1]));
                s2[j] = add2(s2[j], exp2_2(fma2(z, c2, nr[j])));
              }
              if (lim < 32) s2[2] = s2[3] = 0ull;  // not query rows
#pragma unroll
              for (int j = 0; j < 4; ++j) unpack2(s2[j], v[2 * j], v[2 * j + 1]);
            }
            float colsum = sum_over_keys(v, lane);
            int col = bcol;
            // an exponent above 2^64 shows in its column's sum (inf/NaN
            // when above 2^128 or with the references still -inf)
            if (__any_sync(0xffffffffu, !(colsum <= kRaiseSum))) {
              const int tok = tok0 + lane;
              colsum = p1_raise_group(taddr + c0, ref + c0, acc_s + c0, sWpos + c0, lim, edge,
                                      tok < L, n - tok, c, lane);
              col = lane;
            }
            acc_s[c0 + col] += colsum;
            __syncwarp();
          }
          first = false;
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty(b));
        }
        if (stop) break;
        // the warpgroup's (M, S) pairs for this chunk, then its ticket
        if (!wg_sync()) break;
        float2* part = p.partials +
                       (static_cast<long long>(d.chunk) * kFusedPartsPerChunk + wg) * p.part_stride;
        for (int q = tw; q < N; q += 128) {
          float m = kNegInf;
          for (int w = 0; w < 4; ++w) m = fmaxf(m, sRef[(wg * 4 + w) * rstride + q]);
          float z = 0.f;
          for (int w = 0; w < 4; ++w) {
            const float rw = sRef[(wg * 4 + w) * rstride + q];
            if (rw != kNegInf) z += sAcc[(wg * 4 + w) * rstride + q] * ex2_approx(rw - m);
          }
          part[q] = make_float2(m, z);
        }
        if (!wg_sync()) break;  // every row read (the next chunk reuses them)
        if (!publish(ci)) break;
      } else {
        // ---------------------------------------- pass 2: raw scores
        // log2 D_q of every query row into this warp's row of sRef
        if (p.given_lse) {
          const uint32_t bits = p.srh_bits[F.list(s, g)];
          for (int q = lane; q < N; q += 32) {
            const int hi = q / W;
            const int w = q - hi * W;
            const int head = g * G + nth_bit(bits, hi);
            ref[q] = p.lse[static_cast<long long>(s) * p.lse_bs +
                           static_cast<long long>(head) * p.lse_hs + w] *
                     1.4426950408889634f;
          }
        } else {
          // published only after its claimer saw the unit's denominators
          // merged (acquire), before the descriptor barrier
          const float* bias = p.bias + static_cast<long long>(u) * p.part_stride;
          for (int q = lane; q < N; q += 32) ref[q] = __ldcg(bias + q);
        }
        __syncwarp();
        for (int tile = d.t0 + wg; tile < d.t1; tile += nwg) {
          const int kk = kc++;
          const int b = wg + nwg * (kk & (bpw - 1));
          const uint32_t use = static_cast<uint32_t>(kk >> lbpw) & 1u;
          const bool ok = F.wait_bar(tfull(b), use);
          if (!__all_sync(0xffffffffu, ok)) {
            stop = true;
            break;
          }
          tc_fence_after();
          const uint32_t taddr = tbase + (static_cast<uint32_t>(qd * 32) << 16) +
                                 static_cast<uint32_t>(b * p.tstride);
          // 2^(z c - log2 D_q) summed over the query rows.  (Causality needs
          // no mask: every query row sees every prefix key, and the scores of
          // later keys are not kept.)
          uint64_t rs2[4] = {0ull, 0ull, 0ull, 0ull};  // the lane's four keys
#pragma unroll 1
          for (int c0 = 0; c0 < N; c0 += 32) {
            uint32_t r[32];
            tmem_load_block(taddr + c0, r);
            const float2* lq = reinterpret_cast<const float2*>(ref + c0) + (lane & 3);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              if (j == 2 && N - c0 == 16) break;  // the last 16 columns are not query rows
              const float2 x = lq[4 * j];
              const uint64_t nl = pack2(-x.x, -x.y);
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const int e = 16 * (k >> 1) + 4 * j + 2 * (k & 1);
                const uint64_t z = pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1]));
                rs2[k] = add2(rs2[k], exp2_2(fma2(z, c2, nl)));
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty(b));
          float rs[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            float x, y;
            unpack2(rs2[k], x, y);
            rs[k] = x + y;
          }
          const float v = sum_over_cols(rs, lane);
          const int tok = tile * kTileTokens + qd * 32 + block_key(lane);
          if (tok < n) p.raw[soff + tok] = v;
        }
        if (stop) break;
        if (!publish(ci)) break;
      }
    }
  } else if (warp >= kCWarp0 && warp < kCWarp0 + kCThreads / 32) {
    // ------------------------------------------------------------ merge / select
    const int ct = threadIdx.x - kCWarp0 * 32;
    TaskPos T{-1, 0, 0, -1, -1, 0};
    for (;;) {
      if (ct == 0) {
        claim_ticket<kKind>(F, T, s_task);
      }
      cbar();
      const int type = s_task[0];
      const int idx = s_task[1];
      const int piece = s_task[2];
      cbar();
      if (type == kTaskEnd) break;
      if (type == kTaskMerge) {
        merge_unit(F, idx, creg, ct);
      } else if (p.do_select) {
        const int s = idx / Hkv;
        const int g = idx - s * Hkv;
        SelUnit U;
        U.g = g;
        U.seq0 = p.cu_seqlens[s];
        U.L = F.len(s);
        U.W = W;
        U.out0 = p.cu_out[s];
        U.kept = p.cu_out[s + 1] - U.out0;
        const long long soff = static_cast<long long>(g) * p.p_total + p.cu_prefix[s];
        if constexpr (kKind != kPlain) {
          SelShared& ss = *reinterpret_cast<SelShared*>(creg);
          uint32_t* const rowmax = p.rowmax + row_max_offset(soff, g, s, p.batch);
          if (type == kTaskPool) {
            pool_piece(p.raw + soff, p.pooled + soff, rowmax, U.L - U.W, piece, sel, ss,
                       F.bias_state(idx), 4, ct);
            continue;
          }
          if (ct == 0) ss.rowmax = kKind == kInPieces || s_task[3] > 0 ? rowmax : nullptr;
          cbar();
        }
        select_unit<kKind>(sel, U, p.raw + soff, p.pooled + soff,
                           p.indices + static_cast<long long>(g) * p.o_total + U.out0, creg, ct);
      }
    }
  }

  // ------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tbase, 512);
  }
  if (threadIdx.x == 0) {
    // (the resident kernel of the same call may still run: its words are among
    // those zeroed below, and the next kernel waits for this one alone)
    if (kKind == kMixed) pdl_wait();
    __threadfence();
    *s_last = atomicAdd(p.ctr + kCtrExit, 1) == static_cast<int>(gridDim.x) - 1 ? 1 : 0;
  }
  __syncthreads();
  if (*s_last) {
    // every other CTA has finished: zero the counters for the next call
    __threadfence();
    const int nz = kFusedCtrHead + 3 * p.n_units;
    for (int i = threadIdx.x; i < nz; i += kFThreads) p.ctr[i] = 0;
  }
}

}  // namespace

size_t fused_smem_bytes(int q_half_bytes, int q_bufs, int stages, int row_stride) {
  return 1024 + static_cast<size_t>(stages) * kTileBytes +
         2 * static_cast<size_t>(q_bufs) * q_half_bytes +
         2 * static_cast<size_t>(4 * kNwg) * row_stride * 4 + kFixedBytes + kSelRegion;
}

cudaError_t fused_set_smem_limit(size_t bytes) {
  for (auto kernel : {fused_kernel<kPlain>, fused_kernel<kInPieces>, fused_kernel<kMixed>}) {
    const cudaError_t e = cudaFuncSetAttribute(
        kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_fused(const FusedParams& p, int grid, size_t smem, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(kFThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  // After the resident kernel of the same call: its CTAs start where that
  // kernel's have ended (the two share nothing but the call's inputs).
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.mixed ? 1 : 0;
  return cudaLaunchKernelEx(&cfg,
                            p.mixed       ? fused_kernel<kMixed>
                            : p.in_pieces ? fused_kernel<kInPieces>
                                          : fused_kernel<kPlain>,
                            p);
}

}  // namespace ckv
