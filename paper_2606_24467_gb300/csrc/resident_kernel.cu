// Persistent fused layer call for short prompts (CompressKV Sec. 3.3 token
// selection with the SnapKV-style window of Sec. 4, per-group selection): one
// launch scores every unit (sequence, KV group) of a call, pools the scores,
// takes the budgeted top-k, appends the window and gathers the retained K/V
// rows.
//
// For unit (s, g), with Q_S the N = |S_g| * W window-query rows of the
// group's SRH heads, z = <q, k> * scale and c = log2(e), query q (window
// position p_q) attends key j <= p_q with 2^(z_qj c) / D_q,
// D_q = sum_{j <= p_q} 2^(z_qj c), and the raw score of prefix key j is the
// sum of that over q.  Every score needs every key's share of D first, so a
// plain kernel reads K twice.  Here the logits stay on the chip instead: a
// unit's K tiles are spread over all SMs at once (chunk x of the call goes to
// CTA x mod grid, a chunk being one to four tiles of 128 keys), every SM keeps
// the fp32 logits of its chunks in tensor memory (512 columns: 16 tiles of 32
// query rows, 8 of 64, 4 of 128, 2 of 192) while the chunks' sums of
// exponentials are added up over the SMs, and the scores are then taken from
// the same logits:
//   pass 1  S_q = sum 2^(z c) over the chunk's keys, per query row; added to
//           the unit's accumulators in global memory by one 64-bit integer
//           reduction per query row (below);
//   pass 2  raw_j = sum_q 2^(z_qj c - R_q) w_q, 2^R_q / w_q = D_q, from the
//           same tensor memory once the unit's D_q are complete.
// The worker warps (unit_select.cuh) then pool, pooled_j = (sum_{t=-h..h}
// raw_{j+t}) / P with zeros outside [0, n), take the k = kept - W largest
// pooled scores (ties to the lower position) in ascending position and the
// window, and copy the K/V rows.
// With the window queries' log-sum-exp given (given_lse) pass 1 is skipped
// and log2 D_q = LSE_q * log2(e).
//
// The sum over the SMs (kAccWords 64-bit words per unit and query row): a
// chunk's S_q, an fp32 number, is rounded to an integer multiple of a power
// of two that its exponent selects (one of kAccBins bins, spaced so that no
// bit of a sum of 2^-10 or more is lost) and added to the bin's word, whose low
// bits count the contributions.  Integer addition has no
// order, so D_q is the same whatever the order of arrival; a reader that
// finds as many contributions as the unit has chunks has the complete sum, so
// one reduction and one read carry it between SMs, with no fence, ticket or
// merge in between (measured on 152 SMs: 2.1 us for 64 rows with a ticket and
// fence, 6 us when every SM reads every other's partial sums).  Rows whose
// sums leave the bins' range are added up again against the unit's largest
// chunk exponent (slow_denominators): a chunk's sum of 2^142 and more in a
// unit of one chunk, of 2^86 in one of 128, or a D below 2^-48 and 2^-27 in
// these (every logit above about +60 or below about -25).
//
// One CTA per SM runs for the whole call.  The chunks of a unit wait for one
// another, so the CTAs that take part are those that are resident when the call
// starts (take_part): all, but where another kernel holds SMs for longer than
// kStartWaitNs.  A unit's sums and scores do not depend on how many they are.
// Warps:
//   warp 0      loads each unit's SRH query rows (one TMA box of W rows per
//               head and 64-column half) into one of two or three Q buffers
//               and streams the K tiles, by TMA, into a shared-memory ring;
//   warp 1      issues the UMMAs (M = 128 keys, N = query rows) into tensor
//               memory, taken as a ring of columns; allocates it;
//   warp 2      writes the chunk descriptors;
//   warp 3      adds the four pass-1 warps' sums and reduces them into the
//               unit's accumulators;
//   warps 4-7   pass 1 (warpgroup 0; with the LSE given: every other chunk
//               of pass 2);
//   warps 8-11  pass 2 (warpgroup 1);
//   warps 12-19 workers: zero the accumulators when the call starts, then
//               select and gather the units u = id, id + grid...
//               as their chunks are scored;
//   warps 20,22 read the units' complete sums, one unit ahead of pass 2
//               (alternate units);
//   warp 21     tells the selection which chunks are scored.
// What a chunk needs to know of its sequence travels in its descriptor: the
// roles share one instruction and one constant cache, and looking the tables
// up in the kernel parameters cost each of them 300 clocks a miss.
// The epilogue reads tensor memory in the 16x256b shape: a lane holds 4 keys
// x 8 query rows of a 32 x 32 block, so the sum over keys (pass 1) takes 3
// exchange steps of 7 shuffles after all tiles of a chunk, and the sum over
// query rows (pass 2) 3 shuffles a tile, where one lane per key takes 31
// shuffles per block for the first.
// What bounds it: a short call the chain of its steps (one 777-token layer,
// 29 us a call against 73 in the two-pass kernel before it: start 4, scores 9,
// selection 8, the rest the host's), a full one the time that tensor memory is
// held: a chunk's logits wait for the sums of the unit's slowest chunk, and the
// memory holds few chunks (32 layers of 32768 tokens: 622 us, 3.5 TB/s of the K
// that is read once; 32 layers of 8 prompts of 300 to 4000 tokens: 0.48 ms
// against 3.5).
// Every wait is bounded (ResidentParams::wait_ns, kWaitTimeoutNs unless a test
// shortens it) and on expiry records CKV_ERR_DEVICE_TIMEOUT and stops the
// call.  A wait depends only on chunks of the same or earlier units, which
// every CTA takes in the same order, so a call completes.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cfloat>

#include "ckv_device.cuh"
#include "tile_math.cuh"
#include "unit_select.cuh"

namespace ckv {

namespace {

constexpr int kRWarps = 23;
constexpr int kRThreads = 32 * kRWarps;
constexpr int kProdWarp = 0;
constexpr int kMmaWarp = 1;
constexpr int kSchedWarp = 2;
constexpr int kSumWarp = 3;
constexpr int kEpiWarp0 = 4;  // warps 4..11: two warpgroups (TMEM lane quarter = warp % 4)
constexpr int kEpiWarps = 8;
constexpr int kCWarp0 = 12;   // warps 12..19
constexpr int kDenWarp = 20;
constexpr int kAnnWarp = 21;
constexpr int kDenWarp2 = 22;
constexpr int kDescs = 32;    // chunk descriptors in flight: more than the chunks the tensor memory
                              // (16) and the K ring (8) can hold at once
constexpr int kTiles = 16;       // K tiles whose logits are in tensor memory (512 columns / 32)
constexpr int kMaxStages = 8;   // K ring stages
constexpr int kPub = 8;       // chunks scored, not yet announced to the selection
constexpr float kNegInf = -INFINITY;

// A unit's accumulators: words 0..kAccBins-1 the bins, then the number of
// contributions outside their range, the sum of the second round and its
// largest exponent.
constexpr int kAccBins = 5;
constexpr int kAccOut = kAccBins;
constexpr int kAccSlow = kAccBins + 1;
constexpr int kAccMax = kAccBins + 2;
static_assert(kAccMax + 1 == kAccWords, "accumulator words");
constexpr int kAccE0 = -10;   // sums below 2^kAccE0 share bin 0

// Words of the header's counter block that the two-pass kernel does not use
// (it zeroes them with its own).  The last CTA past the start zeroes the
// start's, also in a call that stops; the number of calls stays, and the abort
// word holds the number of the call that stopped.
constexpr int kCtrNever = 6;   // never set: the test hook's stall waits for it
constexpr int kCtrStop = 8;    // number of the last call in which a wait ran out
constexpr int kCtrCalls = 9;   // calls so far
constexpr int kCtrArrive = 32; // CTAs that have started (16 bits); once closed, how many had then
constexpr int kCtrZeroed = 40; // CTAs taking part that have zeroed their share
constexpr int kCtrPast = 48;   // CTAs past the start
constexpr int kCtrSlots = 56;  // (5 words) numbers given by number_by_sm
constexpr unsigned kClosed = 1u << 31;  // (of kCtrArrive; the 14 bits below kApart: how many take part)
constexpr unsigned kApart = 1u << 30;   // the CTAs did not start together

// How long the first CTA waits for the others to start.  A kernel of another
// stream that ends in this time delays the call by no more than its own time;
// one that holds SMs for longer leaves the call the others.
constexpr uint64_t kStartWaitNs = 1000000ull;
constexpr uint64_t kStartApartNs = 8000ull;  // (together: within 2 us)

constexpr int kModeP1 = 1;    // the chunk's sums of exponentials
constexpr int kModeP2 = 2;    // the chunk's scores

struct alignas(16) ChunkDesc {
  int mode, wg, new_q, unit;      // mode 0: no more chunks; the unit whose pass 2 is in hand
  int s, g, t0, nt;               // sequence, group, K tiles [t0, t0 + nt)
  int n_rows, nch;                // query rows, chunks of the unit
  int tile, sum_unit;             // number of the first tile; the unit that pass 1 adds to
  int n, L, row0, soff;           // prefix, length, first row of K, offset of the scores
  uint32_t bits;                  // SRH heads of the group
  int ct, last_q;                 // tiles per chunk; the Q buffer's last chunk
  int x, x_last;                  // number of the chunk, of the unit's last of this CTA
  int col, width;                 // tensor-memory columns: tile i at col + i * width
};

// Position in the list of this CTA's chunks, and what the chunk's sequence
// and unit are.
struct ListPos {
  int x, sq, off, off_next, nch, ct, row0, L;
  int unit, gr, n_rows, soff, width, unit_end;
  uint32_t bits;
};

// What the warp roles need of the call's parameters, in shared memory.  Each
// role is a function of its own, so that its registers are its own and
// nothing of it lives on the stack (beside 227 KB of shared memory the L1
// cache holds a small part of 21 warps' stacks, and a miss costs an L2 round
// trip); a reference to the kernel's parameters would be read through L1 too.
struct CallInfo {
  int* status;
  int* abort_word;
  int number;                      // of this call on this workspace, from 1
  unsigned long long wait_ns;
  unsigned long long* acc;
  int* slow_ticket;
  float* raw;
  float* pooled;
  const float* lse;
  long long lse_bs, lse_hs;
  const void* tmap_k;
  const void* tmap_q;
  uint8_t* sK;
  uint8_t* sQ;
  float2* rows;
  uint32_t tbase;
  float c;
  int id, grid;                    // of this CTA among those that take part (id -1: not one)
  int ring;                        // chunk sums that each keeps in `pairs`
  int acc_rows, stages, q_bufs, q_half_bytes;
  int window, group_size, is_bf16, given_lse;
  float2* pairs;                   // (M, S) of this CTA's latest chunks, a row each
  SelCall sel;
};

// Shared memory beside the K ring, the Q buffers and the workers' region.
struct ResidentShared {
  CallInfo call;
  uint64_t full[kMaxStages], empty[kMaxStages];      // K stage landed / consumed
  uint64_t tfull[2][kTiles], tempty[kTiles];           // tile written (per warpgroup) / read
  int tile_c0[kTiles], tile_c1[kTiles];                // its tensor-memory columns
  uint64_t dfull[kDescs], dempty[kDescs];              // descriptor written / read by all
  uint64_t qfull[3], qempty[3];                        // Q buffer landed / consumed
  uint64_t p1full[2], p1empty[2];                      // chunk sums written / added up
  uint64_t p2full[kPub], p2empty[kPub];                // chunk scored / announced
  uint64_t dnfull[2][2], dnempty[2][2];                // denominators of a unit, per warpgroup
  uint64_t startbar;
  uint32_t tmem;
  int abort_cta, task, piece, pieces;
  int sum_pos;                                         // chunks below have left their pairs
  int p2_unit[kPub];
  ChunkDesc descs[kDescs];
  ListPos list[2];                                     // ([1]: of pass 2 apart from pass 1)
};

// ... and rows of acc_rows pairs: the chunk sums (M, S) of the four pass-1
// warps, two chunks; (-R_q, w_q) of two units for warpgroup 1 (for warpgroup
// 0, with the LSE given, in the place of the chunk sums).
constexpr int kDenRow = 8, kPairRows = 10;
constexpr int kResidentSharedBytes = (static_cast<int>(sizeof(ResidentShared)) + 15) & ~15;

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_relaxed64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_add64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// Between threads of one CTA: what this thread has waited for happens before
// what the observer of its next relaxed write does after such a fence.
__device__ __forceinline__ void fence_acq_rel_cta() {
  asm volatile("fence.acq_rel.cta;" ::: "memory");
}
__device__ __forceinline__ int ld_volatile(const int* p) {
  return *reinterpret_cast<const volatile int*>(p);
}

// Index of the i-th set bit of `bits` (i < popc(bits)).
__device__ __forceinline__ int nth_bit(uint32_t bits, int i) {
  for (int j = 0; j < i; ++j) bits &= bits - 1u;
  return __ffs(bits) - 1;
}

// 2^e for -126 <= e <= 127; 0 below, infinity above.
__device__ __forceinline__ float pow2i(int e) {
  return e < -126 ? 0.f : (e > 127 ? INFINITY : __int_as_float((e + 127) << 23));
}

// ---------------------------------------------------------------- waits
__device__ __forceinline__ bool aborted(const ResidentShared& sh) {
  return ld_volatile(sh.call.abort_word) == sh.call.number;
}
__device__ __forceinline__ void arrive(uint64_t* bar) { mbar_arrive(smem_u32(bar)); }

// One more turn of a wait that began at t0: false when the call stopped or
// the wait ran out (the status word and the abort word are then set).
__device__ __noinline__ bool still_waiting(ResidentShared& sh, uint64_t t0) {
  assume_shared(&sh);
  volatile int* mine = &sh.abort_cta;
  if (*mine) return false;
  if (aborted(sh)) {
    *mine = 1;  // tell this CTA's other waits
    return false;
  }
  if (globaltimer_ns() - t0 > sh.call.wait_ns) {
    atomicCAS(sh.call.status, 0, CKV_DEV_ERR_TIMEOUT);
    atomicExch(sh.call.abort_word, sh.call.number);
    *mine = 1;
    return false;
  }
  return true;
}
// Waits for an mbarrier phase for up to about kWaitHintNs, suspended: polling
// warps cost the others of this kernel issue slots and instruction cache.
constexpr uint32_t kWaitHintNs = 20000;
__device__ __forceinline__ bool mbar_suspended_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(kWaitHintNs)
      : "memory");
  return ok != 0;
}
// Bounded wait (another CTA's progress) until *ptr >= target; false when the
// call was aborted or the wait ran out.
__device__ __noinline__ bool wait_counter(ResidentShared& sh, const int* ptr, int target) {
  assume_shared(&sh);
  if (ld_acquire(ptr) >= target) return true;
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    __nanosleep(200);
    if (ld_acquire(ptr) >= target) return true;
    if (!still_waiting(sh, t0)) return false;
  }
}
// Bounded wait on one of this CTA's mbarriers; a timeout stops the call.
__device__ __noinline__ bool wait_more(ResidentShared& sh, uint32_t a, uint32_t parity) {
  assume_shared(&sh);
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    if (mbar_suspended_wait(a, parity)) return true;
    if (!still_waiting(sh, t0)) return false;
  }
}
__device__ __forceinline__ bool wait_bar(ResidentShared& sh, const uint64_t* bar, uint32_t parity) {
  const uint32_t a = smem_u32(bar);
  if (mbar_suspended_wait(a, parity)) return true;
  return wait_more(sh, a, parity);
}

// The same by a whole warp.
__device__ __forceinline__ bool wait_all(ResidentShared& sh, const uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, wait_bar(sh, bar, parity));
}

// Row i of pairs, and the denominators of warpgroup wg's k-th unit.
__device__ __forceinline__ float2* pair_row(ResidentShared& sh, int i) {
  float2* const r = sh.call.rows + i * sh.call.acc_rows;
  assume_shared(r);
  return r;
}
// (acc_rows values of -R, then acc_rows of w)
__device__ __forceinline__ float* den_row(ResidentShared& sh, int wg, int k) {
  float* const r = reinterpret_cast<float*>(pair_row(sh, (wg ? kDenRow : 0) + k));
  assume_shared(r);
  return r;
}

// Position in a ring of n slots and the parity of its use.
struct Ring {
  int i = 0;
  uint32_t ph = 0;
  __device__ void next(int n) {
    if (++i == n) {
      i = 0;
      ph ^= 1u;
    }
  }
};

// ---------------------------------------------------------------- the unit's sums
// The bins of a unit of nch chunks: cb bits count contributions; a
// contribution has at most vb bits, so nch of them do not overflow into one
// another (nch 2^vb <= 2^(64 - cb)); bin 0 holds sums below 2^kAccE0, bin
// k >= 1 those in [2^(kAccE0 + (k - 1) width), 2^(kAccE0 + k width)), which
// have at least vb - width = 24 bits there: an fp32 sum is added exactly.
struct Bins {
  int cb, vb, width;
  __device__ explicit Bins(int nch) {
    cb = 32 - __clz(nch);
    vb = 64 - 2 * cb;
    width = vb - 24;
  }
  __device__ int grid(int k) const { return kAccE0 + k * width - vb; }
};

// Adds S 2^m (m integral) to the accumulators of one query row (words acc,
// acc + stride, ...).
__device__ __forceinline__ void add_sum(const Bins& B, unsigned long long* acc, int stride, float m,
                                        float S) {
  const uint32_t bits = __float_as_uint(S);  // S >= 0 or NaN
  const float ef = static_cast<float>(static_cast<int>((bits >> 23) & 255u) - 127) + m;
  const bool fits = ef < static_cast<float>(kAccE0 + (kAccBins - 1) * B.width);  // false for NaN
  if (fits && (bits & 0x7F800000u) != 0x7F800000u) {
    const int e = static_cast<int>(fmaxf(ef, -4096.f)) - kAccE0;
    int k = 0;
#pragma unroll
    for (int i = 0; i < kAccBins - 1; ++i) k += e >= i * B.width ? 1 : 0;
    // S 2^m / 2^grid < 2^vb: scaled in two steps, each within the fp32 range
    const int sc = static_cast<int>(fmaxf(m, -4096.f)) - B.grid(k);
    const float v = S * pow2i(sc >> 1) * pow2i(sc - (sc >> 1));
    red_add64(acc + static_cast<long long>(k) * stride, (__float2ull_rn(v) << B.cb) | 1ull);
  } else {
    red_add64(acc + static_cast<long long>(kAccOut) * stride, 1ull);
  }
}

// -R and w of a denominator D > 0 (finite, fp32): D = 2^R / w, R integral.
__device__ __forceinline__ void split_denominator(float D, float* nR, float* w) {
  const uint32_t bits = __float_as_uint(D);
  *nR = static_cast<float>(127 - static_cast<int>(bits >> 23));
  *w = __frcp_rn(__uint_as_float((bits & 0x7FFFFFu) | 0x3F800000u));
}

// Order-preserving integer of a float (NaN above everything, 0 unused).
__device__ __forceinline__ unsigned long long order_key(float x) {
  if (x != x) return 0xFFFFFFFFull;
  const uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float order_value(unsigned long long k) {
  const uint32_t b = static_cast<uint32_t>(k);
  return __uint_as_float((b & 0x80000000u) ? (b & 0x7FFFFFFFu) : ~b);
}

// ---------------------------------------------------------------- epilogue
// Sums inside these bounds are exact enough in fp32 against 2^0 (no term
// that matters is flushed to zero, nothing overflows).
constexpr float kSumLo = 1.0e-27f, kSumHi = 1.0e27f;

// A warpgroup of the epilogue: four warps, one per TMEM lane quarter.
struct Group {
  ResidentShared& sh;
  int w, quarter, lane;  // warpgroup, TMEM lane quarter, lane
  uint32_t tile_ph = 0;  // parity of the next use of every tile barrier by this group
  __device__ __forceinline__ bool wait_tile(int tile) {
    const int b = tile % kTiles;
    const bool ok = wait_bar(sh, &sh.tfull[w][b], (tile_ph >> b) & 1u);
    tile_ph ^= 1u << b;
    return __all_sync(0xffffffffu, ok);
  }
  __device__ __forceinline__ void free_tile(int tile) {
    __syncwarp();
    if (lane == 0) arrive(&sh.tempty[tile % kTiles]);
  }
};

// Pass 1, rare: 32-column blocks (bits of `bad`) whose sums left the fp32
// range, or of a chunk that reaches the window: the sums over the chunk's
// tiles against the largest scaled logit of each column (rounded up, M), from
// the logits still in tensor memory; (0, 0) when no key is attended.
__device__ __noinline__ void p1_slow(ResidentShared& sh, const ChunkDesc& d, int quarter,
                                     int lane, uint32_t bad, float2* out) {
  assume_shared(&sh);
  const int window = sh.call.window;
  const float c = sh.call.c;
  const int nt = d.nt, n = d.n, L = d.L;
  const int tok0 = d.t0 * kTileTokens + quarter * 32;
  const uint32_t tb = sh.call.tbase + (static_cast<uint32_t>(quarter * 32) << 16);
#pragma unroll 1
  for (; bad != 0u; bad &= bad - 1u) {
    const int c0 = 32 * (__ffs(bad) - 1);
    const int lim = d.n_rows - c0;
    float mx[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) mx[i] = kNegInf;
    bool any = false;
#pragma unroll 1
    for (int t = 0; t < nt; ++t) {
      uint32_t r[32];
      tmem_load_block(tb + static_cast<uint32_t>(d.col + t * d.width + c0), r);
      const uint32_t ok = block_mask(c0, window, lim, tok0 + t * kTileTokens, n, L, lane);
      any |= ok != 0u;
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        const int i = 2 * ((e >> 2) & 3) + (e & 1);
        if ((ok >> e) & 1u) mx[i] = fmaxf(mx[i], __uint_as_float(r[e]) * c);
      }
    }
    float S = 0.f, M = 0.f;
    if (__any_sync(0xffffffffu, any)) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
#pragma unroll
        for (int bit = 16; bit >= 4; bit >>= 1)
          mx[i] = fmaxf(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], bit));
        mx[i] = mx[i] == kNegInf ? 0.f : ceilf(mx[i]);
      }
      float acc[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] = 0.f;
#pragma unroll 1
      for (int t = 0; t < nt; ++t) {
        uint32_t r[32];
        tmem_load_block(tb + static_cast<uint32_t>(d.col + t * d.width + c0), r);
        const uint32_t ok = block_mask(c0, window, lim, tok0 + t * kTileTokens, n, L, lane);
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          const int i = 2 * ((e >> 2) & 3) + (e & 1);
          if ((ok >> e) & 1u) acc[i] += ex2_approx(fmaf(__uint_as_float(r[e]), c, -mx[i]));
        }
      }
      M = mx[0];
#pragma unroll
      for (int i = 1; i < 8; ++i) M = block_slot(lane) == i ? mx[i] : M;
      S = sum_over_keys(acc, lane);
    }
    if (block_col(lane) < lim) out[c0 + block_col(lane)] = make_float2(M, S);
  }
}

// Second round of a unit's sums (one warp), for rows whose chunk sums left
// the bins or whose total is too small for their grid: the largest chunk
// exponent of every row by an atomic maximum (with a ticket: the maximum is
// complete when every chunk has put its own in), then the sums again against
// it.
__device__ __noinline__ bool slow_denominators(ResidentShared& sh, const ChunkDesc& d, float* out,
                                               int lane) {
  assume_shared(&sh);
  const int grid = sh.call.grid;
  const int nown = (d.x_last - d.x) / grid + 1;
  const int first = d.x / grid;  // this chunk's number among the CTA's
  const int nch = d.nch;
  const int rows = sh.call.acc_rows;
  unsigned long long* const acc =
      sh.call.acc + static_cast<long long>(d.unit) * kAccWords * rows;
  int* const ticket = sh.call.slow_ticket + d.unit;
  // the sums are complete, so this CTA's chunks have left theirs, or are about
  // to leave the pairs
  bool ok = true;
  {
    const uint64_t t0 = globaltimer_ns();
    while (ok && ld_volatile(&sh.sum_pos) <= d.x_last) ok = still_waiting(sh, t0);
    if (!__all_sync(0xffffffffu, ok)) return false;
    __threadfence_block();
  }
  auto own = [&](int i, int q) -> float2 {
    return __ldcg(sh.call.pairs + (first + i) % sh.call.ring * rows + q);
  };
#pragma unroll 1
  for (int q = lane; q < d.n_rows; q += 32) {
    unsigned long long mx = 0ull;
#pragma unroll 1
    for (int i = 0; i < nown; ++i) {
      const float2 pr = own(i, q);
      if (!(pr.y == 0.f)) mx = max(mx, order_key(pr.x + __log2f(pr.y)));
    }
    atomicMax(acc + kAccMax * rows + q, mx);
  }
  __syncwarp();
  if (lane == 0) {
    __threadfence();
    atomicAdd(ticket, nown);
    ok = wait_counter(sh, ticket, nch);
    __threadfence();
  }
  if (!__all_sync(0xffffffffu, ok)) return false;
  const Bins B(nch);
  const unsigned long long mask = (1ull << B.cb) - 1ull;
#pragma unroll 1
  for (int q = lane; q < d.n_rows; q += 32) {
    const unsigned long long key = ld_relaxed64(acc + kAccMax * rows + q);
    const float top = key == 0ull ? NAN : ceilf(order_value(key));
    float nR = 0.f, w = NAN;  // no finite denominator: the scores are NaN
    if (top - top == 0.f) {
      unsigned long long* a = acc + kAccSlow * rows + q;
#pragma unroll 1
      for (int i = 0; i < nown; ++i) {
        const float2 pr = own(i, q);
        const float v = pr.y * pow2i(static_cast<int>(fmaxf(pr.x - top, -1024.f)));
        red_add64(a, (__float2ull_rn(v * pow2i(B.vb - 2)) << B.cb) | 1ull);
      }
      const uint64_t t0 = globaltimer_ns();
      unsigned long long x = 0ull;
#pragma unroll 1
      for (uint32_t it = 1;; ++it) {
        x = ld_relaxed64(a);
        if (static_cast<int>(x & mask) == nch) break;
        if ((it & 31u) == 0 && !still_waiting(sh, t0)) {
          ok = false;
          break;
        }
      }
      const float D = __ull2float_rn(x >> B.cb) * pow2i(2 - B.vb);
      if (D > 0.f) {
        split_denominator(D, &nR, &w);
        nR -= top;
      }
    }
    out[q] = nR;
    out[rows + q] = w;
  }
  return __all_sync(0xffffffffu, ok);
}

// (-R_q, w_q) of a unit's query rows from the given LSE (one warp).
__device__ __noinline__ void lse_denominators(ResidentShared& sh, const ChunkDesc& d, float* out,
                                              int lane) {
  assume_shared(&sh);
  const CallInfo& p = sh.call;
  const float* lse = p.lse + static_cast<long long>(d.s) * p.lse_bs +
                     static_cast<long long>(d.g) * p.group_size * p.lse_hs;
  const int W = p.window, rows = p.acc_rows, n_rows = d.n_rows;
  const uint32_t bits = d.bits;
  for (int q = lane; q < n_rows; q += 32) {
    const int hi = q / W;
    const float l2 = lse[static_cast<long long>(nth_bit(bits, hi)) * p.lse_hs + (q - hi * W)] *
                     1.4426950408889634f;
    const float R = rintf(l2);
    out[q] = -R;
    out[rows + q] = R - R == 0.f ? ex2_approx(R - l2) : 1.f;
  }
}

// (-R_q, w_q) of the unit's query rows once all its chunks are in (one warp).
__device__ __forceinline__ bool denominators(ResidentShared& sh, const ChunkDesc& d, float* out,
                                             int lane) {
  const int rows = sh.call.acc_rows;
  const int n_rows = d.n_rows;
  const int nch = d.nch;
  const Bins B(nch);
  const uint32_t mask = (1u << B.cb) - 1u;
  // below this the rounding to bin 0's grid would show in the total
  const float dmin = pow2i(kAccE0 - B.vb + B.cb + 23);
  const unsigned long long* const acc =
      sh.call.acc + static_cast<long long>(d.unit) * kAccWords * rows;
  bool ok = true, slow = false;
#pragma unroll 1
  for (int q = lane; q < n_rows && ok; q += 32) {
    unsigned long long v[kAccBins + 1];
    const uint64_t t0 = globaltimer_ns();
#pragma unroll 1
    for (uint32_t it = 1;; ++it) {
      uint32_t cnt = 0u;
#pragma unroll
      for (int k = 0; k <= kAccBins; ++k) v[k] = ld_relaxed64(acc + k * rows + q);
#pragma unroll
      for (int k = 0; k <= kAccBins; ++k) cnt += static_cast<uint32_t>(v[k]) & mask;
      if (cnt == static_cast<uint32_t>(nch)) break;
      __nanosleep(100);
      if ((it & 31u) == 0 && !still_waiting(sh, t0)) {
        ok = false;
        break;
      }
    }
    // the bins, smallest first, in fp32: D is good to 2^-23
    float D = 0.f, scale = pow2i(B.grid(0));
    const float step = pow2i(B.width);
#pragma unroll
    for (int k = 0; k < kAccBins; ++k) {
      D = fmaf(__ull2float_rn(v[k] >> B.cb), scale, D);
      scale *= step;
    }
    slow |= v[kAccOut] != 0ull || !(D >= dmin && D < 1.0e38f);
    split_denominator(D, out + q, out + rows + q);
  }
  fence_acq_rel_cta();  // (see sum_role)
  if (!__all_sync(0xffffffffu, ok)) return false;
  if (__any_sync(0xffffffffu, slow)) return slow_denominators(sh, d, out, lane);
  return true;
}

// Pass 1 of a 32 x 32 block that reaches the window or the sequence's end (a
// key at distance x >= 0 into the window is seen by the rows of window
// positions >= x, keys past the sequence by none): adds to acc.
__device__ __noinline__ void p1_edge_block(uint32_t taddr, float c, int w0, int W, int lim, int wl,
                                           int lane, uint64_t* acc) {
  uint32_t r[32];
  tmem_load_block(taddr, r);
#pragma unroll
  for (int e = 0; e < 32; e += 2) {
    const int j = (e >> 2) & 3;
    const int k = 16 * (e >> 4) + 8 * ((e >> 1) & 1) + (lane >> 2);
    const int x = k - lim < wl ? k - lim : 1 << 30;
    int w = w0 + 8 * j;  // (W is a multiple of 16: no pair of columns straddles)
    w = w >= W ? w - W : w;
    w = w >= W ? w - W : w;
    const float e0 = ex2_approx(__uint_as_float(r[e]) * c);
    const float e1 = ex2_approx(__uint_as_float(r[e + 1]) * c);
    acc[j] = add2(acc[j], pack2(w >= x ? e0 : 0.f, w + 1 >= x ? e1 : 0.f));
  }
}

// Pass 1 of a chunk (one warp): the sums of 2^(z c) over the warp's keys of
// the chunk's tiles, per query row, as pairs (M, S) with sum = S 2^M (M = 0
// unless the sums would leave the fp32 range).
__device__ __forceinline__ bool pass1(Group& g, const ChunkDesc& d, int nt, int tile0,
                                      float2* out, uint32_t tbase, float c) {
  const int N = d.n_rows;
  const int lane = g.lane;
  const int width = d.width;
  const int tok0 = d.t0 * kTileTokens + g.quarter * 32;  // the warp's first key
  const int lim0 = d.n - tok0;                           // its keys before the window
  const uint32_t tb =
      tbase + (static_cast<uint32_t>(g.quarter * 32) << 16) + static_cast<uint32_t>(d.col);
  uint32_t bad = 0u;  // blocks whose sums are taken the slow way, below
  const uint64_t c2 = pack2(c, c);
  const int bcol = block_col(lane);
#pragma unroll 1
  for (int c0 = 0; c0 < N; c0 += 32) {
    uint64_t acc2[4] = {0ull, 0ull, 0ull, 0ull};
    uint32_t ta = tb + static_cast<uint32_t>(c0);
    int lim = lim0;
#pragma unroll 1
    for (int t = 0; t < nt; ++t) {
      if (c0 == 0) {
        if (!g.wait_tile(tile0 + t)) return false;
        tc_fence_after();
      }
      if (lim >= 32) {
        uint32_t r[32];
        tmem_load_block(ta, r);
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          const int j = (e >> 2) & 3;
          const uint64_t z = pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1]));
          acc2[j] = add2(acc2[j], exp2_2(mul2(z, c2)));
        }
      } else {
        const int W = g.sh.call.window;
        uint64_t a[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) a[j] = acc2[j];
        p1_edge_block(ta, c, (c0 + 2 * (lane & 3)) % W, W, lim, d.L - d.n, lane, a);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc2[j] = a[j];
      }
      ta += static_cast<uint32_t>(width);
      lim -= kTileTokens;
    }
    float acc[8];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      unpack2(acc2[j], acc[2 * j], acc[2 * j + 1]);
    const float S = sum_over_keys(acc, lane);
    const int col = c0 + bcol;
    const bool in = col < N;
    bool out_of_range = in && !(S >= kSumLo && S <= kSumHi);
    if (__any_sync(0xffffffffu, out_of_range)) {
      // (a row that sees no key of the warp has the sum 0)
      if (lim0 < 32) out_of_range = out_of_range && lim0 > d.n - d.L &&
                                    col % g.sh.call.window >= -lim0;
      if (__any_sync(0xffffffffu, out_of_range)) bad |= 1u << (c0 >> 5);
    }
    if (in) out[col] = make_float2(0.f, S);
  }
  if (bad != 0u) p1_slow(g.sh, d, g.quarter, lane, bad, out);
  return true;
}

// Pass 2 of a chunk (one warp): raw scores of its keys.  (Causality needs no
// mask here: every query row sees every prefix key, and the scores of later
// keys are not kept.)
__device__ __forceinline__ bool pass2(Group& g, const ChunkDesc& d, int nt, int tile0,
                                      const float* den, uint32_t tbase, float c) {
  const int N = d.n_rows;
  const int lane = g.lane;
  const int width = d.width;
  const bool wait = d.mode == kModeP2;  // else pass 1 has seen the tiles written
  uint32_t ta =
      tbase + (static_cast<uint32_t>(g.quarter * 32) << 16) + static_cast<uint32_t>(d.col);
  const float* dl = den + 2 * (lane & 3);
  const int rows = g.sh.call.acc_rows;
  const uint64_t c2 = pack2(c, c);
  int tok = d.t0 * kTileTokens + g.quarter * 32 + block_key(lane);
  const int n = d.n;
  float* raw = g.sh.call.raw + d.soff;
  tc_fence_after();
#pragma unroll 1
  for (int t = 0; t < nt; ++t) {
    if (wait) {
      if (!g.wait_tile(tile0 + t)) return false;
      tc_fence_after();
    }
    uint64_t rs2[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 1
    for (int c0 = 0; c0 < N; c0 += 32) {
      uint64_t nr[4], wt[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        nr[j] = *reinterpret_cast<const uint64_t*>(dl + c0 + 8 * j);
        wt[j] = *reinterpret_cast<const uint64_t*>(dl + rows + c0 + 8 * j);
      }
      uint32_t r[32];
      tmem_load_block(ta + static_cast<uint32_t>(c0), r);
      if (N - c0 == 16) {  // the block's last 16 columns are not query rows
#pragma unroll
        for (int j = 2; j < 4; ++j) {
          nr[j] = wt[j] = 0ull;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            r[16 * (k >> 1) + 4 * j + 2 * (k & 1)] = r[16 * (k >> 1) + 4 * j + 2 * (k & 1) + 1] = 0u;
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int e = 16 * (k >> 1) + 4 * j + 2 * (k & 1);
          const uint64_t z = pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1]));
          rs2[k] = fma2(exp2_2(fma2(z, c2, nr[j])), wt[j], rs2[k]);
        }
    }
    tc_fence_before();
    g.free_tile(tile0 + t);
    float rs[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float x, y;
      unpack2(rs2[k], x, y);
      rs[k] = x + y;
    }
    const float v = sum_over_cols(rs, lane);
    if (tok < n) raw[tok] = v;
    tok += kTileTokens;
    ta += static_cast<uint32_t>(width);
  }
  return true;
}

__device__ __forceinline__ void wait_plain(const uint64_t* bar, uint32_t parity,
                                           uint64_t timeout_ns) {
  volatile int never = 0;
  mbar_wait_bounded(smem_u32(bar), parity, &never, nullptr, timeout_ns);
}

// The end of the producer: waits for what may still land in this CTA's
// shared memory (bounded: after an abort some never comes).  After an abort
// the copies already issued; then the UMMA warp's releases of the stages and
// Q buffers, tcgen05.commit arrivals that nobody else waits for at the end.
__device__ __noinline__ void drain_loads(ResidentShared& sh, uint32_t k_used, uint32_t k_phase,
                                         uint32_t q_used, uint32_t q_phase) {
  assume_shared(&sh);
  const bool ab = ld_volatile(&sh.abort_cta) != 0;
#pragma unroll 1
  for (int pass = ab ? 0 : 1; pass < 2; ++pass) {
    const uint64_t ns = pass == 0 ? 100000000ull : (ab ? 1000000ull : sh.call.wait_ns);
#pragma unroll 1
    for (int i = 0; i < kMaxStages + 3; ++i) {
      const bool q = i >= kMaxStages;
      const int b = q ? i - kMaxStages : i;
      if (!(((q ? q_used : k_used) >> b) & 1u)) continue;
      const uint64_t* bar = pass == 0 ? (q ? &sh.qfull[b] : &sh.full[b])
                                      : (q ? &sh.qempty[b] : &sh.empty[b]);
      wait_plain(bar, ((q ? q_phase : k_phase) >> b) & 1u, ns);
    }
  }
}

__device__ __noinline__ void producer_role(ResidentShared& sh, int lane) {
  assume_shared(&sh);
  const CallInfo& p = sh.call;
  const int nst = p.stages, nqb = p.q_bufs, qh = p.q_half_bytes;
  uint8_t* const sK = p.sK;
  uint8_t* const sQ = p.sQ;
  // ------------------------------------------------------------ TMA
  if (lane == 0) {
    // K is read once; the query rows are reused by every chunk.
    const uint64_t pol_once = l2_policy_evict_first();
    const uint64_t pol_keep = l2_policy_evict_last();
    Ring st, qr;
    uint32_t k_used = 0, k_phase = 0, q_used = 0, q_phase = 0;
    for (int c = 0;; ++c) {
      const int ds = c % kDescs;
      if (!wait_bar(sh, &sh.dfull[ds], static_cast<uint32_t>(c / kDescs) & 1u)) break;
      const ChunkDesc& d = sh.descs[ds];
      if (d.mode == 0) break;
      if (d.new_q) {
        // head block hi of the buffer holds the W window rows of the
        // group's hi-th SRH head
        if (!wait_bar(sh, &sh.qempty[qr.i], qr.ph ^ 1u)) break;
        const uint32_t bar = smem_u32(&sh.qfull[qr.i]);
        mbar_arrive_expect_tx(bar, static_cast<uint32_t>(d.n_rows) * (kHeadDim * 2));
        uint32_t dst = smem_u32(sQ + qr.i * 2 * qh);
#pragma unroll 1
        for (uint32_t bits = d.bits; bits != 0u; bits &= bits - 1u) {
          const int head = d.g * p.group_size + (__ffs(bits) - 1);
          tma_load_4d(dst, p.tmap_q, bar, 0, 0, head, d.s, pol_keep);
          tma_load_4d(dst + qh, p.tmap_q, bar, 64, 0, head, d.s, pol_keep);
          dst += static_cast<uint32_t>(p.window * 128);
        }
        q_used |= 1u << qr.i;
        q_phase = (q_phase & ~(1u << qr.i)) | (qr.ph << qr.i);
        qr.next(nqb);
      }
      int row = d.row0 + d.t0 * kTileTokens;
      bool stop = false;
      const int nt = d.nt, gr = d.g;
      arrive(&sh.dempty[ds]);
#pragma unroll 1
      for (int t = 0; t < nt; ++t, row += kTileTokens) {
        if (!wait_bar(sh, &sh.empty[st.i], st.ph ^ 1u)) {
          stop = true;
          break;
        }
        const uint32_t bar = smem_u32(&sh.full[st.i]);
        mbar_arrive_expect_tx(bar, kTileBytes);
        const uint32_t dst = smem_u32(sK + st.i * kTileBytes);
        tma_load_3d(dst, p.tmap_k, bar, 0, gr, row, pol_once);
        tma_load_3d(dst + kHalfTileBytes, p.tmap_k, bar, 64, gr, row, pol_once);
        k_used |= 1u << st.i;
        k_phase = (k_phase & ~(1u << st.i)) | (st.ph << st.i);
        st.next(nst);
      }
      if (stop) break;
    }
    drain_loads(sh, k_used, k_phase, q_used, q_phase);
  }
  __syncwarp();
}

// The UMMA warp.  All its lanes run the same code and one issues (descriptors
// then stay in uniform registers: a tile of up to 64 rows takes 700 clocks
// with its waits instead of 910 from one lane of a diverged warp).  A second
// issuing warp would not help: tensor-memory loads queue behind the UMMAs
// issued, and took 600 to 1000 clocks instead of 190 with two issuers.
__device__ __noinline__ void mma_role(ResidentShared& sh, int lane) {
  assume_shared(&sh);
  const CallInfo& p = sh.call;
  const int nqb = p.q_bufs, qh = p.q_half_bytes, nst = p.stages;
  const bool bf16 = p.is_bf16 != 0;
  const uint32_t tbase = p.tbase;
  const uint64_t dk0 = smem_desc_sw128(smem_u32(p.sK));
  const uint64_t dqb = smem_desc_sw128(smem_u32(p.sQ));
  Ring st, qr;
  int qb = 0;        // Q buffer of the current unit
  int last_st = -1;  // stage (and its phase) of the last UMMAs issued
  uint32_t last_ph = 0;
  // Tensor memory is taken as a ring of columns: a tile takes its columns
  // after those of the tile before, and first waits for the tiles, oldest
  // first, that still hold columns up to there.
  int tile = 0, oldest = 0, end = 0;
  for (int c = 0;; ++c) {
    const int ds = c % kDescs;
    if (!wait_all(sh, &sh.dfull[ds], static_cast<uint32_t>(c / kDescs) & 1u)) break;
    const ChunkDesc& d = sh.descs[ds];
    const int mode = d.mode, nt = d.nt, wg = d.wg;
    const int n_rows = d.n_rows, new_q = d.new_q, last_q = d.last_q, width = d.width;
    int col = d.col;
    __syncwarp();
    if (lane == 0) arrive(&sh.dempty[ds]);
    if (mode == 0) break;
    if (new_q) {
      qb = qr.i;
      if (!wait_all(sh, &sh.qfull[qb], qr.ph)) break;
      qr.next(nqb);
    }
    const uint32_t idesc = umma_idesc_f16(kTileTokens, n_rows, bf16);
    const uint64_t dq0 = dqb + static_cast<uint64_t>((qb * 2 * qh) >> 4);
    const uint64_t qhalf = static_cast<uint64_t>(qh >> 4);
    bool stop = false;
#pragma unroll 1
    for (int t = 0; t < nt; ++t, col += width) {
      const bool wrap = col < end;  // the columns after `end` are skipped
      for (; oldest < tile; ++oldest) {
        const int o = oldest % kTiles;
        const int c0 = sh.tile_c0[o], c1 = sh.tile_c1[o];
        const bool in_way = tile - oldest >= kTiles ||
                            (wrap ? c1 > end || c0 < col + width : c1 > end && c0 < col + width);
        if (!in_way) break;
        if (!wait_all(sh, &sh.tempty[o], static_cast<uint32_t>(oldest / kTiles) & 1u)) {
          stop = true;
          break;
        }
      }
      if (stop || !wait_all(sh, &sh.full[st.i], st.ph)) {
        stop = true;
        break;
      }
      tc_fence_after();
      const int b = tile % kTiles;
      const uint32_t dt = tbase + static_cast<uint32_t>(col);
      const uint64_t dk = dk0 + static_cast<uint64_t>((st.i * kTileBytes) >> 4);
      if (elect_one()) {
        sh.tile_c0[b] = col;
        sh.tile_c1[b] = col + width;
#pragma unroll
        for (int k8 = 0; k8 < kHeadDim / 16; ++k8) {
          const uint64_t koff = ((k8 >> 2) * kHalfTileBytes + (k8 & 3) * 32) >> 4;
          const uint64_t qoff = (k8 >> 2) * qhalf + (((k8 & 3) * 32) >> 4);
          umma_f16(dt, dk + koff, dq0 + qoff, idesc, k8 > 0 ? 1u : 0u);
        }
        // for the warpgroup that reads the tile first
        umma_commit(smem_u32(&sh.tfull[(mode & kModeP1) ? 0 : wg][b]));
        umma_commit(smem_u32(&sh.empty[st.i]));
      }
      __syncwarp();
      end = col + width;
      last_st = st.i;
      last_ph = st.ph;
      st.next(nst);
      ++tile;
    }
    if (stop) break;
    if (last_q && elect_one()) umma_commit(smem_u32(&sh.qempty[qb]));
    __syncwarp();
  }
  if (lane == 0 && ld_volatile(&sh.abort_cta) != 0 && last_st >= 0)
    wait_plain(&sh.empty[last_st], last_ph, 100000000ull);  // MMAs done before TMEM is freed
  __syncwarp();
}

// Sum of four pairs of which some have another power of two than 0 (rare).
__device__ __noinline__ float2 sum_pairs(const float2* src, int rows) {
  float m = kNegInf, S = 0.f;
#pragma unroll 1
  for (int w = 0; w < 4; ++w)
    if (!(src[w * rows].y == 0.f)) m = fmaxf(m, src[w * rows].x);
#pragma unroll 1
  for (int w = 0; w < 4; ++w)
    if (!(src[w * rows].y == 0.f)) S += src[w * rows].y * ex2_approx(src[w * rows].x - m);
  return make_float2(m == kNegInf ? 0.f : m, S);
}

__device__ __noinline__ void sum_role(ResidentShared& sh, int lane) {
  assume_shared(&sh);
  const CallInfo& p = sh.call;
  const int rows = p.acc_rows;
  int k1 = 0;    // pass-1 chunks so far
  int slot = 0;  // ... in the ring of their sums
  bool ok = wait_bar(sh, &sh.startbar, 0);
  for (int c = 0; __all_sync(0xffffffffu, ok); ++c) {
    const int ds = c % kDescs;
    ok = wait_all(sh, &sh.dfull[ds], static_cast<uint32_t>(c / kDescs) & 1u);
    if (!ok) break;
    const ChunkDesc& d = sh.descs[ds];
    if (d.mode == 0) break;
    if (d.mode & kModeP1) {
      const int b = k1 & 1;
      const Bins B(d.nch);
      const int n_rows = d.n_rows;
      unsigned long long* const acc =
          p.acc + static_cast<long long>(d.sum_unit) * kAccWords * rows;
      float2* const keep = p.pairs + slot * rows;
      const float2* src = pair_row(sh, b * 4);
      ok = wait_all(sh, &sh.p1full[b], static_cast<uint32_t>(k1 >> 1) & 1u);
      if (!ok) break;
      // pass 1's reads of the chunk's tiles, and the UMMAs it has waited for,
      // come before pass 2's reads (which begin once a warp of this CTA has
      // seen the sums below) and the tiles' release
      fence_acq_rel_cta();
#pragma unroll 1
      for (int q = lane; q < n_rows; q += 32) {
        const float2 v0 = src[q], v1 = src[rows + q], v2 = src[2 * rows + q], v3 = src[3 * rows + q];
        float2 o = make_float2(0.f, (v0.y + v1.y) + (v2.y + v3.y));
        if (!(v0.x == 0.f && v1.x == 0.f && v2.x == 0.f && v3.x == 0.f))
          o = sum_pairs(src + q, rows);
        add_sum(B, acc + q, rows, o.x, o.y);
        keep[q] = o;  // for the second round of sums that leave the bins
      }
      __syncwarp();
      if (lane == 0) {
        arrive(&sh.p1empty[b]);
        __threadfence_block();  // the pairs, for slow_denominators
        *reinterpret_cast<volatile int*>(&sh.sum_pos) = d.x + 1;
      }
      ++k1;
      slot = slot + 1 == p.ring ? 0 : slot + 1;
      // (tiles that pass 2 does not read from this copy, at most four: freed here)
      if (d.mode == kModeP1 && lane < 4 * d.nt) arrive(&sh.tempty[(d.tile + (lane >> 2)) % kTiles]);
    }
    __syncwarp();
    if (lane == 0) arrive(&sh.dempty[ds]);
  }
  __syncwarp();
}

// Warpgroup 0 without a given LSE.
__device__ __noinline__ void pass1_role(ResidentShared& sh, int warp, int lane) {
  assume_shared(&sh);
  const uint32_t tbase = sh.call.tbase;
  const float c = sh.call.c;
  Group g{sh, 0, warp & 3, lane};
  int k1 = 0;    // pass-1 chunks so far
  int tile = 0;  // K tiles so far
  for (int ci = 0;; ++ci) {
    const int ds = ci % kDescs;
    if (!__all_sync(0xffffffffu,
                    wait_bar(sh, &sh.dfull[ds], static_cast<uint32_t>(ci / kDescs) & 1u)))
      break;
    const ChunkDesc& d = sh.descs[ds];
    const int mode = d.mode;
    const int nt = d.nt;
    if (mode == 0) break;
    if (mode & kModeP1) {
      const int b = k1 & 1;
      const bool ok = wait_bar(sh, &sh.p1empty[b], (static_cast<uint32_t>(k1 >> 1) & 1u) ^ 1u);
      if (!__all_sync(0xffffffffu, ok)) break;
      if (!pass1(g, d, nt, tile, pair_row(sh, b * 4 + g.quarter), tbase, c)) break;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive(&sh.p1full[b]);
      ++k1;
    }
    tile += nt;
    __syncwarp();
    if (lane == 0) arrive(&sh.dempty[ds]);
  }
}

// Warpgroup 1 (warpgroup 0 too when the LSE is given: every other chunk).
template <int w>
__device__ __noinline__ void pass2_role(ResidentShared& sh, int warp, int lane) {
  assume_shared(&sh);
  const uint32_t tbase = sh.call.tbase;
  const float c = sh.call.c;
  Group g{sh, w, warp & 3, lane};
  int k2 = 0;     // pass-2 chunks of the call so far
  int tile = 0;  // K tiles so far
  int unit = -1;  // unit whose denominators this warpgroup holds
  int kd = -1;    // units whose denominators it has taken, minus one
  for (int ci = 0;; ++ci) {
    const int ds = ci % kDescs;
    if (!__all_sync(0xffffffffu,
                    wait_bar(sh, &sh.dfull[ds], static_cast<uint32_t>(ci / kDescs) & 1u)))
      break;
    const ChunkDesc& d = sh.descs[ds];
    const int mode = d.mode;
    const int nt = d.nt;
    if (mode == 0) break;
    if (mode & kModeP2) {
      if (d.wg == w) {
        if (d.unit != unit) {
          __syncwarp();
          if (kd >= 0 && lane == 0) arrive(&sh.dnempty[w][kd & 1]);
          ++kd;
          const bool ok =
              wait_bar(sh, &sh.dnfull[w][kd & 1], static_cast<uint32_t>(kd >> 1) & 1u);
          if (!__all_sync(0xffffffffu, ok)) break;
          unit = d.unit;
        }
        if (!pass2(g, d, nt, tile, den_row(sh, w, kd & 1), tbase, c)) break;
        // announced by the scheduler thread, off this path
        const int k = k2 % kPub;
        __syncwarp();
        bool ok = true;
        if (lane == 0)
          ok = wait_bar(sh, &sh.p2empty[k], (static_cast<uint32_t>(k2 / kPub) & 1u) ^ 1u);
        if (!__all_sync(0xffffffffu, ok)) break;
        if (lane == 0) {
          if (g.quarter == 0) sh.p2_unit[k] = unit;
          arrive(&sh.p2full[k]);
        }
      }
      ++k2;
    }
    tile += nt;
    __syncwarp();
    if (lane == 0) arrive(&sh.dempty[ds]);
  }
}

// Tells the selection which chunks are scored, in order: after the
// warpgroup's arrivals (CTA-scope release/acquire) one GPU-scope fence covers
// the chunks that are ready, then each adds to its unit's count.
__device__ __noinline__ void announce_role(ResidentShared& sh, int* p2done, int lane) {
  assume_shared(&sh);
  if (lane == 0 && wait_bar(sh, &sh.startbar, 0)) {  // every CTA has zeroed its counts
    int next = 0, issued = 0;  // first chunk not yet announced, pass-2 chunks listed
    for (int ci = 0;;) {
      // the next pass-2 chunk
      bool end = false;
      while (issued == next && !end) {
        const int ds = ci % kDescs;
        if (!wait_bar(sh, &sh.dfull[ds], static_cast<uint32_t>(ci / kDescs) & 1u)) end = true;
        const int mode = end ? 0 : sh.descs[ds].mode;
        if (mode == 0) end = true;
        if (mode & kModeP2) ++issued;
        arrive(&sh.dempty[ds]);
        ++ci;
      }
      if (end) break;
      const int k = next % kPub;
      if (!wait_bar(sh, &sh.p2full[k], static_cast<uint32_t>(next / kPub) & 1u)) break;
      fence_acq_rel_gpu();
      atomicAdd(p2done + sh.p2_unit[k], 1);
      arrive(&sh.p2empty[k]);
      ++next;
    }
  }
  __syncwarp();
}

// Two warps, each every other unit of a warpgroup (its buffer of two).
__device__ __noinline__ void denominator_role(ResidentShared& sh, int mine, int lane) {
  assume_shared(&sh);
  const bool given_lse = sh.call.given_lse != 0;
  int unit[2] = {-1, -1}, k[2] = {0, 0};  // per warpgroup: last unit, units so far
  bool ok = given_lse || wait_bar(sh, &sh.startbar, 0);  // no stale sums from here on
  for (int ci = 0; __all_sync(0xffffffffu, ok); ++ci) {
    const int ds = ci % kDescs;
    if (!wait_all(sh, &sh.dfull[ds], static_cast<uint32_t>(ci / kDescs) & 1u)) break;
    const ChunkDesc& d = sh.descs[ds];
    if (d.mode == 0) break;
    const int w = d.wg;
    if (d.unit != (w ? unit[1] : unit[0])) {
      const int kw = w ? k[1]++ : k[0]++;
      if (w) unit[1] = d.unit; else unit[0] = d.unit;
      if ((kw & 1) == mine) {
        ok = wait_all(sh, &sh.dnempty[w][mine], (static_cast<uint32_t>(kw >> 1) & 1u) ^ 1u);
        if (!ok) break;
        float* const out = den_row(sh, w, mine);
        if (given_lse) {
          lse_denominators(sh, d, out, lane);
        } else {
          ok = denominators(sh, d, out, lane);
        }
        if (!ok) break;
        __syncwarp();
        if (lane == 0) arrive(&sh.dnfull[w][mine]);
      }
    }
    __syncwarp();
    if (lane == 0) arrive(&sh.dempty[ds]);
  }
  __syncwarp();
}

// A number of its own for every CTA, by the SM it is on: neighbours on one TPC
// get neighbouring numbers, as in a launch on an idle GPU (chunks of a unit on
// SMs far apart, as CTAs that start one by one behind another kernel have them,
// cost 5 to 20%).  A slot taken already (an SM's number may change) goes on to
// the next free one; -1 (the CTA leaves) when none is, in a workspace that was
// not initialised.
__device__ __noinline__ int number_by_sm(int* ctr) {
  uint32_t sm;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
  const uint32_t all = gridDim.x;
  sm %= all;
#pragma unroll 1
  for (uint32_t left = all; left; --left) {
    const uint32_t bit = 1u << (sm & 31u);
    if (!(atomicOr(reinterpret_cast<unsigned*>(ctr + kCtrSlots) + (sm >> 5), bit) & bit))
      return static_cast<int>(sm);
    if (++sm == all) sm = 0;
  }
  return -1;
}

// Whether this CTA takes part in the call (one thread, first thing): all do once
// all have started; when not all have kStartWaitNs after one has, the call is
// closed to the others, which leave.  Whatever the words held before, a CTA ends
// with a number below a grid of at most gridDim.x, or leaves.
__device__ __forceinline__ void take_part(ResidentShared& sh, int* ctr) {
  const unsigned all = gridDim.x;
  unsigned* const word = reinterpret_cast<unsigned*>(ctr + kCtrArrive);
  const unsigned old = atomicAdd(word, 1u);
  int id = static_cast<int>(blockIdx.x), grid = static_cast<int>(all);
  const uint64_t t0 = globaltimer_ns();
#pragma unroll 1
  for (unsigned w = old + 1u; w != all; w = static_cast<unsigned>(ld_acquire(ctr + kCtrArrive))) {
    if (w & kClosed) {
      id = old & kClosed ? -1 : static_cast<int>(old & 0xFFFFu);
      grid = static_cast<int>((w >> 16) & 0x3FFFu);
      break;
    }
    const unsigned n = w & 0xFFFFu;
    if (n == all) {  // kApart
      id = number_by_sm(ctr);
      break;
    }
    const uint64_t t = globaltimer_ns() - t0;
    if (t > kStartWaitNs) {
      atomicCAS(word, w, kClosed | (n << 16) | n);
    } else if (t > kStartApartNs && !(w & kApart)) {
      atomicCAS(word, w, w | kApart);
    }
  }
  if (id >= grid || grid > static_cast<int>(all)) id = -1;
  sh.call.id = id;
  sh.call.grid = grid;
}

// Once every CTA has come here, nothing reads the start's words any more.
__device__ __forceinline__ void past_start(ResidentShared& sh, int* ctr) {
  if (atomicAdd(ctr + kCtrPast, 1) == static_cast<int>(gridDim.x) - 1) {
    ctr[kCtrArrive] = ctr[kCtrZeroed] = ctr[kCtrPast] = 0;
    for (int i = 0; i < (kResidentMaxGrid + 31) / 32; ++i) ctr[kCtrSlots + i] = 0;
    ctr[kCtrCalls] = sh.call.number;
  }
}

// The list of a CTA's chunks, id, id + grid, ...: what chunk l.x belongs to.
__device__ __forceinline__ void locate_chunk(const ResidentParams& p, ListPos& l) {
  if (l.x >= p.n_chunks) return;
  if (l.x >= l.off_next) {
    int sq = l.sq, off, off_next = l.off_next;
#pragma unroll 1
    do {
      ++sq;
      off = off_next;
      off_next = p.chunk_off[sq + 1];
    } while (l.x >= off_next);
    l.sq = sq;
    l.off = off;
    l.off_next = off_next;
    l.row0 = p.cu_seqlens[sq];
    l.L = p.cu_seqlens[sq + 1] - l.row0;
    l.nch = (off_next - off) / p.num_kv_heads;
    l.ct = p.seq_chunk[sq];
  }
  const int gr = (l.x - l.off) / l.nch;
  const int unit = l.sq * p.num_kv_heads + gr;
  if (unit != l.unit) {
    l.unit = unit;
    l.gr = gr;
    l.unit_end = l.off + (gr + 1) * l.nch;
    l.bits = p.srh_bits[srh_group(l.sq, gr, p.seqs_per_mask, p.num_kv_heads)];
    l.n_rows = __popc(l.bits) * p.window;
    l.width = (l.n_rows + 31) & ~31;
    l.soff = gr * p.p_total + p.cu_prefix[l.sq];
  }
}
__device__ __forceinline__ void first_chunk(const ResidentParams& p, ListPos& l, int id) {
  l.x = id;
  l.sq = l.unit = -1;
  l.off_next = 0;
  locate_chunk(p, l);
}
// Chunk l.x's descriptor; end: of the last chunk's tensor-memory columns, tile:
// tiles so far, unit: whose pass 2 is in hand.
__device__ __forceinline__ void write_chunk(const ResidentParams& p, const ListPos& l, ChunkDesc& d,
                                            int mode, int wg, int new_q, int grid, int& end,
                                            int& tile, int& unit) {
  const int ct = l.ct;
  const int width = l.width;
  const int cc = l.x - (l.unit_end - l.nch);
  const int nt = min(((l.L + kTileTokens - 1) / kTileTokens) - cc * ct, ct);
  d.new_q = new_q;
  d.last_q = l.x + grid >= l.unit_end ? 1 : 0;  // this CTA's last chunk of the unit
  d.mode = mode;
  d.wg = wg;
  unit = mode == kModeP1 ? unit : l.unit;
  d.unit = unit;
  d.sum_unit = l.unit;
  d.s = l.sq;
  d.g = l.gr;
  d.t0 = cc * ct;
  d.nt = nt;
  d.n_rows = l.n_rows;
  d.nch = l.nch;
  d.n = l.L - p.window;
  d.L = l.L;
  d.row0 = l.row0;
  d.soff = l.soff;
  d.bits = l.bits;
  d.ct = ct;
  // the chunk's columns: the next multiple of their number, so that
  // floor(512 / number) chunks of a unit never stand in one another's way
  const int all = ct * width;
  int col = (end + all - 1) / all * all;
  if (col + all > 512) col = 0;
  end = col + all;
  d.col = col;
  d.width = width;
  d.tile = tile;
  tile += nt;
  d.x = l.x;
  d.x_last = l.x + (l.unit_end - 1 - l.x) / grid * grid;
}
// No more chunks: descriptor c.
__device__ __forceinline__ void write_end(ResidentShared& sh, int c) {
  const int ds = c % kDescs;
  wait_bar(sh, &sh.dempty[ds], (static_cast<uint32_t>(c / kDescs) & 1u) ^ 1u);
  sh.descs[ds].mode = 0;
  arrive(&sh.dfull[ds]);
}

template <int kKind>
__global__ void __launch_bounds__(kRThreads, 1) resident_kernel(const __grid_constant__ ResidentParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const int nst = p.stages;
  const int nqb = p.q_bufs;
  const int qh = p.q_half_bytes;
  uint8_t* sK = base;
  uint8_t* sQ = base + nst * kTileBytes;  // nqb buffers of two 64-column halves
  float2* sRows = reinterpret_cast<float2*>(sQ + 2 * nqb * qh);  // kPairRows rows
  ResidentShared& sh = *reinterpret_cast<ResidentShared*>(sRows + kPairRows * p.acc_rows);
  uint8_t* creg = reinterpret_cast<uint8_t*>(&sh) + kResidentSharedBytes;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  constexpr bool kPieces = kKind != kPlain;

  if (threadIdx.x == kAnnWarp * 32) take_part(sh, p.ctr);
  if (threadIdx.x == 0) {
    auto init = [](uint64_t* b, int n) { mbar_init(smem_u32(b), static_cast<uint32_t>(n)); };
    for (int i = 0; i < nst; ++i) {
      init(&sh.full[i], 1);
      init(&sh.empty[i], 1);
    }
    for (int i = 0; i < kTiles; ++i) {
      init(&sh.tfull[0][i], 1);
      init(&sh.tfull[1][i], 1);
      init(&sh.tempty[i], 4);  // the four warps of the warpgroup that reads it last
    }
#pragma unroll 1
    for (int i = 0; i < kDescs; ++i) {
      init(&sh.dfull[i], 1);
      init(&sh.dempty[i], 6 + kEpiWarps);  // TMA, UMMA, sum, denominator (2) and announcing warps, epilogue
    }
    for (int i = 0; i < nqb; ++i) {
      init(&sh.qfull[i], 1);
      init(&sh.qempty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      init(&sh.p1full[i], 4);
      init(&sh.p1empty[i], 1);
      for (int k = 0; k < 2; ++k) {
        init(&sh.dnfull[i][k], 1);
        init(&sh.dnempty[i][k], 4);
      }
    }
    for (int i = 0; i < kPub; ++i) {
      init(&sh.p2full[i], 4);
      init(&sh.p2empty[i], 1);
    }
    init(&sh.startbar, 1);
    sh.call.status = p.status;
    sh.call.sel.status = p.status;
    sh.call.abort_word = p.ctr + kCtrStop;
    // (stays until every CTA is past the start)
    sh.call.number = ld_volatile(p.ctr + kCtrCalls) + 1;
    sh.call.wait_ns = p.wait_ns;
    sh.call.acc = p.acc;
    sh.call.slow_ticket = p.unit_ctr + p.n_units;
    sh.call.raw = p.raw;
    sh.call.pooled = p.pooled;
    sh.call.lse = p.lse;
    sh.call.lse_bs = p.lse_bs;
    sh.call.lse_hs = p.lse_hs;
    sh.call.tmap_k = &p.tmap_k;
    sh.call.tmap_q = &p.tmap_q;
    sh.call.sK = sK;
    sh.call.sQ = sQ;
    sh.call.rows = sRows;
    sh.call.c = p.c;
    sh.call.stages = nst;
    sh.call.q_bufs = nqb;
    sh.call.q_half_bytes = qh;
    sh.call.window = p.window;
    sh.call.group_size = p.group_size;
    sh.call.is_bf16 = p.is_bf16;
    sh.call.given_lse = p.given_lse;
    sh.call.acc_rows = p.acc_rows;
    sh.call.sel.num_kv_heads = p.num_kv_heads;
    sh.call.sel.pool_width = p.pool_width;
    sh.call.sel.raw_scratch = p.raw_scratch;
    sh.call.sel.k = p.k;
    sh.call.sel.v = p.v;
    sh.call.sel.k_out = p.k_out;
    sh.call.sel.v_out = p.v_out;
    sh.call.sel.tok_stride_v16 = p.tok_stride_v16;
    sh.call.sel.head_stride_v16 = p.head_stride_v16;
    sh.abort_cta = 0;
    sh.sum_pos = 0;
    fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(smem_u32(&sh.tmem), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = sh.tmem;
  const int id = sh.call.id, grid = sh.call.grid;
  if (threadIdx.x == 0) {
    sh.call.tbase = tbase;
    sh.call.ring = grid == kResidentMaxGrid ? kPairRing : kResidentMaxGrid * kPairRing / grid;
    sh.call.pairs = p.pairs + static_cast<long long>(id) * sh.call.ring * p.acc_rows;
  }
  __syncthreads();

  if (kKind == kMixed) pdl_launch_dependents();  // the two-pass kernel of the same call
  if (id < 0) {
    if (threadIdx.x == 0) past_start(sh, p.ctr);
  } else if (warp == kSchedWarp) {
    // ------------------------------------------------------------ descriptors
    if (lane == 0) {
      // test hook: a wait that cannot complete, before anything is issued;
      // it runs out after p.wait_ns and stops the call
      if (p.stall && id == 0) wait_counter(sh, p.ctr + kCtrNever, 1);
      if (p.given_lse || grid >= p.min_grid) {
        ListPos& l = sh.list[0];
        first_chunk(p, l, id);
        int c = 0, last_unit = -1, end = 0, tile = 0, unit = -1;
#pragma unroll 1
        for (; l.x < p.n_chunks; ++c) {
          const int ds = c % kDescs;
          if (!wait_bar(sh, &sh.dempty[ds], (static_cast<uint32_t>(c / kDescs) & 1u) ^ 1u)) break;
          const int new_q = l.unit != last_unit ? 1 : 0;
          last_unit = l.unit;
          write_chunk(p, l, sh.descs[ds], p.given_lse ? kModeP2 : kModeP1 | kModeP2,
                      p.given_lse ? (c & 1) : 1, new_q, grid, end, tile, unit);
          arrive(&sh.dfull[ds]);
          l.x += grid;
          locate_chunk(p, l);
        }
        write_end(sh, c);
      } else {
        // Too few CTAs for a unit's logits to be in tensor memory all at once:
        // its chunks go through pass 1 alone and, after the next unit's pass 1,
        // through pass 2 with K read again.  (The same sums of the same chunks:
        // the same bits.  A loop of its own: the two as one cost 1%, this one as
        // a function 3-6%.)
        ListPos* l = sh.list;
        first_chunk(p, sh.list[0], id);
        first_chunk(p, sh.list[1], id);
        int mode = kModeP1;
        int run = l->x < p.n_chunks ? l->unit : -1;  // the unit in hand
        int prev = -1;                               // and the one before, pass 2 to come
        int c = 0, last_unit = -1, end = 0, tile = 0, unit = -1;
#pragma unroll 1
        for (;;) {
          if (l->x >= p.n_chunks || l->unit != run) {
            const int next = sh.list[0].x < p.n_chunks ? sh.list[0].unit : -1;
            if (mode == kModeP2) {
              if (prev < 0) break;
              mode = kModeP1;
              run = next;
            } else if (prev >= 0) {
              mode = kModeP2;
              const int u = run;
              run = prev;
              prev = u;
            } else {
              prev = run;
              if (prev < 0) break;
              run = next;
            }
            l = sh.list + (mode == kModeP2 ? 1 : 0);
            last_unit = -1;
            continue;
          }
          const int ds = c % kDescs;
          if (!wait_bar(sh, &sh.dempty[ds], (static_cast<uint32_t>(c / kDescs) & 1u) ^ 1u)) break;
          const int new_q = l->unit != last_unit ? 1 : 0;
          last_unit = l->unit;
          write_chunk(p, *l, sh.descs[ds], mode, 1, new_q, grid, end, tile, unit);
          arrive(&sh.dfull[ds]);
          l->x += grid;
          locate_chunk(p, *l);
          ++c;
        }
        write_end(sh, c);
      }
    }
    __syncwarp();
  } else if (warp == kProdWarp) {
    producer_role(sh, lane);
  } else if (warp == kMmaWarp) {
    mma_role(sh, lane);
  } else if (warp == kSumWarp) {
    sum_role(sh, lane);
  } else if (warp >= kEpiWarp0 && warp < kEpiWarp0 + kEpiWarps) {
    if (warp >= kEpiWarp0 + 4) {
      pass2_role<1>(sh, warp, lane);
    } else if (p.given_lse) {
      pass2_role<0>(sh, warp, lane);
    } else {
      pass1_role(sh, warp, lane);
    }
  } else if (warp == kAnnWarp) {
    announce_role(sh, p.unit_ctr, lane);
  } else if (warp == kDenWarp || warp == kDenWarp2) {
    denominator_role(sh, warp == kDenWarp ? 0 : 1, lane);
  } else {
    // ------------------------------------------------------------ workers
    const int ct = threadIdx.x - kCWarp0 * 32;
    {
      // this CTA's share of the accumulators and counters
      const long long who = static_cast<long long>(id) * kCThreads + ct;
      const long long all = static_cast<long long>(grid) * kCThreads;
      if (!p.given_lse) {
        uint4* a = reinterpret_cast<uint4*>(p.acc);
        const long long na = static_cast<long long>(p.n_units) * kAccWords * p.acc_rows / 2;
        for (long long i = who; i < na; i += all) a[i] = make_uint4(0u, 0u, 0u, 0u);
      }
      const long long nc = (kPieces ? 3 : 2) * static_cast<long long>(p.n_units) + (kPieces ? 1 : 0);
      for (long long i = who; i < nc; i += all) p.unit_ctr[i] = 0;
      cbar();
      if (ct == 0) {
        __threadfence();
        atomicAdd(p.ctr + kCtrZeroed, 1);
        const uint64_t t0 = globaltimer_ns();
        while (ld_acquire(p.ctr + kCtrZeroed) < grid && still_waiting(sh, t0)) {
        }
        arrive(&sh.startbar);
        past_start(sh, p.ctr);
      }
    }
#pragma unroll 1
    for (int u = id; !kPieces && p.do_select && u < p.n_units; u += grid) {
      const int s = u / p.num_kv_heads;
      const int g = u - s * p.num_kv_heads;
      const int nch = (p.chunk_off[s + 1] - p.chunk_off[s]) / p.num_kv_heads;
      if (ct == 0) sh.task = wait_counter(sh, p.unit_ctr + u, nch) ? 1 : 0;
      cbar();
      const int go = sh.task;
      cbar();
      if (!go) break;
      SelUnit U;
      U.g = g;
      U.seq0 = p.cu_seqlens[s];
      U.L = p.cu_seqlens[s + 1] - U.seq0;
      U.W = p.window;
      U.out0 = p.cu_out[s];
      U.kept = p.cu_out[s + 1] - U.out0;
      const long long soff = static_cast<long long>(g) * p.p_total + p.cu_prefix[s];
      select_unit<kPlain>(sh.call.sel, U, p.raw + soff, p.pooled + soff,
                  p.indices + static_cast<long long>(g) * p.o_total + U.out0, creg, ct);
    }
    TaskPos T{-1, 0, 0, -1, -1, 0};
#pragma unroll 1
    while (kPieces && (kKind != kMixed || p.do_select)) {
      if (ct == 0) {
        take_ticket(T, p.unit_ctr + 3 * p.n_units, p.batch, p.num_kv_heads, [&](int s) {
          if (kKind == kMixed && p.seq_chunk[s] == 0) return -1;
          return kKind == kInPieces || p.in_pieces
                     ? pool_pieces(p.cu_seqlens[s + 1] - p.cu_seqlens[s] - p.window)
                     : 0;
        });
        bool ok = T.unit >= 0;
        if (ok)
          ok = T.piece < 0 && T.pieces > 0
                   ? wait_counter(sh, p.unit_ctr + 2 * p.n_units + T.unit, T.pieces)
                   : wait_counter(sh, p.unit_ctr + T.unit,
                                  (p.chunk_off[T.s + 1] - p.chunk_off[T.s]) / p.num_kv_heads);
        sh.task = ok ? T.unit : -1;
        sh.piece = T.piece;
        if (kKind == kMixed) sh.pieces = T.pieces;
      }
      cbar();
      const int u = sh.task;
      const int piece = sh.piece;
      cbar();
      if (u < 0) break;
      const int s = u / p.num_kv_heads;
      const int g = u - s * p.num_kv_heads;
      SelUnit U;
      U.g = g;
      U.seq0 = p.cu_seqlens[s];
      U.L = p.cu_seqlens[s + 1] - U.seq0;
      U.W = p.window;
      U.out0 = p.cu_out[s];
      U.kept = p.cu_out[s + 1] - U.out0;
      const long long soff = static_cast<long long>(g) * p.p_total + p.cu_prefix[s];
      SelShared& ss = *reinterpret_cast<SelShared*>(creg);
      uint32_t* const rowmax = p.rowmax + row_max_offset(soff, g, s, p.batch);
      if (piece >= 0) {
        pool_piece(p.raw + soff, p.pooled + soff, rowmax, U.L - U.W, piece, sh.call.sel, ss,
                   p.unit_ctr + 2 * p.n_units + u, 1, ct);
        continue;
      }
      if (ct == 0) ss.rowmax = kKind == kInPieces || sh.pieces > 0 ? rowmax : nullptr;
      cbar();
      select_unit<kKind>(sh.call.sel, U, p.raw + soff, p.pooled + soff,
                        p.indices + static_cast<long long>(g) * p.o_total + U.out0, creg, ct);
    }
  }

  // ------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tbase, 512);
  }
}

}  // namespace

size_t resident_smem_bytes(int q_half_bytes, int q_bufs, int stages, int acc_rows) {
  return 1024 + static_cast<size_t>(stages) * kTileBytes +
         2 * static_cast<size_t>(q_bufs) * q_half_bytes +
         kPairRows * static_cast<size_t>(acc_rows) * sizeof(float2) + kResidentSharedBytes +
         kSelRegion;
}

cudaError_t resident_set_smem_limit(size_t bytes) {
  for (auto kernel : {resident_kernel<kPlain>, resident_kernel<kInPieces>, resident_kernel<kMixed>}) {
    const cudaError_t e = cudaFuncSetAttribute(
        kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_resident(const ResidentParams& p, int grid, size_t smem, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(kRThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = nullptr;
  cfg.numAttrs = 0;
  return cudaLaunchKernelEx(&cfg,
                            p.mixed       ? resident_kernel<kMixed>
                            : p.in_pieces ? resident_kernel<kInPieces>
                                          : resident_kernel<kPlain>,
                            p);
}

}  // namespace ckv
