// Population replay (sm_100a): one CTA of six warps replays one candidate.
//
// Requests are strictly ordered inside a candidate and every step depends on the one before, so a
// replay is bound by the latency of that chain, not by bandwidth.  What is on the chain is kept small:
//  * Cached blocks are tracked per ATOM (see Touch): a long prompt is a handful of atoms instead of
//    its 60 blocks.  Per candidate one word per atom says which replicas hold (a leading part of) the
//    atom; per replica at most one atom is held in part, the one the eviction cursor stands in.
//  * Exact LRU without stamps: the recency order of replica i is the order of the requests routed
//    to it, deepest atom first inside a request; a touch is the atom's latest touch on i iff no
//    later occurrence of the atom (static links) belongs to a request routed to i.
//  * Completions: a request that finishes before one of the next kNear - 1 arrivals is filed in shared
//    memory, any other is pushed onto the list, in memory, of the first request that arrives at or
//    after its finish time.
// Roles, one warp each:
//   route    the chain itself: score (Eq. 3), argmin, cache commit;
//   stage    prefix hits of the coming requests, up to kStages ahead, several requests at once;
//   time     slots, start / first-token / finish times of routed requests, several at once;
//   expiry   in-flight signal that has left each replica by every request's arrival, ahead;
//   scout    lists the coming victims of every replica whose cache is close to full;
//   file     32 requests at a time, one per lane: outputs, completion lists, and the lists' entries
//            for the expiry warp.
// A staged request may have been read before the last commits; the route warp notes the coming
// occurrences of every atom that it changes and stages those requests again, so results never depend
// on the timing of the warps.
//
// Why six warps and not more: the loops of all warps have to stay in the SM's instruction cache.
// Measured with straight-line loops on eight warps, an SM runs at full rate up to about 28 KB of code
// and fetches about one instruction per cycle beyond.  Splitting the route warp further (argmin and
// commits apart, two commit warps) gave 1.07 us per request at one candidate per SM and 1.8 at two;
// this split gives 0.73, 0.84, 1.09 and 1.32 at one to four (long-context trace, 16 replicas, 20,000 requests,
// 4,000 blocks a cache; the twelve-warp kernel on blocks before it 1.09, 1.39, 2.65 and 2.77).  The loops are
// still over the cache: with three or four candidates an SM 128 bytes more in one of them cost about 3 %,
// so what is rare is out of line, and loops that could share a body do.  Three builds share this source
// (launch_replay_n says which a launch takes).  16 / 148 / 256 / 444 / 592 candidates, long contexts (8,000 requests, 2,000
// blocks a cache) with the dense build 0.87 / 0.89 / 0.96 / 1.35 / 1.64 us per request, with the three 0.79 / 0.84 / 0.94 / 1.35 /
// 1.64; shared prompts 0.76 / 0.80 / 0.85 / 1.05 / 1.22 and 0.74 / 0.78 / 0.85 / 1.05 / 1.22; 64 replicas (6,000
// requests) 1.32 / 1.51 / 1.68 / 2.36 / 3.91 and 1.29 / 1.40 / 1.61 / 2.36 / 3.91.
#include "gorgo_device.cuh"

namespace gorgo {
namespace {

// Cycle accounting of the warps (built only with -DGORGO_PROF; the normal library carries none of
// it).  Every lap adds the SM clock ticks since the previous lap of the same warp to one of 16
// accumulators per role; the totals of all candidates end up in g_prof.  What functions out of line spend
// is added by themselves, from 96 on.
#ifdef GORGO_PROF
__device__ unsigned long long g_prof[112];
#define PROF_BEGIN() unsigned long long pf[16] = {}; long long pf_t = clock64()
#define PROF_LAP(k) do { const long long pf_n = clock64(); pf[k] += (unsigned long long)(pf_n - pf_t); pf_t = pf_n; } while (0)
#define PROF_ADD(k, v) pf[k] += (unsigned long long)(v)
#define PROF_MARK(t) const long long t = clock64()
#define PROF_SINCE(k, t) do { if ((threadIdx.x & 31u) == 0) atomicAdd(&g_prof[k], (unsigned long long)(clock64() - t)); } while (0)
#define PROF_COUNT(k) do { if ((threadIdx.x & 31u) == 0) atomicAdd(&g_prof[k], 1ull); } while (0)
#define PROF_END(base) do { if (lane == 0) { _Pragma("unroll") for (int pf_i = 0; pf_i < 16; ++pf_i) atomicAdd(&g_prof[(base) + pf_i], pf[pf_i]); } } while (0)
#else
#define PROF_BEGIN() do {} while (0)
#define PROF_LAP(k) do {} while (0)
#define PROF_ADD(k, v) do {} while (0)
#define PROF_MARK(t) do {} while (0)
#define PROF_SINCE(k, t) do {} while (0)
#define PROF_COUNT(k) do {} while (0)
#define PROF_END(base) do {} while (0)
#endif

// Builds of the kernel that share this source (launch_replay_n says which a launch takes).
enum Build : uint32_t { kSparse = 1, kPaired = 2, kDense = 3 };

constexpr uint32_t kStages = 16;      // requests staged ahead of the commits
constexpr uint32_t kPublish = 8;      // commits are published that many at a time
constexpr uint32_t kFar = 0xFFFFu;    // the touches of a request are not in shared memory
constexpr uint32_t kGroup = 8;        // most requests staged at once
constexpr uint32_t kChunkRing = 64;   // requests whose static data is in shared memory, in chunks
constexpr uint32_t kChunkMin = 4;     // fewest requests of a chunk
constexpr uint32_t kRing = 128;       // requests by request number: routes, completions
constexpr uint32_t kTimes = 64;       // the same where only those between the file warp and the route warp are needed (> kLead)
constexpr uint32_t kLead = 60;        // the route warp runs at most this far ahead of the file warp
constexpr uint32_t kRecent = 62;      // routes of that many requests before a commit are in the ring, older ones in the log
constexpr uint32_t kNear = 64;        // completions within fewer than this many requests skip the lists in memory
constexpr uint32_t kFiled = 16;      // requests the file warp waits for
constexpr uint32_t kList = 64;        // requests whose lists the file warp hands over ahead
constexpr uint32_t kInline = 3;       // list entries of a request handed over in shared memory
// (Rules of the scout.  The times are us per request on reduced cases unless they say otherwise.)
// List victims once a cache is this close to full (blocks).  64, 512 and 2,048 give the same times everywhere
// (within 1 %): a cache passes the margin once, and a list holds 16 or 32 entries.  A few prompts' worth.
constexpr uint32_t kMargin = 512;
// Occurrences looked at before the replica's next requests are asked.  2 / 4 / 8 / 16, shared prompts: 8 replicas
// 0.96 / 0.80 / 0.77 / 0.82, and with a cache of one long prompt 0.77 / 0.79 / 0.83 / 0.88; 32 replicas 2.1 / 2.13 /
// 2.28 / 2.60; 56 replicas 3.87 / 3.90 / 4.04 / 4.47.  Prompts that are not shared: no difference.
constexpr uint32_t kHops = 4;
// Quarters of a list up to which it is filled again.  A commit that takes more victims than are listed waits for a
// scout round, 5,000 to 10,000 ticks.  Filled again from half a list down, that was 7 commits in 100 on small caches (lists
// of 16, found with 10 entries, 14 taken) and 2 with shared prompts; the scout idles for two thirds of the time.
// Half / 5 eighths / 3 quarters / 7 eighths: 32 replicas, 148 candidates 1.18 / 1.13 / 1.11 / 1.11 us per request, 480 candidates
// 1.64 / 1.59 / 1.57 / 1.57; 64 replicas, 60 candidates 1.25 / 1.20 / 1.19 / 1.19; 16 replicas 0.79 / 0.78 / 0.78 / 0.78, four an
// SM 1.46 / 1.46 / 1.47 / 1.47; shared prompts 0.81 / 0.81 / 0.82 / 0.82, four an SM 1.38 / 1.35 / 1.34 / 1.35.
constexpr uint32_t kRefill = 3;
// Requests after which a replica whose order ran out is looked at again.  1 / 4 / 16, a cache of one long prompt:
// 1 replica 1.00 / 1.18 / 1.51, 2 replicas 0.93 / 0.96 / 1.35, 16 replicas 0.99 / 0.95 / 0.95, 64 replicas 1.32 / 1.27 /
// 1.23; larger caches run out of nothing.
constexpr uint32_t kNews = 4;
// Requests of a launch up to which victims are listed only when a commit waits for one.  A proxy waits for every
// launch, and the round the scout is in when the last request is done is part of that: appended and routed one by
// one 39 us (regions) and 45 us (long context), with lists made ahead 44 and 50; two at a time 41 and 48 (regions);
// four to eight within 5 % either way; at 16 the lists win, 91 and 84.  Launches of an uploaded trace that follow one
// another without a wait would take them from two requests on: 8 requests 26.5 and 21.8 us.
constexpr uint32_t kFew = 8;
// Sleeps of the waits, of the idle file and scout warps.  With three and four candidates an SM instruction fetch is what
// the warps share, and polls take part of it.  Waits 20, file and scout 100 / 40 and 500 / 100 and 300 ns: 16 replicas
// three an SM 1.171 / 1.156 / 1.157 us per request, four 1.453 / 1.429 / 1.429; 32 replicas, 480 candidates 1.563 / 1.545 / 1.544; 64
// replicas, 400 candidates 1.938 / 1.924 / 1.925.  One candidate an SM: no difference, but a launch of one request ends when
// the file warp has seen it, so there that sleep stays short.
constexpr uint32_t kWaitNs = 40;
template <uint32_t kBuild> constexpr uint32_t kIdleNs = kBuild == kSparse ? 100 : 500;
constexpr uint32_t kMatches = 32;     // requests of a replica looked at per scout round: one per lane

// Counters the warps hand work over with; first in shared memory, so that their addresses do not depend
// on the build.  committed: commits whose words are visible; decided: commits made; want: the route warp
// waits for a victim of this replica (+ 1); steps, walk, marks: see at_limit.
struct Control {
  volatile uint32_t routed, timed, filed, listed, exp_ready, committed, decided, want, want_timed, abort_flag;
  volatile int32_t status;
  volatile uint32_t steps, walk, marks[6];
  uint32_t scan_pos[64], scan_req[64];   // scout, per replica: next request of the log, request it stands at,
  int32_t scan_k[64];                    //   touch of it
};

// Shared memory of one candidate.  Everything with a fixed size comes first: its addresses are
// constants of the instructions (a layout computed from R, G, K and S cost tens of instructions per
// access).
template <typename MaskT, bool kExt>
struct Shared {
  static constexpr uint32_t kR = sizeof(MaskT) == 8 ? 64 : 32;
  static constexpr uint32_t kRows = sizeof(MaskT) == 8 ? 8 : 16;   // completion rows published ahead of the route warp
  // Listed victims of all replicas together, [R][ring_cap].  Of a victim the route warp needs its atom,
  // the blocks listed for the replica up to and with it (so that the victims of a commit are found by
  // one comparison per entry, without a scan over their lengths) and the request of the atom's first
  // occurrence after the listing.  The rest (that occurrence's touch, the victim's request, its index there,
  // its touch) is read rarely; with 64 replicas it lies in memory, so that three candidates fit an SM.
  static constexpr uint32_t kVictims = sizeof(MaskT) == 8 ? 1024 : 512;
  static constexpr uint32_t kMore = sizeof(MaskT) == 8 ? 1 : kVictims;
  Control c;
  uint64_t mbar[kChunkRing / kChunkMin];
  // stages: request + 1; (input tokens, -, blocks | origin << 16, where its touches are in shared
  // memory (kFar: nowhere) | touches << 16)
  uint4 facts[kStages];
  uint32_t tag[kStages];
  uint16_t hits[kStages][kR];         // prefix hit in blocks
  uint16_t ihits[kExt ? kStages : 1][kExt ? kR : 1];   // and in the proxy's index
  uint32_t epoch[kExt ? kStages : 1];                  // epoch under a time-varying network
  MaskT words[kStages][32];           // mask words of the first 32 atoms
  MaskT iwords[kExt ? kStages : 1][kExt ? 32 : 1];     // and of the proxy's index
  double2 times[kTimes];              // first-token and finish time
  uint2 what[kTimes];                 // (tokens, replica) of a routed request
  uint32_t near_head[kRing];          // request whose completion is seen first by request x, near ones (kNone: none)
  uint32_t near_next[kTimes];         // next of the same x
  double ts[2 * kNear];               // arrivals around the time warp's position
  uint2 listed_e[kList][kInline + 1]; // (rest of the list, entries), (tokens, replica) x 3
  double rows[kRows][kR];             // queue signal gone by the request's arrival
  double w[3 + 64];                   // weights
  uint32_t route_ring[kRing];         // replica | prefix hit << 8
  uint2 part[kR];                     // atom held in part (kNone: none), blocks of it
  uint32_t occ[kR];                   // cached blocks
  uint2 take[kR];                     // victims taken from the ring, blocks taken from the list
  uint32_t cur_req[kR];               // eviction cursor at the start
  int32_t cur_k[kR];
  volatile uint32_t ring_tail[kR];    // victims listed
  uint32_t scan_cum[kR], scan_plen[kR];   // scout: blocks listed, blocks of a partly evicted touch
  uint32_t scan_list[kMatches];       // requests found in the log in a pass
  ReqRec c_req[kChunkRing];           // static data of the requests
  uint32_t c_at[kChunkRing];          // index of a request's touches in c_touch (kNone: they are not all there)
  uint4 victim_more[kMore];
  uint2 victims[kVictims];            // (atom, blocks listed)
  uint32_t victim_next[kVictims];     // request of its next occurrence
  Touch c_touch[1];                   // [chunks][chunk_cap], then the regions of Dyn
};
// Regions whose size depends on the model: [G*R] RTT, [G*R] w_net * RTT, [R*S] time each slot frees.
struct Dyn { double *rtt, *wrtt, *free_at; };

template <typename MaskT, bool kExt>
size_t shared_bytes(const Model& m, uint32_t chunk_req, uint32_t chunk_cap, bool slots_in_smem) {
  return sizeof(Shared<MaskT, kExt>) + (size_t)(kChunkRing / chunk_req) * chunk_cap * sizeof(Touch) +
         ((size_t)m.G * m.R * 2 + (slots_in_smem ? (size_t)m.R * m.S : 0)) * 8;
}

// ---------------------------------------------------------------------------- small helpers
// Keeps a converged warp's plain shared-memory accesses on their side of a counter another warp hands
// data over with.  (The hardware performs a warp's shared-memory accesses in program order; a fence
// would also wait for the warp's global loads in flight.)
__device__ __forceinline__ void smem_order() { __syncwarp(); }
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// A loop-invariant condition the compiler must not see as one: it would clone the loop for each of its
// values, and code size matters here (the loops of all warps together have to stay in the 32 KB
// instruction cache: beyond it the SM fetches about one instruction per cycle for all its warps).
__device__ __forceinline__ uint32_t opaque(uint32_t x) { asm volatile("" : "+r"(x)); return x; }

// Shared-memory accesses of data another warp hands over: they stay where they are written and are
// one transaction per lane.  (A load wider than 4 bytes reaches the lanes in several steps, between
// which another warp's store may fall; lanes that must agree agree on a 4-byte load.)
__device__ __forceinline__ uint4 lds128(uint32_t p) {
  uint4 v;
  asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t p) {
  uint2 v;
  asm volatile("ld.volatile.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t p) {
  uint32_t v;
  asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t p) {
  uint16_t v;
  asm volatile("ld.volatile.shared.u16 %0, [%1];" : "=h"(v) : "r"(p) : "memory");
  return v;
}
__device__ __forceinline__ double lds_f64(uint32_t p) {
  double v;
  asm volatile("ld.volatile.shared.f64 %0, [%1];" : "=d"(v) : "r"(p) : "memory");
  return v;
}
__device__ __forceinline__ void sts128(uint32_t p, uint4 v) {
  asm volatile("st.volatile.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t p, uint2 v) {
  asm volatile("st.volatile.shared.v2.u32 [%0], {%1, %2};" ::"r"(p), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void sts_f64(uint32_t p, double v) {
  asm volatile("st.volatile.shared.f64 [%0], %1;" ::"r"(p), "d"(v) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t p, uint32_t v) {
  asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}

// A walk over the occurrences of an atom, over a replica's order or over a list of completions can be as long
// as the trace: millions of steps behind a single request.  Those that wait meanwhile have to see that it
// goes on: the route and expiry warps count their steps here, the scout leaves the number of its step in
// `walk` and where it stands in scan_*.  (Every such walk is finite: its position only moves forward.)
__device__ __forceinline__ void count_step(uint32_t sb) {
  asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(sb + (uint32_t)offsetof(Control, steps)) : "memory");
}
// A wait has run into its limit.  It starts again if a decision or a walk has moved since this warp was here
// before; else the candidate is marked failed, which ends every wait.  (Out of line, and only at the limit: the
// same look in every poll cost four candidates an SM 8 %.)
__device__ __noinline__ void at_limit(uint32_t sb) {
  if ((threadIdx.x & 31u) != 0) return;
  const uint32_t want = lds32(sb + (uint32_t)offsetof(Control, want)), mark = sb + (uint32_t)offsetof(Control, marks) + threadIdx.x / 32u * 4u;
  uint32_t now = lds32(sb + (uint32_t)offsetof(Control, decided)) + lds32(sb + (uint32_t)offsetof(Control, steps)) + lds32(sb + (uint32_t)offsetof(Control, walk));
  if (want != 0) {
    const uint32_t i = sb + (want - 1u) * 4u;
    now += 0x9E3779B9u * (lds32(i + (uint32_t)offsetof(Control, scan_pos)) + lds32(i + (uint32_t)offsetof(Control, scan_req)) -
                          lds32(i + (uint32_t)offsetof(Control, scan_k)));
  }
  if (now == lds32(mark)) { sts32(sb + offsetof(Control, status), (uint32_t)-6); sts32(sb + offsetof(Control, abort_flag), 1u); }
  sts32(mark, now);
}

// Polls the counter at shared address `p` until (int)(counter - want) >= 0, one lane for the warp.  If
// the limit runs out while nothing moves (or another warp already gave up) the candidate is marked failed
// and every later wait returns at once, so the CTA still terminates.  Called by converged warps; every lane
// gets the same value.  (Out of line: one copy for all waits.)
__device__ __noinline__ uint32_t wait_slow(uint32_t p, uint32_t want, uint32_t sb, uint32_t limit) {
  uint32_t v = 0;
  if ((threadIdx.x & 31u) == 0) {
    v = lds32(p);
    #pragma unroll 1
    for (uint32_t polls = 0; (int32_t)(v - want) < 0; ++polls) {
      if (lds32(sb + offsetof(Control, abort_flag))) break;
      if (polls >= limit) { at_limit(sb); polls = 0; }
      if (polls > 4) __nanosleep(kWaitNs);
      v = lds32(p);
    }
  }
  return __shfl_sync(kFull, v, 0);
}
__device__ __forceinline__ uint32_t wait_counter(uint32_t p, uint32_t want, uint32_t sb, uint32_t limit) {
  const uint32_t v = __shfl_sync(kFull, lds32(p), 0);   // (every lane has to see the same value)
  return (int32_t)(v - want) >= 0 ? v : wait_slow(p, want, sb, limit);
}
__device__ __forceinline__ bool aborted(uint32_t sb) { return __any_sync(kFull, lds32(sb + offsetof(Control, abort_flag)) != 0); }

__device__ __forceinline__ void mbar_init(uint64_t* b) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok) : "r"(smem_addr(b)), "r"(parity) : "memory");
  return ok != 0;
}
// Both addresses 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* b) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(b)) : "memory");
}
// Order-preserving 64-bit key of a score: -0.0 is folded onto +0.0 so that the two zeros tie, as they
// do under '<'; a NaN counts as +inf, and as -inf on replica 0 (what a strict '<' scan from replica 0
// makes of it).
__device__ __forceinline__ uint64_t score_key(double v, bool first) {
  uint64_t b = (uint64_t)__double_as_longlong(__dadd_rn(v, 0.0));
  const uint32_t hi = (uint32_t)(b >> 32);
  if ((hi & 0x7FFFFFFFu) >= 0x7FF00000u && v != v) b = first ? 0xFFF0000000000000ULL : 0x7FF0000000000000ULL;
  return (b >> 63) ? ~b : (b | 0x8000000000000000ULL);
}
// The lowest `index` among the lanes that hold the smallest key.
__device__ __forceinline__ uint32_t argmin(uint64_t key, uint32_t index) {
  const uint32_t hi = (uint32_t)(key >> 32), lo = (uint32_t)key;
  const uint32_t mh = __reduce_min_sync(kFull, hi);
  const uint32_t ml = __reduce_min_sync(kFull, hi == mh ? lo : 0xFFFFFFFFu);
  return __reduce_min_sync(kFull, hi == mh && lo == ml ? index : 0xFFFFFFFFu);
}

// Set / clear `bit` of mask[a] without reading it back (reductions performed in L2).
__device__ __forceinline__ void mask_set(uint32_t* mask, uint32_t a, uint32_t bit) { atomicOr(mask + a, bit); }
__device__ __forceinline__ void mask_set(unsigned long long* mask, uint32_t a, unsigned long long bit) {
  atomicOr(mask + a, bit);
}
__device__ __forceinline__ void mask_clear(uint32_t* mask, uint32_t a, uint32_t bit) { atomicAnd(mask + a, ~bit); }
__device__ __forceinline__ void mask_clear(unsigned long long* mask, uint32_t a, unsigned long long bit) {
  atomicAnd(mask + a, ~bit);
}

// Epoch of the (scaled) time t under a time-varying network: the largest k in [0, n_epochs-1]
// with k * epoch_ms <= t (a quotient as first guess, then the defining comparison).
__device__ __forceinline__ uint32_t epoch_of(const ReplayArgs& a, double t) {
  const double q = t / a.epoch_ms;
  uint32_t k = q >= (double)(a.n_epochs - 1) ? a.n_epochs - 1 : (uint32_t)q;
  #pragma unroll 1
  while (k + 1 < a.n_epochs && __dmul_rn((double)(k + 1), a.epoch_ms) <= t) ++k;
  #pragma unroll 1
  while (k > 0 && __dmul_rn((double)k, a.epoch_ms) > t) --k;
  return k;
}

// Pointers of one candidate into global memory.
template <typename MaskT>
struct Cand {
  MaskT *mask, *index;        // cached-on words, proxy-index words (routed-to ever), one per atom
  CandHeader* hdr;
  RepState* rep;
  double* finish_log;
  uint32_t* exp_head;
  uint4* exp_rec;
  uint8_t* route_log;
  unsigned long long* slot_kv;
  const double* params;
  double scale;
};

// ------------------------------------------------------------------------------- stage warp
// Static data of the requests comes in chunks of chunk_req requests by bulk copies into a ring of
// kChunkRing requests.
struct Chunks {
  uint32_t shift, cap, n_chunks, n_req, n_touch;
  uint32_t next, landed;         // next chunk to request, chunks < landed are in
  uint32_t first_c, buf_mask;    // chunk of the first request, buffers - 1
};
// Requests the next chunk.
template <typename Sh>
__device__ __forceinline__ void chunk_request(const ReplayArgs& a, Sh& sh, const Chunks& ch, uint32_t lane) {
  const uint32_t c = ch.next, buf = c & ch.buf_mask;
  const uint32_t r0 = c << ch.shift, r1 = min(r0 + (1u << ch.shift), ch.n_req);
  const uint32_t off0 = __ldg(&a.tr.req[r0].off);
  const uint32_t off1 = r1 < ch.n_req ? __ldg(&a.tr.req[r1].off) : ch.n_touch;
  if (lane == 0) {
    const uint32_t nt = min(off1 - off0, ch.cap);
    mbar_expect(sh.mbar + buf, (r1 - r0) * 32u + nt * 16u);
    bulk_load(sh.c_req + (buf << ch.shift), a.tr.req + r0, (r1 - r0) * 32u, sh.mbar + buf);
    if (nt) bulk_load(sh.c_touch + buf * ch.cap, a.tr.touch + off0, nt * 16u, sh.mbar + buf);
  }
  __syncwarp();
}
// Waits (bounded) for the next chunk and notes where the touches of its requests are.
template <typename Sh>
__device__ __forceinline__ bool chunk_wait(Sh& sh, const Chunks& ch, uint32_t limit, uint32_t lane) {
  const uint32_t k = ch.landed, buf = k & ch.buf_mask, parity = ((k - ch.first_c) / (ch.buf_mask + 1u)) & 1u;
  bool in = mbar_try(sh.mbar + buf, parity);
  #pragma unroll 1
  for (uint32_t polls = 0; !in && polls < limit; ++polls) { __nanosleep(20); in = mbar_try(sh.mbar + buf, parity); }
  if (!__all_sync(kFull, in)) { sh.c.status = -6; sh.c.abort_flag = 1; return false; }
  const ReqRec* q = sh.c_req + (buf << ch.shift);
  const uint32_t nr = min(1u << ch.shift, ch.n_req - (k << ch.shift));
  if (lane < nr) {
    const uint32_t rel = q[lane].off - q[0].off;
    sh.c_at[(buf << ch.shift) + lane] = rel + q[lane].m <= ch.cap ? buf * ch.cap + rel : kNone;
  }
  __syncwarp();
  return true;
}

template <typename MaskT> __device__ __forceinline__ int first_bit(MaskT v) {
  return sizeof(MaskT) == 8 ? __ffsll((long long)v) - 1 : __ffs((int)v) - 1;
}
__device__ __forceinline__ uint32_t low_bits(uint32_t n) { return n >= 32u ? kFull : (1u << n) - 1u; }

// The atoms of up to kGroup consecutive requests, one per lane: lane j < n passes the number of atoms
// of the j-th request.  As many requests as fit 32 lanes are packed; every lane learns its request and
// the lane of that request's first atom.
// (start, in lane j: the first lane of the j-th request)
struct Pack { uint32_t n, total, g, seg, start; };
__device__ __forceinline__ Pack pack_lanes(uint32_t m, uint32_t n, uint32_t lane) {
  const uint32_t mm = lane < n ? max(m, 1u) : 64u;   // (a request without blocks takes a lane all the same)
  uint32_t incl = mm;
#pragma unroll
  for (int d = 1; d < (int)kGroup; d <<= 1) {
    const uint32_t up = __shfl_up_sync(kFull, incl, d);
    if (lane >= (uint32_t)d) incl += up;
  }
  const unsigned fit = __ballot_sync(kFull, lane < kGroup && incl <= 32u);
  Pack p;
  p.n = (uint32_t)__popc(fit);
  p.start = incl - mm;
  const uint32_t starts = __reduce_or_sync(kFull, lane < p.n ? 1u << p.start : 0u);
  p.total = p.n ? __shfl_sync(kFull, incl, p.n - 1u) : 0u;
  const uint32_t below = starts & (kFull >> (31u - lane));
  p.g = (uint32_t)__popc(below) - 1u;
  p.seg = 31u - (uint32_t)__clz((int)below);
  return p;
}

// What staging needs of the candidate.
template <typename MaskT>
struct StageArgs { MaskT *mask, *index; double scale; };

template <typename MaskT, bool kExt>
__device__ __forceinline__ void stage_facts(const ReplayArgs& a, Shared<MaskT, kExt>& sh, const StageArgs<MaskT>& sa,
                                            uint32_t r) {
  const ReqRec& q = sh.c_req[r % kChunkRing];
  if (kExt && opaque(a.rtt_ewma != nullptr)) sh.epoch[kExt ? r % kStages : 0] = epoch_of(a, __dmul_rn(sa.scale, q.ts_ms));
  sts128(smem_addr(&sh.facts[r % kStages]), make_uint4(q.in_tok, 0u, q.nblk | (uint32_t)q.origin << 16, min(sh.c_at[r % kChunkRing], kFar) | (uint32_t)q.m << 16));
  sts32(smem_addr(&sh.tag[r % kStages]), r + 1u);
}

// Stages one request with the whole warp, from the words in memory as they are now: requests with more
// than 32 atoms, or whose touches are not in shared memory, or that are staged again.
template <typename MaskT, bool kExt>
__device__ __noinline__ void stage_now(const ReplayArgs& a, Shared<MaskT, kExt>& sh, const StageArgs<MaskT> sa,
                                       uint32_t r) {
  constexpr bool kWide = sizeof(MaskT) == 8;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t R = a.m.R, slot = r % kStages;
  const ReqRec& q = sh.c_req[r % kChunkRing];
  const uint32_t at = sh.c_at[r % kChunkRing], m = q.m, nblk = q.nblk;
  const bool index = kExt && opaque(a.proxy_index);
  MaskT alive = R >= sizeof(MaskT) * 8 ? ~(MaskT)0 : (((MaskT)1 << R) - 1), ialive = index ? alive : 0;
  // per replica (lane and lane + 32): leading atoms held at least in part, the first of them that is
  // its partly held atom; the same for the index
  uint32_t run0 = 0, run1 = 0, irun0 = 0, irun1 = 0, kp0 = kNone, kp1 = kNone;
  #pragma unroll 1
  for (uint32_t base = 0; base < m; base += 32) {
    const uint32_t k = base + lane, cnt = min(m - base, 32u);
    MaskT word = 0, iword = 0;
    uint32_t atom = kNone;
    if (k < m) {
      atom = at != kNone ? sh.c_touch[at + k].atom : __ldg(&a.tr.touch[q.off + k].atom);
      word = __ldcg(sa.mask + atom);
      if (index) iword = __ldcg(sa.index + atom);
      if (base == 0) {
        sh.words[slot][lane] = word;
        if (index) sh.iwords[kExt ? slot : 0][kExt ? lane : 0] = iword;
      }
    }
    const MaskT w0 = __shfl_sync(kFull, word, 0);
    MaskT hold = w0 & alive, all = 0;
    #pragma unroll 1
    while (hold) {
      const uint32_t i = (uint32_t)first_bit<MaskT>(hold);
      hold &= hold - 1;
      const uint32_t b = __ballot_sync(kFull, (word >> i) & 1), full = low_bits(cnt);
      const uint32_t rr = (b & full) == full ? cnt : (uint32_t)__ffs((int)~b) - 1u;
      const uint32_t pb = __ballot_sync(kFull, atom == sh.part[i].x && atom != kNone) & low_bits(rr);
      const uint32_t kp = pb ? base + (uint32_t)__ffs((int)pb) - 1u : kNone;
      if (kWide && i >= 32u) { if (lane == i - 32u) { run1 += rr; kp1 = min(kp1, kp); } }
      else if (lane == i) { run0 += rr; kp0 = min(kp0, kp); }
      if (rr == cnt) all |= (MaskT)1 << i;
    }
    alive = all;
    if (index) {
      hold = __shfl_sync(kFull, iword, 0) & ialive; all = 0;
      #pragma unroll 1
      while (hold) {
        const uint32_t i = (uint32_t)first_bit<MaskT>(hold);
        hold &= hold - 1;
        const uint32_t b = __ballot_sync(kFull, (iword >> i) & 1), full = low_bits(cnt);
        const uint32_t rr = (b & full) == full ? cnt : (uint32_t)__ffs((int)~b) - 1u;
        if (kWide && i >= 32u) { if (lane == i - 32u) irun1 += rr; }
        else if (lane == i) irun0 += rr;
        if (rr == cnt) all |= (MaskT)1 << i;
      }
      ialive = all;
    }
  }
  auto blocks_of = [&](uint32_t run, uint32_t kp, uint32_t plen) -> uint32_t {
    const uint32_t k = min(run, kp);
    if (k >= m) return nblk;
    const uint32_t pos = (at != kNone ? sh.c_touch[at + k].len_pos : __ldg(&a.tr.touch[q.off + k].len_pos)) >> 16;
    return pos + (kp < run ? plen : 0u);
  };
  sh.hits[slot][lane] = (uint16_t)blocks_of(run0, kp0, sh.part[lane].y);
  if (kWide) sh.hits[slot][kWide ? lane + 32u : 0u] = (uint16_t)blocks_of(run1, kp1, sh.part[kWide ? lane + 32u : 0u].y);
  if (index) {
    sh.ihits[kExt ? slot : 0][kExt ? lane : 0] = (uint16_t)blocks_of(irun0, kNone, 0u);
    if (kWide) sh.ihits[kExt ? slot : 0][kExt && kWide ? lane + 32u : 0u] = (uint16_t)blocks_of(irun1, kNone, 0u);
  }
  __syncwarp();
  if (lane == 0) stage_facts<MaskT, kExt>(a, sh, sa, r);
  __syncwarp();
}

// Stages the coming requests, up to kGroup of them at once with one atom per lane; the words of the
// next group are requested before those of the current one are looked at.
template <typename MaskT, bool kExt>
__device__ __forceinline__ void stage_warp(const ReplayArgs& a, Shared<MaskT, kExt>& sh, uint32_t sb,
                                           const StageArgs<MaskT>& sa, uint32_t lane) {
  using Sh = Shared<MaskT, kExt>;
  const uint32_t end = a.first + a.count;
  Chunks ch;
  ch.shift = 31 - __clz((int)a.tr.chunk_req);
  ch.cap = a.tr.chunk_cap;
  ch.buf_mask = kChunkRing / a.tr.chunk_req - 1u;
  ch.first_c = ch.next = ch.landed = a.first >> ch.shift;
  ch.n_req = end;                                   // (nothing behind the launch's requests is needed)
  ch.n_touch = end < a.tr.n_req ? __ldg(&a.tr.req[end].off) : a.tr.n_touch;
  ch.n_chunks = ((end - 1) >> ch.shift) + 1;
  // the group whose words are on their way: its first request, its size (0: none);
  // per lane: request and atom of it, its first lane, word and atom
  uint32_t q = a.first, n = 0, g = 0, seg = 0, m_seg = 0, atom = kNone, pos = 0;
  MaskT word = 0, iword = 0;
  const bool use_index = kExt && opaque(a.proxy_index);
  uint32_t next_q = a.first;                        // first request that is not in a group yet
  PROF_BEGIN();
  #pragma unroll 1
  while (q < end) {
    // ---- the next group: as many requests as there are free stages, landed chunks and lanes
    uint32_t n2 = 0, view2 = 0, g2 = 0, seg2 = 0, m2 = 0, atom2 = kNone, pos2 = 0;
    MaskT word2 = 0, iword2 = 0;
    bool slow = false;
    if (next_q < end) {
      view2 = __shfl_sync(kFull, lds32(sb + offsetof(Control, committed)), 0);
      uint32_t room = min(end, view2 + kStages) - next_q;
      if (room == 0 && n == 0) {                    // nothing to do before another commit
        view2 = wait_counter(sb + offsetof(Control, committed), view2 + 1u, sb, a.poll_limit);
        room = min(end, view2 + kStages) - next_q;
        if (room == 0) break;                       // gave up
      }
      PROF_LAP(0);
      if (room > 0) {
        const uint32_t c = next_q >> ch.shift;
        if (ch.landed <= c) {                       // the first request of a chunk
          // chunks up to c + 2, as far as the requests in their buffers are committed and timed
          const uint32_t done = min(view2, __shfl_sync(kFull, lds32(sb + offsetof(Control, timed)), 0));
          #pragma unroll 1
          while (ch.next <= c + 2u && ch.next < ch.n_chunks) {
            if (ch.next - ch.first_c > ch.buf_mask && ((ch.next - ch.buf_mask) << ch.shift) > done) {
              if (ch.next > c) break;
              wait_counter(sb + offsetof(Control, timed), (ch.next - ch.buf_mask) << ch.shift, sb, a.poll_limit);
              if (aborted(sb)) break;
            }
            chunk_request(a, sh, ch, lane);
            ++ch.next;
          }
          if (aborted(sb) || !chunk_wait(sh, ch, a.poll_limit, lane)) break;
          ++ch.landed;
        }
        room = min(room, (ch.landed << ch.shift) - next_q);
        uint32_t m = 64u, at = 0;
        if (lane < kGroup && lane < room) {
          at = sh.c_at[(next_q + lane) % kChunkRing];
          m = sh.c_req[(next_q + lane) % kChunkRing].m;
          if (at == kNone || opaque(a.probe_off)) m = 64u;
        }
        const Pack pk = pack_lanes(m, min(room, kGroup), lane);
        n2 = pk.n;
        slow = n2 == 0;
        g2 = pk.g; seg2 = pk.seg;
        const uint32_t k = lane - seg2;
        m2 = __shfl_sync(kFull, m, g2 & 31u);
        at = __shfl_sync(kFull, at, g2 & 31u);
        if (lane < pk.total && k < m2) {
          const uint2 x = *reinterpret_cast<const uint2*>(&sh.c_touch[at + k]);
          atom2 = x.x; pos2 = x.y >> 16;
          word2 = __ldcg(sa.mask + atom2);
          if (use_index) iword2 = __ldcg(sa.index + atom2);
        }
        if (lane >= pk.total) { g2 = kNone; m2 = 0; }
      }
    }
    PROF_LAP(1);
    // ---- hits of the current group
    if (n > 0) {
      // (hit rows start from 0)
      const uint32_t row_words = Sh::kR / 2u;
      #pragma unroll 1
      for (uint32_t t = lane; t < n * row_words; t += 32)
        reinterpret_cast<uint32_t*>(&sh.hits[(q + t / row_words) % kStages][0])[t % row_words] = 0u;
      if (use_index) {
        #pragma unroll 1
        for (uint32_t t = lane; t < n * row_words; t += 32)
          reinterpret_cast<uint32_t*>(&sh.ihits[kExt ? (q + t / row_words) % kStages : 0][0])[kExt ? t % row_words : 0] = 0u;
      }
      __syncwarp();
      const uint32_t r = q + g, k = lane - seg;
      if (k < m_seg) {
        sh.words[r % kStages][k] = word;
        if (use_index) sh.iwords[kExt ? r % kStages : 0][kExt ? k : 0] = iword;
      }
      const uint32_t full = low_bits(m_seg);
      auto prefixes = [&](MaskT wd, bool parts, uint16_t* rows) {   // (rows: [kStages][kR] hits)
        const MaskT first = __shfl_sync(kFull, wd, seg);
        MaskT hold = g < n ? first : 0;
        #pragma unroll 1
        while (__any_sync(kFull, hold != 0)) {      // once per replica that holds the first atom: usually 0 to 2
          const uint32_t i = hold ? (uint32_t)first_bit<MaskT>(hold) : 0u;
          uint2 part = make_uint2(kNone, 0u);
          if (parts) part = lds64(sb + (uint32_t)offsetof(Sh, part) + i * 8u);
          const uint32_t b = __ballot_sync(kFull, (wd >> i) & 1) >> seg;
          const uint32_t pb = __ballot_sync(kFull, k < m_seg && atom == part.x) >> seg;
          const uint32_t run = (b & full) == full ? m_seg : (uint32_t)__ffs((int)~b) - 1u;
          const uint32_t pm = pb & low_bits(run);   // its partly held atom among the leading ones
          const uint32_t kk = pm ? (uint32_t)__ffs((int)pm) - 1u : run;
          const uint32_t ps = __shfl_sync(kFull, pos, min(seg + kk, 31u));
          if (hold && k == 0)
            rows[(r % kStages) * Sh::kR + i] = (uint16_t)(pm ? ps + part.y : run == m_seg ? sh.c_req[r % kChunkRing].nblk : ps);
          hold &= hold - 1;
        }
      };
      prefixes(word, true, &sh.hits[0][0]);
      if (use_index) prefixes(iword, false, &sh.ihits[0][0]);
      __syncwarp();
      if (g < n && k == 0) stage_facts<MaskT, kExt>(a, sh, sa, r);
      q += n;
    }
    PROF_LAP(2);
    if (slow) {
      stage_now<MaskT, kExt>(a, sh, sa, next_q);
      n2 = 0;
      ++next_q;
      q = next_q;
      n = 0;
    } else {
      next_q += n2;
      n = n2; g = g2; seg = seg2; m_seg = m2; atom = atom2; pos = pos2; word = word2; iword = iword2;
    }
    if (aborted(sb)) break;
  }
  PROF_END(80);
  #pragma unroll 1
  while (ch.landed < ch.next) {                     // no bulk copy is in flight when the block ends
    if (!chunk_wait(sh, ch, 1u << 24, lane)) break;
    ++ch.landed;
  }
}

// ------------------------------------------------------------------------------ route warp
// Requests after r, within the reach of the stage warp, that contain an atom that changes (`next`: its
// first occurrence after the touch at hand); bit k: request r + 1 + k.
__device__ __forceinline__ uint32_t dirty_from(const Touch* touch, uint32_t next, uint32_t next_req, uint32_t r) {
  uint32_t d = 0;
  #pragma unroll 1
  while (next != kNone && next_req - r < kStages) {
    d |= 1u << (next_req - r - 1u);
    const uint2 nx = __ldg(reinterpret_cast<const uint2*>(&touch[next].next));
    next = nx.x; next_req = nx.y;
  }
  return d;
}
// A listed victim whose atom occurs again before r + kStages, first at touch `next` of request
// `next_req`: is its touch still the latest on replica `rep` as of the commit of request r there?
// `dirty` gets what comes after r.
__device__ __forceinline__ bool victim_live(const Touch* touch, const uint8_t* route_log, uint32_t sb, uint32_t ring, uint32_t next,
                                            uint32_t next_req, uint32_t r, uint32_t first, uint32_t rep, uint32_t& dirty) {
  #pragma unroll 1
  while (next != kNone && next_req <= r) {
    count_step(sb);
    const uint2 nx = __ldg(reinterpret_cast<const uint2*>(&touch[next].next));
    const uint32_t rt = next_req == r ? rep : r - next_req < kRecent && next_req >= first ? (lds32(ring + (next_req % kRing) * 4u) & 0xFFu)
                                                                     : (uint32_t)__ldcg(route_log + next_req);
    if (rt == rep) return false;
    next = nx.x; next_req = nx.y;
  }
  dirty = dirty_from(touch, next, next_req, r);
  return true;
}

// Evicts `need` blocks from replica `rep` for the commit of request r, victims in the order the scout
// lists them, one entry per lane; waits for the scout where its list is too short.  Returns the
// requests that are dirty now (see route_warp).  (Out of line: the route warp handles the usual case
// itself.)
//   The list usually holds more than the commit takes.  The entries behind the first that is enough if all before it are
// victims are left for another round of the loop: the walks of 32 lanes over later occurrences take as long as the
// longest.  (One candidate an SM, half-full lists against full ones: 16 replicas, 639 blocks a cache 1.69 -> 1.49 us per request,
// 64 replicas 1.35 -> 1.31; without the limit and otherwise the same, 148 candidates 0.88 -> 0.85 and, 64 replicas, 1.51 -> 1.43.
// Not in the dense build: with three and four candidates an SM the loops are larger than the instruction cache, and the
// few instructions cost 1 to 2 %, 592 candidates with 64 replicas 5 %.)
template <typename MaskT, bool kExt, uint32_t kBuild>
__device__ __noinline__ uint32_t evict_slow(const ReplayArgs& a, Shared<MaskT, kExt>& sh, MaskT* mask,
                                            const uint8_t* route_log, const uint4* more, uint32_t rep, uint32_t r, uint32_t need) {
  using Sh = Shared<MaskT, kExt>;
  const uint32_t lane = threadIdx.x & 31u, sb = smem_addr(&sh), cap_mask = a.ring_cap - 1u;
  const uint32_t p_take = sb + (uint32_t)offsetof(Sh, take) + rep * 8u;
  const uint32_t p_tail = sb + (uint32_t)offsetof(Sh, ring_tail) + rep * 4u;
  const MaskT bit = (MaskT)1 << rep;
  uint32_t dirty = 0;
  uint32_t head = __shfl_sync(kFull, lds32(p_take), 0), cons = lds32(p_take + 4u);   // entries taken, blocks taken from the list
  #pragma unroll 1
  while (true) {
    uint32_t avail = __shfl_sync(kFull, lds32(p_tail), 0) - head;
    if (avail == 0) {                               // the scout is behind: it lists this replica next
      if (lane == 0) {
        sts64(p_take, make_uint2(head, cons));
        sts32(sb + offsetof(Control, want), rep + 1u);
      }
      PROF_MARK(waited);
      avail = wait_slow(p_tail, head + 1u, sb, a.poll_limit) - head;
      PROF_SINCE(96, waited);
      PROF_COUNT(97);
      if (lane == 0) sts32(sb + offsetof(Control, want), 0u);
      if ((int32_t)avail <= 0) break;               // gave up
    }
    const uint32_t e = rep * a.ring_cap + ((head + lane) & cap_mask);
    const uint2 v = lds64(sb + (uint32_t)offsetof(Sh, victims) + e * 8u);
    const uint32_t next_req = lds32(sb + (uint32_t)offsetof(Sh, victim_next) + e * 4u);
    const uint32_t upto = v.y - cons;               // blocks gone with this entry
    if (kBuild != kDense) {
      const uint32_t most = __ballot_sync(kFull, lane < avail && upto >= need);
      if (most) avail = min(avail, (uint32_t)__ffs((int)most));
    }
    const bool listed = lane < avail;
    bool live = listed;
    uint32_t d = 0;
    PROF_MARK(walked);
    if (listed && next_req < r + kStages) {         // it occurred again since it was listed, or will soon
      const uint32_t next = sizeof(MaskT) == 8 ? __ldcg(&more[e].x) : lds32(sb + (uint32_t)offsetof(Sh, victim_more) + e * 16u);
      live = victim_live(a.tr.touch, route_log, sb, sb + (uint32_t)offsetof(Sh, route_ring), next, next_req, r, a.first, rep, d);
    }
    dirty |= __reduce_or_sync(kFull, d);
    PROF_SINCE(98, walked);
    PROF_COUNT(99);
    const uint32_t prev = __shfl_up_sync(kFull, upto, 1);
    uint32_t dead = listed && !live ? upto - (lane ? prev : 0u) : 0u;   // blocks that are no victims
    if (kBuild == kDense || __any_sync(kFull, dead != 0u)) {
      #pragma unroll 1
      for (uint32_t w = 1; w < 32u; w <<= 1) {
        const uint32_t below = __shfl_up_sync(kFull, dead, w);
        if (lane >= w) dead += below;
      }
    }
    const uint32_t freed = upto - dead;             // blocks that are freed up to this entry
    const uint32_t enough = __ballot_sync(kFull, live && freed >= need);
    // lanes up to the first that is enough (all that are listed, if there is none)
    const uint32_t last = enough ? (uint32_t)__ffs((int)enough) - 1u : min(avail, 32u) - 1u;
    const uint32_t got = __shfl_sync(kFull, freed, last), gone = __shfl_sync(kFull, upto, last);
    const uint32_t atom = __shfl_sync(kFull, v.x, last);
    const uint32_t keep = enough ? got - need : 0u;   // blocks the last victim keeps
    if (live && lane <= last && !(keep && lane == last)) mask_clear(mask, v.x, bit);
    head += last + (keep ? 0u : 1u);
    cons += gone - keep;
    if (lane == 0) sts64(sb + (uint32_t)offsetof(Sh, part) + rep * 8u, make_uint2(keep ? atom : kNone, keep));
    if (enough) break;
    need -= got;
  }
  if (lane == 0) sts64(p_take, make_uint2(head, cons));
  __syncwarp();
  return dirty;
}

// Sets the bit of replica `rep` on the atoms of request r that do not have it.  Returns the blocks that
// were missing; `dirty` gets the requests that are dirty now.  (Out of line, for any number of atoms.)
template <typename MaskT, bool kExt>
__device__ __noinline__ uint32_t commit_slow(const ReplayArgs& a, Shared<MaskT, kExt>& sh, const StageArgs<MaskT> sa,
                                             uint32_t rep, uint32_t r, uint32_t& dirty) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t at = sh.c_at[r % kChunkRing], m = sh.c_req[r % kChunkRing].m;
  const MaskT bit = (MaskT)1 << rep;
  const uint2 part = lds64(smem_addr(&sh.part[rep]));
  uint32_t missing = 0, later = 0;
  bool filled = false;
  #pragma unroll 1
  for (uint32_t k = lane; k < m; k += 32u) {
    const uint4 x = at != kNone ? *reinterpret_cast<const uint4*>(&sh.c_touch[at + k])
                                : __ldg(reinterpret_cast<const uint4*>(a.tr.touch + sh.c_req[r % kChunkRing].off + k));
    const MaskT word = k < 32u ? *const_cast<const volatile MaskT*>(&sh.words[r % kStages][k]) : (MaskT)__ldcg(sa.mask + x.x);
    const bool fills = (word & bit) && x.x == part.x;   // the partly held atom becomes whole
    bool changes = !(word & bit);
    if (changes) mask_set(sa.mask, x.x, bit);
    changes = changes || fills;
    if (changes) missing += (x.y & 0xFFFFu) - (fills ? part.y : 0u);
    filled = filled || fills;
    if (kExt && opaque(a.proxy_index)) {
      const MaskT iword = k < 32u ? *const_cast<const volatile MaskT*>(&sh.iwords[kExt ? r % kStages : 0][kExt ? k : 0])
                                  : (MaskT)__ldcg(sa.index + x.x);
      if (!(iword & bit)) { mask_set(sa.index, x.x, bit); changes = true; }
    }
    if (changes && x.w - r < kStages) later |= dirty_from(a.tr.touch, x.z, x.w, r);
  }
  dirty |= __reduce_or_sync(kFull, later);
  if (__any_sync(kFull, filled) && lane == 0) sts64(smem_addr(&sh.part[rep]), make_uint2(kNone, 0u));
  __syncwarp();
  return __reduce_add_sync(kFull, missing);
}

// The serial chain.  Lane i (and i+32 when kWide) keeps replica i's in-flight signal (an exact integer in
// a double).  Per request: subtract what has completed, score, argmin by reductions and one vote, hand
// the route over, commit: set the replica's bit on the request's atoms (one per lane) and evict what
// the scout has listed (one victim per lane).  An atom that a commit changes is changed for its coming
// occurrences too: those that may be staged already are noted (`dirty`) and staged again when their
// turn comes.
//   What bounds it is the latency of its own instructions.  The usual request takes one straight path in
// which the commit of request q - 1 and the score of q run side by side, their shared-memory reads and
// reductions interleaved, before it is known whether q is ready and its stage up to date; if not
// (about 1.5 requests in 100), q is decided once more with nothing to commit.  Everything unusual is out of line
// behind one vote.  (Commit after score: 0.85 us per request at one candidate per SM; side by side 0.73.)
template <typename MaskT, bool kExt, uint32_t kBuild>
__device__ __forceinline__ void route_warp(const ReplayArgs& a, Shared<MaskT, kExt>& sh, uint32_t sb, const Dyn& dy,
                                           const StageArgs<MaskT>& sa, const uint8_t* route_log, const uint4* more, const RepState* rep,
                                           uint32_t p, uint32_t lane) {
  using Sh = Shared<MaskT, kExt>;
  constexpr bool kWide = sizeof(MaskT) == 8;
  const uint32_t R = a.m.R, K = a.m.K, end = a.first + a.count;
  const bool in0 = lane < R, in1 = kWide && lane + 32u < R;
  const double w_pre = sh.w[1], w_que = sh.w[2];
  double ld0 = 0.0, ld1 = 0.0, nrm0 = 1.0, nrm1 = 1.0;
  if (in0) { ld0 = (double)rep[lane].load; if (K != 3) nrm0 = sh.w[3 + lane]; }
  if (in1) { ld1 = (double)rep[lane + 32].load; if (K != 3) nrm1 = sh.w[35 + lane]; }
  const uint32_t i0 = min(lane, R - 1u), i1 = min(lane + 32u, R - 1u);
  const uint32_t cap_mask = a.ring_cap - 1u;
  const uint32_t C = a.m.C < 0xFFFFFFF0ull ? (uint32_t)a.m.C : 0xFFFFFFF0u;   // (its domain)
  uint32_t dirty = 0;                               // bit k: an atom of request q + k has changed since it was staged
  unsigned long long st_probe = 0, st_hit = 0, st_blk = 0, st_evict = 0;
  // What a request has to wait for, one counter per lane: its stage (lane 0), its completions (lane 1),
  // the file warp (the others).
  const uint32_t p_wait = sb + (lane == 0 ? (uint32_t)offsetof(Sh, tag) : lane == 1 ? (uint32_t)offsetof(Control, exp_ready)
                                                                                   : (uint32_t)offsetof(Control, filed));
  const uint32_t ahead = lane < 2u ? 1u : 1u - kLead;
  // The request that awaits its commit, q - 1 (if `pend`): its replica, this lane's atom of it (lanes
  // without one have all bits set in the word), and whether the commit is an unusual one.
  bool pend = false, odd = false;
  uint32_t istar = 0, atom = kNone - 1u, len = 0, next_req = kNone;
  MaskT word = ~(MaskT)0, iword = ~(MaskT)0;         // (iword: of the proxy's index)
  const bool use_index = kExt && opaque(a.proxy_index);
  uint32_t q = a.first;
  PROF_BEGIN();
  #pragma unroll 1
  while (true) {
    // ---- what the commit of q - 1 and the score of q need from shared memory
    const MaskT bit = (MaskT)1 << istar;
    const uint32_t p_part = sb + (uint32_t)offsetof(Sh, part) + istar * 8u;
    const uint32_t p_occ = sb + (uint32_t)offsetof(Sh, occ) + istar * 4u;
    const uint32_t p_take = sb + (uint32_t)offsetof(Sh, take) + istar * 8u;
    const uint2 tk = lds64(p_take);                             // entries taken, blocks taken from the list
    const uint32_t tail = lds32(sb + (uint32_t)offsetof(Sh, ring_tail) + istar * 4u);
    const uint32_t slot = q % kStages;
    const bool rdy = (int32_t)(lds32(p_wait + (lane == 0 ? slot * 4u : 0u)) - (q + ahead)) >= 0;
    // (valid if q is ready: read after that)
    const uint4 f = lds128(sb + (uint32_t)offsetof(Sh, facts) + slot * 16u);
    const uint32_t p_hit = sb + (uint32_t)offsetof(Sh, hits) + (slot * Sh::kR + lane) * 2u;
    const uint32_t p_row = sb + (uint32_t)offsetof(Sh, rows) + ((q % Sh::kRows) * Sh::kR + lane) * 8u;
    const uint32_t hit0 = lds16(p_hit), hit1 = kWide ? lds16(p_hit + 64u) : 0u;
    const double gone0 = lds_f64(p_row), gone1 = kWide ? lds_f64(p_row + 256u) : 0.0;
    const uint32_t part = lds32(p_part), occ = lds32(p_occ);
    // ---- commit: set the replica's bit on the atoms that do not have it
    const bool changes = !(word & bit);
    if (changes) mask_set(sa.mask, atom, bit);
    const bool indexed = use_index && !(iword & bit);
    if (indexed) mask_set(sa.index, atom, bit);
    uint32_t missing = __reduce_add_sync(kFull, changes ? len & 0xFFFFu : 0u);
    const uint32_t entry = istar * a.ring_cap + ((tk.x + lane) & cap_mask);
    const uint2 v = lds64(sb + (uint32_t)offsetof(Sh, victims) + entry * 8u);
    const uint32_t v_next = lds32(sb + (uint32_t)offsetof(Sh, victim_next) + entry * 4u);
    const bool special = odd || atom == part || ((changes || indexed) && next_req - (q - 1u) < kStages);
    // ---- score of Eq. 3 (fixed order, no FMA) and lowest-index argmin
    const uint32_t in_tok = f.x, nblk = f.z & 0xFFFFu, at = f.w & 0xFFFFu, m = f.w >> 16;
    const double* net = dy.wrtt + (f.z >> 16) * R;
    uint32_t s0 = hit0, s1 = hit1;
    if (use_index) {
      s0 = sh.ihits[kExt ? slot : 0][kExt ? lane : 0];
      if (kWide) s1 = sh.ihits[kExt ? slot : 0][kExt && kWide ? lane + 32u : 0u];
    }
    auto score = [&](uint32_t i, uint32_t h, double load, double nrm) {   // (h < n blocks: h * B < input tokens)
      const double qd = K != 3 ? __dmul_rn(load, nrm) : load;
      const uint32_t unc = h >= nblk ? 0u : in_tok - h * a.m.B;
      double nt = net[i];
      if (kExt && opaque(a.rtt_ewma != nullptr))     // time-varying network: signal of the request's epoch
        nt = __dmul_rn(sh.w[0], __ldg(a.rtt_ewma + ((size_t)sh.epoch[kExt ? slot : 0] * a.m.G + (f.z >> 16)) * R + i));
      return __dadd_rn(__dadd_rn(nt, __dmul_rn(w_pre, (double)unc)), __dmul_rn(w_que, qd));
    };
    uint64_t key = score_key(score(i0, s0, ld0 - gone0, nrm0), lane == 0);
    if (!in0) key = ~0ull;
    uint32_t index = lane;
    if (kWide) {
      uint64_t k1 = score_key(score(i1, s1, ld1 - gone1, nrm1), false);
      if (!in1) k1 = ~0ull;
      if (k1 < key) { key = k1; index = lane + 32u; }
    }
    PROF_LAP(0);
    uint32_t sel = argmin(key, index);
    // ---- this lane's atom of q
    const bool far = at == kFar || m > 32u;
    const bool has = lane < m && !far;
    const uint4 x = *reinterpret_cast<const uint4*>(&sh.c_touch[has ? at + lane : 0u]);
    const MaskT x_word = *const_cast<const volatile MaskT*>(&sh.words[slot][lane]);
    const MaskT x_iword = use_index ? *const_cast<const volatile MaskT*>(&sh.iwords[kExt ? slot : 0][kExt ? lane : 0]) : ~(MaskT)0;
    // ---- eviction for q - 1: the victims are listed, none occurred again since, none occurs again soon
    dirty >>= pend ? 1u : 0u;
    uint32_t held = occ + missing, need = held > C ? held - C : 0u;
    const uint32_t upto = v.y - tk.y;                           // blocks gone with this entry
    const unsigned enough = __ballot_sync(kFull, lane < tail - tk.x && upto >= need);
    const unsigned taken = enough ^ (enough - 1u);              // lanes up to the first that is enough (all if none)
    const bool soon = (taken >> lane & 1u) && v_next < q - 1u + kStages;
    bool valid = !(dirty & 1u);
    PROF_LAP(1);
    if (__any_sync(kFull, special || !rdy || (need != 0u && (soon || enough == 0u)))) {
      PROF_LAP(2);
      const bool again = __any_sync(kFull, special);
      if (again) {
        PROF_ADD(10, 1);
        uint32_t d = dirty;
        missing = commit_slow<MaskT, kExt>(a, sh, sa, istar, q - 1u, d);
        dirty = d;
        held = occ + missing;
        need = held > C ? held - C : 0u;
      }
      PROF_LAP(6);
      if (need != 0u && (again || enough == 0u || __any_sync(kFull, soon))) {
        PROF_ADD(9, 1);
        dirty |= evict_slow<MaskT, kExt, kBuild>(a, sh, sa.mask, route_log, more, istar, q - 1u, need);
        if (kExt) st_evict += need;
        need = 0u;
        held = C;
      }
      PROF_LAP(11);
      valid = __all_sync(kFull, rdy) && !(dirty & 1u);
    }
    PROF_LAP(2);
    PROF_LAP(12);                                               // (nothing: what a lap itself costs)
    if (need != 0u) {
      const uint32_t keep = upto - need;                        // (last of them: blocks the last victim keeps)
      const bool last = taken >> lane == 1u;
      if ((taken >> lane & 1u) && !(last && keep)) mask_clear(sa.mask, v.x, bit);
      if (last) {
        sts64(p_part, make_uint2(keep ? v.x : kNone, keep));
        sts64(p_take, make_uint2(tk.x + lane + (keep ? 0u : 1u), tk.y + need));
      }
      if (kExt) st_evict += need;
      held = C;
    }
    if (lane == 0) {
      sts32(p_occ, held);
      sts32(sb + offsetof(Control, decided), q);
    }
    PROF_LAP(3);
    // words are visible with `committed`; the fence waits for the reductions in flight, so it is made
    // only every kPublish requests
    if (pend && (q % kPublish == 0u || q == end)) {
      __syncwarp();
      __threadfence_block();
      if (lane == 0) sts32(sb + offsetof(Control, committed), q);
      if (q == end || aborted(sb)) break;
    }
    if (!valid) {
      // ---- q was not ready, or its stage has changed: decide again, with nothing to commit
      wait_slow(sb + (uint32_t)offsetof(Sh, tag) + slot * 4u, q + 1u, sb, a.poll_limit);
      wait_slow(sb + offsetof(Control, exp_ready), q + 1u, sb, a.poll_limit);
      wait_slow(sb + offsetof(Control, filed), q + 1u - kLead, sb, a.poll_limit);
      if (aborted(sb)) break;                                   // gave up
      if (dirty & 1u) {
        PROF_ADD(8, 1);
        __syncwarp();
        __threadfence_block();                                  // (the words of the last commits)
        stage_now<MaskT, kExt>(a, sh, sa, q);
        dirty &= ~1u;
      }
      PROF_ADD(7, 1);
      pend = odd = false;
      word = iword = ~(MaskT)0;
      atom = kNone - 1u;
      PROF_LAP(4);
      continue;
    }
    // ---- hand the route over; q awaits its commit
    if (kExt && opaque(a.forced_route != nullptr)) sel = __ldg(a.forced_route + q);
    const bool mine = lane == (sel & 31u), up = kWide && sel >= 32u;
    double add = (double)in_tok;
    if (kExt && opaque(a.queue_in_requests)) add = 1.0;         // baseline "least-request"
    if (mine) {
      sts32(sb + (uint32_t)offsetof(Sh, route_ring) + (q % kRing) * 4u, sel | (up ? hit1 : hit0) << 8);
      sts32(sb + offsetof(Control, routed), q + 1u);
    }
    ld0 += mine && !up ? add : 0.0;
    if (kWide) ld1 += mine && up ? add : 0.0;
    if (kExt && opaque(a.stats != nullptr)) {
      if (in0) st_probe += min(hit0 + 1u, nblk);
      if (in1) st_probe += min(hit1 + 1u, nblk);
      if (mine) st_hit += up ? hit1 : hit0;
      st_blk += nblk;
    }
    istar = sel;
    odd = far;
    atom = has ? x.x : kNone - 1u;
    len = x.y;
    next_req = x.w;
    word = has ? x_word : ~(MaskT)0;
    if (use_index) iword = has ? x_iword : ~(MaskT)0;
    pend = true;
    ++q;
    PROF_LAP(5);
  }
  PROF_END(0);
  const uint32_t last_row = (end - 1u) % Sh::kRows;
  if (in0) sh.rows[last_row][lane] = ld0 - sh.rows[last_row][lane];   // (the signal left)
  if (in1) sh.rows[last_row][kWide ? lane + 32u : 0u] = ld1 - sh.rows[last_row][kWide ? lane + 32u : 0u];
  if (kExt && a.stats) {
    unsigned long long* s4 = reinterpret_cast<unsigned long long*>(a.stats) + (size_t)p * 4;
    atomicAdd(s4, st_probe);
    if (st_hit) atomicAdd(s4 + 1, st_hit);
    if (lane == 0) { atomicAdd(s4 + 2, st_blk); atomicAdd(s4 + 3, st_evict); }
  }
}

// ------------------------------------------------------------------------------- time warp
// Service model of the routed requests (paper Eq. 1: network, queue wait, prefill): up to kTimed
// consecutive requests that went to different replicas at once, 32 / kTimed lanes each (a request takes
// the slot its predecessors on the replica left).  A request that completes before one of the next
// kNear - 1 arrivals is filed here, in shared memory.
constexpr uint32_t kTimed = 4, kTimeLanes = 32 / kTimed;
template <typename MaskT, bool kExt>
__device__ __forceinline__ void time_warp(const ReplayArgs& a, Shared<MaskT, kExt>& sh, uint32_t sb, const Dyn& dy,
                                          unsigned long long* slot_kv, double scale, uint32_t lane) {
  using Sh = Shared<MaskT, kExt>;
  const uint32_t R = a.m.R, S = a.m.S, end = a.first + a.count;
  const uint32_t j = lane / kTimeLanes, sub = lane % kTimeLanes, lead = lane - sub;
  const uint32_t seg_mask = (1u << kTimeLanes) - 1u;
  // arrivals base .. base + 127 are in the ring for s in [base, base + 64)
  uint32_t base = a.first;
#pragma unroll
  for (uint32_t t = lane; t < 2u * kNear; t += 32)
    sh.ts[(base + t) % (2u * kNear)] = base + t < end ? __dmul_rn(scale, __ldg(a.tr.ts + base + t)) : d_inf();
  __syncwarp();
  uint32_t s0 = a.first;
  PROF_BEGIN();
  #pragma unroll 1
  while (s0 < end) {
    // a full round, unless the expiry warp waits for less
    uint32_t seen = wait_counter(sb + offsetof(Control, routed), s0 + 1u, sb, a.poll_limit);
    if ((int32_t)(seen - (s0 + 1u)) < 0) break;            // gave up
    const uint32_t full = min(s0 + kTimed, end);
    #pragma unroll 1
    for (uint32_t polls = 0; (int32_t)(seen - full) < 0 && polls < 64u; ++polls) {
      if ((int32_t)(__shfl_sync(kFull, lds32(sb + offsetof(Control, want_timed)), 0) - s0) > 0) break;
      __nanosleep(50);
      seen = __shfl_sync(kFull, lds32(sb + offsetof(Control, routed)), 0);
    }
    PROF_LAP(0);
    if (s0 - base >= 32u) {                                // the next 32 arrivals
      base += 32u;
      const uint32_t t = base + 3u * 32u + lane;
      sh.ts[t % (2u * kNear)] = t < end ? __dmul_rn(scale, __ldg(a.tr.ts + t)) : d_inf();
      __syncwarp();
    }
    uint32_t n = min(seen - s0, kTimed);
    const uint32_t rq0 = lds32(sb + (uint32_t)offsetof(Sh, route_ring) + ((s0 + j) % kRing) * 4u);
    // requests of a replica already taken in this pass wait for the next one
    {
      const unsigned peers = __match_any_sync(kFull, j < n ? rq0 & 0xFFu : 0x100u + j);
      const unsigned again = __ballot_sync(kFull, (peers & ((1u << lead) - 1u)) != 0u);
      if (again) n = min(n, ((uint32_t)__ffs((int)again) - 1u) / kTimeLanes);
    }
    const bool on = j < n;
    const uint32_t s = s0 + (on ? j : 0u);
    const uint32_t rq_0 = __shfl_sync(kFull, rq0, 0), rq = on ? rq0 : rq_0;
    const ReqRec& q = sh.c_req[s % kChunkRing];
    const uint32_t i = rq & 0xFFu, h = rq >> 8;
    double* fa = dy.free_at + i * S;
    const double t = sh.ts[s % (2u * kNear)];
    const uint32_t in_tok = q.in_tok, out_tok = q.out_tok;
    const uint32_t unc = h >= q.nblk ? 0u : in_tok - h * a.m.B;
    double delay = dy.rtt[q.origin * R + i];
    if (kExt && opaque(a.rtt_raw != nullptr))              // time-varying network: the probe of the request's epoch
      delay = a.rtt_raw[((size_t)epoch_of(a, t) * a.m.G + q.origin) * R + i];
    const double arrive = __dadd_rn(t, delay);
    const double pre_ms = (kExt && opaque(a.rep_prefill_ms != nullptr)) ? a.rep_prefill_ms[i] : a.m.prefill_ms;
    double tok_ms = (kExt && opaque(a.rep_tpot_ms != nullptr)) ? a.rep_tpot_ms[i] : a.m.tpot_ms;
    // earliest-free slot, lowest index on ties
    double bv = d_inf();
    uint32_t bs = kNone;
    #pragma unroll 1
    for (uint32_t s2 = sub; s2 < S; s2 += kTimeLanes) {
      const double v = fa[s2];
      if (v < bv || bs == kNone) { bv = v; bs = s2; }
    }
#pragma unroll
    for (int d = 1; d < (int)kTimeLanes; d <<= 1) {
      const double ov = __shfl_xor_sync(kFull, bv, d);
      const uint32_t os = __shfl_xor_sync(kFull, bs, d);
      if (ov < bv || (ov == bv && os < bs)) { bv = ov; bs = os; }
    }
    double start = bv > arrive ? bv : arrive;
    const unsigned long long need_kv = (unsigned long long)in_tok + out_tok;
    if (kExt && opaque(a.kv_budget > 0)) {
      // admission under the KV budget: wait for other slots to finish until the request fits
      const unsigned long long* kv = slot_kv + (size_t)i * S;
      bool fits = !on;
      #pragma unroll 1
      for (uint32_t round = 0; round <= S; ++round) {
        unsigned long long usage = 0;
        double nf = d_inf();                               // earliest finish among the other busy slots
        #pragma unroll 1
        for (uint32_t s2 = sub; s2 < S; s2 += kTimeLanes) {
          const double f = fa[s2];
          if (s2 != bs && f > start) { usage += kv[s2]; nf = fmin(nf, f); }
        }
#pragma unroll
        for (int d = 1; d < (int)kTimeLanes; d <<= 1) {
          usage += __shfl_xor_sync(kFull, usage, d);
          nf = fmin(nf, __shfl_xor_sync(kFull, nf, d));
        }
        fits = fits || nf == d_inf() || usage + need_kv <= a.kv_budget;
        if (__all_sync(kFull, fits)) break;
        if (!fits) start = nf;
      }
    }
    const double first = __dadd_rn(start, __dmul_rn(pre_ms, (double)unc));
    if (kExt && opaque(a.decode_slowdown > 0.0)) {
      // a fuller batch decodes slower: busy slots at the first token, this one included
      uint32_t busy = 0;
      #pragma unroll 1
      for (uint32_t s2 = sub; s2 < S; s2 += kTimeLanes) busy += (s2 != bs && fa[s2] > first) ? 1u : 0u;
#pragma unroll
      for (int d = 1; d < (int)kTimeLanes; d <<= 1) busy += __shfl_xor_sync(kFull, busy, d);
      tok_ms = __dmul_rn(tok_ms, __dadd_rn(1.0, __dmul_rn(a.decode_slowdown, (double)busy)));
    }
    const double finish = __dadd_rn(first, __dmul_rn(tok_ms, (double)(out_tok > 0 ? out_tok - 1u : 0u)));
    // the first of the next kNear - 1 arrivals that is not before the finish: its eighth, then its place
    const uint32_t e8 = (__ballot_sync(kFull, sh.ts[(s + 1u + sub * 8u + (sub == 7u ? 6u : 7u)) % (2u * kNear)] >= finish) >> lead) & seg_mask;
    const uint32_t blk = e8 ? (uint32_t)__ffs((int)e8) - 1u : 0u;
    const uint32_t e1 = (__ballot_sync(kFull, sh.ts[(s + 1u + blk * 8u + sub) % (2u * kNear)] >= finish) >> lead) & seg_mask;
    const uint32_t x = s + blk * 8u + (uint32_t)__ffs((int)e1);   // (e1 != 0 when e8 != 0)
    __syncwarp();                                          // every lane has read the slots
    if (on && sub == 0) {
      if (kExt && opaque(a.kv_budget > 0)) slot_kv[(size_t)i * S + bs] = need_kv;
      fa[bs] = finish;
      sts_f64(sb + (uint32_t)offsetof(Sh, times) + (s % kTimes) * 16u, first);
      sts_f64(sb + (uint32_t)offsetof(Sh, times) + (s % kTimes) * 16u + 8u, finish);
      sts64(sb + (uint32_t)offsetof(Sh, what) + (s % kTimes) * 8u, make_uint2(in_tok, i));
      if (e8 && x < end) sts32(sb + (uint32_t)offsetof(Sh, near_next) + (s % kTimes) * 4u, atomicExch(&sh.near_head[x % kRing], s));
    }
    __syncwarp();
    s0 += n;
    if (lane == 0) sts32(sb + offsetof(Control, timed), s0);
    PROF_LAP(1);
  }
  PROF_END(16);
}

// ----------------------------------------------------------------------------- expiry warp
// For every request r, ahead of the route warp: the queue signal whose completion the proxy has seen
// by r's arrival, cumulative since the start of the launch, one row per request.  A request j < r is
// due at r only if lb_j = t_j + tpot * decode tokens <= t_r (network, waiting and prefill only add to
// it), so the row waits for the time warp only up to the latest such j.  Completions come from two
// lists of r: near ones (time warp), others (handed over by the file warp).
template <typename MaskT, bool kExt>
__device__ __forceinline__ void expiry_warp(const ReplayArgs& a, Shared<MaskT, kExt>& sh, uint32_t sb,
                                            const uint4* exp_rec, double scale, uint32_t lane) {
  using Sh = Shared<MaskT, kExt>;
  constexpr bool kWide = sizeof(MaskT) == 8;
  const uint32_t R = a.m.R, end = a.first + a.count;
  double tok_ms = a.m.tpot_ms;                         // smallest time per output token over the replicas
  if (kExt && a.rep_tpot_ms) {
    tok_ms = a.rep_tpot_ms[0];
    #pragma unroll 1
    for (uint32_t i = 1; i < R; ++i) tok_ms = fmin(tok_ms, a.rep_tpot_ms[i]);
  }
  // requests base..base+31, one per lane: arrival, and how far the time warp has to be for its row
  double t = 0.0, lb = d_inf(), t_nx = 0.0, lb_nx = d_inf();
  uint32_t need = 0;
  auto load_block = [&](uint32_t b) {
    const uint32_t r = min(b + lane, end - 1u);
    t_nx = __dmul_rn(scale, __ldg(a.tr.ts + r));
    const uint32_t out = __ldg(&a.tr.req[r].out_tok);
    lb_nx = __dadd_rn(t_nx, __dmul_rn(tok_ms, (double)(out > 0 ? out - 1u : 0u)));
  };
  load_block(a.first);
  double cum0 = 0.0, cum1 = 0.0;
  uint32_t timed = a.first, routed = a.first, listed = a.first;
  auto take = [&](uint2 x) {                           // (tokens, replica)
    double v = (double)x.x;
    if (kExt && opaque(a.queue_in_requests)) v = 1.0;
    if (x.y == lane) cum0 += v;
    if (kWide && x.y == lane + 32u) cum1 += v;
  };
  PROF_BEGIN();
  #pragma unroll 1
  for (uint32_t r = a.first; r < end; ++r) {
    if (((r - a.first) & 31u) == 0) {                  // next block: its values were loaded one block ago
      const double lb_old = lb;
      t = t_nx; lb = lb_nx;
      load_block(r + 32u);
      // the latest earlier request of the last 32 that can be due at this lane's request (+ 1)
      need = r + lane - min(r + lane - a.first, 32u);
      #pragma unroll 1
      for (int k = 0; k < 32; ++k) {
        const double old = __shfl_sync(kFull, lb_old, k), now = __shfl_sync(kFull, lb, k);
        if (old <= t && (uint32_t)k >= lane) need = max(need, r - 31u + (uint32_t)k);
        if (now <= t && (uint32_t)k < lane) need = max(need, r + 1u + (uint32_t)k);
      }
      if (aborted(sb)) break;
    }
    const uint32_t cur = (r - a.first) & 31u;
    const double tr = __shfl_sync(kFull, t, cur);
    const uint32_t want = __shfl_sync(kFull, need, cur);
    // the row is free once the route warp has used its previous occupant
    if (r - a.first >= Sh::kRows && (int32_t)(routed - (r + 1u - Sh::kRows)) < 0)
      routed = wait_counter(sb + offsetof(Control, routed), r + 1u - Sh::kRows, sb, a.poll_limit);
    if ((int32_t)(listed - (r + 1u)) < 0) listed = wait_counter(sb + offsetof(Control, listed), r + 1u, sb, a.poll_limit);
    if ((int32_t)(timed - want) < 0) {
      if (lane == 0) sts32(sb + offsetof(Control, want_timed), want);
      timed = wait_counter(sb + offsetof(Control, timed), want, sb, a.poll_limit);
    }
    PROF_LAP(0);
    // near completions
    const uint32_t p_head = sb + (uint32_t)offsetof(Sh, near_head) + (r % kRing) * 4u;
    uint32_t nj = __shfl_sync(kFull, lds32(p_head), 0);
    if (nj != kNone) {
      #pragma unroll 1
      for (uint32_t guard = 0; nj != kNone && guard < kNear; ++guard) {
        take(lds64(sb + (uint32_t)offsetof(Sh, what) + (nj % kTimes) * 8u));
        nj = __shfl_sync(kFull, lds32(sb + (uint32_t)offsetof(Sh, near_next) + (nj % kTimes) * 4u), 0);
      }
      if (lane == 0) sts32(p_head, kNone);
    }
    // the list of r
    const uint32_t p_le = sb + (uint32_t)offsetof(Sh, listed_e) + (r % kList) * ((kInline + 1u) * 8u);
    const uint2 hd = lds64(p_le);
    #pragma unroll 1
    for (uint32_t k = 1; k <= hd.y; ++k) take(lds64(p_le + k * 8u));
    uint32_t e = hd.x;
    #pragma unroll 1
    for (uint32_t guard = 0; e != kNone && guard < a.tr.n_req; ++guard) {   // (rarely: more than kInline entries)
      if (lane == 0) count_step(sb);
      const uint4 rec = __ldcg(exp_rec + e);
      take(make_uint2(rec.y, rec.z));
      e = rec.x;
    }
    sh.rows[r % Sh::kRows][lane] = cum0;
    if (kWide) sh.rows[r % Sh::kRows][kWide ? lane + 32u : 0u] = cum1;
    __syncwarp();
    if (lane == 0) sts32(sb + offsetof(Control, exp_ready), r + 1u);
    PROF_LAP(1);
  }
  PROF_END(32);
}

// ------------------------------------------------------------------------------- file warp
// Everything about a routed request that may lag behind, up to 32 requests at a time, one per lane:
// outputs (coalesced), the route log, the list of the request at whose arrival its completion is seen
// (found through the time grid over the arrivals, then a short scan), and the hand-over of finished
// lists to the expiry warp.  The list of request r gains entries only from requests <= r - kNear, so
// it is final once the file warp has passed r - kNear.
template <typename MaskT, bool kExt, uint32_t kBuild>
__device__ __forceinline__ void file_warp(const ReplayArgs& a, Shared<MaskT, kExt>& sh, const Cand<MaskT>& cd, uint32_t p,
                                          uint32_t lane) {
  const uint32_t end = a.first + a.count, N = a.tr.n_req;
  const double scale = cd.scale;
  const double t_last = __dmul_rn(scale, a.tr.ts[N - 1]);
  // grid bucket of a time: (time / scale) / grid_dt, as one multiplication; the search starts one
  // bucket early, which covers the rounding of this product many times over
  const bool use_grid = a.tr.grid_n > 0 && scale * a.tr.grid_dt >= 1e-280;
  const double to_bucket = use_grid ? 1.0 / (scale * a.tr.grid_dt) : 0.0;
  uint32_t filed = a.first, listed = a.first;
  uint32_t idle = 0;
  PROF_BEGIN();
  #pragma unroll 1
  while (true) {
    bool progress = false;
    // ---- hand lists over: requests < min(end, filed + kNear), not further than the expiry warp has room for
    {
      uint32_t upto = min(end, filed + kNear);
      const uint32_t room = __shfl_sync(kFull, sh.c.exp_ready, 0) + kList;
      smem_order();
      if ((int32_t)(upto - room) > 0) upto = room;
      uint32_t n = upto - listed;
      if (n > 0 && (n >= 16u || upto == end || listed - filed < 40u)) {
        n = min(n, 32u);
        if (lane < n) {
          const uint32_t r = listed + lane;
          uint2* le = sh.listed_e[r % kList];
          uint32_t e = __ldcg(cd.exp_head + r), cnt = 0;
          #pragma unroll 1
          while (e != kNone && cnt < kInline) {
            const uint4 rec = __ldcg(cd.exp_rec + e);
            le[++cnt] = make_uint2(rec.y, rec.z);
            e = rec.x;
          }
          le[0] = make_uint2(e, cnt);
        }
        __syncwarp();
        smem_order();
        listed += n;
        if (lane == 0) sh.c.listed = listed;
        progress = true;
      }
    }
    PROF_LAP(0);
    if (filed == end) { if (listed == end) break; }
    else {
      // ---- file the requests whose times are known
      const uint32_t timed = __shfl_sync(kFull, sh.c.timed, 0);
      smem_order();
      const uint32_t n = min(timed - filed, 32u);
      // many at a time: a pass costs the same for one and for 32
      if (n >= kFiled || (n > 0 && timed == end)) {
        uint32_t old = kNone, x = kNone;
        const uint32_t j = filed + lane;
        if (lane < n) {
          const double2 tm = sh.times[j % kTimes];
          const uint32_t rq = sh.route_ring[j % kRing];
          const uint2 what = sh.what[j % kTimes];
          const uint32_t istar = rq & 0xFFu;
          const double t = __dmul_rn(scale, a.tr.ts[j]);
          const double t_far = __dmul_rn(scale, a.tr.ts[min(j + kNear - 1u, end - 1)]);
          const size_t o = (size_t)p * a.out_stride + (j - a.first);
          cd.route_log[j] = (uint8_t)istar;
          if (opaque(a.route_out != nullptr)) a.route_out[o] = (uint8_t)istar;
          if (opaque(a.hit_out != nullptr)) a.hit_out[o] = (uint16_t)(rq >> 8);
          if (opaque(a.ttft_out != nullptr)) a.ttft_out[o] = __dsub_rn(tm.x, t);
          if (opaque(a.e2e_out != nullptr)) a.e2e_out[o] = __dsub_rn(tm.y, t);
          const double f = tm.y;
          auto record = [&](uint32_t next) {           // (the fourth word is the state's list of late completions)
            *reinterpret_cast<uint2*>(cd.exp_rec + j) = make_uint2(next, what.x);
            cd.exp_rec[j].z = istar;
          };
          if (f > t_far) {
            const uint32_t lo = max(j + 1u, min(j + kNear, end));      // (later than every near request)
            if (lo < N && t_last >= f) {
              uint32_t g = lo;
              if (opaque(use_grid)) {
                const double bf = __dmul_rn(f, to_bucket);
                uint32_t b = 0;
                if (bf >= 2.0) b = (bf >= (double)a.tr.grid_n ? a.tr.grid_n : (uint32_t)bf) - 1u;
                g = max(lo, __ldg(a.tr.grid + b));
              }
              // a few requests on from the grid's lower bound, four at a time; then bisection
              bool found = false;
              #pragma unroll 1
              for (uint32_t step = 0; step < 4 && !found; ++step) {
                double v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = __dmul_rn(scale, __ldg(a.tr.ts + min(g + u, N - 1)));
                uint32_t adv = 0;
#pragma unroll
                for (int u = 3; u >= 0; --u) if (v[u] >= f) { found = true; adv = u; }
                g += found ? adv : 4u;
              }
              x = found ? min(g, N - 1) : first_arrival_at_or_after(a.tr.ts, scale, f, min(g, N - 1), N - 1);
              old = atomicExch(cd.exp_head + x, j);
              record(old);
            } else if (opaque(cd.finish_log != nullptr)) {
              // completes after the last known arrival: listed in the state (read by the next launch)
              cd.finish_log[j] = f;
              reinterpret_cast<uint32_t*>(cd.exp_rec)[4 * (size_t)atomicAdd(&cd.hdr->overflow, 1u) + 3] = j;
              record(kNone);
            }
          }
        }
        __threadfence_block();                         // lists and route log are visible with `filed`
        __syncwarp();
        filed += n;
        if (lane == 0) sh.c.filed = filed;
        progress = true;
      }
    }
    PROF_LAP(1);
    if (progress) idle = 0;
    else {
      if (__any_sync(kFull, sh.c.abort_flag != 0)) break;
      // (whom it waits for is at work or in a wait of its own; 2^31 rounds are longer than any walk)
      if (++idle >> 31) break;
      __nanosleep(kIdleNs<kBuild>);
    }
  }
  PROF_END(48);
}

// Asks the replica's next requests (one per lane, `n` of them: number, first touch, touches) for the atom that
// this lane's touch, the my_k-th of request my_q, holds (kNone: nothing to ask).  True if one has it at the same index.
//   Usually a few lanes ask and twenty or thirty requests are asked, so the requests go by lane and the askers one
// after the other (kAsk of them with their loads in flight together): one memory latency per asker.  (The askers by lane
// and the requests one after the other, four at a time: shared prompts, 8 replicas, 64 candidates 0.81 us per request,
// with this 0.78.  Inlined, one asker is in flight: the code of four inside the scout's loop costs four candidates an
// SM 5 %, two 1 to 3 % and with 64 replicas 7 to 9 % (1.79 -> 1.95 us).  With one candidate an SM and shared prompts four
// gain 1 % (8 replicas, 16 candidates 0.738 -> 0.729), so the build for few candidates has four.  With more than 32
// replicas it is called, with four: 1, 2, 4 and 8 take 2.02, 1.98, 1.97 and 2.05 us.)
template <uint32_t kAsk>
__device__ __forceinline__ bool touched_again(const Touch* touch, uint32_t atom, uint32_t my_q, uint32_t my_k, uint32_t rq, uint32_t off,
                                              uint32_t m, uint32_t n) {
  const uint32_t lane = threadIdx.x & 31u;
  unsigned open = __ballot_sync(kFull, atom != kNone);
  bool again = false;
  #pragma unroll 1
  while (open) {
    uint32_t got[kAsk], want[kAsk], src[kAsk];
#pragma unroll
    for (uint32_t u = 0; u < kAsk; ++u) {
      src[u] = open ? (uint32_t)__ffs((int)open) - 1u : 32u;
      open &= open - 1u;
      const uint32_t from = src[u] & 31u, q = __shfl_sync(kFull, my_q, from), k = __shfl_sync(kFull, my_k, from);
      want[u] = __shfl_sync(kFull, atom, from);
      got[u] = src[u] < 32u && lane < n && rq > q && k < m ? __ldg(&touch[off + k].atom) : kNone;
    }
#pragma unroll
    for (uint32_t u = 0; u < kAsk; ++u) {
      const bool has = __any_sync(kFull, got[u] == want[u] && got[u] != kNone);
      again = again || (lane == src[u] && has);
    }
  }
  return again;
}

// With more than 32 replicas it is called, not inlined: where prompts are not shared it is not reached, and inside
// the scout's loop its code alone cost 64 replicas with 400 candidates 3 % and a small cache with 444 candidates 5 %
// (1.81 -> 1.66 and 2.35 -> 2.05 us per request out of line; 1.76 and 2.24 without it, where shared prompts
// take 5.2 instead of 3.9).  Up to 32 replicas the call costs shared prompts 7 % at four candidates an SM.
__device__ __noinline__ bool touched_again_called(const Touch* touch, uint32_t atom, uint32_t my_q, uint32_t my_k, uint32_t rq, uint32_t off,
                                                  uint32_t m, uint32_t n) {
  return touched_again<4>(touch, atom, my_q, my_k, rq, off, m, n);
}

// ------------------------------------------------------------------------------ scout warp
// Lists coming victims: for the active replica with the emptiest ring it walks the recency order
// (the requests of the route log with that replica, deepest touch first) from where it stopped, up to
// 32 touches per round, one per lane, and appends those that are still the latest touch of their
// atom.  The route warp checks again what occurs between the listing and the eviction.
template <typename MaskT, bool kExt, uint32_t kBuild>
__device__ __forceinline__ void scout_warp(const ReplayArgs& a, Shared<MaskT, kExt>& sh, const Cand<MaskT>& cd, uint4* more,
                                           uint32_t lane) {
  const uint32_t R = a.m.R, end = a.first + a.count;
  const Touch* touch = a.tr.touch;
  const bool ahead = !a.scout_off && a.count > kFew;
  uint32_t dry0 = a.first - kNews, dry1 = dry0;        // requests known when the replica's order ran out
  uint32_t idle = 0;
  const uint32_t sb = smem_addr(&sh), ring = smem_addr(sh.route_ring);
  PROF_BEGIN();
  #pragma unroll 1
  while (true) {
    // requests known: those whose commits are made (a touch that a later request touches again is
    // still a victim of the commits in between).  Routes the file warp has not logged are in the ring.
    const uint32_t filed = __shfl_sync(kFull, sh.c.filed, 0);
    const uint32_t seen = __shfl_sync(kFull, sh.c.decided, 0);
    if (__any_sync(kFull, sh.c.abort_flag != 0 || (int32_t)(seen - end) >= 0)) break;
    const uint32_t want = __shfl_sync(kFull, sh.c.want, 0);
    smem_order();
    uint32_t best = kNone;
#pragma unroll
    for (int half = 0; half < (sizeof(MaskT) == 8 ? 2 : 1); ++half) {
      const uint32_t i = lane + 32u * half;
      if (i < R && (want == i + 1u || (ahead && (uint64_t)*(volatile uint32_t*)&sh.occ[i] + kMargin >= a.m.C))) {
        const uint32_t fill = sh.ring_tail[i] - *(volatile uint32_t*)&sh.take[i].x;
        const uint32_t news = seen - (half ? dry1 : dry0);
        if (fill * 4u <= a.ring_cap * kRefill && (news >= kNews || (news && want == i + 1u))) best = min(best, (want == i + 1u ? 0u : 1u << 16) | (fill << 8) | i);
      }
    }
    best = __reduce_min_sync(kFull, best);
    if (best == kNone) {
      // Only rounds in which the route warp waits for a victim count: a launch may go on for long before a cache
      // fills, and it ends this warp when it ends.  (The route warp's own limit reports the failure.)
      idle += want != 0 ? 1u : 0u;
      if (idle > a.poll_limit) break;
      __nanosleep(kIdleNs<kBuild>);
      continue;
    }
    idle = 0;
    const uint32_t i = best & 255u;                    // (what is waited for, else the emptiest list)
    uint32_t tail = sh.ring_tail[i];
    uint32_t room = a.ring_cap - 1u - (best >> 8 & 255u);   // (the last victim taken stays readable)
    if (room > 32u) room = 32u;
    uint32_t pos = sh.c.scan_pos[i], vq = sh.c.scan_req[i];
    int32_t vk = sh.c.scan_k[i];
    // ---- requests of the replica in the next stretch of the log, in order (the first kMatches)
    uint32_t n_match = 0, off = 0, m = 0, rq = 0;
    uint32_t stop = pos;                               // requests < stop are looked at in this pass
    const uint32_t budget = room - min(room, (uint32_t)(vk + 1));
    if (budget > 0 && pos < seen) {
      // (a word of four routes per lane and load; the loads of a stretch are in flight together)
      const uint32_t mis = (uint32_t)(uintptr_t)cd.route_log & 3u, log_end = min(filed, seen);
      const uint32_t lo = pos + mis, hi = max(lo, log_end + mis), word0 = lo & ~3u;
      auto routes = [&](uint32_t u) -> uint32_t {
        const uint32_t x = word0 + 128u * u + 4u * lane;
        return x < hi ? __ldcg(reinterpret_cast<const uint32_t*>(cd.route_log - mis + x)) : 0u;
      };
      uint32_t rt = routes(0), rt1 = routes(1), rt2 = routes(2), rt3 = routes(3);
      #pragma unroll 1
      for (uint32_t u = 0; u < 4u && n_match < budget && stop < log_end; ++u) {
        const uint32_t x = word0 + 128u * u + 4u * lane;
        uint32_t hit = x < hi ? __vcmpeq4(rt, i * 0x01010101u) : 0u;   // 0xFF in the bytes that are equal
        if (x < lo) hit &= kFull << (8u * (lo - x));
        if (x < hi && hi - x < 4u) hit &= kFull >> (8u * (4u - (hi - x)));
        const uint32_t cnt = (uint32_t)__popc(hit) / 8u;
        uint32_t at = cnt;
        #pragma unroll 1
        for (uint32_t d = 1; d < 32u; d <<= 1) {
          const uint32_t up = __shfl_up_sync(kFull, at, d);
          if (lane >= d) at += up;
        }
        const uint32_t total = __shfl_sync(kFull, at, 31);
        at += n_match - cnt;
        #pragma unroll 1
        while (hit && at < kMatches) {
          const uint32_t b = ((uint32_t)__ffs((int)hit) - 1u) / 8u;
          sh.scan_list[at++] = x + b - mis;
          hit &= ~(0xFFu << (8u * b));
        }
        n_match += total;
        stop = min(word0 + 128u * (u + 1u) - mis, log_end);
        rt = rt1; rt1 = rt2; rt2 = rt3;
      }
      #pragma unroll 1
      while (stop >= log_end && stop < seen && n_match < budget) {
        const uint32_t r = stop + lane, v = lds32(ring + (r % kRing) * 4u) & 0xFFu;
        // (none of the entries has been written again: else all these are in the log by now)
        if (__shfl_sync(kFull, sh.c.routed, 0) - stop >= kRing) break;
        const unsigned bal = __ballot_sync(kFull, r < seen && v == i);
        const uint32_t at = n_match + (uint32_t)__popc(bal & ((1u << lane) - 1u));
        if ((bal >> lane & 1u) && at < kMatches) sh.scan_list[at] = r;
        n_match += (uint32_t)__popc(bal);
        stop = min(stop + 32u, seen);
      }
      __syncwarp();
      if (n_match > kMatches) { n_match = kMatches; stop = sh.scan_list[kMatches - 1] + 1u; }
      if (lane < n_match) {
        rq = sh.scan_list[lane];
        off = a.tr.req[rq].off;
        m = a.tr.req[rq].m;
      }
    }
    PROF_LAP(0);
    // ---- up to `room` touches, one per lane, in recency order
    uint32_t my_q = kNone, my_k = 0, my_off = 0;
    uint32_t used = 0, mi = 0, v_off = vk >= 0 ? a.tr.req[vq].off : 0u;
    #pragma unroll 1
    while (used < room) {
      if (vk < 0) {
        if (mi == n_match) break;
        vq = __shfl_sync(kFull, rq, mi);
        v_off = __shfl_sync(kFull, off, mi);
        vk = (int32_t)__shfl_sync(kFull, m, mi) - 1;
        ++mi;
        continue;
      }
      const uint32_t take = min((uint32_t)vk + 1u, room - used);
      if (lane - used < take) { my_q = vq; my_k = (uint32_t)vk - (lane - used); my_off = v_off; }
      used += take;
      vk -= (int32_t)take;
    }
    // requests of the stretch that were not reached are looked at again next time
    pos = mi < n_match ? __shfl_sync(kFull, rq, mi & 31u) : stop;
    uint32_t len = 0;
    Touch t = {0u, 0u, kNone, kNone};
    bool live = my_q != kNone;
    if (live) {
      t = touch[my_off + my_k];
      len = t.len_pos & 0xFFFFu;
      if (sh.scan_plen[i] && my_q == sh.cur_req[i] && (int32_t)my_k == sh.cur_k[i]) len = sh.scan_plen[i];   // (partly evicted before)
    }
    // later occurrences known to the log: the touch is none of the latest if one of them is this replica's
    bool open = live && t.next != kNone && t.next_req < seen;
    auto step = [&]() {
      const uint2 nx = __ldg(reinterpret_cast<const uint2*>(&touch[t.next].next));
      const uint32_t r = t.next_req;
      bool logged = r < filed;
      uint32_t rt = 0;
      if (!logged) {
        rt = lds32(ring + (r % kRing) * 4u) & 0xFFu;
        logged = sh.c.routed - r >= kRing;
      }
      if (logged) rt = (uint32_t)__ldcg(cd.route_log + r);
      if (rt == i) live = open = false;
      else { t.next = nx.x; t.next_req = nx.y; open = t.next != kNone && t.next_req < seen; }
    };
    // One occurrence after the other.  An atom that occurs in request after request (a prompt many share) would
    // take about R steps.  The replica's next requests, found above, usually have it at the same index: they are
    // asked after the first kHops.  (Shared prompts: 8 replicas, 64 candidates 1.09 us per request with the walk
    // alone, 0.80 with this; 32 replicas 3.85 and 2.13; 56 replicas, 241 candidates 5.2 and 3.9.)
    //   If the route warp waits meanwhile, for what is found already or for another replica, the touches from the
    // first undecided one on are looked at again next time.  (Found already: the first lane that is live is decided.)
    //   (One copy of the step for both phases: with two, four candidates an SM take 1.41 instead of 1.33 us.)
    #pragma unroll 1
    for (uint32_t hop = 0;; ++hop) {
      unsigned rest = __ballot_sync(kFull, open);
      if (!rest) break;
      if (hop >= kHops) {
        if (hop == kHops && n_match) {
          const uint32_t asked = open ? t.atom : kNone;
          if (sizeof(MaskT) == 8 ? touched_again_called(touch, asked, my_q, my_k, rq, off, m, n_match)
                                : touched_again<kBuild == kSparse ? 4 : 1>(touch, asked, my_q, my_k, rq, off, m, n_match)) live = open = false;
          rest = __ballot_sync(kFull, open);
          if (!rest) break;
        }
        const uint32_t w = __shfl_sync(kFull, sh.c.want, 0);
        const unsigned found = __ballot_sync(kFull, live);
        if (w != 0 && (w != i + 1u || !(found & (0u - found) & rest))) {
          const uint32_t cut = (uint32_t)__ffs((int)rest) - 1u;
          live = live && lane < cut;
          vq = __shfl_sync(kFull, my_q, cut);
          vk = (int32_t)__shfl_sync(kFull, my_k, cut);
          pos = vq + 1u;
          break;
        }
        sts32(sb + (uint32_t)offsetof(Control, walk), hop);
      }
      if (open) step();
    }
    const unsigned lv = __ballot_sync(kFull, live);
    uint32_t cum = live ? len : 0u;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t up = __shfl_up_sync(kFull, cum, d);
      if (lane >= (uint32_t)d) cum += up;
    }
    cum += sh.scan_cum[i];
    if (live) {
      const uint32_t slot = i * a.ring_cap + ((tail + (uint32_t)__popc(lv & ((1u << lane) - 1u))) & (a.ring_cap - 1u));
      sh.victims[slot] = make_uint2(t.atom, cum);
      sh.victim_next[slot] = t.next == kNone ? kNone : t.next_req;
      more[slot] = make_uint4(t.next, my_q, my_k, my_off + my_k);
    }
    cum = __shfl_sync(kFull, cum, 31);
    // every lane's entries are stored before lane 0 publishes the new tail
    if (sizeof(MaskT) == 8) __threadfence_block();
    __syncwarp();
    smem_order();
    if (lane == 0) {
      sh.c.scan_pos[i] = pos; sh.c.scan_req[i] = vq; sh.c.scan_k[i] = vk; sh.scan_cum[i] = cum;
      sh.ring_tail[i] = tail + (uint32_t)__popc(lv);
    }
    if (used == 0 && pos == seen) {                    // the order ran out
      if ((i & 31u) == lane) { if (i < 32) dry0 = seen; else dry1 = seen; }
    }
    __syncwarp();
    PROF_LAP(1);
  }
  PROF_END(64);
}

enum Role : uint32_t { kRoleRoute, kRoleStage, kRoleTime, kRoleExpiry, kRoleScout, kRoleFile, kRoles };
constexpr uint32_t kReplayThreads = 32 * kRoles;
// Candidates an SM holds, which caps the registers: four (80 registers a thread), three with more than 32 replicas (96).
// A launch does not see what other streams run on the GPU, so a build that large launches take leaves room for as
// many: with two an SM (98 registers, no spills; 1 to 4 % faster alone) three populations of 148 on three streams took
// 1.91 us per request instead of 1.41 (16 replicas), 1.69 instead of 1.10 (shared prompts) and 2.40 instead of 1.68 (32
// replicas), and two of 256 1.96 instead of 1.62.  The build for few candidates has room for two
// (three with more than 32 replicas, where two gain nothing).  With 96 registers three would fit, 1 % slower, but only if
// their warps begin on alternate schedulers, as those of one launch do; three streams of 148 took two turns all the same.
template <typename MaskT, uint32_t kBuild> constexpr int kReplayMinCtas = sizeof(MaskT) == 8 ? 3 : kBuild == kSparse ? 2 : 4;
// The lists of the launch before (the end of the kernel says why).  (Out of line: inlined it costs the
// loops registers.)
template <typename MaskT, bool kExt>
__device__ __noinline__ void lists_in(const ReplayArgs& a, Shared<MaskT, kExt>& sh, const uint4* listed, uint4* more) {
  #pragma unroll 1
  for (uint32_t x = threadIdx.x; x < a.m.R * a.ring_cap; x += blockDim.x) {
    const uint32_t i = x / a.ring_cap, e = x % a.ring_cap;
    if (e < sh.ring_tail[i]) {
      const uint4* l = listed + (size_t)i * (2u * a.ring_cap + 1u) + 1u + 2u * e;
      uint4 v = l[0], y = l[1];
      if (y.x == kNone && a.tr.growing) {              // (it may have grown: any occurrence after the listed one will do)
        const Touch t = a.tr.touch[y.w];
        y.x = t.next; v.z = t.next_req;
      }
      sh.victims[x] = make_uint2(v.x, v.y);
      sh.victim_next[x] = v.z;
      more[x] = y;
    }
  }
}

template <typename MaskT, bool kExt, uint32_t kBuild>
__global__ void __launch_bounds__(kReplayThreads, (kReplayMinCtas<MaskT, kBuild>)) replay_kernel(const __grid_constant__ ReplayArgs a) {
  const uint32_t p = blockIdx.x;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t w_id = __shfl_sync(kFull, threadIdx.x >> 5, 0);   // (known to be the same for all lanes)
  // Role of the warp.  The hardware gives an SM's four schedulers a block's warps in turn, so the third and fourth of six
  // have a scheduler alone.  In a launch of at most one candidate an SM the order is scout, stage, route, expiry, time,
  // file: with the route warp alone 148 candidates take 0.844 us per request instead of 0.863, 32 replicas 1.07 instead
  // of 1.09, 64 replicas 1.40 instead of 1.43.  Two an SM put three warps on every scheduler, and the order of Role is
  // the faster one (256 candidates 0.94, in the other order 0.98).  (The form matters more than its few instructions: as
  // a table or a select, which move the roles' code, 256 candidates took 0.97 and 0.98 in the order of Role too.)
  uint32_t warp = w_id;
  if (kBuild != kDense && (kBuild == kSparse || a.alone) && !(w_id & 1u)) {
    warp += 4u;
    if (warp >= kRoles) warp -= kRoles;
  }
  const uint32_t R = a.m.R, K = a.m.K, GR = a.m.G * a.m.R, RS = a.m.R * a.m.S;
  const uint32_t N = a.tr.n_req;

  extern __shared__ __align__(128) unsigned char smem_raw[];
  Shared<MaskT, kExt>& sh = *reinterpret_cast<Shared<MaskT, kExt>*>(smem_raw);
  Dyn dy;
  dy.rtt = reinterpret_cast<double*>(smem_raw + sizeof(sh) + (size_t)(kChunkRing / a.tr.chunk_req) * a.tr.chunk_cap * sizeof(Touch));
  dy.wrtt = dy.rtt + GR;
  dy.free_at = dy.wrtt + GR;

  unsigned char* st = a.states + (size_t)p * a.lay.bytes;
  double* g_slot = reinterpret_cast<double*>(st + a.lay.slot_off);     // [R*S] slot free times
  if (!a.slots_in_smem) dy.free_at = g_slot;
  Cand<MaskT> cd;
  cd.hdr = reinterpret_cast<CandHeader*>(st);
  cd.rep = reinterpret_cast<RepState*>(st + a.lay.rep_off);
  cd.slot_kv = reinterpret_cast<unsigned long long*>(st + a.lay.slot_kv_off);
  cd.mask = reinterpret_cast<MaskT*>(a.masks + (size_t)p * a.mask_stride);
  cd.index = reinterpret_cast<MaskT*>(a.masks + (size_t)p * a.mask_stride + a.index_off);
  cd.finish_log = a.finish_log ? a.finish_log + (size_t)p * N : nullptr;
  cd.exp_head = a.exp_head + (size_t)p * N;
  cd.exp_rec = a.exp_rec + (size_t)p * N;
  cd.route_log = a.route_log + (size_t)p * a.route_log_stride;
  cd.params = a.params ? a.params + (size_t)p * K : a.inline_params;
  cd.scale = a.scales ? a.scales[p] : a.scale;

  const uint4* listed = reinterpret_cast<const uint4*>(st + a.lay.list_off);
  // (the first value of every table below: in flight together, a short launch is mostly such latencies)
  const uint32_t tid = threadIdx.x;
  const uint32_t processed = cd.hdr->processed;
  const double w_net = cd.params[0], rtt_0 = tid < GR ? a.tr.rtt[tid] : 0.0, par_0 = tid < K ? cd.params[tid] : 0.0,
               slot_0 = tid < RS && a.slots_in_smem ? g_slot[tid] : 0.0;
  RepState rep_0 = {};
  if (tid < R) rep_0 = cd.rep[tid];
  if (a.check_order && processed != a.first) {   // uniform over the CTA
    if (threadIdx.x == 0) {
      cd.hdr->status = -8;
      if (a.status_out) a.status_out[p] = -8;
    }
    return;
  }

  for (uint32_t i = tid; i < GR; i += blockDim.x) {
    const double v = i == tid ? rtt_0 : a.tr.rtt[i];
    dy.rtt[i] = v;
    dy.wrtt[i] = __dmul_rn(w_net, v);                    // first product of the score
  }
  if (tid < K) sh.w[tid] = par_0;                        // (K <= 67)
  if (tid < R) {
    const uint32_t i = tid;
    const RepState rs = rep_0;
    sh.cur_req[i] = rs.cur_req; sh.cur_k[i] = rs.cur_k;
    sh.take[i] = make_uint2(0u, 0u); sh.ring_tail[i] = 0; sh.scan_cum[i] = 0;
    sh.scan_plen[i] = rs.part != kNone ? rs.part_len : 0u;
    sh.part[i] = make_uint2(rs.part, rs.part_len); sh.occ[i] = rs.occ;
    sh.c.scan_pos[i] = rs.cur_req == kNone ? 0u : rs.cur_req + 1u;
    sh.c.scan_req[i] = rs.cur_req;
    sh.c.scan_k[i] = rs.cur_req == kNone ? -1 : rs.cur_k;
    if (a.check_order && rs.listed) {                    // the list of the launch before, and where its scout stood
      const uint4 g = listed[(size_t)i * (2u * a.ring_cap + 1u)];
      sh.ring_tail[i] = rs.listed;
      sh.c.scan_pos[i] = g.x; sh.c.scan_req[i] = g.y; sh.c.scan_k[i] = (int32_t)g.z; sh.scan_cum[i] = g.w;
    }
  }
  if (a.slots_in_smem)
    for (uint32_t x = threadIdx.x; x < RS; x += blockDim.x) dy.free_at[x] = x == threadIdx.x ? slot_0 : g_slot[x];
  for (uint32_t i = R + threadIdx.x; i < Shared<MaskT, kExt>::kR; i += blockDim.x) sh.part[i] = make_uint2(kNone, 0u);
  if (threadIdx.x < kRing) sh.near_head[threadIdx.x] = kNone;
  if (threadIdx.x < 6u) sh.c.marks[threadIdx.x] = 0u;
  if (threadIdx.x < kStages) {                               // (stages are read before it is known that they are ready)
    sh.tag[threadIdx.x] = 0u;
    sh.facts[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
    if (kExt) sh.epoch[kExt ? threadIdx.x : 0] = 0u;
  }
  if (threadIdx.x == 0) {
    sh.c.routed = a.first; sh.c.timed = a.first; sh.c.filed = a.first; sh.c.listed = a.first; sh.c.exp_ready = a.first;
    sh.c.abort_flag = 0; sh.c.status = 0; sh.c.steps = 0; sh.c.walk = 0;
    sh.c.committed = a.first; sh.c.decided = a.first; sh.c.want = 0; sh.c.want_timed = a.first;
#pragma unroll
    for (uint32_t k = 0; k < kChunkRing / kChunkMin; ++k) mbar_init(sh.mbar + k);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (a.check_order) {
    __syncthreads();
    lists_in<MaskT, kExt>(a, sh, listed, sizeof(MaskT) == 8 ? reinterpret_cast<uint4*>(st + a.lay.more_off) : sh.victim_more);
  }
  if (cd.finish_log) {
    // The trace may have grown since the last batch: requests that were to complete after its old
    // end are filed under the first request, not yet replayed, that arrives at or after their finish
    // time; the rest stay listed.  (Their list is an array, in the fourth words of the completion
    // records: as a chain, one thread followed it in every launch, one memory latency per request in flight.)
    uint32_t* list = reinterpret_cast<uint32_t*>(cd.exp_rec) + 3;
    const uint32_t n = cd.hdr->overflow;
    uint32_t& kept = sh.scan_list[0];
    if (threadIdx.x == 0) kept = 0;
    const double t_last = __dmul_rn(cd.scale, a.tr.ts[N - 1]);
    #pragma unroll 1
    for (uint32_t base = 0; base < n; base += blockDim.x) {
      const bool on = base + threadIdx.x < n;
      bool keep = false;
      uint32_t e = 0;
      if (on) {
        e = list[4 * (size_t)(base + threadIdx.x)];
        const double f = cd.finish_log[e];
        keep = !(e + 1 < N && t_last >= f);
        if (!keep) {
          const uint32_t x = first_arrival_at_or_after(a.tr.ts, cd.scale, f, max(e + 1u, a.first), N - 1);
          cd.exp_rec[e].x = atomicExch(cd.exp_head + x, e);
        }
      }
      __syncthreads();                                 // (entries move down only, to places that are read)
      if (keep) list[4 * (size_t)atomicAdd(&kept, 1u)] = e;
    }
    __syncthreads();
    if (threadIdx.x == 0 && n > 0) cd.hdr->overflow = kept;
  }
  __syncthreads();

  const uint32_t sb = smem_addr(smem_raw);
  const StageArgs<MaskT> sa = {cd.mask, cd.index, cd.scale};
  uint4* more = sizeof(MaskT) == 8 ? reinterpret_cast<uint4*>(st + a.lay.more_off) : sh.victim_more;
  if (warp == kRoleRoute) route_warp<MaskT, kExt, kBuild>(a, sh, sb, dy, sa, cd.route_log, more, cd.rep, p, lane);
  else if (warp == kRoleStage) stage_warp<MaskT, kExt>(a, sh, sb, sa, lane);
  else if (warp == kRoleTime) time_warp<MaskT, kExt>(a, sh, sb, dy, cd.slot_kv, cd.scale, lane);
  else if (warp == kRoleExpiry) expiry_warp<MaskT, kExt>(a, sh, sb, cd.exp_rec, cd.scale, lane);
  else if (warp == kRoleFile) file_warp<MaskT, kExt, kBuild>(a, sh, cd, p, lane);
  else scout_warp<MaskT, kExt, kBuild>(a, sh, cd, more, lane);
  __syncthreads();

  // (pointers computed again: registers less in the loops)
  unsigned char* st_end = a.states + (size_t)opaque(blockIdx.x) * a.lay.bytes;
  RepState* rep_end = reinterpret_cast<RepState*>(st_end + a.lay.rep_off);
  uint4* lists = reinterpret_cast<uint4*>(st_end + a.lay.list_off);
  const uint4* more_end = sizeof(MaskT) == 8 ? reinterpret_cast<const uint4*>(st_end + a.lay.more_off) : sh.victim_more;
  // ---- write the small state back; the eviction cursor stands at the next listed touch, or behind
  //      the last one taken
  for (uint32_t i = threadIdx.x; i < R; i += blockDim.x) {
    const uint32_t head = sh.take[i].x, tail = sh.ring_tail[i];
    RepState s = {(long long)sh.rows[(a.first + a.count - 1u) % Shared<MaskT, kExt>::kRows][i], sh.occ[i], sh.cur_req[i], sh.cur_k[i], sh.part[i].x, sh.part[i].y,
                  a.check_order ? tail - head : 0u};
    const uint32_t b = i * a.ring_cap, cap_mask = a.ring_cap - 1u;
    if (tail != head) {
      const uint4 x = more_end[b + (head & cap_mask)];
      s.cur_req = x.y;
      s.cur_k = (int32_t)x.z;
    } else if (head != 0) {
      const uint32_t e = b + ((head - 1u) & cap_mask);
      s.cur_req = more_end[e].y;
      s.cur_k = (int32_t)more_end[e].z - 1;
    }
    rep_end[i] = s;
    if (s.listed) lists[(size_t)i * (2u * a.ring_cap + 1u)] = make_uint4(sh.c.scan_pos[i], sh.c.scan_req[i], (uint32_t)sh.c.scan_k[i], sh.scan_cum[i] - sh.take[i].y);
  }
  // A state that goes on keeps the lists: short launches (a tuner's hop, a proxy's request) would else
  // begin with a scout round per replica, most of it looking again at touches that are superseded.
  // (Hops of 32 requests, two tuners: 13.4 -> 6.8 ms for 190 launches.)
  if (a.check_order) {
    #pragma unroll 1
    for (uint32_t x = threadIdx.x; x < R * a.ring_cap; x += blockDim.x) {
      const uint32_t i = x / a.ring_cap, e = x % a.ring_cap;
      const uint2 tk = sh.take[i];
      if (e < sh.ring_tail[i] - tk.x) {
        const uint32_t slot = i * a.ring_cap + ((tk.x + e) & (a.ring_cap - 1u));
        const uint2 v = sh.victims[slot];
        uint4* l = lists + (size_t)i * (2u * a.ring_cap + 1u) + 1u + 2u * e;
        l[0] = make_uint4(v.x, v.y - tk.y, sh.victim_next[slot], 0u);
        l[1] = more_end[slot];
      }
    }
  }
  if (a.slots_in_smem)
    for (uint32_t x = threadIdx.x; x < RS; x += blockDim.x) reinterpret_cast<double*>(st_end + a.lay.slot_off)[x] = dy.free_at[x];
  if (threadIdx.x == 0) {
    const int32_t status = sh.c.status;
    reinterpret_cast<CandHeader*>(st_end)->processed = a.first + a.count;
    if (status != 0) reinterpret_cast<CandHeader*>(st_end)->status = status;
    if (a.status_out && (status != 0 || !a.check_order)) a.status_out[opaque(blockIdx.x)] = status;
  }
}

// Slots live in shared memory up to this size, else in global memory.
constexpr size_t kSlotBytes = 40 * 1024;

template <typename MaskT, bool kExt>
size_t replay_smem_bytes(ReplayArgs& a) {
  a.slots_in_smem = (size_t)a.m.R * a.m.S * 8 <= kSlotBytes ? 1u : 0u;
  a.ring_cap = listed_victims(a.m.R);
  return shared_bytes<MaskT, kExt>(a.m, a.tr.chunk_req, a.tr.chunk_cap, a.slots_in_smem != 0);
}

template <typename MaskT, bool kExt, uint32_t kBuild>
cudaError_t prepare_replay(size_t smem) {
  cudaError_t e = cudaFuncSetAttribute(replay_kernel<MaskT, kExt, kBuild>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // several candidates share an SM: the per-CTA footprint, not the default carve-out, decides
  return cudaFuncSetAttribute(replay_kernel<MaskT, kExt, kBuild>, cudaFuncAttributePreferredSharedMemoryCarveout,
                              (int)cudaSharedmemCarveoutMaxShared);
}

template <typename MaskT, bool kExt, uint32_t kBuild>
cudaError_t launch_replay_t(ReplayArgs a, uint32_t n_cand, cudaStream_t st) {
  const size_t smem = replay_smem_bytes<MaskT, kExt>(a);
  cudaError_t e = prepare_replay<MaskT, kExt, kBuild>(smem);
  if (e != cudaSuccess) return e;
  replay_kernel<MaskT, kExt, kBuild><<<n_cand, kReplayThreads, smem, st>>>(a);
  return cudaGetLastError();
}

// The build of a launch.  Up to a quarter of the SMs: the one for few candidates, 1 to 4 % faster than the next (16
// candidates, long contexts 0.79 and 0.82 us per request, shared prompts 0.74 and 0.75, 32 replicas 1.02 and 1.05).  A GPU
// takes launches of eight streams at once unless it is told otherwise: even then there are at most two of these an SM, and
// two fit (eight populations of 37 at once: 1.09 us per request).  Up to half of the SMs, six populations of 74
// would take 1.85 instead of 1.55.  Up to two candidates an SM: the build with the limited
// eviction (see evict_slow).  More: the dense one.  Around the line, 296 candidates 1.05 and 1.05, 32 replicas 1.23 and 1.24,
// 64 replicas 1.77 and 1.82; 444 candidates 1.37 and 1.35, 32 replicas 1.61 and 1.59, 64 replicas 2.33 and 2.35.
// Where shared memory lets only two an SM fit, the line could lie elsewhere, but does not matter: 600 candidates on a
// grown trace 4.86 and 4.87 (shared prompts), 15.9 and 16.4 (long contexts), with 38 KB of slots 2.83 and 2.84, 32
// replicas 3.35 and 3.27, 64 replicas 4.29 and 4.19.
template <typename MaskT, bool kExt>
cudaError_t launch_replay_n(ReplayArgs a, uint32_t n_cand, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  a.alone = n_cand <= (uint32_t)sms ? 1u : 0u;
  const uint32_t build = a.build ? a.build : n_cand <= (uint32_t)sms / 4u ? kSparse : n_cand <= 2u * (uint32_t)sms ? kPaired : kDense;
  return build == kSparse ? launch_replay_t<MaskT, kExt, kSparse>(a, n_cand, st)
         : build == kPaired ? launch_replay_t<MaskT, kExt, kPaired>(a, n_cand, st)
                            : launch_replay_t<MaskT, kExt, kDense>(a, n_cand, st);
}

template <typename MaskT, uint32_t kBuild>
int replay_occupancy_t(ReplayArgs& a, size_t* smem_out) {
  *smem_out = replay_smem_bytes<MaskT, false>(a);
  int n = 0;
  if (prepare_replay<MaskT, false, kBuild>(*smem_out) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, replay_kernel<MaskT, false, kBuild>, (int)kReplayThreads,
                                                    *smem_out) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  return n;
}
template <typename MaskT>
int replay_occupancy_n(ReplayArgs& a, size_t* smem_out) {
  return a.build == kSparse ? replay_occupancy_t<MaskT, kSparse>(a, smem_out)
         : a.build == kPaired ? replay_occupancy_t<MaskT, kPaired>(a, smem_out) : replay_occupancy_t<MaskT, kDense>(a, smem_out);
}

}  // namespace

int replay_occupancy(const Model& m, const TraceView& tr, uint32_t build, uint64_t* smem_bytes) {
  ReplayArgs a = {};
  a.m = m;
  a.tr = tr;
  a.build = build;
  size_t smem = 0;
  const int n = m.R <= 32 ? replay_occupancy_n<uint32_t>(a, &smem) : replay_occupancy_n<unsigned long long>(a, &smem);
  if (smem_bytes) *smem_bytes = smem;
  return n;
}

cudaError_t load_replay() {
  cudaFuncAttributes fa;
  cudaError_t e = cudaSuccess;
  const auto load = [&](auto kernel) { if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel); };
  load(replay_kernel<uint32_t, false, kSparse>); load(replay_kernel<uint32_t, true, kSparse>);
  load(replay_kernel<uint32_t, false, kPaired>); load(replay_kernel<uint32_t, true, kPaired>);
  load(replay_kernel<uint32_t, false, kDense>); load(replay_kernel<uint32_t, true, kDense>);
  load(replay_kernel<unsigned long long, false, kSparse>); load(replay_kernel<unsigned long long, true, kSparse>);
  load(replay_kernel<unsigned long long, false, kPaired>); load(replay_kernel<unsigned long long, true, kPaired>);
  load(replay_kernel<unsigned long long, false, kDense>); load(replay_kernel<unsigned long long, true, kDense>);
  return e;
}

uint32_t mask_bytes_for(uint32_t n_replicas) { return n_replicas <= 32 ? 4u : 8u; }

cudaError_t launch_replay(const ReplayArgs& a, uint32_t n_cand, cudaStream_t st) {
  // the plain cost-model replay carries none of the optional model parts
  const bool ext = a.queue_in_requests || a.forced_route || a.rep_prefill_ms || a.rep_tpot_ms ||
                   a.decode_slowdown > 0.0 || a.kv_budget > 0 || a.rtt_ewma || a.proxy_index || a.stats;
  if (a.m.R <= 32) return ext ? launch_replay_n<uint32_t, true>(a, n_cand, st) : launch_replay_n<uint32_t, false>(a, n_cand, st);
  return ext ? launch_replay_n<unsigned long long, true>(a, n_cand, st)
             : launch_replay_n<unsigned long long, false>(a, n_cand, st);
}

#ifdef GORGO_PROF
cudaError_t prof_read(unsigned long long* out112, bool reset) {
  cudaError_t e = cudaMemcpyFromSymbol(out112, g_prof, sizeof(g_prof));
  if (e != cudaSuccess || !reset) return e;
  unsigned long long zero[112] = {};
  return cudaMemcpyToSymbol(g_prof, zero, sizeof(zero));
}
#endif

}  // namespace gorgo
