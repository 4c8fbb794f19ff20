// dpm_queue.cu -- persistent transport kernel with device-wide particle queues.
//
// The paper runs one history per thread, so the 32 threads of a warp follow
// statistically independent paths and execute mostly one at a time (its
// Sec. 4 diagnosis of the C1060 speed-up).  Here every warp holds particles of
// ONE type (photons or electrons/positrons) in its lanes, steps them together,
// and refills lanes that have finished from a stash of its own in shared
// memory.  The stash is filled 32 particles at a time: with new histories, which
// all lanes make together, or from per-type particle queues.  Secondaries of
// the warp's type go to its stash, the others by way of a buffer to the queues.
// The physics of a particle is the same code as in the per-history kernel and
// its random numbers are keyed by its identity, so both kernels produce the
// same integer tally.
//
// Queues: for each type, one ring per CTA ("shard") in global memory, with a
// sequence number per slot (a producer publishes position p by writing p+1,
// the consumer frees the slot for position p+capacity), so that producers and
// consumers on different SMs never read a half-written record.  A warp pushes
// to its CTA's shard and pops from it first, stealing from other shards when it
// is empty.  The grid alternates between a source phase and a secondary
// phase (see the scheduler below) so that all SMs run one particle type's
// code at a time.  The run ends when every started warp is idle (its stash and
// buffer empty), every queue is empty and the source is exhausted.  Every wait
// is bounded by a time limit read from %globaltimer; on expiry the kernel
// records an error and returns.
//
// What bounds the kernel: instruction issue (73 to 78 % of the slots on long
// launches, at 21 of 32 lanes), then instruction fetch and the latency of table
// lookups, not memory bandwidth.  Four things follow.
// - Code size.  The kernel took 276 KB when every secondary was queued where it
//   is made, every refill was spelled out and the photon interaction stood
//   after each of two flights; "no instruction" was the leading stall (4.7 of
//   17 cycles per issue on 6 MV, 5.0 on 20 MeV electrons).  With one copy of
//   each it takes 81 KB (1.2 and 1.7 cycles).
// - Full warps.  Lanes that wait for a refill waste issue slots, and a refill
//   from the device-wide queues costs several L2 round trips.  Taking from the
//   stash costs some 60 instructions, so it happens at 2 idle lanes.  What few
//   lanes of a warp do at a time waits for company: see kHardEvery.
// - Few instructions per step: see Num<float> and electron_step in
//   dpm_device.cuh.
// - Nothing at the ends of a launch that grows with the grid: see any_work and
//   queue_fresh.
// Transport times, before and with all four: 10^7 6 MV histories 14.6 and
// 8.3 ms, 5x10^6 20 MeV electrons on the 128^3 blobs 52.4 and 25.8 ms, 2x10^4
// on the slabs 1.58 and 0.59 ms, 2000 photons of 15 MeV 0.63 and 0.34 ms.
#include <cuda_runtime.h>

#include "dpm_device.cuh"
#include "dpm_queue.h"

namespace dpm {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kQBlock = 128;
#ifndef DPM_STEAL_PROBES
#define DPM_STEAL_PROBES 8
#endif
// The whole grid alternates between a source phase (histories start, warps
// track particles of the beam's type) and a secondary phase (no history
// starts, warps track the queued particles of the other type).  The
// secondary phase starts when the other type's particles queued in all
// shards exceed K * (capacity >> HIGH) and ends when they fall below
// K * (capacity >> LOW); photon beams queue electrons, electron beams queue
// bremsstrahlung and annihilation photons.  A CTA whose own shards hold more
// than capacity >> GUARD particles starts no history.
// Every switch drains the warps of the other type, whose last particles step in
// nearly empty warps, so a phase goes on until there are 32 particles per shard
// left; at 512 (photon beams) and 256 (electron beams), 2x10^7 6 MV histories in the
// lung slab took 15.4 ms for 14.9, 10^7 on the slab phantom 8.83 for 8.46, 5x10^6
// 20 MeV electrons on the 128^3 blobs 26.7 for 26.0.
#ifndef DPM_PHASE_HIGH_SHIFT_G
#define DPM_PHASE_HIGH_SHIFT_G 2
#endif
#ifndef DPM_PHASE_LOW_SHIFT_G
#define DPM_PHASE_LOW_SHIFT_G 9
#endif
#ifndef DPM_PHASE_GUARD_SHIFT_G
#define DPM_PHASE_GUARD_SHIFT_G 1
#endif
#ifndef DPM_PHASE_HIGH_SHIFT_E
#define DPM_PHASE_HIGH_SHIFT_E 4
#endif
#ifndef DPM_PHASE_LOW_SHIFT_E
#define DPM_PHASE_LOW_SHIFT_E 10
#endif
#ifndef DPM_PHASE_GUARD_SHIFT_E
#define DPM_PHASE_GUARD_SHIFT_E 2
#endif
constexpr int kStealProbes = DPM_STEAL_PROBES;
// Idle lanes at which a warp takes particles from its stash, by particle type:
// 1 to 4 measured within 1 % of each other, 8 and 12 1 to 2 % slower.
#ifndef DPM_REFILL_MIN_G
#define DPM_REFILL_MIN_G 2
#endif
#ifndef DPM_REFILL_MIN_E
#define DPM_REFILL_MIN_E 2
#endif
// Idle lanes at which a warp with an empty stash looks for more (4 and 16:
// -4 and -1 %).
#ifndef DPM_FETCH_MIN
#define DPM_FETCH_MIN 8
#endif
// On shards below 2^kFullFetchLog2 slots a warp fetches only when it is empty (its
// pause after a fetch outlasts its particles), and a photon beam's secondary phase
// starts at half the backlog: with photons in the stash as well as in the lanes,
// what they still leave after their phase has ended is more than such a shard holds
// (six photon beams of 10^5 to 5x10^6 histories on 256-slot shards: 108 of 240 runs
// overflowed, now none; without stashes 1 of 240).  Runs on larger shards take the
// same time as before (within 0.2 %).
constexpr int kFullFetchLog2 = 9;
// Calls of electron_step between two that make hard events: an event is some 300
// instructions with its secondary, and one or two lanes of a warp have one in
// half of all calls.  Waiting in its lane for the next such call it meets
// others: 5x10^6 20 MeV electrons on the 128^3 blobs 30.8 (every call), 29.9
// (every 2nd), 28.9 (4th), 28.9 (8th) ms; 2x10^4 on the slab 0.70, 0.68, 0.67,
// 0.68 ms.
#ifndef DPM_HARD_EVERY
#define DPM_HARD_EVERY 4
#endif
constexpr unsigned kHardEvery = DPM_HARD_EVERY;
// Records of a warp's stash and of its out buffer, and how many in the buffer
// are sent to the queues by a warp of photons and one of electrons: the buffer
// has room for a step's 32 always.  Sending is a chain of four L2 round trips,
// and the 17 electrons that a call of a full photon warp leaves on the slab
// phantom went to the queues in nearly every call while 16 were kept; now 32 go
// at a time (10^7 6 MV histories 8.44 -> 8.29 ms; 24 kept: 8.38).  An electron
// warp leaves a photon or two per call, which other warps may be waiting for.
constexpr int kStash = 32;
constexpr int kOut = 64;
constexpr int kKeepG = 32, kKeepE = 16;
// Fetch pause: a warp with particles waits this many steps, after it found no
// work for its stash, before it looks again.  A look costs several dependent L2
// round trips, and in the phase of the other type, or at the end of a launch,
// it finds nothing for hundreds of steps (10^7 20 MeV electrons on the blobs
// -5 %, 3x10^7 6 MV histories -2 % against no pause).
#ifndef DPM_REFILL_COOLDOWN
#define DPM_REFILL_COOLDOWN 128
#endif
constexpr unsigned kSleepMaxNs = 1024;  // longest sleep of an idle warp between two looks (16 us ended launches 1 % later)
constexpr int kSpillProbes = 8;

// Where a warp looks for particles (see the refill loop of k_queue).
constexpr unsigned kAskOBit = 2, kAskProbeBit = 4;
constexpr unsigned kAskS = 1, kAskO = 1 | kAskOBit, kAskSProbe = 1 | kAskProbeBit, kAskOProbe = 1 | kAskOBit | kAskProbeBit,
                   kAskSource = 8;

struct alignas(128) Ctl {
  unsigned long long v;
  unsigned long long pad[15];
};

// A queued particle: three 16-byte words, so that a lane writes or reads its
// record with three vector accesses.  (One array per component took twelve
// 4-byte accesses, each with its own 64-bit address, and a sector each where
// one or two lanes push, which is the usual case.)
struct alignas(16) Rec {
  float4 a;  // x, y, z, u
  float4 b;  // v, w, E, packed voxel index
  uint4 c;   // id low, id high, history (bit 31: positron), tag
};

// A particle's tag: the index of its history's batch, and in a shared launch
// its job (at most 1024 batches and kSharedJobs jobs).
constexpr int kTagJobShift = 16;
constexpr uint32_t kTagPhoton = 0x80000000u;   // a photon in an out buffer
constexpr uint32_t kTagPrimary = 0x40000000u;  // a source particle in a stash: its first random block is used

struct QType {
  Rec *rec;
  uint32_t *seq;
  Ctl *head, *tail;  // [K]
};

struct QDev {
  QType q[2];  // 0 photons, 1 electrons and positrons
  int K, log2cs;
  uint32_t mask;
  Ctl *dirty;     // nonzero: a launch gave up a wait, the queues are not in order
  Ctl *n_init;    // blocks of k_queue_init that are done
  Ctl *next_hist, *idle, *started;
  Ctl *backlog;   // queued particles of each type, all shards (signed; pushes add, claims subtract) [2]
  Ctl *phase;     // 0 source phase, 1 secondary phase
  Ctl *cur_job;   // batch launches: the first job that may still have histories to
                  // start (word 0; word 1 unused)
  Ctl *job_next;  // batch launches: next history of each job [kMaxJobs]
  int refill_min[2];  // idle lanes before a warp takes from its stash, by its particle type (photon, electron)
  int pause[2];       // steps a warp with particles waits after a fetch that found none, some
  uint32_t guard[2];               // per-shard bound for sources, by beam type
  long long phase_high[2], phase_low[2];  // global backlog thresholds, by beam type
  uint32_t limit;  // pushes beyond this occupancy of a shard spill over (fault injection can lower it)
  unsigned long long timeout_ns;   // bound on any single wait
  unsigned long long deadline_ns;  // bound on the whole launch (from kernel start)
  // single runs: the batch of a history below 2^31 is its index divided by the
  // batch size d, here by a multiplication: with l = ceil(log2 d) and
  // m = ceil(2^(31+l) / d), floor(h / d) = floor(m h / 2^(31+l)) (Granlund and
  // Montgomery, PLDI 1994); m = 0 stands for d = 1
  uint32_t batch_mul, batch_shift;
  __device__ __forceinline__ uint32_t batch_of(uint32_t h) const {
    return batch_mul ? __umulhi(h, batch_mul) >> batch_shift : h;
  }
};

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned long long ld_volatile(const unsigned long long *p) {
  return *(const volatile unsigned long long *)p;
}

// Slot sequence words: the producer publishes a record and the consumer
// frees its slot with a release store; both wait for the word with acquire
// loads, so the record's plain loads and stores are ordered around them.
__device__ __forceinline__ uint32_t ld_acquire32(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release32(uint32_t *p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}

// Wait until a slot's sequence word is `want`; false when the time limit runs out.
__device__ __forceinline__ bool wait_seq(const uint32_t *seq, uint32_t want, unsigned long long timeout_ns) {
  if (ld_acquire32(seq) == want) return true;
  const unsigned long long t0 = now_ns();
  while (ld_acquire32(seq) != want) {
    if (now_ns() - t0 > timeout_ns) return false;
    __nanosleep(32);
  }
  return true;
}

// Occupancy of a shard from two relaxed loads.  The loads of head and tail
// may be observed in either order, so a concurrent consumer can make head
// appear ahead of tail: the difference saturates at zero.
__device__ __forceinline__ unsigned long long occupancy(unsigned long long head, unsigned long long tail) {
  return tail > head ? tail - head : 0ull;
}

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// What a particle step of a batch job reads of its job: the phantom, the
// history numbering and the tally.  A shared launch copies these records of all
// its jobs into shared memory at the start (at most kSharedJobs), so that a
// step reads them from shared memory instead of the job table.
struct JobHot {
  DevPhantom P;
  uint64_t first;
  uint32_t key0, key1;
  unsigned long long *slabs;
  uint32_t V;
};

// A warp's part of shared memory.
struct WarpBox {
  Rec stash[kStash];  // particles of the warp's own type, for its idle lanes (last in, first out)
  Rec out[kOut];      // secondaries on their way to the queues
  long long esc[32];  // energy that left the phantom, by lane
  float held[3][32];  // numbers kept for the lanes' particles (QSink::hold)
  long long emit, miss;            // emitted and missed energy (lane 0)
  unsigned long long t_start;      // launch time of the warp
  int cool;                        // steps before the warp, with particles, looks for work again
  unsigned retry_ns;               // pause of an idle warp before it looks for work again
  int err;
};

// energy counters (coarser quantum than the tally's, see kCounterScale)
__device__ __forceinline__ long long fxc(float e) { return __float2ll_rn(e * kCounterScaleF); }

// Lane-level sink: tally with run-length coalescing and counters.  kMulti: a
// batch launch, whose particles carry their job index.  kCount: also count
// events (steps, flights, interactions, tally atomics, pushes) for the run
// statistics; the energy counters (emitted, escaped, missed) are always kept.
// The event counts live in registers across the whole loop and cost 8 to 9 % of
// the transport time (10^7 6 MV histories 8.76 -> 9.45 ms, 10^6 20 MeV electrons on
// the slabs 6.11 -> 6.67 ms), so runs count them only on request
// (dpm_run_opts.count_events).  kSauter_: compile in the photoelectron angle
// option (DPM_SAUTER); its code alone, unused, measured 4-6 % slower, so only
// the single-run launches that ask for it carry it.
template <bool kMulti, bool kCount, bool kSauter_ = false>
struct QSink {
  static constexpr bool kSauter = kSauter_;
  const RunParams &R;
  const QDev &Q;
  const JobHot *sjobs;
  WarpBox *box;
  uint32_t tag = 0;  // of the particle in the lane (batch launches)
  const uint32_t *hist;  // the particle's history
  long long pend_q = 0;
  unsigned calls = 0;  // of the warp (uniform)
  __device__ __forceinline__ bool hard_waits() const { return calls % kHardEvery != 0; }
  long long cnt[C_N];  // event counts only (kCount)

  __device__ QSink(const RunParams &r, const QDev &q, const JobHot *sj, WarpBox *w, const uint32_t *h)
      : R(r), Q(q), sjobs(sj), box(w), hist(h) {
#pragma unroll
    for (int i = 0; i < C_N; ++i) cnt[i] = 0;
  }
  __device__ __forceinline__ static long long fx(float e) { return __float2ll_rn(e * 4294967296.0f); }
  // Run-length coalescing: a particle's deposits in one voxel are summed and
  // added to the tally when it leaves the voxel or ends (photons, which deposit
  // only where they interact, after the step).
  __device__ __forceinline__ void deposit(int, float dE) { pend_q += fx(dE); }
  __device__ __forceinline__ void leave(int v) {
    if (pend_q != 0) {
      unsigned long long *slabs = R.slabs;
      uint32_t V = uint32_t(R.P.nx) * uint32_t(R.P.ny) * uint32_t(R.P.nz), b;
      if (kMulti) {
        const JobHot &J = sjobs[tag >> kTagJobShift];
        slabs = J.slabs;
        V = J.V;
        b = tag & ((1u << kTagJobShift) - 1);
      } else {
        b = Q.batch_of(*hist);
      }
      atomicAdd(slabs + (uint64_t(b) * V + uint32_t(v)), (unsigned long long)pend_q);
      if (kCount) ++cnt[C_ATOM];
      pend_q = 0;
    }
  }
  __device__ __forceinline__ void escape(float E) { box->esc[threadIdx.x & 31] += fxc(E); }
  __device__ __forceinline__ void error(int e) { atomicOr(&box->err, e); }
  // volatile: these are here so that no register holds them through the step
  __device__ __forceinline__ volatile float *held_at(int k) const { return &box->held[k][threadIdx.x & 31]; }
  __device__ __forceinline__ void hold(float R, float S, float Sigma) {
    *held_at(0) = R;
    *held_at(1) = S;
    *held_at(2) = Sigma;
  }
  __device__ __forceinline__ float held_range() const { return *held_at(0); }
  __device__ __forceinline__ float held_power() const { return *held_at(1); }
  __device__ __forceinline__ float held_sigma() const { return *held_at(2); }
  __device__ __forceinline__ void count_step() {
    if (kCount) ++cnt[C_ESTEP];
  }
  __device__ __forceinline__ void count_flight() {
    if (kCount) ++cnt[C_GFLIGHT];
  }
  __device__ __forceinline__ void count_interaction() {
    if (kCount) ++cnt[C_GINT];
  }
  // record of secondary o of p
  __device__ __forceinline__ Rec record(const Part &p, const Emission &o) const {
    Rec r;
    r.a = make_float4(p.x, p.y, p.z, o.u);
    r.b = make_float4(o.v, o.w, o.E, __uint_as_float(p.vx));
    r.c = make_uint4(o.id_lo, o.id_hi, p.hist | (o.type == POSITRON ? 0x80000000u : 0u),
                     (kMulti ? tag : 0u) | (o.type == PHOTON ? kTagPhoton : 0u));
    return r;
  }
};

// 16 bytes at a time: the lane's own state stays in registers meanwhile.
__device__ __forceinline__ void copy_rec(Rec *to, const Rec *from) {
  to->a = from->a;
  to->b = from->b;
  to->c = from->c;
}

// Reserve n positions of queue t in the CTA's own shard, else in one of the next
// ones (a full shard spills over): the shard and the first position, or -1.
__device__ __forceinline__ int reserve(const QDev &Q, int t, int n, unsigned long long &base) {
  const QType &Qt = Q.q[t];
  int s = blockIdx.x % Q.K;
#pragma unroll 1
  for (int k = 0; k <= kSpillProbes && k < Q.K; ++k) {
    if (occupancy(ld_volatile(&Qt.head[s].v), ld_volatile(&Qt.tail[s].v)) + n <= Q.limit) {
      base = atomicAdd(&Qt.tail[s].v, (unsigned long long)n);
      atomicAdd(&Q.backlog[t].v, (unsigned long long)n);
      return s;
    }
    s = s + 1 == Q.K ? 0 : s + 1;
  }
  return -1;
}

// Queue records [from, n) of the warp's out buffer: one atomic per 32 records on
// the shard's tail and the backlog of each type.
__device__ __forceinline__ void flush_out(const QDev &Q, WarpBox *w, int from, int n) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll 1
  for (int i = from + lane; i - lane < n; i += 32) {
    const bool have = i < n;
    const int t = have && (w->out[i].c.w & kTagPhoton) ? 0 : 1;
    const unsigned m0 = __ballot_sync(kFull, have && t == 0), m1 = __ballot_sync(kFull, have && t == 1);
    const unsigned mask = t ? m1 : m0;
    const int leader = (mask ? __ffs(mask) : 1) - 1;
    const QType &Qt = Q.q[t];
    unsigned long long base = 0;
    int shard = -1;
    if (have && lane == leader) shard = reserve(Q, t, __popc(mask), base);
    base = __shfl_sync(kFull, base, leader) + __popc(mask & lanemask_lt());
    shard = __shfl_sync(kFull, shard, leader);
    if (have && shard < 0) shard = reserve(Q, t, 1, base);  // small queues: one by one where 32 do not fit
    if (have) {
      if (shard < 0) {
        atomicOr(&w->err, ERR_OVERFLOW);
        w->esc[lane] += fxc(w->out[i].b.z + ((w->out[i].c.z >> 31) ? 2.f * kMc2f : 0.f));
      } else {
        const unsigned long long pos = base;
        const size_t idx = (size_t(shard) << Q.log2cs) + (uint32_t(pos) & Q.mask);
        // wait for the consumer of position pos - capacity to have freed the slot
        if (!wait_seq(Qt.seq + idx, uint32_t(pos), Q.timeout_ns)) {
          atomicOr(&w->err, ERR_TIMEOUT);
        } else {
          copy_rec(Qt.rec + idx, w->out + i);
          st_release32(Qt.seq + idx, uint32_t(pos + 1));
        }
      }
    }
  }
  __syncwarp();
}

// Leader claims up to `want` queued positions of shard s with a CAS on its
// head; returns the count (warp-uniform) and the first position.
__device__ __forceinline__ int claim(const QType &Qt, int s, int want, unsigned long long &base) {
  int n = 0;
  unsigned long long b = 0;
  if ((threadIdx.x & 31) == 0) {
#pragma unroll 1
    for (int tries = 0; tries < 32; ++tries) {
      const unsigned long long h = ld_volatile(&Qt.head[s].v);
      const unsigned long long t = ld_volatile(&Qt.tail[s].v);
      if (t <= h) break;
      const unsigned long long k = min(t - h, (unsigned long long)want);
      if (atomicCAS(&Qt.head[s].v, h, h + k) == h) {
        n = int(k);
        b = h;
        break;
      }
    }
  }
  n = __shfl_sync(kFull, n, 0);
  base = __shfl_sync(kFull, b, 0);
  return n;
}

// Read the record at position p of shard s (waiting for its publication) and
// free the slot for the producer one lap later.
__device__ __forceinline__ void take(const QDev &Q, int t, int s, unsigned long long p, Rec *to, int *err) {
  const QType &Qt = Q.q[t];
  const size_t idx = (size_t(s) << Q.log2cs) + (uint32_t(p) & Q.mask);
  if (!wait_seq(Qt.seq + idx, uint32_t(p + 1), Q.timeout_ns)) {
    atomicOr(err, ERR_TIMEOUT);
    // a particle without energy in its place: its first step ends it
    to->a = to->b = make_float4(0.f, 0.f, 0.f, 0.f);
    to->c = make_uint4(0u, 0u, 0u, 0u);
    return;
  }
  to->a = __ldcg(&Qt.rec[idx].a);
  to->b = __ldcg(&Qt.rec[idx].b);
  to->c = __ldcg(&Qt.rec[idx].c);
  st_release32(Qt.seq + idx, uint32_t(p + (1ull << Q.log2cs)));
}

// Up to `want` particles of type t into the stash (home shard first, then
// `probes` others).  Returns their number (warp-uniform).
__device__ __forceinline__ int fetch_queue(const QDev &Q, int t, int probes, int want, WarpBox *w) {
  const int lane = threadIdx.x & 31;
  unsigned long long base;
  int s = blockIdx.x % Q.K, n = 0;
#pragma unroll 1
  for (int k = 0; k <= probes && k < Q.K; ++k) {
    n = claim(Q.q[t], s, want, base);
    if (n) break;
    s = (s + 97) % Q.K;
  }
  if (n == 0) return 0;
  if (lane == 0) atomicAdd(&Q.backlog[t].v, (unsigned long long)(-(long long)n));
  if (lane < n) take(Q, t, s, base + lane, w->stash + lane, &w->err);
  return n;
}

struct JobStepCtx {
  const DevTables &T;
  const DevPhantom &P;
  uint64_t first;
  uint32_t key0, key1;
};

__device__ __forceinline__ JobStepCtx job_step_ctx(const RunParams &R, const JobHot *sj, uint32_t tag) {
  const JobHot &J = sj[tag >> kTagJobShift];
  return JobStepCtx{R.T, J.P, J.first, J.key0, J.key1};
}

// Context of a batch job for the source (the job table lives in global memory).
__device__ __forceinline__ JobCtx job_ctx(const RunParams &R, int j) {
  const DevJob &J = R.jobs[j];
  return JobCtx{R.T, J.P, J.S, J.first, J.key0, J.key1};
}

// Queued particles anywhere, or histories left to start, by the global per-type
// backlog counters (warp-uniform).  With pushes and claims in flight they may be
// off; once every warp is idle (each is counted after all it did) they are exact,
// and end the run.  Until then every warp looked through the heads and tails of
// all shards, which for K shards and 4 K warps is 16 K^2 loads: one history took
// 0.10 ms with 3 blocks per SM and 0.22 ms with 7.
template <bool kMulti>
__device__ bool any_work(const RunParams &R, const QDev &Q) {
  bool w = false;
  if ((threadIdx.x & 31) == 0) {
    w = (long long)ld_volatile(&Q.backlog[0].v) > 0 || (long long)ld_volatile(&Q.backlog[1].v) > 0;
    if (!kMulti && ld_volatile(&Q.next_hist->v) < R.n) w = true;
    if (kMulti && ld_volatile(&Q.cur_job[0].v) < (unsigned long long)R.n_jobs) w = true;
  }
  return __shfl_sync(kFull, w, 0);
}

// True while both of the CTA's shards hold at most `bound` particles (warp-uniform).
__device__ bool source_allowed(const QDev &Q, int home, unsigned long long bound) {
  bool ok = true;
  if ((threadIdx.x & 31) == 0) {
    for (int t = 0; t < 2; ++t)
      if (occupancy(ld_volatile(&Q.q[t].head[home].v), ld_volatile(&Q.q[t].tail[home].v)) > bound) ok = false;
  }
  return __shfl_sync(kFull, ok, 0);
}

// The grid-wide phase (0 source, 1 secondary) for beam type S, switched
// with hysteresis on the global backlog of the other type by whichever warp
// sees the threshold crossed first (warp-uniform).
__device__ int grid_phase(const QDev &Q, int S, unsigned long long *counters) {
  int ph = 0;
  if ((threadIdx.x & 31) == 0) {
    ph = int(ld_volatile(&Q.phase->v));
    const long long b = (long long)ld_volatile(&Q.backlog[1 - S].v);
    if (ph == 0 && b > Q.phase_high[S]) {
      ph = 1;
      if (atomicExch(&Q.phase->v, 1ull) == 0ull) atomicAdd(counters + C_SWITCH, 1ull);
    } else if (ph == 1 && b < Q.phase_low[S]) {
      ph = 0;
      if (atomicExch(&Q.phase->v, 0ull) == 1ull) atomicAdd(counters + C_SWITCH, 1ull);
    }
  }
  return __shfl_sync(kFull, ph, 0);
}

// Beam type of the batch job being started (the table lists photon beams
// first); once every job has been started, that of the last job
// (warp-uniform).
__device__ __forceinline__ int current_source_type(const RunParams &R, const QDev &Q) {
  int t = 0;
  if ((threadIdx.x & 31) == 0) {
    const unsigned long long j = ld_volatile(&Q.cur_job[0].v);
    t = (j < (unsigned long long)R.n_photon_jobs || R.n_photon_jobs == R.n_jobs) ? 0 : 1;
  }
  return __shfl_sync(kFull, t, 0);
}

// True once every source history of the launch has been started (warp-uniform).
template <bool kMulti>
__device__ __forceinline__ bool source_exhausted(const RunParams &R, const QDev &Q) {
  bool e = false;
  if ((threadIdx.x & 31) == 0)
    e = kMulti ? ld_volatile(&Q.cur_job[0].v) >= (unsigned long long)R.n_jobs : ld_volatile(&Q.next_hist->v) >= R.n;
  return __shfl_sync(kFull, e, 0);
}

// A lane's state set aside in local memory while its warp starts histories.
// The source's code needs some 50 registers; were the lane's state to live
// through it, the compiler would keep part of that state in local memory for
// the whole loop and store it on every step.
struct Parked {
  volatile uint32_t w[16];
};

__device__ __forceinline__ void park(Parked &k, const Part &p, uint32_t tag, long long pend_q) {
  k.w[0] = __float_as_uint(p.x);
  k.w[1] = __float_as_uint(p.y);
  k.w[2] = __float_as_uint(p.z);
  k.w[3] = __float_as_uint(p.u);
  k.w[4] = __float_as_uint(p.v);
  k.w[5] = __float_as_uint(p.w);
  k.w[6] = __float_as_uint(p.E);
  k.w[7] = p.vx;
  k.w[8] = p.id_lo;
  k.w[9] = p.id_hi;
  k.w[10] = p.ctr;
  k.w[11] = p.hist;
  k.w[12] = uint32_t(p.type);
  k.w[13] = tag;
  k.w[14] = uint32_t(pend_q);
  k.w[15] = uint32_t(uint64_t(pend_q) >> 32);
}

__device__ __forceinline__ void unpark(const Parked &k, Part &p, uint32_t &tag, long long &pend_q) {
  p.x = __uint_as_float(k.w[0]);
  p.y = __uint_as_float(k.w[1]);
  p.z = __uint_as_float(k.w[2]);
  p.u = __uint_as_float(k.w[3]);
  p.v = __uint_as_float(k.w[4]);
  p.w = __uint_as_float(k.w[5]);
  p.E = __uint_as_float(k.w[6]);
  p.vx = k.w[7];
  p.id_lo = k.w[8];
  p.id_hi = k.w[9];
  p.ctr = k.w[10];
  p.hist = k.w[11];
  p.type = int(k.w[12]);
  tag = k.w[13];
  const uint32_t lo = k.w[14], hi = k.w[15];
  pend_q = (long long)((uint64_t(hi) << 32) | lo);
}

// Start up to 32 new source histories of beam type S into the (empty) stash:
// from the run's range, or (batch) from the current job of the batch, job after
// job, so that one job's phantom and tally are hot in L2 at a time.  All lanes
// make a primary each, whatever their own particle is doing.  Returns the
// number of particles in the stash, or -1 if no history was left to start.
template <bool kMulti>
__device__ __noinline__ int fetch_source(const RunParams &R, const QDev &Q, WarpBox *w, int S) {
  const int lane = threadIdx.x & 31;
  unsigned long long b = ~0ull, n = 0;
  int j = 0;
  if (lane == 0) {
    if (!kMulti) {
      n = R.n;
      if (ld_volatile(&Q.next_hist->v) < R.n) b = atomicAdd(&Q.next_hist->v, 32ull);
    } else {
#pragma unroll 1
      for (int tries = 0; tries <= R.n_jobs; ++tries) {
        j = int(ld_volatile(&Q.cur_job[0].v));
        if (j >= R.n_jobs) break;
        if ((R.jobs[j].S.particle == 0 ? 0 : 1) != S) break;  // the current job has the other beam type
        n = R.jobs[j].n;
        if (ld_volatile(&Q.job_next[j].v) < n) {
          b = atomicAdd(&Q.job_next[j].v, 32ull);
          if (b < n) break;
        }
        atomicCAS(&Q.cur_job[0].v, (unsigned long long)j, (unsigned long long)(j + 1));  // job exhausted
        b = ~0ull;
      }
    }
  }
  b = __shfl_sync(kFull, b, 0);
  n = __shfl_sync(kFull, n, 0);
  j = __shfl_sync(kFull, j, 0);
  if (b >= n) return -1;
  const unsigned long long hl = b + lane;
  bool hit = false;
  long long e_emit = 0, e_miss = 0;
  Part q;
  if (hl < n) {
    hit = kMulti ? make_primary(q, job_ctx(R, j), uint32_t(hl)) : make_primary(q, R, uint32_t(hl));
    e_emit = fxc(q.E);
    e_miss = hit ? 0 : e_emit;
  }
  const unsigned hits = __ballot_sync(kFull, hit);
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    e_emit += __shfl_down_sync(kFull, e_emit, o);
    e_miss += __shfl_down_sync(kFull, e_miss, o);
  }
  if (lane == 0) {
    w->emit += e_emit;
    w->miss += e_miss;
  }
  if (hit) {
    uint32_t tag = kTagPrimary;
    if (kMulti) tag |= uint32_t(hl) / uint32_t(R.jobs[j].batch_size) | uint32_t(j) << kTagJobShift;
    Rec &r = w->stash[__popc(hits & lanemask_lt())];
    r.a = make_float4(q.x, q.y, q.z, q.u);
    r.b = make_float4(q.v, q.w, q.E, __uint_as_float(q.vx));
    r.c = make_uint4(q.id_lo, q.id_hi, q.hist, tag);
  }
  return __popc(hits);
}

// What fetch() found: particles in the stash (n may be 0 when a batch of
// histories missed the phantom), their type, and whether the source is dry.
struct Fetched {
  int n, mode;
  bool found, dry;
};

// Fill the empty stash of a warp of type `mode` (-1: no particles in its lanes)
// with up to 32 particles, or `few` (its idle lanes) once the source is dry: near
// the end of a launch the queued particles are spread over the warps.
//
// Source phase: warps start histories and track particles of the beam's type
// while the secondaries of the other type pile up in the queues; secondary
// phase: no history starts and warps track the queued particles in full warps.
// Warps of the type out of phase finish their particles and turn over.  A
// grid-wide phase keeps the SMs on one of the two code paths at a time.
template <bool kMulti>
__device__ __forceinline__ Fetched fetch(const RunParams &R, const QDev &Q, WarpBox *w, int mode, int few, bool dry, Part &p,
                                 uint32_t &tag, long long &pend_q) {
  const int S = kMulti ? current_source_type(R, Q) : (R.S.particle == 0 ? 0 : 1);
  const int O = 1 - S;
  const int ph = grid_phase(Q, S, R.counters);
  dry = dry || source_exhausted<kMulti>(R, Q);
  // the places to look for work, first to last, four bits each; one loop
  // over them keeps a single copy of the code
  unsigned todo = 0;
  Fetched f{0, mode, false, dry};
  if (mode < 0)
    todo = ph == 1 ? (kAskO | kAskOProbe << 4 | kAskS << 8 | kAskSProbe << 12)
                   : (kAskS | kAskSource << 4 | kAskO << 8 | kAskOProbe << 12 | kAskSProbe << 16);
  else if (mode == S)
    todo = ph == 0 ? (kAskS | kAskSource << 4) : 0u;
  else if (ph == 1 || dry)
    todo = kAskOProbe;
#pragma unroll 1
  for (; todo != 0 && !f.found; todo >>= 4) {
    const unsigned ask = todo & 15u;
    if (ask == kAskSource) {
      if (source_allowed(Q, blockIdx.x % Q.K, Q.guard[S])) {
        Parked k;
        park(k, p, tag, pend_q);
        const int k_src = fetch_source<kMulti>(R, Q, w, S);
        f.found = k_src >= 0;
        f.n = max(k_src, 0);
        unpark(k, p, tag, pend_q);
        f.dry = !f.found;
        if (f.found) f.mode = S;
      }
    } else {
      const int t = (ask & kAskOBit) ? O : S;
      f.n = fetch_queue(Q, t, (ask & kAskProbeBit) ? kStealProbes : 0, f.dry ? few : 32, w);
      f.found = f.n != 0;
      if (f.found) f.mode = t;
    }
  }
  if (f.found && (threadIdx.x & 31) == 0) w->retry_ns = 32;
  __syncwarp();
  return f;
}

// A warp without particles waits until there is work within reach (true: look
// again), or until the run is over or a time limit has passed (false).
template <bool kMulti>
__device__ __forceinline__ bool idle_wait(const RunParams &R, const QDev &Q, WarpBox *w) {
  const int lane = threadIdx.x & 31;
  const unsigned long long t0 = __shfl_sync(kFull, now_ns(), 0);
  unsigned sleep_ns = 128;
  __threadfence();
  if (lane == 0) atomicAdd(&Q.idle->v, 1ull);
#pragma unroll 1
  for (;;) {
    if (any_work<kMulti>(R, Q)) {
      // work exists but this warp found none within reach: retry after a
      // short, growing pause instead of rescanning at once
      if (lane == 0) atomicAdd(&Q.idle->v, ~0ull);  // -1
      if (__shfl_sync(kFull, now_ns() - w->t_start > Q.deadline_ns, 0)) {
        if (lane == 0) atomicOr(&w->err, ERR_TIMEOUT);
        return false;
      }
      const unsigned ns = w->retry_ns;
      __syncwarp();
      __nanosleep(ns);
      if (lane == 0) w->retry_ns = min(ns * 2, 2048u);
      __syncwarp();
      return true;
    }
    bool done = false;
    if (lane == 0) {
      const unsigned long long idle = ld_volatile(&Q.idle->v);  // before the number of those started
      done = idle == ld_volatile(&Q.started->v);
    }
    done = __shfl_sync(kFull, done, 0);
    if (done) {
      __threadfence();
      if (!any_work<kMulti>(R, Q)) return false;
    }
    if (__shfl_sync(kFull, now_ns() - t0 > Q.timeout_ns, 0)) {
      if (lane == 0) atomicOr(&w->err, ERR_TIMEOUT);
      return false;
    }
    __nanosleep(sleep_ns);
    sleep_ns = min(sleep_ns * 2, kSleepMaxNs);
  }
}

__device__ void reduce_counters_q(const long long *cnt, const WarpBox *w, const RunParams &R, const QDev &Q) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < C_N; ++i) {
    long long v = i == C_ESC ? w->esc[lane] : i == C_EMIT ? (lane == 0 ? w->emit : 0) : i == C_MISS ? (lane == 0 ? w->miss : 0) : cnt[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    if (lane == 0 && v != 0) atomicAdd(R.counters + i, (unsigned long long)v);
  }
  if (lane == 0 && w->err) {
    atomicOr(R.err, w->err);
    if (w->err & ERR_TIMEOUT) atomicExch(&Q.dirty->v, 1ull);
  }
}

// Seven resident blocks per SM: 28 warps with up to 72 registers each, and
// nothing spilled in the hot loop.  6, 7 and 8 blocks (80, 72 and 64 registers):
// 10^7 6 MV histories 9.68, 8.83 and 9.98 ms, 5x10^6 20 MeV electrons on the
// 128^3 blobs 28.9, 26.4 and 29.8 ms, 2x10^4 on the slab 0.57, 0.58 and 0.70 ms.
// (6 blocks that are held to 72 registers: 9.29, 28.1 and 0.56 ms.)
#ifndef DPM_QUEUE_MIN_BLOCKS
#define DPM_QUEUE_MIN_BLOCKS 7
#endif
template <bool kMulti, bool kCount, bool kSauter = false>
__global__ void __launch_bounds__(kQBlock, DPM_QUEUE_MIN_BLOCKS)
    k_queue(const __grid_constant__ RunParams R, const __grid_constant__ QDev Q) {
  __shared__ WarpBox s_box[kQBlock / 32];
  extern __shared__ JobHot sjobs[];
  const int lane = threadIdx.x & 31;
  WarpBox *box = s_box + (threadIdx.x >> 5);
  box->esc[lane] = 0;
  if (lane == 0) {
    box->emit = box->miss = 0;
    box->t_start = now_ns();
    box->retry_ns = 32;
    box->cool = 0;
    box->err = 0;
    atomicAdd(&Q.started->v, 1ull);
  }
  // batch launches: the jobs' step records in shared memory (all threads of
  // the block are here, before any divergent code)
  if (kMulti) {
    for (int j = threadIdx.x; j < R.n_jobs; j += blockDim.x) {
      const DevJob &J = R.jobs[j];
      sjobs[j] = JobHot{J.P, J.first, J.key0, J.key1, J.slabs, uint32_t(J.V)};
    }
  }
  __syncthreads();
  Part p{};
  QSink<kMulti, kCount, kSauter> sk(R, Q, sjobs, box, &p.hist);
  bool alive = false;
  // warp-uniform from here on
  int n_stash = 0, n_out = 0;  // records in the stash (all of type `mode`) and in the out buffer
  int mode = -1;               // type of the particles in the lanes, -1 without any
  bool dry = false;            // the source had nothing left when last asked
  for (;;) {
    const unsigned live = __ballot_sync(kFull, alive);
    const int n_idle = 32 - __popc(live);
    // near the end of a launch every particle is for whoever is idle
    const bool send = n_out > (mode == 0 ? kKeepG : kKeepE) || (n_out != 0 && (dry || live == 0));
    bool look = live == 0 && n_stash == 0;
    if (live == 0 && n_stash == 0) {
      mode = -1;
    } else if (n_stash == 0 && n_idle >= DPM_FETCH_MIN) {
      const int c = box->cool;
      __syncwarp();
      if (lane == 0 && c > 0) box->cool = c - 1;
      look = c == 0;
    }
    if (send) {
      const int from = dry || live == 0 ? 0 : max(n_out - 32, 0);  // the newest 32, or all
      flush_out(Q, box, from, n_out);
      n_out = from;
    }
    if (look) {
      const Fetched f = fetch<kMulti>(R, Q, box, mode, n_idle, dry, p, sk.tag, sk.pend_q);
      n_stash = int(__reduce_max_sync(kFull, unsigned(f.n)));
      mode = int(__reduce_max_sync(kFull, unsigned(f.mode + 1))) - 1;
      dry = __any_sync(kFull, f.dry);
      if (lane == 0) box->cool = Q.pause[f.found ? 1 : 0];
      __syncwarp();
    }
    if (n_idle >= Q.refill_min[mode > 0 ? 1 : 0] || live == 0) {
      if (n_stash != 0) {
        // the newest records into the idle lanes
        __syncwarp();
        const int rank = __popc(~live & lanemask_lt());
        if (!alive && rank < n_stash) {
          const Rec &r = box->stash[n_stash - 1 - rank];
          const float4 a = r.a, b = r.b;
          const uint4 c = r.c;
          p.x = a.x;
          p.y = a.y;
          p.z = a.z;
          p.u = a.w;
          p.v = b.x;
          p.w = b.y;
          p.E = b.z;
          p.vx = __float_as_uint(b.w);
          p.id_lo = c.x;
          p.id_hi = c.y;
          p.hist = c.z & 0x7fffffffu;
          p.type = mode == 0 ? PHOTON : (c.z >> 31) ? POSITRON : ELECTRON;
          p.ctr = (c.w & kTagPrimary) ? 1u : 0u;
          if (kMulti) sk.tag = c.w & ~(kTagPhoton | kTagPrimary);
          alive = true;
        }
        __syncwarp();
        n_stash = max(n_stash - n_idle, 0);
      } else if (live == 0) {
        if (!__any_sync(kFull, idle_wait<kMulti>(R, Q, box))) break;
        p = Part{};  // nothing in the lanes: no state to keep through the wait
        sk.tag = 0;
        sk.pend_q = 0;
        continue;
      }
    }
    const bool was = alive;
    ++sk.calls;
    Emission o;
    if (alive) {
      if (p.type & CHAIN)
        alive = kMulti ? chain_step(p, job_step_ctx(R, sjobs, sk.tag), sk, o) : chain_step(p, R, sk, o);
      else if (mode == 0)
        alive = kMulti ? photon_flight(p, job_step_ctx(R, sjobs, sk.tag), sk, o) : photon_flight(p, R, sk, o);
      else
        alive = kMulti ? electron_step(p, job_step_ctx(R, sjobs, sk.tag), sk, o) : electron_step(p, R, sk, o);
      if (alive && p.ctr >= (mode == 0 ? kMaxPhotonBlocks : kMaxElectronBlocks)) {
        sk.error(ERR_STEPCAP);
        sk.deposit(kMulti ? vox(p, job_step_ctx(R, sjobs, sk.tag).P) : vox(p, R.P), p.E);
        alive = false;
      }
    }
    // The step's secondaries, in one place for the whole warp whatever made
    // them: those of the warp's own type go to its stash while it has room,
    // the others to the queues by way of the out buffer (which has room for 32).
    bool want = false;
    if (o.kind != EM_NONE) want = kMulti ? settle(p, o, job_step_ctx(R, sjobs, sk.tag), sk) : settle(p, o, R, sk);
    if (was && (!alive || mode == 0)) sk.leave(kMulti ? vox(p, job_step_ctx(R, sjobs, sk.tag).P) : vox(p, R.P));
    const unsigned all = __ballot_sync(kFull, want);
    if (all != 0) {
      if (kCount && want) ++sk.cnt[C_PUSH];
      const unsigned own = __ballot_sync(kFull, want && (o.type == PHOTON) == (mode == 0));
      const bool keep = !dry && n_stash + __popc(own) <= kStash;
      const unsigned to_out = keep ? all & ~own : all;
      if (want) {
        const bool st = keep && (own >> lane & 1u);
        Rec *dst = st ? box->stash + n_stash + __popc(own & lanemask_lt()) : box->out + n_out + __popc(to_out & lanemask_lt());
        *dst = sk.record(p, o);
      }
      if (keep) n_stash += __popc(own);
      n_out += __popc(to_out);
    }
  }
  __syncwarp();
  reduce_counters_q(sk.cnt, box, R, Q);
}

// Prepares the queues for a launch: the control words zero and, on a fresh
// layout (`fresh`) or after a launch that gave up a wait (*dirty), the shards
// empty.  Positions of a shard go on counting from launch to launch: a launch
// that ends in order leaves every shard empty with its sequence words ready for
// the next position, so nothing else has to be written.  Writing the sequence
// words of the default queues (120 to 240 MB) before every launch, and three
// fills, took 40 to 60 us (one 6 MV history, call and wait: 0.27 -> 0.21 ms).
__global__ void k_queue_init(QDev Q, Ctl *ctl, int n_ctl, size_t n, bool fresh) {
  const size_t i0 = size_t(blockIdx.x) * blockDim.x + threadIdx.x, stride = size_t(gridDim.x) * blockDim.x;
  for (size_t i = i0; i < size_t(n_ctl); i += stride) ctl[i].v = 0;
  if (fresh || ld_volatile(&Q.dirty->v) != 0) {
    for (int t = 0; t < 2; ++t) {
      for (size_t i = i0; i < size_t(Q.K); i += stride) Q.q[t].head[i].v = Q.q[t].tail[i].v = 0;
      for (size_t i = i0; i < n; i += stride) Q.q[t].seq[i] = uint32_t(i) & Q.mask;
    }
  }
  // the last block to come here, when all have read the word, clears it
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&Q.n_init->v, 1ull) == gridDim.x - 1) Q.dirty->v = Q.n_init->v = 0;
  }
}

}  // namespace

// The queue kernel's instantiations: single run or batch launch (kMulti) x
// event counts, and the single runs with the photoelectron angle option.
using QKernel = void (*)(RunParams, QDev);
struct QKernelEntry {
  QKernel k;
  bool multi;
};
const QKernelEntry kQueueKernels[6] = {
    {k_queue<false, false>, false},      {k_queue<false, true>, false},      {k_queue<true, false>, true},
    {k_queue<true, true>, true},         {k_queue<false, false, true>, false}, {k_queue<false, true, true>, false}};

QKernel queue_kernel(bool multi, bool count, bool sauter) {
  if (sauter) return count ? k_queue<false, true, true> : k_queue<false, false, true>;
  if (multi) return count ? k_queue<true, true> : k_queue<true, false>;
  return count ? k_queue<false, true> : k_queue<false, false>;
}

int queue_blocks_per_sm() {
  // Shared memory for the resident blocks (21 KB of stashes and buffers each,
  // in a batch launch also the step records of up to kSharedJobs jobs, and 1 KB
  // reserved), the rest to L1, where the tables are cached: at 84 % for batch
  // launches, which takes the next larger split, serving took 5 % longer.
  int best = 1 << 30;
  for (const QKernelEntry &e : kQueueKernels) {
    const QKernel k = e.k;
    int per_sm = 0;
    const bool multi = e.multi;
    const size_t smem = multi ? kSharedJobs * sizeof(JobHot) : 0;
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, multi ? 80 : 70);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kQBlock, smem) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    best = std::min(best, per_sm);
  }
  return best;
}

int queue_preload() {
  // cudaFuncGetAttributes loads a kernel under lazy module loading
  cudaFuncAttributes a;
  bool ok = cudaFuncGetAttributes(&a, k_queue_init) == cudaSuccess;
  for (const QKernelEntry &e : kQueueKernels) ok = ok && cudaFuncGetAttributes(&a, e.k) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    return 0;
  }
  return queue_blocks_per_sm();
}

constexpr int kWordsPerSlot = 13;  // a record and its sequence word
static_assert(sizeof(Rec) + 4 == kWordsPerSlot * 4, "record layout");
// dirty n_init | next_hist idle started cur_job[2] backlog[2] phase job_next[kMaxJobs], zeroed before every launch
constexpr int kKeptWords = 2;
constexpr int kCtlWords = kKeptWords + 8 + kMaxJobs;

size_t queue_bytes(int K, int log2cs) {
  const size_t slots = size_t(K) << log2cs;
  const size_t per_type = slots * kWordsPerSlot * sizeof(uint32_t) + 2 * size_t(K) * sizeof(Ctl);
  return 2 * per_type + kCtlWords * sizeof(Ctl) + 128;
}

// The queues of K shards of 2^log2cs slots in `mem`.
static QDev queue_layout(void *mem, int K, int log2cs) {
  const size_t slots = size_t(K) << log2cs;
  const size_t per_type = slots * kWordsPerSlot * sizeof(uint32_t) + 2 * size_t(K) * sizeof(Ctl);
  QDev Q{};
  char *m = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(mem) + 127) & ~uintptr_t(127));
  Q.dirty = reinterpret_cast<Ctl *>(m);
  Q.n_init = Q.dirty + 1;
  Q.next_hist = Q.dirty + kKeptWords;
  Q.idle = Q.next_hist + 1;
  Q.started = Q.next_hist + 2;
  Q.cur_job = Q.next_hist + 3;  // two words
  Q.backlog = Q.next_hist + 5;  // two words
  Q.phase = Q.next_hist + 7;
  Q.job_next = Q.next_hist + 8;
  char *ctl_end = m + kCtlWords * sizeof(Ctl);
  for (int t = 0; t < 2; ++t) {
    QType &T = Q.q[t];
    char *b = ctl_end + t * per_type;
    T.head = reinterpret_cast<Ctl *>(b);
    T.tail = T.head + K;
    T.rec = reinterpret_cast<Rec *>(b + 2 * size_t(K) * sizeof(Ctl));
    T.seq = reinterpret_cast<uint32_t *>(T.rec + slots);
  }
  Q.K = K;
  Q.log2cs = log2cs;
  Q.mask = uint32_t((size_t(1) << log2cs) - 1);
  return Q;
}

int queue_fresh(void *mem, int K, int log2cs, int sm_count, cudaStream_t st, std::string &err) {
  const QDev Q = queue_layout(mem, K, log2cs);
  cudaError_t e = cudaMemsetAsync(Q.dirty, 0, kKeptWords * sizeof(Ctl), st);
  if (e == cudaSuccess) {
    k_queue_init<<<sm_count * 4, 256, 0, st>>>(Q, Q.next_hist, 0, size_t(K) << log2cs, true);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    err = cudaGetErrorString(e);
    return DPM_ECUDA;
  }
  return DPM_OK;
}

int queue_launch(void *mem, int K, int log2cs, int log2use, const RunParams &R, uint64_t batch_size,
                 const dpm_run_opts &o, cudaStream_t st, cudaEvent_t start, std::string &err) {
  if (R.jobs && (R.T.flags & DPM_SAUTER)) {
    err = "the photoelectron angle option (DPM_SAUTER) runs in single runs only";
    return DPM_EINVAL;
  }
  if (R.jobs && (R.n_jobs < 1 || R.n_jobs > kSharedJobs)) {
    err = "a shared launch takes 1 to kSharedJobs jobs";
    return DPM_EINVAL;
  }
  QDev Q = queue_layout(mem, K, log2cs);
  const size_t cs = size_t(1) << log2use;
  Q.refill_min[0] = o.refill_min > 0 ? std::min(o.refill_min, 32) : DPM_REFILL_MIN_G;
  Q.refill_min[1] = o.refill_min > 0 ? std::min(o.refill_min, 32) : DPM_REFILL_MIN_E;
  const bool small = log2use < kFullFetchLog2;
  Q.guard[0] = uint32_t(cs >> (small ? 2 : DPM_PHASE_GUARD_SHIFT_G));
  Q.guard[1] = uint32_t(cs >> DPM_PHASE_GUARD_SHIFT_E);
  Q.phase_high[0] = (long long)K * (long long)(cs >> (small ? 3 : DPM_PHASE_HIGH_SHIFT_G));
  // at least one particle per shard: a phase that ended below 0 would never end
  Q.phase_low[0] = (long long)K * (long long)std::max(cs >> DPM_PHASE_LOW_SHIFT_G, decltype(cs)(1));
  Q.phase_high[1] = (long long)K * (long long)(cs >> DPM_PHASE_HIGH_SHIFT_E);
  Q.phase_low[1] = (long long)K * (long long)std::max(cs >> DPM_PHASE_LOW_SHIFT_E, decltype(cs)(1));
  Q.limit = uint32_t(cs - 64);
  if (o.queue_limit > 0) Q.limit = std::min<uint32_t>(Q.limit, uint32_t(o.queue_limit));
  const double tmo = o.timeout_s > 0 ? o.timeout_s : 20.0;
  Q.timeout_ns = (unsigned long long)(tmo * 1e9);
  // the whole launch: the wait bound plus 2 us per history (a hundred times the
  // cost of a 20 MeV electron history on this path)
  Q.deadline_ns = Q.timeout_ns + (unsigned long long)(double(R.n) * 2000.0);
  if (batch_size > 1) {
    int l = 0;
    while ((uint64_t(1) << l) < batch_size) ++l;
    Q.batch_mul = uint32_t(((uint64_t(1) << (31 + l)) + batch_size - 1) / batch_size);
    Q.batch_shift = uint32_t(l - 1);
  }
  k_queue_init<<<16, 256, 0, st>>>(Q, Q.next_hist, R.jobs ? 8 + R.n_jobs : 8, size_t(K) << log2cs, false);
  if (start) cudaEventRecord(start, st);
  const bool count = o.count_events != 0;
  const bool sauter = (R.T.flags & DPM_SAUTER) != 0;
  const bool pause = o.refill_pause >= 0;  // callers on queues below 2^kPauseMinLog2 slots pass -1 for 0
  Q.pause[0] = small ? 1 << 30 : pause ? DPM_REFILL_COOLDOWN : 0;
  Q.pause[1] = small ? 1 << 30 : 0;
  const size_t smem = R.jobs ? size_t(R.n_jobs) * sizeof(JobHot) : 0;
  queue_kernel(R.jobs != nullptr, count, sauter)<<<K, kQBlock, smem, st>>>(R, Q);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    err = cudaGetErrorString(e);
    return DPM_ECUDA;
  }
  return DPM_OK;
}

// Default shard capacity: 2^14 slots; 2^15 for a single electron-beam run,
// whose secondary (photon) phase then starts later and runs longer (20 MeV
// electrons +2 % on the slab phantom, +1.5 % on the 128^3 blobs; 6 MV photons
// -0.3 %, so photon beams keep 2^14).
int default_queue_log2(const RunParams &R) { return (!R.jobs && R.S.particle == 1) ? 15 : 14; }

int queue_prepare(QueueState &q, const dpm_run_opts &o, int sm_count, cudaStream_t st, int &K, int &log2cs, int &log2use,
                  std::string &err) {
  if (q.per_sm < 1) q.per_sm = queue_blocks_per_sm();
  if (q.per_sm < 1) {
    err = "occupancy query failed";
    return DPM_ECUDA;
  }
  const int bps = o.blocks_per_sm > 0 ? std::min(o.blocks_per_sm, q.per_sm) : q.per_sm;
  K = sm_count * bps;
  log2use = o.queue_log2 > 0 ? o.queue_log2 : 14;
  if (log2use < 7 || log2use > 20) {
    err = "queue_log2 must be in [7, 20]";
    return DPM_EINVAL;
  }
  // a layout with the same shards and room enough stays (photon and electron
  // beams, with their 2^14 and 2^15 slots, then take turns without a new one)
  log2cs = q.mem && q.K == K && q.log2_cap >= log2use ? q.log2_cap : log2use;
  const size_t bytes = queue_bytes(K, log2cs);
  if (q.bytes < bytes) {
    if (q.budget && q.in_use && *q.in_use - q.bytes + bytes > q.budget) {
      err = "device-memory budget of the context exceeded by the particle queues (" + std::to_string(bytes) +
            " bytes)";
      return DPM_ENOMEM;
    }
    if (q.mem) cudaFree(q.mem);
    if (q.in_use) *q.in_use -= q.bytes;
    q.mem = nullptr;
    q.bytes = 0;
    q.K = 0;
    cudaError_t e = cudaMalloc(&q.mem, bytes);
    if (e != cudaSuccess) {
      cudaGetLastError();
      err = std::string("queue allocation: ") + cudaGetErrorString(e);
      return DPM_ENOMEM;
    }
    q.bytes = bytes;
    if (q.in_use) *q.in_use += bytes;
  }
  if (q.K != K || q.log2_cap != log2cs) {
    q.K = 0;
    const int rc = queue_fresh(q.mem, K, log2cs, sm_count, st, err);
    if (rc) return rc;
    q.K = K;
    q.log2_cap = log2cs;
  }
  return DPM_OK;
}

int queue_run(QueueState &q, const RunParams &R, uint64_t batch_size, const dpm_run_opts &o, int sm_count,
              cudaStream_t st, cudaEvent_t start, std::string &err) {
  if (R.n > 0x7fffffffull) {
    err = "the queue kernel takes at most 2^31-1 histories per call";
    return DPM_EINVAL;
  }
  if (R.jobs && (R.n_jobs < 1 || R.n_jobs > kSharedJobs)) {
    err = "bad job count";
    return DPM_EINVAL;
  }
  int K = 0, log2cs = 0, log2use = 0;
  dpm_run_opts oq = o;
  if (oq.queue_log2 <= 0) oq.queue_log2 = default_queue_log2(R);
  const int rc = queue_prepare(q, oq, sm_count, st, K, log2cs, log2use, err);
  if (rc) return rc;
  return queue_launch(q.mem, K, log2cs, log2use, R, batch_size, o, st, start, err);
}

void queue_free(QueueState &q) {
  if (q.mem) cudaFree(q.mem);
  if (q.in_use) *q.in_use -= q.bytes;
  q.mem = nullptr;
  q.bytes = 0;
  q.K = 0;
}

}  // namespace dpm
