// dpm_history.cu -- one-history-per-thread transport (the paper's own layout,
// Sec. 2.2: each thread follows a source particle and all its secondaries
// with a private stack), the batch fold and the dose normalisation.
#include <cuda_runtime.h>

#include "dpm_device.cuh"
#include "dpm_kernels.h"

namespace dpm {

// The particle that emission o of p creates: at p's place, with its own random
// stream.
template <class Real>
__device__ __forceinline__ PartT<Real> secondary(const PartT<Real> &p, const EmissionT<Real> &o) {
  PartT<Real> c = p;
  c.type = o.type;
  c.E = o.E;
  c.u = o.u;
  c.v = o.v;
  c.w = o.w;
  c.id_lo = o.id_lo;
  c.id_hi = o.id_hi;
  c.ctr = 0;
  return c;
}

// Tally sink with run-length coalescing: consecutive deposits of one thread
// into the same voxel are summed in a register and issued as one 64-bit
// atomic add (exact, order-independent fixed point, 2^-32 MeV).  Real: the
// transport's arithmetic (float; double for the precision ablation).
template <class Real>
struct HistSinkT {
  static constexpr bool kSauter = true;  // DPM_SAUTER compiled in
  const RunParamsT<Real> &R;
  unsigned long long *slab = nullptr;
  int pend_v = -1;
  long long pend_q = 0;
  long long cnt[C_N];
  int err = 0;
  PartT<Real> *stack;
  int sp = 0, cap;

  __device__ HistSinkT(const RunParamsT<Real> &r, PartT<Real> *st, int c) : R(r), stack(st), cap(c) {
#pragma unroll
    for (int i = 0; i < C_N; ++i) cnt[i] = 0;
  }
  __device__ __forceinline__ static long long fx(Real e) { return Num<Real>::round_ll(e * Real(4294967296.0f)); }
  // energy counters (coarser quantum, see kCounterScale)
  __device__ __forceinline__ static long long fxc(Real e) { return Num<Real>::round_ll(e * Real(kCounterScaleF)); }
  __device__ __forceinline__ void flush() {
    if (pend_v >= 0 && pend_q != 0) {
      atomicAdd(slab + pend_v, (unsigned long long)pend_q);
      ++cnt[C_ATOM];
    }
    pend_v = -1;
    pend_q = 0;
  }
  __device__ __forceinline__ void deposit(int v, Real dE) {
    const long long q = fx(dE);
    if (v == pend_v) {
      pend_q += q;
    } else {
      flush();
      pend_v = v;
      pend_q = q;
    }
  }
  __device__ __forceinline__ void leave(int) {}
  __device__ __forceinline__ void escape(Real E) { cnt[C_ESC] += fxc(E); }
  Real held_[3];
  __device__ __forceinline__ void hold(Real R, Real S, Real Sigma) {
    held_[0] = R;
    held_[1] = S;
    held_[2] = Sigma;
  }
  static __device__ __forceinline__ bool hard_waits() { return false; }
  __device__ __forceinline__ Real held_range() const { return held_[0]; }
  __device__ __forceinline__ Real held_power() const { return held_[1]; }
  __device__ __forceinline__ Real held_sigma() const { return held_[2]; }
  // secondary o of particle p
  __device__ __forceinline__ void push(const PartT<Real> &p, const EmissionT<Real> &o) {
    ++cnt[C_PUSH];
    if (sp < cap) {
      stack[sp++] = secondary(p, o);
    } else {
      err |= ERR_OVERFLOW;
      cnt[C_ESC] += fxc(o.E + (o.type == POSITRON ? Real(2) * Num<Real>::mc2 : Real(0)));
    }
  }
  __device__ __forceinline__ void error(int e) { err |= e; }
  __device__ __forceinline__ void count_step() { ++cnt[C_ESTEP]; }
  __device__ __forceinline__ void count_flight() { ++cnt[C_GFLIGHT]; }
  __device__ __forceinline__ void count_interaction() { ++cnt[C_GINT]; }
};
using HistSink = HistSinkT<float>;

template <class RP>
__device__ void reduce_counters(const long long *cnt, int err, const RP &R) {
#pragma unroll
  for (int i = 0; i < C_N; ++i) {
    long long v = cnt[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && v != 0) atomicAdd(R.counters + i, (unsigned long long)v);
  }
  int e = err;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e |= __shfl_down_sync(0xffffffffu, e, o);
  if ((threadIdx.x & 31) == 0 && e) atomicOr(R.err, e);
}

constexpr int kHistStack = 64;

// Transport every particle on the thread's stack, secondaries included.
template <class Real, class Sink>
__device__ __forceinline__ void run_stack(const RunParamsT<Real> &R, Sink &s) {
  while (s.sp > 0) {
    PartT<Real> q = s.stack[--s.sp];
    const bool photon = q.type == PHOTON;
    uint32_t cap = photon ? kMaxPhotonBlocks : kMaxElectronBlocks;
    Real E_seen = q.E;
    EmissionT<Real> o;
    for (;;) {
      o.kind = EM_NONE;
      const bool alive = (q.type & CHAIN)      ? chain_step(q, R, s, o)
                         : photon              ? photon_flight(q, R, s, o)
                                               : electron_step(q, R, s, o);
      if (o.kind != EM_NONE && settle(q, o, R, s)) s.push(q, o);
      if (!alive) break;
      if (q.ctr >= cap) {
        if (photon && q.E != E_seen) {  // a photon that has scattered since: as many again
          E_seen = q.E;
          cap += kMaxPhotonBlocks;
          continue;
        }
        s.error(ERR_STEPCAP);
        s.deposit(vox(q, R.P), q.E);
        break;
      }
    }
  }
}

// 8 resident blocks of 128 threads cap the registers at 64: the extra spills cost
// less than the doubled occupancy gains (+26 % on 6 MV, +30 % on 20 MeV electrons
// against 128 registers).
template <class Real>
__global__ void __launch_bounds__(128, 8) k_history(const __grid_constant__ RunParamsT<Real> R, uint64_t batch_size) {
  PartT<Real> stack[kHistStack];
  HistSinkT<Real> s(R, stack, kHistStack);
  const size_t V = size_t(R.P.nx) * R.P.ny * R.P.nz;
  const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
  for (uint64_t hl = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; hl < R.n; hl += stride) {
    s.slab = R.slabs + (hl / batch_size) * V;
    PartT<Real> p;
    const bool hit = make_primary(p, R, uint32_t(hl));
    s.cnt[C_EMIT] += HistSinkT<Real>::fxc(p.E);
    if (!hit) {
      s.cnt[C_MISS] += HistSinkT<Real>::fxc(p.E);
      continue;
    }
    s.sp = 0;
    s.stack[s.sp++] = p;
    run_stack(R, s);
    s.flush();
  }
  reduce_counters(s.cnt, s.err, R);
}

template <class Real>
static void launch_history_t(const RunParamsT<Real> &R, uint64_t batch_size, int sm_count, cudaStream_t st) {
  const int block = 128;  // the kernel's launch bound
  const uint64_t need = (R.n + block - 1) / block;
  const uint64_t cap = uint64_t(sm_count) * 16;
  const int grid = int(need < cap ? need : cap);
  cudaFuncSetAttribute(k_history<Real>, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
  k_history<Real><<<grid > 0 ? grid : 1, block, 0, st>>>(R, batch_size);
}

void launch_history(const RunParams &R, uint64_t batch_size, int sm_count, int block, cudaStream_t st) {
  (void)block;
  launch_history_t(R, batch_size, sm_count, st);
}

void launch_history_f64(const RunParamsT<double> &R, uint64_t batch_size, int sm_count, cudaStream_t st) {
  launch_history_t(R, batch_size, sm_count, st);
}

// ---------------------------------------------------------------------------
// The paper's own tally (Sec. 2.4), kept as an ablation of the exact one above.
// Each thread holds a sparse dose counter of kPaperCounter (voxel, energy)
// entries in its own memory: a deposit adds to its voxel's entry (searched
// from the newest, since consecutive deposits usually share a voxel) or opens
// a new one.  When the history ends, or the counter is full, the entries are
// added to a float dose array with atomic float additions.  kCas emulates the
// float addition with a compare-and-swap loop on the 32-bit word, the scheme
// the paper uses on a GPU without float atomics; otherwise the native float
// atomic add is used.  Float sums depend on the order of the additions, so
// this tally is not reproducible bit for bit; k_f32_to_fixed rounds it to
// the fixed-point slabs for the common fold.
// ---------------------------------------------------------------------------
constexpr int kPaperCounter = 128;
constexpr int kCasTries = 1 << 20;  // a bound on one CAS addition's retries

template <bool kCas>
__device__ __forceinline__ bool add_f32(float *a, float x) {
  if (!kCas) {
    atomicAdd(a, x);
    return true;
  }
  unsigned int *w = reinterpret_cast<unsigned int *>(a);
  unsigned int old = *w;
  for (int t = 0; t < kCasTries; ++t) {
    const unsigned int seen = old;
    old = atomicCAS(w, seen, __float_as_uint(__uint_as_float(seen) + x));
    if (old == seen) return true;
  }
  return false;
}

template <bool kCas>
struct PaperSink {
  static constexpr bool kSauter = false;
  const RunParams &R;
  float *fslab = nullptr;
  int n = 0;
  int lv[kPaperCounter];
  float le[kPaperCounter];
  long long cnt[C_N];
  int err = 0;
  Part *stack;
  int sp = 0, cap;

  __device__ PaperSink(const RunParams &r, Part *st, int c) : R(r), stack(st), cap(c) {
#pragma unroll
    for (int i = 0; i < C_N; ++i) cnt[i] = 0;
  }
  __device__ void flush() {
    for (int i = 0; i < n; ++i) {
      if (!add_f32<kCas>(fslab + lv[i], le[i])) err |= ERR_TIMEOUT;
    }
    cnt[C_ATOM] += n;
    n = 0;
  }
  __device__ void deposit(int v, float dE) {
    for (int i = n - 1; i >= 0; --i) {
      if (lv[i] == v) {
        le[i] += dE;
        return;
      }
    }
    if (n == kPaperCounter) flush();
    lv[n] = v;
    le[n] = dE;
    ++n;
  }
  // run counters exactly as HistSink keeps them, so that the energy balance
  // of both tallies is the same
  __device__ __forceinline__ void leave(int) {}
  __device__ __forceinline__ void escape(float E) { cnt[C_ESC] += HistSink::fxc(E); }
  float held_[3];
  __device__ __forceinline__ void hold(float R, float S, float Sigma) {
    held_[0] = R;
    held_[1] = S;
    held_[2] = Sigma;
  }
  static __device__ __forceinline__ bool hard_waits() { return false; }
  __device__ __forceinline__ float held_range() const { return held_[0]; }
  __device__ __forceinline__ float held_power() const { return held_[1]; }
  __device__ __forceinline__ float held_sigma() const { return held_[2]; }
  __device__ __forceinline__ void push(const Part &p, const Emission &o) {
    ++cnt[C_PUSH];
    if (sp < cap) {
      stack[sp++] = secondary(p, o);
    } else {
      err |= ERR_OVERFLOW;
      cnt[C_ESC] += HistSink::fxc(o.E + (o.type == POSITRON ? 2.f * kMc2f : 0.f));
    }
  }
  __device__ __forceinline__ void error(int e) { err |= e; }
  __device__ __forceinline__ void count_step() { ++cnt[C_ESTEP]; }
  __device__ __forceinline__ void count_flight() { ++cnt[C_GFLIGHT]; }
  __device__ __forceinline__ void count_interaction() { ++cnt[C_GINT]; }
};

template <bool kCas>
__global__ void __launch_bounds__(128) k_history_paper(const __grid_constant__ RunParams R, uint64_t batch_size,
                                                       float *fslabs) {
  Part stack[kHistStack];
  PaperSink<kCas> s(R, stack, kHistStack);
  const size_t V = size_t(R.P.nx) * R.P.ny * R.P.nz;
  const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
  for (uint64_t hl = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; hl < R.n; hl += stride) {
    s.fslab = fslabs + (hl / batch_size) * V;
    Part p;
    const bool hit = make_primary(p, R, uint32_t(hl));
    s.cnt[C_EMIT] += HistSink::fxc(p.E);
    if (!hit) {
      s.cnt[C_MISS] += HistSink::fxc(p.E);
      continue;
    }
    s.sp = 0;
    s.stack[s.sp++] = p;
    run_stack(R, s);
    s.flush();
  }
  reduce_counters(s.cnt, s.err, R);
}

// Float dose slabs to the fixed-point slabs (nearest multiple of 2^-32 MeV).
__global__ void k_f32_to_fixed(const float *f, unsigned long long *slabs, size_t n) {
  for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x)
    slabs[i] = (unsigned long long)__double2ll_rn(double(f[i]) * 4294967296.0);
}

void launch_history_paper(const RunParams &R, uint64_t batch_size, bool cas, float *fslabs, size_t n_slab,
                          int sm_count, cudaStream_t st) {
  const int block = 128;
  const uint64_t need = (R.n + block - 1) / block;
  const uint64_t cap = uint64_t(sm_count) * 16;
  const int grid = int(need < cap ? need : cap);
  if (cas) {
    cudaFuncSetAttribute(k_history_paper<true>, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
    k_history_paper<true><<<grid > 0 ? grid : 1, block, 0, st>>>(R, batch_size, fslabs);
  } else {
    cudaFuncSetAttribute(k_history_paper<false>, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
    k_history_paper<false><<<grid > 0 ? grid : 1, block, 0, st>>>(R, batch_size, fslabs);
  }
  const size_t cgrid = (n_slab + 255) / 256 < size_t(sm_count) * 8 ? (n_slab + 255) / 256 : size_t(sm_count) * 8;
  k_f32_to_fixed<<<cgrid > 0 ? int(cgrid) : 1, 256, 0, st>>>(fslabs, R.slabs, n_slab);
}

// Sum the batch slabs of one run into S1 (exact int64) and Q = sum_b d_b^2/n_b.
// The squares of all batches but the last, which have the same n_b, are summed
// exactly in 128-bit integers and rounded once per voxel.  FP64 is scarce on
// this chip (2 operations per SM and cycle): a conversion, two products and a
// sum in FP64 per entry took 0.82 ms on 50 slabs of 128^3 voxels, where reading
// them takes 0.13 ms.  Now 0.18 ms there, and 0.096 -> 0.029 ms on 50 slabs
// of 61x61x60 (in L2).  Groups of entries that are all zero, most of a large
// phantom's, are skipped.
__global__ void __launch_bounds__(256, 4)
    k_fold(const unsigned long long *slabs, int nb, size_t V, double inv_n, double inv_n_last, long long *S1, double *Q) {
  constexpr int kAhead = 10;  // loads in flight per thread
  for (size_t v = size_t(blockIdx.x) * blockDim.x + threadIdx.x; v < V; v += size_t(gridDim.x) * blockDim.x) {
    const unsigned long long *p = slabs + v;
    const long long last = (long long)p[size_t(nb - 1) * V];
    long long s = last;
    unsigned long long sq_lo = 0, sq_hi = 0;
    for (int b0 = 0; b0 < nb - 1; b0 += kAhead) {
      long long d[kAhead], any = 0;
#pragma unroll
      for (int k = 0; k < kAhead; ++k) d[k] = b0 + k < nb - 1 ? (long long)p[size_t(b0 + k) * V] : 0;
#pragma unroll
      for (int k = 0; k < kAhead; ++k) any |= d[k];
      if (any != 0) {
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
          s += d[k];
          const unsigned long long m = (unsigned long long)(d[k] < 0 ? -d[k] : d[k]);
          const unsigned long long lo = m * m;
          sq_lo += lo;
          sq_hi += __umul64hi(m, m) + (sq_lo < lo ? 1ull : 0ull);
        }
      }
    }
    if (s != 0 || last != 0 || (sq_lo | sq_hi) != 0) {
      const double dl = double(last);
      S1[v] += s;
      Q[v] += (double(sq_hi) * 18446744073709551616.0 + double(sq_lo)) * inv_n + dl * dl * inv_n_last;
    }
  }
}

void launch_fold(const unsigned long long *slabs, int nb, size_t V, double inv_n, double inv_n_last, long long *S1, double *Q,
                 int sm_count, cudaStream_t st) {
  const size_t need = (V + 255) / 256;
  const size_t cap = size_t(sm_count) * 8;
  const int grid = int(need < cap ? need : cap);
  k_fold<<<grid > 0 ? grid : 1, 256, 0, st>>>(slabs, nb, V, inv_n, inv_n_last, S1, Q);
}

// Density and material of each voxel in one 8-byte word, as the transport reads
// them: one access and one sector per step or flight instead of two (with the
// photon coefficient's table of its own 1 % of the transport time).
__global__ void k_pack_voxels(const uint8_t *mat, const float *rho, size_t V, float2 *vox) {
  for (size_t v = size_t(blockIdx.x) * blockDim.x + threadIdx.x; v < V; v += size_t(gridDim.x) * blockDim.x)
    vox[v] = make_float2(rho[v], __int_as_float(mat[v]));
}

void launch_pack_voxels(const uint8_t *mat, const float *rho, size_t V, float2 *vox, int sm_count, cudaStream_t st) {
  const size_t need = (V + 255) / 256;
  const size_t cap = size_t(sm_count) * 8;
  const int grid = int(need < cap ? need : cap);
  k_pack_voxels<<<grid > 0 ? grid : 1, 256, 0, st>>>(mat, rho, V, vox);
}

// Validity and largest densities of a phantom's arrays: out[m] becomes the
// largest density (as bits, which order like positive floats) of material m, and
// out[DPM_MAX_MAT] nonzero if an index is out of range or a density not positive
// and finite.  The host's scan of 128^3 voxels took 2.6 of the 2.8 ms in which a
// resident phantom got new contents.
__global__ void k_scan_voxels(const uint8_t *mat, const float *rho, size_t V, unsigned *out) {
  __shared__ unsigned s_max[DPM_MAX_MAT + 1];
  if (threadIdx.x <= DPM_MAX_MAT) s_max[threadIdx.x] = 0;
  __syncthreads();
  for (size_t v = size_t(blockIdx.x) * blockDim.x + threadIdx.x; v < V; v += size_t(gridDim.x) * blockDim.x) {
    const unsigned m = mat[v];
    const float r = rho[v];
    const bool ok = m < DPM_MAX_MAT && r > 0.f && r <= 3.402823466e38f;  // not NaN, not infinite
    const unsigned k = ok ? m : DPM_MAX_MAT, bits = ok ? __float_as_uint(r) : 1u;
    if (bits > *(volatile unsigned *)&s_max[k]) atomicMax(&s_max[k], bits);
  }
  __syncthreads();
  if (threadIdx.x <= DPM_MAX_MAT && s_max[threadIdx.x]) atomicMax(out + threadIdx.x, s_max[threadIdx.x]);
}

void launch_scan_voxels(const uint8_t *mat, const float *rho, size_t V, unsigned *out, int sm_count, cudaStream_t st) {
  cudaMemsetAsync(out, 0, (DPM_MAX_MAT + 1) * sizeof(unsigned), st);
  const size_t need = (V + 1023) / 1024;  // four voxels per thread
  const size_t cap = size_t(sm_count) * 8;
  const int grid = int(need < cap ? need : cap);
  k_scan_voxels<<<grid > 0 ? grid : 1, 256, 0, st>>>(mat, rho, V, out);
}

// Sum of the integer tally over the voxels, exact: the high (signed) and low
// 32-bit halves apart, neither of which can overflow 64 bits below 2^32 voxels
// (the largest phantom has fewer).  out[0] += high, out[1] += low.
__global__ void k_sum_tally(const long long *S1, size_t V, unsigned long long *out) {
  long long hi = 0, lo = 0;
  for (size_t v = size_t(blockIdx.x) * blockDim.x + threadIdx.x; v < V; v += size_t(gridDim.x) * blockDim.x) {
    const long long x = S1[v];
    hi += x >> 32;  // arithmetic shift: floor(x / 2^32)
    lo += x & 0xffffffffll;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    hi += __shfl_down_sync(0xffffffffu, hi, o);
    lo += __shfl_down_sync(0xffffffffu, lo, o);
  }
  if ((threadIdx.x & 31) == 0 && (hi | lo) != 0) {
    atomicAdd(out, (unsigned long long)hi);
    atomicAdd(out + 1, (unsigned long long)lo);
  }
}

void launch_sum_tally(const long long *S1, size_t V, unsigned long long *out, int sm_count, cudaStream_t st) {
  cudaMemsetAsync(out, 0, 2 * sizeof(unsigned long long), st);
  const size_t need = (V + 1023) / 1024;  // four voxels per thread
  const size_t cap = size_t(sm_count) * 4;
  const int grid = int(need < cap ? need : cap);
  k_sum_tally<<<grid > 0 ? grid : 1, 256, 0, st>>>(S1, V, out);
}

// Dose (Gy per history) and its standard error from the batch statistics:
// per-history variance (Q - S1^2/n)/(B - 1), sigma of the mean sqrt(var/n).
// FP64 bound (2 operations per SM and cycle), so it takes few of them: none for
// untouched voxels (most of a large phantom); S1/n as S1 r_n (r_n = 1/n) for the
// dose and, in one fused operation whose rounding the difference Q - S1 (S1/n)
// keeps small, for the variance; one factor r_v = 1/((B - 1) n); and the division
// by the density only where it differs from the thread's voxel before (128^3
// voxels with half of them touched: 0.19 -> 0.085 ms).
__global__ void k_normalize(const long long *S1, const double *Q, const float2 *vox, size_t V, double r_n, double r_v,
                            double conv_1, double *dose, double *sigma) {
  float rho = 1.f;
  double conv = conv_1;
  for (size_t v = size_t(blockIdx.x) * blockDim.x + threadIdx.x; v < V; v += size_t(gridDim.x) * blockDim.x) {
    const long long s = S1[v];
    const double qv = Q[v];
    double d = 0.0, sg = 0.0;
    if (s != 0 || qv != 0.0) {
      const float r = vox[v].x;
      if (r != rho) {
        rho = r;
        conv = conv_1 / double(r);
      }
      const double s1 = double(s), mean = s1 * r_n;
      d = mean * conv;
      const double x = fma(-s1, mean, qv);
      if (x > 0.0) sg = sqrt(x * r_v) * conv;
    }
    if (dose) dose[v] = d;
    if (sigma) sigma[v] = sg;
  }
}

void launch_normalize(const long long *S1, const double *Q, const float2 *vox, size_t V, double n, double B,
                      double vox_cm3, double *dose, double *sigma, int sm_count, cudaStream_t st) {
  const size_t need = (V + 255) / 256;
  const size_t cap = size_t(sm_count) * 8;
  const int grid = int(need < cap ? need : cap);
  const double r_n = n > 0 ? 1.0 / n : 0.0, r_v = n > 0 && B > 1 ? 1.0 / ((B - 1.0) * n) : 0.0;
  k_normalize<<<grid > 0 ? grid : 1, 256, 0, st>>>(S1, Q, vox, V, r_n, r_v, kMeVtoJ / (vox_cm3 * 1e-3) / kTallyScale, dose,
                                                   sigma);
}

// D_max search for the stop rule: a 64-bit key (dose as float bits, which order
// like the values for non-negative doses, above the voxel index) reduced with
// atomicMax; then one thread evaluates dose and sigma at the winner.  The dose
// takes an FP64 division, so only voxels that may win get it: those within 4e-6
// of the block's largest single-precision estimate, whose own error is below
// 5e-7 (128^3 voxels, most of them in a 6 MV field: 0.10 -> 0.05 ms).
// (Densities below 1e-30, whose estimate would not hold, always get it.)
__global__ void k_dmax_key(const long long *S1, const float2 *vox, size_t V, double vox_cm3,
                           unsigned long long *key) {
  __shared__ float s_top[8];
  const size_t v0 = size_t(blockIdx.x) * blockDim.x + threadIdx.x, stride = size_t(gridDim.x) * blockDim.x;
  float top = 0.f;
  for (size_t v = v0; v < V; v += stride) {
    const long long s = S1[v];
    if (s > 0 && vox[v].x > 1e-30f) top = fmaxf(top, __fdividef(__ll2float_rn(s), vox[v].x));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_down_sync(0xffffffffu, top, o));
  if ((threadIdx.x & 31) == 0) s_top[threadIdx.x >> 5] = top;
  __syncthreads();
  for (int w = 0; w < 8; ++w) top = fmaxf(top, s_top[w]);
  top = __shfl_sync(0xffffffffu, top, 0) * (1.f - 4e-6f);
  unsigned long long best = 0;
  for (size_t v = v0; v < V; v += stride) {
    const long long s = S1[v];
    if (s <= 0 || (vox[v].x > 1e-30f && __fdividef(__ll2float_rn(s), vox[v].x) < top)) continue;
    const double s1 = double(s);
    const float dose = float(s1 * kMeVtoJ / (double(vox[v].x) * vox_cm3 * 1e-3));
    const unsigned long long k = (uint64_t(__float_as_uint(dose)) << 32) | uint64_t(uint32_t(v));
    best = k > best ? k : best;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long other = __shfl_down_sync(0xffffffffu, best, o);
    best = other > best ? other : best;
  }
  if ((threadIdx.x & 31) == 0 && best) atomicMax(key, best);
}

__global__ void k_dmax_eval(const long long *S1, const double *Q, const float2 *vox, double n, double B,
                            double vox_cm3, const unsigned long long *key, double *out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  out[0] = out[1] = 0.0;
  out[2] = -1.0;
  if (*key == 0 || n <= 0) return;
  const size_t v = size_t(uint32_t(*key));
  const double s1 = double(S1[v]);
  const double conv = kMeVtoJ / (double(vox[v].x) * vox_cm3 * 1e-3) / kTallyScale;
  const double var = B > 1.0 ? fmax(Q[v] - s1 * s1 / n, 0.0) / (B - 1.0) : 0.0;
  out[0] = s1 / n * conv;
  out[1] = sqrt(var / n) * conv;
  out[2] = double(v);
}

void launch_dmax(const long long *S1, const double *Q, const float2 *vox, size_t V, double n, double B, double vox_cm3,
                 unsigned long long *key, double *out, int sm_count, cudaStream_t st) {
  cudaMemsetAsync(key, 0, sizeof(unsigned long long), st);
  const size_t need = (V + 1023) / 1024;  // four voxels per thread
  const size_t cap = size_t(sm_count) * 8;
  const int grid = int(need < cap ? need : cap);
  k_dmax_key<<<grid > 0 ? grid : 1, 256, 0, st>>>(S1, vox, V, vox_cm3, key);
  k_dmax_eval<<<1, 32, 0, st>>>(S1, Q, vox, n, B, vox_cm3, key, out);
}

}  // namespace dpm
