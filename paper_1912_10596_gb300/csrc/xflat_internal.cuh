// Internal device-side data structures of the bulb-model solver (not part of the C ABI).
//
// Work decomposition.  All instances' beams live in one set of SoA planes.  The beams of the whole
// problem are cut into G equal contiguous slices, one per persistent block; the intersection of a
// slice with an instance is a "piece".  A block processes its pieces one after the other and adds
// each piece's moments to its instance's fixed-point accumulators; after the device-wide barrier every
// block derives the next stage's constants from them in its set-up.  Only a step's final barrier (and the
// moment launch's) has a serial section: its last block runs the step bookkeeping before it releases the
// others.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace xflat {

constexpr int kMaxStages = 12;      // stage slots 0..11 (Richardson-controlled CF4: 11 stages)
constexpr int kStateRingDepth = 3;  // FP32 two-flavour bulb passes: state vectors in flight per thread
constexpr int kNM2 = 6;             // 2 flavours: j0 (3) and j1 (3) Bloch components
constexpr int kNM3 = 18;            // 3 flavours: j0 and j1, 9 reals each
constexpr int kNSC2 = 8;            // stage constants: mu*j0 (3), mu*j1 (3), lambda, R^2/r^2
constexpr int kNSC3 = 20;           // mu*j0 (9), mu*j1 (9), lambda, R^2/r^2
constexpr int kNMMax = 18;
constexpr int kNSCMax = 20;
// Blocks add their moment partials to one of kAccCopies copies of an instance's accumulators
// (block index mod kAccCopies), so the integer atomics of hundreds of blocks spread over several
// L2 lines instead of queueing on one; every reader sums the copies (exact integer sums).
constexpr int kAccCopies = 8;
// accumulator words: [stage slot][copy][component][2] per instance; FP64 kernels have one copy more, whose
// words hold the upper parts of partials of 8 and more (fx_add)
constexpr int acc_words_per_slot(size_t real_size) { return (kAccCopies + (real_size == 8 ? 1 : 0)) * kNMMax * 2; }
constexpr int acc_words_per_inst(size_t real_size) { return kMaxStages * acc_words_per_slot(real_size); }

enum Integrator : int { kRK4 = 0, kDP45 = 1, kLieRK4 = 2, kExpMid = 3, kLieAdaptive = 4 };
enum Matter : int { kMatterNone = 0, kMatterPower = 1, kMatterConst = 2, kMatterTable = 3 };
enum Geometry : int { kGeomBulb = 0, kGeomSingleAngle = 1, kGeomHomogeneous = 2 };
enum ShardMode : int { kShardOff = 0, kShardPass = 1, kShardSerialInit = 2, kShardSerialFinal = 3 };

// Instance constants, written by the host before a launch.
struct InstConst {
  uint64_t beam_off;        // first beam of the instance in the planes
  uint32_t n_beams;         // 2 * n_angle * n_energy
  uint32_t n_energy, n_angle;
  uint32_t e_off, a_off;    // offsets into the energy and angle tables
  uint32_t n_phi;           // azimuthal bins of the extended bulb model (n_angle counts u x phi)
  uint64_t div_magic;       // floor(2^40 / n_energy) + 1: q = (l * magic) >> 40 is l / n_energy
  double R2;                // R^2 (km^2)
  double mu_coef;           // mu(r) = mu_coef / r^2, includes the weight scale wscale
  double wscale;            // physical per-bin number luminosity of a unit table weight (1/s)
  double acc_unit;          // mixed kernels: value of one unit of the fixed-point moment sums (2^-S)
  float wmax, pad_wmax;     // mixed kernels: largest weight |du_j g_k| of a beam, in those units
  double lam_coef, power, lam_const, r_ref;   // lambda(r) = lam_coef (r_ref / r)^power
  const double* mtab;       // matter table: [mt_n][3] (r_i, lambda_i, exponent p_i of the interval
  int32_t mt_n;             // after r_i: lambda = lambda_i (r/r_i)^p_i), device memory, or null
  int32_t geom;             // Geometry
  uint32_t rec_start;       // first beam of the instance this handle integrates (beam shards; else 0):
                            // the block holding it records the stage moments and constants
  double mu_const;          // homogeneous geometry: the constant nu-nu strength mu0 (1/km)
  int32_t matter;
  int32_t adaptive;
  double B[3];              // 2 flavours: unit vacuum vector (sin 2th, 0, -cos 2th)
  double rtol, atol, h_min, h_max;
};

// Instance dynamics, owned by the device during a launch.
struct InstDyn {
  double r, h, r_end;       // current radius, next step size, target
  double r0_fixed, h_fixed; // fixed-step grid: r_n = r0_fixed + n h_fixed
  long long n_fixed, n_fixed_total;
  double err;               // last error norm
  double rs[kMaxStages];    // stage radii of the current step
  double xs[kMaxStages];    // R^2 / rs^2
  double mus[kMaxStages];   // mu(rs): nu-nu strength at the stage radii
  double lams[kMaxStages];  // lambda(rs): matter strength at the stage radii
  int32_t status, done, last, parity;
  int32_t geo_pending, pad_geo;   // stage geometry of the next step still to be computed
  unsigned long long accepted, rejected, stage_evals;
  double mom[kMaxStages][kNMMax];   // raw moments (weights normalised by wscale) per stage
  double sc[kMaxStages][kNSCMax];   // stage constants per stage
};

struct Piece {
  int32_t inst;
  uint32_t start;           // first local beam of the piece within the instance
  uint32_t len;             // beams in the piece
  uint32_t jj_lo;           // first combined angle index (species * n_angle + j) touched
  uint32_t n_jj;            // combined angle indices touched
  uint32_t pad;
};

struct Barrier {
  unsigned int count;
  unsigned int pad0[31];
  unsigned int gen;
  unsigned int pad1[31];
  unsigned long long passes;   // arrivals at the barriers without a serial section (pass_barrier)
  unsigned int pad3[30];
  int abort;
  int timeout_hits;
  unsigned int extra;       // test hook: additional arrivals expected
  // dynamic piece scheduling: the pass after barrier generation g (which steps by 2, bit 0 being a
  // flag) takes pieces from chunk[(g >> 1) & 1]; the last block at a barrier zeroes the counter
  // of the pass that follows it before the release
  unsigned int chunk[2];
  // checked build (-DXFLAT_BOUNDS): the first access found outside its allocation (site number,
  // byte offset from the allocation's start)
  int bounds_site;
  long long bounds_off;
  int pad2[24];
};

// Checked build: the allocations the step kernel's pass body reads and writes, by role.
struct Span {
  const char* lo;
  unsigned long long bytes;
};
enum SpanId : int { kSpanPlanes = 0, kSpanEscr, kSpanKst, kSpanEtab, kSpanU, kSpanDu, kSpanCount };

// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned int ld_acquire(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ int ld_acquire_int(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ uint32_t fast_div(uint32_t l, uint64_t magic) {
  return (uint32_t)(((uint64_t)l * magic) >> 40);
}

// Device-wide barrier.  Returns kBarLast in every thread of the one block that arrived last (that
// block must call barrier_release after its serial work), kBarReleased elsewhere after the
// release, or kBarAbort.  Every wait is bounded by timeout_ns: on expiry the block records
// XFLAT_ERR_TIMEOUT in *status_word, raises the abort flag and returns kBarAbort; a block that sees
// the abort flag while waiting also returns kBarAbort, so every block leaves the kernel.
enum BarrierResult : int { kBarReleased = 0, kBarLast = 1, kBarAbort = 2 };

__device__ __forceinline__ int barrier_arrive(Barrier* bar, unsigned int n_blocks,
                                             unsigned long long timeout_ns, int* status_word,
                                             int* s_flag, unsigned int* s_gen) {
  // *s_gen: in, the generation this block last saw; out (released blocks), the new one
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned int g = *s_gen;                 // generation of the last barrier this block passed
    __threadfence();                               // this block's writes before its arrival
    const unsigned int ticket = atomicAdd(&bar->count, 1u);
    const unsigned int expected = n_blocks + bar->extra;
    int res = (ticket == expected - 1) ? kBarLast : kBarReleased;
    unsigned int gnow = g;
    if (res == kBarLast) {
      __threadfence();                             // acquire: every other block's writes
    } else {
      const unsigned long long t0 = globaltimer_ns();
      while ((gnow = ld_acquire(&bar->gen)) == g) {   // acquire load: no further fence needed
        if (ld_acquire_int(&bar->abort)) { res = kBarAbort; break; }
        if (globaltimer_ns() - t0 > timeout_ns) {
          atomicAdd(&bar->timeout_hits, 1);
          atomicCAS(status_word, 0, 4 /* XFLAT_ERR_TIMEOUT */);
          atomicExch(&bar->abort, 1);
          res = kBarAbort;
          break;
        }
        __nanosleep(20);
      }
    }
    if (res == kBarReleased) *s_gen = gnow;
    *s_flag = res | (int)((gnow & 1u) << 4);       // bit 4: the flag carried by the release
  }
  __syncthreads();
  return *s_flag;
}

// Release the barrier (last block only, after its serial work; every thread that wrote shared
// results must have executed __threadfence() before the __syncthreads here).  The generation word
// advances by 2 and its low bit carries one flag to every waiting block (the kernels use it for
// "every instance finished"), so a released block learns it from the load that saw the release.
// The count is reset before the new generation is published with release ordering.
__device__ __forceinline__ void barrier_release(Barrier* bar, int flag, unsigned int* s_gen) {
  __syncthreads();
  if (threadIdx.x == 0) {
    bar->count = 0;
    const unsigned int ng = ((*s_gen & ~1u) + 2u) | (flag ? 1u : 0u);
    *s_gen = ng;
    unsigned int old;
    asm volatile("atom.release.gpu.global.exch.b32 %0, [%1], %2;" : "=r"(old) : "l"(&bar->gen), "r"(ng) : "memory");
  }
}

// Device-wide barrier without a serial section: every block adds one to a counter that only grows and
// waits for the count itself, so the way from the last arrival to the waiting blocks is one hop (the last
// block neither learns that it is the last nor opens a second word).  *s_next: the count at which the
// barrier before this one was complete (pass_barrier_base at the kernel's start), advanced here.
// expected: arrivals a barrier waits for (the blocks, or more under the test hook).  Returns false in every
// thread on a timeout or an abort, as barrier_arrive.  (GB300, 152 blocks, from the last block's end of work
// to the first start after it: 1.8 us with a last-block release, 1.0 us so; and the blocks leave it within 0.3 us of one
// another instead of 0.9.  24 mixed DP45 steps of 159,594 beams 1665 -> 1491 us, 16 FP64 RK4 steps of 4096
// beams 707 -> 647 us, 12 mixed steps of 4M beams 2.65 -> 2.55 ms.)
__device__ __forceinline__ unsigned long long pass_barrier_base(const Barrier* bar, unsigned int n_blocks) {
  // whole barriers only have completed before this block's first arrival
  const unsigned long long v = ld_acquire64(&bar->passes);
  return v - v % n_blocks;
}
__device__ __forceinline__ bool pass_barrier(Barrier* bar, unsigned int n_blocks, unsigned int expected,
                                             unsigned long long timeout_ns, int* status_word, int* s_flag,
                                             unsigned long long* s_next) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long base = *s_next, target = base + expected;
    *s_next = base + n_blocks;
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(&bar->passes), "l"(1ull) : "memory");
    int res = kBarReleased;
    unsigned long long t0 = 0;
    for (unsigned int poll = 1; ld_acquire64(&bar->passes) < target; ++poll) {
      if (poll % 16u != 0) continue;
      if (ld_acquire_int(&bar->abort)) { res = kBarAbort; break; }
      const unsigned long long now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      if (now - t0 > timeout_ns) {
        atomicAdd(&bar->timeout_hits, 1);
        atomicCAS(status_word, 0, 4 /* XFLAT_ERR_TIMEOUT */);
        atomicExch(&bar->abort, 1);
        res = kBarAbort;
        break;
      }
    }
    *s_flag = res;
  }
  __syncthreads();
  return *s_flag != kBarAbort;
}

}  // namespace xflat
