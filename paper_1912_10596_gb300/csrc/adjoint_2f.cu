// Discrete adjoint of classical RK4 for the two-flavour bulb model, FP64.
//
// Forward map (Sec. 2, Eq. eom in the Bloch form of the step kernel): every beam b obeys
// ds_b/dr = K_b x s_b with K_b = q_b [eta omega_k B(theta_v) + lambda(r) z + mu(r) (D + t2_b J1)],
// q = 1/cos th_b, t2 = 1 - cos th_b, and the moments D = sum_b w_b t1_b s_b, J1 = sum_b w_b s_b,
// t1 = 1/cos - 1, w_b = du_j g_{sigma,k}.  Objective: J = sum over nu beams of
// du_j objw_k (1 + s_z)/2, the number-flux weighted mean survival probability.
//
// Adjoint of one evaluation k = f(s) with cotangent v (per beam):
//   p_b = s_b x v_b                        (adjoint of K_b)
//   Dbar = mu sum_b q_b p_b,  J1bar = mu sum_b t1_b p_b    (two grid reductions of 3-vectors)
//   sbar_b = v_b x K_b + w_b (t1_b Dbar + J1bar)
//   dJ/dw_b      += s_b . (t1_b Dbar + J1bar)
//   dJ/dtheta_v  += q_b eta omega_k p_b . dB/dtheta
// and RK4 is reversed stage by stage (a' the adjoint of the step's result):
//   v4 = h/6 a',  v3 = h/3 a' + h sbar4,  v2 = h/3 a' + h/2 sbar3,  v1 = h/6 a' + h/2 sbar2,
//   a = a' + sbar4 + sbar3 + sbar2 + sbar1.
//
// What bounds it: FP64 operations on GB300's two-lane pipe and the fixed time of a pass (12 a step).  So
// everything that the beams of an angle row share is tabulated once a step and stage (AdjRow, AdjBack: an
// assembled K is two FMAs), moments are summed within rows, reductions spread over the lanes, and the
// next stage's strengths are computed beside the sum over blocks.  200 E x 400 u, 128 steps, K = 64:
// 43.1 ms with per-beam assembly and five geometries a pass, 32.1 ms so (30.0 with grid_reduce as it is).
//
// Memory: the forward launch stores the state every K steps (checkpoints); each backward launch
// re-runs one segment of K steps forward from its checkpoint, storing every step's start state and
// stage constants, then runs the segment's steps backwards.  Every pass over the beams ends in a
// device-wide barrier, after which every block sums the block partials in block order (deterministic).
#include "adjoint.cuh"
#include "step_kernel.cuh"

namespace xflat {
namespace {

constexpr int kAdjSlots = 5;         // stages whose rows are tabulated at a time
constexpr int kAdjRows = 64;         // angle rows per block the tables hold

// What the beams of an angle row share at a stage: the geometry (q = 1/cos th, t1 = 1/cos th - 1,
// t2 = 1 - cos th), and K = eta omega (qb0, 0, qb2) + g.
struct AdjRow { double q, t1, t2, qb0, qb2, g[3]; };
// ... and at the stage whose adjoint is finished: brd = du (t1 Dbar + J1bar), and q dB/dtheta.
struct AdjBack { double brd[3], qd0, qd2; };

struct AdjShared {
  AdjRow row[kAdjSlots][kAdjRows];
  AdjBack back[kAdjRows];
  double scratch[32 * 6];
  double tot[8];
  double str[2];                        // mu, lambda of the formed stage (forward)
  double scf[kAdjStageVals];            // constants of the stage finished in this pass
  double scs[4][kAdjStageVals];         // constants of the formed stage's step (backward: all 4)
  double gl[8];                         // broadcast adjoint moments of the finished stage
  int flag;
  unsigned int reduces;                 // grid_reduce calls of this launch (the partials' buffer)
  unsigned long long pass_next;         // pass_barrier's count
};

__device__ __forceinline__ void row_geometry(const AdjParams& p, uint32_t jj, double x, AdjRow& r) {
  const uint32_t j = jj >= p.n_angle ? jj - p.n_angle : jj;
  const Geo g = geometry(p.u[j], x);
  r.q = g.q;
  r.t1 = g.t1;
  r.t2 = g.t2;
  r.qb0 = g.q * p.ic.B[0];
  r.qb2 = g.q * p.ic.B[2];
}
// sc: mu D, mu J1, lambda
__device__ __forceinline__ void row_coupling(const double* sc, AdjRow& r) {
  r.g[0] = r.q * (sc[0] + r.t2 * sc[3]);
  r.g[1] = r.q * (sc[1] + r.t2 * sc[4]);
  r.g[2] = r.q * (sc[6] + sc[2] + r.t2 * sc[5]);
}
__device__ __forceinline__ AdjBack row_back(const AdjParams& p, uint32_t jj, const AdjRow& r, const double* gl) {
  const double du = p.du[jj >= p.n_angle ? jj - p.n_angle : jj];
  const double c2 = -p.ic.B[2], s2 = p.ic.B[0];              // B = (sin 2th, 0, -cos 2th)
  AdjBack b;
  for (int i = 0; i < 3; ++i) b.brd[i] = du * (r.t1 * gl[i] + gl[3 + i]);
  b.qd0 = r.q * (2.0 * c2);                                   // dB/dtheta = (2 cos 2th, 0, 2 sin 2th)
  b.qd2 = r.q * (2.0 * s2);
  return b;
}

// This block's beams [b0, b1), its rows from row0 on (tab: they fit the tables; the same in every thread.
// If not, the row values are computed per beam), and this thread's share: each warp a contiguous run, so
// that a thread stays in one row for many beams (row sums of the moments, as in the step kernel).
struct AdjShare {
  uint32_t b0, b1, row0, rows, first, end;
  bool tab;
  __device__ explicit AdjShare(const AdjParams& p) {
    const uint64_t n = p.n_beams;
    b0 = (uint32_t)(n * blockIdx.x / gridDim.x);
    b1 = (uint32_t)(n * (blockIdx.x + 1) / gridDim.x);
    row0 = fast_div(b0, p.ic.div_magic);
    rows = b1 > b0 ? fast_div(b1 - 1, p.ic.div_magic) - row0 + 1 : 0;
    tab = rows > 0 && rows <= kAdjRows;
    const uint32_t run = (b1 - b0 + blockDim.x - 1) / blockDim.x * 32u, w = threadIdx.x >> 5;
    first = b0 + w * run + (threadIdx.x & 31);
    end = min(b1, b0 + (w + 1) * run);
  }
};

__device__ __forceinline__ void ld3(const double* base, uint64_t n, uint32_t b, double (&x)[3]) {
  x[0] = base[b];
  x[1] = base[n + b];
  x[2] = base[2 * n + b];
}
__device__ __forceinline__ void st3(double* base, uint64_t n, uint32_t b, const double (&x)[3]) {
  base[b] = x[0];
  base[n + b] = x[1];
  base[2 * n + b] = x[2];
}
__device__ __forceinline__ void cross(const double (&a)[3], const double (&b)[3], double (&c)[3]) {
  c[0] = a[1] * b[2] - a[2] * b[1];
  c[1] = a[2] * b[0] - a[0] * b[2];
  c[2] = a[0] * b[1] - a[1] * b[0];
}
__device__ __forceinline__ double dot(const double (&a)[3], const double (&b)[3]) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

__device__ __forceinline__ void kvec(const AdjRow& r, double eo, double (&K)[3]) {
  K[0] = fma(eo, r.qb0, r.g[0]);
  K[1] = r.g[1];
  K[2] = fma(eo, r.qb2, r.g[2]);
}

// RK4: stage s (1..4) forms Y_s = y + a_s h k_{s-1}; weights of k_s in the update.
__device__ __forceinline__ double rk_a(int s) { return s == 4 ? 1.0 : 0.5; }
__device__ __forceinline__ double rk_w(int s) { return (s == 1 || s == 4) ? 1.0 : 2.0; }
__device__ __forceinline__ double rk_c(int s) { return s == 1 ? 0.0 : (s == 4 ? 1.0 : 0.5); }

__device__ __forceinline__ double stage_radius(const AdjParams& p, int n, int s) {
  return (p.r0 + (double)n * p.h) + rk_c(s) * p.h;
}

// Block partials -> grid barrier -> every block sums them in block order into S.tot (the same bits
// everywhere), while one of its idle warps runs `beside` (work that does not need the sums): what follows
// from the totals needs no serial section and no second hop through memory.  The partials alternate
// between two buffers: a block can be at most one reduction ahead of another.  Returns false on a timeout
// or an abort.  (One last block summing and broadcasting: 200 E x 400 u, 128 steps, 32.1 ms; 30.0 ms so;
// 64 E x 32 u, 64 steps, 7.3 and 6.2 ms.)
template <int NV, class Beside>
__device__ bool grid_reduce(const AdjParams& p, AdjShared& S, double (&v)[NV], Beside beside) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  double* part = p.part + (size_t)(S.reduces & 1u) * gridDim.x * kAdjPartStride;
  int idx = 0, left = NV;
  bool valid = true;
  const double s = reduce_scatter<NV, 16, double>(v, lane, idx, left, valid);
  if (valid) S.scratch[warp * NV + idx] = s;
  __syncthreads();
  for (int t = threadIdx.x; t < (NV * 16 + 31) / 32 * 32; t += blockDim.x) {
    const int c = t >> 4, w = t & 15;
    double x = w < nw && c < NV ? S.scratch[w * NV + c] : 0.0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (w == 0 && c < NV) part[(size_t)blockIdx.x * kAdjPartStride + c] = x;
  }
  if (!pass_barrier(p.bar, gridDim.x, gridDim.x, p.timeout_ns, p.status, &S.flag, &S.pass_next)) return false;
  if (threadIdx.x == 0) S.reduces++;
  if (warp < NV) {
    double s = 0.0;
    for (unsigned b = lane; b < gridDim.x; b += 32) s += __ldcg(&part[(size_t)b * kAdjPartStride + warp]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) S.tot[warp] = s;
  } else if (warp == NV && lane == 0) {
    beside();
  }
  __syncthreads();
  return true;
}

// Forward RK4 over steps [n_first, n_first + count) from p.y.  store_seg: each step's start state
// to seg[m] and its stage constants to stage_sc[m]; store_ck: the start state of every step with
// n % K == 0 to ck[n / K]; finish: complete the last step (else stop after its last reduction).
__device__ bool forward_steps(const AdjParams& p, AdjShared& S, int n_first, int count, bool store_seg,
                              bool store_ck, bool finish) {
  const uint64_t n = p.n_beams;
  const AdjShare sh(p);
  const int P = 4 * count;
  for (int pp = 0; pp <= P; ++pp) {
    if (pp == P && !finish) break;
    const int sp = pp > 0 ? ((pp - 1) & 3) + 1 : 0;        // stage finished in this pass
    const int s = (pp & 3) + 1, m = pp >> 2;                // stage formed in this pass
    const int nstep = n_first + m;
    const int slot = pp & 1;                                // rows of the formed stage; the other: the finished one's
    double x_s = 0.0;
    if (pp < P) {
      const double r = stage_radius(p, nstep, s);
      x_s = p.ic.R2 / (r * r);
    }
    // the formed stage's geometry; the finished stage's, tabulated in the pass before, gets its couplings
    if (sh.tab) {
      for (uint32_t t = threadIdx.x; t < 2 * sh.rows; t += blockDim.x) {
        const uint32_t r = t < sh.rows ? t : t - sh.rows;
        if (t < sh.rows) {
          if (pp < P) row_geometry(p, sh.row0 + r, x_s, S.row[slot][r]);
        } else if (pp > 0) {
          row_coupling(S.scf, S.row[slot ^ 1][r]);
        }
      }
    }
    __syncthreads();
    auto finished = [&](uint32_t jj) {
      if (sh.tab) return S.row[slot ^ 1][jj - sh.row0];
      AdjRow r;
      row_geometry(p, jj, S.scf[7], r);
      row_coupling(S.scf, r);
      return r;
    };
    double acc[6] = {0, 0, 0, 0, 0, 0}, rs[3] = {0, 0, 0};
    auto flush = [&](uint32_t jj) {
      const double du = p.du[jj >= p.n_angle ? jj - p.n_angle : jj];
      double t1;
      if (sh.tab) {
        t1 = S.row[slot][jj - sh.row0].t1;
      } else {
        AdjRow r;
        row_geometry(p, jj, x_s, r);
        t1 = r.t1;
      }
      const double dt = du * t1;
      for (int i = 0; i < 3; ++i) {
        acc[i] = fma(dt, rs[i], acc[i]);
        acc[3 + i] = fma(du, rs[i], acc[3 + i]);
        rs[i] = 0.0;
      }
    };
    uint32_t cur = 0xffffffffu;
    for (uint32_t b = sh.first; b < sh.end; b += 32) {
      const uint32_t jj = fast_div(b, p.ic.div_magic), k = b - jj * p.n_energy;
      const bool bar = jj >= p.n_angle;
      double y[3], kl[3];
      ld3(p.y, n, b, y);
      ld3(p.klast, n, b, kl);
      if (pp > 0) {
        const double om = p.omega[k], eo = bar ? -om : om;
        double ys[3], K[3], kk[3], ks[3];
        const double as = sp == 1 ? 0.0 : rk_a(sp) * p.h;
        for (int i = 0; i < 3; ++i) ys[i] = sp == 1 ? y[i] : y[i] + as * kl[i];
        kvec(finished(jj), eo, K);
        cross(K, ys, kk);
        if (sp == 1) {
          for (int i = 0; i < 3; ++i) ks[i] = kk[i];
        } else {
          ld3(p.ksum, n, b, ks);
          for (int i = 0; i < 3; ++i) ks[i] += rk_w(sp) * kk[i];
        }
        if (sp == 4) {
          for (int i = 0; i < 3; ++i) y[i] = y[i] + (p.h / 6.0) * ks[i];
          st3(p.y, n, b, y);
        } else {
          st3(p.ksum, n, b, ks);
        }
        for (int i = 0; i < 3; ++i) kl[i] = kk[i];
        st3(p.klast, n, b, kl);
      }
      if (pp < P) {
        if (s == 1) {
          if (store_seg) st3(p.seg + (size_t)m * 3 * n, n, b, y);
          if (store_ck && nstep % p.ck_every == 0) st3(p.ck + (size_t)(nstep / p.ck_every) * 3 * n, n, b, y);
        }
        if (jj != cur) {
          if (cur != 0xffffffffu) flush(cur);
          cur = jj;
        }
        const double as = s == 1 ? 0.0 : rk_a(s) * p.h, g = p.g[(bar ? p.n_energy : 0u) + k];
        for (int i = 0; i < 3; ++i) rs[i] = fma(g, s == 1 ? y[i] : y[i] + as * kl[i], rs[i]);
      }
    }
    if (pp == P) break;
    if (cur != 0xffffffffu) flush(cur);
    if (!grid_reduce<6>(p, S, acc, [&] { strengths(p.ic, stage_radius(p, nstep, s), S.str[0], S.str[1]); })) return false;
    if (threadIdx.x < kAdjStageVals) {
      const int i = threadIdx.x;
      const double mu = S.str[0];
      const double v = i < 6 ? mu * S.tot[i] : i == 6 ? S.str[1] : i == 7 ? x_s : i == 8 ? mu : 0.0;
      S.scf[i] = v;
      if (store_seg && blockIdx.x == 0) p.stage_sc[((size_t)m * 4 + (s - 1)) * kAdjStageVals + i] = v;
    }
    __syncthreads();
  }
  // block 0's last stage constants, for the backward sweep of every block
  return !store_seg || pass_barrier(p.bar, gridDim.x, gridDim.x, p.timeout_ns, p.status, &S.flag, &S.pass_next);
}

// Objective J and the adjoint of the final state; zero the parameter accumulators.
__device__ bool objective(const AdjParams& p, AdjShared& S) {
  const uint64_t n = p.n_beams;
  const AdjShare sh(p);                  // the beams of forward_steps: each thread reads what it wrote
  double acc[1] = {0.0};
  for (uint32_t b = sh.first; b < sh.end; b += 32) {
    const uint32_t jj = fast_div(b, p.ic.div_magic), k = b - jj * p.n_energy;
    const double ow = jj >= p.n_angle ? 0.0 : p.du[jj] * p.objw[k];      // objective weight: nu beams only
    const double sz = p.y[2 * n + b];
    acc[0] += ow * 0.5 * (1.0 + sz);
    const double a[3] = {0.0, 0.0, 0.5 * ow};
    st3(p.a, n, b, a);
    p.gw[b] = 0.0;
    p.gth[b] = 0.0;
  }
  if (!grid_reduce<1>(p, S, acc, [] {})) return false;
  if (blockIdx.x == 0 && threadIdx.x == 0) p.glob[kGlobJ] = S.tot[0];
  return true;
}

// Backward over the segment's steps [seg_first, seg_first + seg_count), stage by stage.
__device__ bool backward_steps(const AdjParams& p, AdjShared& S) {
  const uint64_t n = p.n_beams;
  const AdjShare sh(p);
  const int count = p.seg_count;
  const int P = 4 * count;
  const double h = p.h;
  for (int pp = 0; pp <= P; ++pp) {
    const int sp = pp > 0 ? 4 - ((pp - 1) & 3) : 0;         // stage finished (its moments reduced)
    const int mp = pp > 0 ? count - 1 - ((pp - 1) >> 2) : 0;
    const int s = 4 - (pp & 3), m = count - 1 - (pp >> 2);  // stage formed
    if (threadIdx.x < 4 * kAdjStageVals && pp < P)
      S.scs[threadIdx.x / kAdjStageVals][threadIdx.x % kAdjStageVals] =
          __ldcg(&p.stage_sc[(size_t)m * 4 * kAdjStageVals + threadIdx.x]);
    if (pp > 0) {
      if (threadIdx.x < kAdjStageVals)
        S.scf[threadIdx.x] = __ldcg(&p.stage_sc[((size_t)mp * 4 + (sp - 1)) * kAdjStageVals + threadIdx.x]);
    }
    __syncthreads();
    // rows: slots 1..4 hold the stages of the formed stage's step, filled once a step (s = 4); slot 0
    // keeps the step before's stage 1 for the pass that finishes it
    const bool step_start = s == 4;
    const int fslot = sp == 1 ? 0 : sp;
    if (sh.tab) {
      if (step_start) {
        for (uint32_t t = threadIdx.x; t < 4 * sh.rows; t += blockDim.x) {
          const uint32_t st = 1 + t / sh.rows, r = t % sh.rows;
          if (st == 1 && pp > 0) {
            S.row[0][r] = S.row[1][r];
            S.back[r] = row_back(p, sh.row0 + r, S.row[0][r], S.gl);
          }
          if (pp < P) {
            row_geometry(p, sh.row0 + r, S.scs[st - 1][7], S.row[st][r]);
            row_coupling(S.scs[st - 1], S.row[st][r]);
          }
        }
      } else {
        for (uint32_t r = threadIdx.x; r < sh.rows; r += blockDim.x)
          S.back[r] = row_back(p, sh.row0 + r, S.row[fslot][r], S.gl);
      }
    }
    __syncthreads();
    auto stage_row = [&](int slot, const double* sc, uint32_t jj) {
      if (sh.tab) return S.row[slot][jj - sh.row0];
      AdjRow r;
      row_geometry(p, jj, sc[7], r);
      row_coupling(sc, r);
      return r;
    };
    double acc[6] = {0, 0, 0, 0, 0, 0}, rs[3] = {0, 0, 0};
    auto flush = [&](uint32_t jj) {
      const AdjRow r = stage_row(s, S.scs[s - 1], jj);
      for (int i = 0; i < 3; ++i) {
        acc[i] = fma(r.q, rs[i], acc[i]);
        acc[3 + i] = fma(r.t1, rs[i], acc[3 + i]);
        rs[i] = 0.0;
      }
    };
    uint32_t cur = 0xffffffffu;
    for (uint32_t b = sh.first; b < sh.end; b += 32) {
      const uint32_t jj = fast_div(b, p.ic.div_magic), k = b - jj * p.n_energy;
      const bool bar = jj >= p.n_angle;
      const double om = p.omega[k], eo = bar ? -om : om;
      double a[3];
      ld3(p.a, n, b, a);
      double vnext[3] = {0, 0, 0};
      if (pp > 0) {
        double ys[3], v[3], K[3], pv[3], t[3];
        if (sp == 1) ld3(p.seg + (size_t)mp * 3 * n, n, b, ys);
        else ld3(p.ystage + (size_t)(sp - 2) * 3 * n, n, b, ys);
        ld3(p.v, n, b, v);
        const AdjRow row = stage_row(fslot, S.scf, jj);
        const AdjBack bk = sh.tab ? S.back[jj - sh.row0] : row_back(p, jj, row, S.gl);
        kvec(row, eo, K);
        cross(v, K, t);
        const double g = p.g[(bar ? p.n_energy : 0u) + k];
        double sb[3];
        for (int i = 0; i < 3; ++i) sb[i] = fma(g, bk.brd[i], t[i]);
        p.gw[b] += dot(ys, bk.brd);
        cross(ys, v, pv);
        p.gth[b] = fma(eo, fma(pv[0], bk.qd0, pv[2] * bk.qd2), p.gth[b]);
        double yb[3];
        if (sp == 4) {
          for (int i = 0; i < 3; ++i) { yb[i] = sb[i]; vnext[i] = (h / 3.0) * a[i] + h * sb[i]; }
        } else {
          ld3(p.ybar, n, b, yb);
          for (int i = 0; i < 3; ++i) yb[i] += sb[i];
          if (sp == 3) for (int i = 0; i < 3; ++i) vnext[i] = (h / 3.0) * a[i] + (0.5 * h) * sb[i];
          if (sp == 2) for (int i = 0; i < 3; ++i) vnext[i] = (h / 6.0) * a[i] + (0.5 * h) * sb[i];
        }
        if (sp == 1) {
          for (int i = 0; i < 3; ++i) a[i] += yb[i];
          st3(p.a, n, b, a);
        } else {
          st3(p.ybar, n, b, yb);
        }
      }
      if (pp < P) {
        double ys[3], v[3];
        if (s == 4) {
          // stage states of step m from its start state and stored stage constants
          double y[3], kk[3], K[3], yy[3];
          ld3(p.seg + (size_t)m * 3 * n, n, b, y);
          for (int i = 0; i < 3; ++i) yy[i] = y[i];
          for (int st = 1; st <= 3; ++st) {
            kvec(stage_row(st, S.scs[st - 1], jj), eo, K);
            cross(K, yy, kk);
            const double as = rk_a(st + 1) * h;
            for (int i = 0; i < 3; ++i) yy[i] = y[i] + as * kk[i];
            st3(p.ystage + (size_t)(st - 1) * 3 * n, n, b, yy);
          }
          for (int i = 0; i < 3; ++i) { ys[i] = yy[i]; v[i] = (h / 6.0) * a[i]; }
        } else {
          if (s == 1) ld3(p.seg + (size_t)m * 3 * n, n, b, ys);
          else ld3(p.ystage + (size_t)(s - 2) * 3 * n, n, b, ys);
          for (int i = 0; i < 3; ++i) v[i] = vnext[i];
        }
        st3(p.v, n, b, v);
        if (jj != cur) {
          if (cur != 0xffffffffu) flush(cur);
          cur = jj;
        }
        double pv[3];
        cross(ys, v, pv);
        for (int i = 0; i < 3; ++i) rs[i] += pv[i];
      }
    }
    if (pp == P) break;
    if (cur != 0xffffffffu) flush(cur);
    if (!grid_reduce<6>(p, S, acc, [] {})) return false;
    if (threadIdx.x < 6) S.gl[threadIdx.x] = S.scs[s - 1][8] * S.tot[threadIdx.x];
    __syncthreads();
  }
  return true;
}

__global__ void __launch_bounds__(kAdjBlock, 1) adjoint_kernel(const __grid_constant__ AdjParams p) {
  __shared__ AdjShared S;
  if (threadIdx.x == 0) {
    S.pass_next = pass_barrier_base(p.bar, gridDim.x);
    S.reduces = 0;
  }
  __syncthreads();
  if (p.mode == kAdjForward) {
    if (!forward_steps(p, S, 0, p.n_steps, false, true, true)) return;
    objective(p, S);
    return;
  }
  // backward over one segment: re-run it forward from its checkpoint, then reverse it
  const uint64_t n = p.n_beams;
  const AdjShare sh(p);                  // the beams of forward_steps: each thread reads what it wrote
  const double* ck = p.ck + (size_t)(p.seg_first / p.ck_every) * 3 * n;
  for (uint32_t b = sh.first; b < sh.end; b += 32) {
    double y[3];
    ld3(ck, n, b, y);
    st3(p.y, n, b, y);
  }
  if (!forward_steps(p, S, p.seg_first, p.seg_count, true, false, false)) return;
  backward_steps(p, S);
}

__global__ void adjoint_sums_kernel(AdjParams p, double* pee_sum, double* gw_sum, double* gth_sum) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * p.n_energy) return;
  const uint32_t sig = t / p.n_energy, k = t - sig * p.n_energy;
  const uint64_t n = p.n_beams;
  const double J = p.glob[kGlobJ];
  double ps = 0.0, gs = 0.0, ts = 0.0;
  for (uint32_t j = 0; j < p.n_angle; ++j) {
    const uint32_t b = (sig * p.n_angle + j) * p.n_energy + k;
    if (!sig) ps += p.du[j] * (0.5 * (1.0 + p.y[2 * n + b]) - J);
    gs += p.gw[b];
    ts += p.gth[b];
  }
  if (!sig) pee_sum[k] = ps;
  gw_sum[t] = gs;
  gth_sum[t] = ts;
}

}  // namespace

cudaError_t adjoint_launch(const AdjParams& p, int grid, cudaStream_t stream) {
  AdjParams q = p;
  void* args[] = {&q};
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kAdjBlock);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, (const void*)adjoint_kernel, args);
}

int adjoint_blocks_per_sm() {
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, adjoint_kernel, kAdjBlock, 0) != cudaSuccess) return 0;
  return occ;
}

cudaError_t adjoint_energy_sums(const AdjParams& p, double* pee_sum, double* gw_sum, double* gth_sum,
                                cudaStream_t stream) {
  const unsigned nt = 2 * p.n_energy;
  adjoint_sums_kernel<<<(nt + 127) / 128, 128, 0, stream>>>(p, pee_sum, gw_sum, gth_sum);
  return cudaGetLastError();
}

}  // namespace xflat
