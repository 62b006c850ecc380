// kernels.cu -- CUDA kernels of the OPMM estimation path (sm_103a).
//
//   k_gather      copy caller traces into the packed, 16-byte aligned buffer
//   k_nominal     box centres: Table 1, W = D - 6 ms, calibrated agonist pulse
//   k_simulate    trajectories of (OPC, saccade) pairs
//   k_score       objective of many OPC vectors against one saccade
//   k_search      persistent multi-start parallel Nelder-Mead (Algorithm 1)
//   k_finalize    per-saccade winner and FP64 re-computation of its error
//   k_refine      Levenberg-Marquardt refinement of search results
//   k_refine_check  FP64 error of the refined vectors
//   k_admit, k_advance  request loop: slot admission and iteration progress
//
// The hot loop is k_search's candidate evaluation: one thread integrates one
// trial OPC vector's plant in registers (plant.cuh), scoring each sample against
// the trace staged once per block in shared memory by a TMA bulk copy, with a
// compensated FP32 sum.  Per block, two groups of G simplices of one saccade
// advance side by side: all 22 trial points of every simplex of a group are
// evaluated in one wave (Sec. 3.3: all simplex transformations are computed at
// once), ordered by their simplices' pulse widths and taken in 32-candidate
// chunks by all of the block's warps; the warp that completes a group's wave takes that group's
// Lagarias decisions and publishes its next wave while the other warps
// evaluate the other group's.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/opmm.h"
#include "common.cuh"
#include "launch.h"
#include "plant.cuh"

namespace opmm {

__device__ __forceinline__ SacConst sac_const(const DevSac& d) {
  SacConst s;
  s.L = d.L; s.onset = d.onset; s.nsub = d.nsub;
  s.fs = d.fs; s.h = d.h; s.th0 = d.th0; s.thf = d.thf;
  return s;
}

// ------------------------------------------------------------------ gather
__global__ void k_gather(const float* const* src, const DevSac* sacs, float* dst, int n) {
  const int b = blockIdx.x;
  if (b >= n) return;
  const DevSac d = sacs[b];
  const float* s = src[b];
  float* o = dst + d.off;
  const int Lp = (d.L + 3) & ~3;
  for (int k = threadIdx.x; k < Lp; k += blockDim.x) o[k] = k < d.L ? s[k] : 0.0f;
}

// ------------------------------------------------------------------ sinks
// Blocked compensated summation: the squared errors of each block of samples
// (the sample loops run in blocks of 4) are summed plainly, and each block sum
// is added to the running total with Kahan compensation, so the relative error
// stays O(4 eps) per block instead of growing with the window length.
struct KahanSink {
  const float* z;   // trace minus end fixation, positive frame
  float sum, c;
  float part;
  __device__ __forceinline__ void emit(int k, float dth) {
    const float d = dth - z[k];
    part = fmaf(d, d, part);
  }
  __device__ __forceinline__ void block_end() {
    const float y = part - c;
    const float t = sum + y;
    c = (t - sum) - y;
    sum = t;
    part = 0.0f;
  }
  // mean over L samples, +inf when it is not finite
  __device__ __forceinline__ float mean(int L) {
    block_end();
    const float f = (sum - c) / (float)L;
    return isfinite(f) ? f : INFINITY;
  }
};

// Writes a trajectory after its samples at rest.  Every thread of a warp writes
// its own row, so a store of single samples touches 32 sectors for 128 bytes;
// GROUPS: four at a time where they fill an aligned 16-byte group, which takes
// a quarter of the transactions (rows with three samples at rest or more: no
// later group then begins before the row).  The last three samples shift
// through registers, which the unrolled sample loops resolve by renaming; an
// array position chosen per sample (compares, selects and a branch) took 65 ns
// a sample where these take 27, and more than the whole walk of one row.
template <bool GROUPS>
struct WriteSink {
  float* out;
  float sign, thf;
  float b1, b2, b3;    // the last three samples
  // all samples so far have the value v
  __device__ __forceinline__ WriteSink(float* o, float sg, float th, float v) : out(o), sign(sg), thf(th), b1(v), b2(v), b3(v) {}
  __device__ __forceinline__ void emit(int k, float dth) {
    const float v = sign * (thf + dth);
    float* o = out + k;
    if constexpr (!GROUPS) {
      *o = v;
    } else {
      if ((~(unsigned)reinterpret_cast<uintptr_t>(o) & 12u) == 0) *reinterpret_cast<float4*>(o - 3) = make_float4(b1, b2, b3, v);
      b1 = b2;
      b2 = b3;
      b3 = v;
    }
  }
  __device__ __forceinline__ void block_end() {}
  // the n samples' last, partial group
  __device__ __forceinline__ void finish(int n) {
    if constexpr (GROUPS) {
      const int s = (int)((reinterpret_cast<uintptr_t>(out + n) >> 2) & 3);
      if (s > 0) out[n - 1] = b3;
      if (s > 1) out[n - 2] = b2;
      if (s > 2) out[n - 3] = b1;
    }
  }
};

// Samples 0 .. n - 1 of a row have the value v.
__device__ __forceinline__ void write_rest(float* out, int n, float v) {
  int k = 0;
  for (; k < n && (reinterpret_cast<uintptr_t>(out + k) & 15u); ++k) out[k] = v;
  for (; k + 4 <= n; k += 4) *reinterpret_cast<float4*>(out + k) = make_float4(v, v, v, v);
  for (; k < n; ++k) out[k] = v;
}

struct PeakSink {
  float m;
  __device__ __forceinline__ void emit(int, float dth) { m = fmaxf(m, dth); }
  __device__ __forceinline__ void block_end() {}
};

// Objective of one OPC vector: mean squared error over the window; the
// samples up to onset (the plant at rest) are folded into (sum0, c0).
// pe (optional): set to 1 when the pulse ends inside the window.
template <bool PACK>
__device__ __forceinline__ float objective(const float* p, const SacConst& sc, const float* z,
                                           float sum0, float c0, float* qs, int qstride, int* pe, unsigned mask) {
  KahanSink s{z, sum0, c0, 0.0f};
  if (walk<KahanSink, true, PACK>(p, sc, s, qs, qstride, true, pe, mask) < 0) return INFINITY;
  return s.mean(sc.L);
}

// Parameter sources of the register-lean walk: each load() re-derives the
// candidate's OPC vector instead of keeping it live.
struct PtrSrc {
  const float* p;
  __device__ __forceinline__ void load(float (&o)[kNumParams]) const {
#pragma unroll
    for (int j = 0; j < kNumParams; ++j) o[j] = p[j];
  }
};

// Candidate in ln-parameter space, from two rows in shared memory: a vertex
// (u = a), or the search's trial-point form u = a + (b - a) / 2 (a = b for the
// deciding warp's four trial points, best vertex and vertex q - 3 for a shrink
// point).
struct ULinSrc {
  const float* a;   // first row
  const float* b;   // second row
  bool half;        // u = a + (b - a) / 2, else u = a
  const float* pc;  // box centre
  float lnlo, lnhi;
  __device__ __forceinline__ void load(float (&o)[kNumParams]) const;
};


// Stage one saccade for a block: TMA bulk copy of the raw trace, then the
// positive-frame trace minus the end fixation and the compensated sum of the
// rest samples.  All threads call it; returns false on a wait timeout.
struct TraceStage {
  float sum0, c0;
};

// The positive-frame trace minus the end fixation into z, and the compensated
// sum of the rest samples (all threads; y in shared or global memory).
__device__ __forceinline__ void shift_trace(const DevSac& d, const float* y, float* z, TraceStage* st) {
  for (int k = threadIdx.x; k < d.L; k += blockDim.x) z[k] = d.sign * y[k] - d.thf;
  if (threadIdx.x == 0) {
    float sum = 0.0f, c = 0.0f;
    const int kend = min(d.onset, d.L - 1);
    for (int k = 0; k <= kend; ++k) {
      const float e = d.th0 - d.sign * y[k];
      const float q = fmaf(e, e, -c);
      const float t = sum + q;
      c = (t - sum) - q;
      sum = t;
    }
    st->sum0 = sum;
    st->c0 = c;
  }
  __syncthreads();
}

__device__ bool stage_trace(const DevSac& d, const float* traces, float* yraw, float* z, uint64_t* bar,
                            uint32_t& phase, TraceStage* st) {
  if (threadIdx.x == 0) {
    fence_proxy_async_smem();
    const uint32_t bytes = (uint32_t)(((d.L + 3) & ~3) * 4);
    mbar_arrive_expect_tx(bar, bytes);
    tma_load_1d(yraw, traces + d.off, bytes, bar);
  }
  const bool ok = mbar_wait(bar, phase, kMaxWaitTries);
  phase ^= 1u;
  if (__syncthreads_or(!ok)) return false;
  shift_trace(d, yraw, z, st);
  return true;
}

// ------------------------------------------------------------------ nominal
// The default plant's saccade from 0 to A, 1 kHz grid, 250 ms after onset; its
// propagators do not depend on the agonist pulse, so one set-up serves all the
// pulses tried (a set-up per pulse, in scalar arithmetic: 615 us against 507 for
// 10,000 saccades).
struct NominalWalk {
  SacConst sc;
  PackedWalk w;
  __device__ __forceinline__ NominalWalk(const float* p, float A) {
    sc.L = 251; sc.onset = 0; sc.nsub = 10; sc.fs = 1000.0f; sc.h = 1.0e-4f; sc.th0 = 0.0f; sc.thf = A;
    w.setup(p, sc);
  }
  // largest sample with agonist pulse nsac
  __device__ __forceinline__ float peak(float* p, float nsac) {
    p[kNsacAg] = nsac;
    PeakSink pk{-sc.thf};
    w.samples(p, sc, pk);
    return sc.thf + pk.m;
  }
};

// One warp per saccade.  Calibrated mode: the agonist pulse for which the
// default plant's saccade peaks at its amplitude A; round 0 brackets the
// crossing between lo 2^(i-1) and lo 2^i (lo = step level of A), six rounds of
// a 32-point search narrow the bracket; if the step level already reaches A
// it is used as is.
__global__ void k_nominal(const DevSac* sacs, int n, int pulse_mode, const float* init_opc, float* pc) {
  const int lane = threadIdx.x & 31;
  const int b = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (b >= n) return;
  float* out = pc + (size_t)b * kNumParams;
  if (init_opc) {
    if (lane < kNumParams) out[lane] = init_opc[(size_t)b * kNumParams + lane];
    return;
  }
  const DevSac d = sacs[b];
  float p[kNumParams];
#pragma unroll
  for (int j = 0; j < kNumParams; ++j) p[j] = kTable1[j];
  p[kPw] = d.dur_ms - 6.0f;
  float nsac = kTable1[kNsacAg];
  if (pulse_mode == OPMM_PULSE_CALIBRATED) {
    const float A = d.thf - d.th0;
    float s[6];
    rest_state(p, A, s);
    const float lo = s[4];
    NominalWalk nw(p, A);
    float pk = nw.peak(p, lo * ldexpf(1.0f, lane));
    unsigned hit = __ballot_sync(0xffffffffu, pk >= A);
    if (hit & 1u) {
      nsac = lo;
    } else if (hit == 0u) {
      nsac = lo * ldexpf(1.0f, 31);
    } else {
      const int i0 = __ffs(hit) - 1;
      float a = lo * ldexpf(1.0f, i0 - 1);
      float bb = lo * ldexpf(1.0f, i0);
#pragma unroll 1
      for (int round = 0; round < 6; ++round) {
        const float x = a + (bb - a) * ((float)(lane + 1) * (1.0f / 33.0f));
        pk = nw.peak(p, x);
        const unsigned h = __ballot_sync(0xffffffffu, pk >= A);
        const int i = h ? __ffs(h) - 1 : 32;
        const float xlo = __shfl_sync(0xffffffffu, x, i > 0 ? i - 1 : 0);
        const float xhi = __shfl_sync(0xffffffffu, x, i < 32 ? i : 31);
        const float na = i == 0 ? a : xlo;
        const float nb = i == 32 ? bb : xhi;
        a = na;
        bb = nb;
      }
      nsac = 0.5f * (a + bb);
    }
  }
  p[kNsacAg] = nsac;
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < kNumParams; ++j) out[j] = p[j];
  }
}

// ------------------------------------------------------------------ simulate
__global__ void __launch_bounds__(256) k_simulate(const float* opc, int n, const DevSac* sacs, const int* sac_of,
                           const long long* out_off, float* out, bool groups) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float p[kNumParams];
#pragma unroll
  for (int j = 0; j < kNumParams; ++j) p[j] = opc[(size_t)i * kNumParams + j];
  const DevSac d = sacs[sac_of ? sac_of[i] : i];
  const SacConst sc = sac_const(d);
  float* row = out + out_off[i];
  const int rest = min(d.onset, d.L - 1) + 1;
  const float v0 = d.sign * d.th0;
  write_rest(row, rest, v0);
  PackedWalk pw;
  pw.setup(p, sc);
  if (groups && rest >= 3) {
    WriteSink<true> w(row, d.sign, d.thf, v0);
    pw.samples(p, sc, w);
    w.finish(d.L);
  } else {
    WriteSink<false> w(row, d.sign, d.thf, v0);
    pw.samples(p, sc, w);
  }
}

// ------------------------------------------------------------------ score
constexpr int kScoreThreads = 128;

// One launch and nothing around it: the descriptor is an argument, and each
// block reads the trace where the caller keeps it (any alignment, a few
// hundred samples) instead of a padded copy by TMA, whose staging, error word
// and second synchronisation were half of a call's time.
__global__ void __launch_bounds__(kScoreThreads) k_score(const float* opc, int m, const __grid_constant__ DevSac d,
                                                         const float* trace, float* f) {
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ TraceStage st;
  float* z = reinterpret_cast<float*>(smraw);
  shift_trace(d, trace, z, &st);
  const SacConst sc = sac_const(d);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    float p[kNumParams];
#pragma unroll
    for (int j = 0; j < kNumParams; ++j) p[j] = opc[(size_t)i * kNumParams + j];
    KahanSink s{z, st.sum0, st.c0, 0.0f};
    f[i] = walk(p, sc, s, nullptr, 0, true) < 0 ? INFINITY : s.mean(sc.L);
  }
}

// ------------------------------------------------------------------ search
// Unit record (kUnitRecFloats words): [0] best f, [1] winning simplex (int),
// [2] its iterations (int), [3] candidate evaluations of the unit (int),
// [4..21] best vertex (ln units), [22] evaluations whose pulse ends inside the
// window (int), [23] unused.  With the 9-parameter model the vertex takes
// [4..12].
constexpr int kUnitRec = kUnitRecFloats;

// The search runs over N coordinates: N = 18, the OPC entries themselves, or
// N = 9, the 9-parameter model (Sec. 2.2.2, Table 2).  A simplex has N + 1
// vertices and each iteration N + 4 trial points.
template <int N>
__host__ __device__ constexpr int verts() { return N + 1; }
template <int N>
__host__ __device__ constexpr int trials() { return N + 4; }

// Search coordinate that scales OPC entry j (Fig. 4 order): j itself for N =
// 18; for N = 9 the coordinate of the Table 2 quantity the entry carries, in
// the table's order (K_SE, K_LT, B_AG, B_ANT, B_P, N_C_AG, N_C_ANT, J,
// N_C_FIX; the shared series elasticity and length-tension coefficient scale
// both muscles' entries), or -1 for the neural control signal, which that
// model does not estimate (activation and deactivation times, pulse heights
// and width stay at the box centre).
template <int N>
__host__ __device__ constexpr int search_coord(int j) {
  if (N == kNumParams) return j;
  switch (j) {
    case kSeAg: case kSeAnt: return 0;
    case kLtAg: case kLtAnt: return 1;
    case kBAg: return 2;
    case kBAnt: return 3;
    case kBp: return 4;
    case kNcAg: return 5;
    case kNcAnt: return 6;
    case kJ: return 7;
    case kNcFix: return 8;
    default: return -1;
  }
}

// OPC vector of search point u: p_j = pc_j exp(clamp(u_c)) for c =
// search_coord(j) >= 0, else pc_j.
template <int N>
__device__ __forceinline__ void u_to_p(const float* u, const float* pc, float lnlo, float lnhi, float (&p)[kNumParams]) {
#pragma unroll
  for (int j = 0; j < kNumParams; ++j) {
    const int c = search_coord<N>(j);
    p[j] = c < 0 ? pc[j] : pc[j] * __expf(fminf(fmaxf(u[c < 0 ? 0 : c], lnlo), lnhi));
  }
}

// Saved simplex (serving): vertices, values, order, active, iterations (the
// centroid and the trial points follow from these).
template <int N>
__host__ __device__ constexpr int state_floats() { return verts<N>() * N + 2 * verts<N>() + 2; }
static_assert(state_floats<kNumParams>() == kSearchStateFloats, "saved simplex layout");

// One block runs G simplices in each of two groups (a unit of 2G simplices of
// one saccade) with twelve warps, all of which evaluate: a group's wave (its
// 22 trial points per simplex, or its initial vertices) is published in
// chunks of 32 candidates that the warps claim in turn; the warp that
// completes a wave's last chunk takes that group's Nelder-Mead decisions,
// orders and publishes its next wave, while the other warps work on the other
// group's wave.  There is no block barrier between steps.  Twelve warps at 168
// registers per thread fill the SM's register file (3 warps per SM
// sub-partition).
constexpr int kSearchWarps = 12;
// Longest a search warp waits with nothing to claim (SM clock cycles, about
// four seconds): far above one chunk's evaluation plus one group's decisions;
// past it the warp raises kErrWaitTimeout and the block leaves the kernel.
constexpr long long kMaxIdleCycles = 8000000000LL;
template <int G, int N>
__host__ __device__ constexpr int search_threads() { return 32 * kSearchWarps; }
// State of one group of G simplices over N coordinates.
template <int G, int N>
struct alignas(16) GroupSmem {
  static constexpr int kNV = verts<N>();
  static constexpr int kNT = trials<N>();
  static_assert(G <= 32, "the deciding warp takes one simplex per lane");
  float U[G][kNV][N];            // vertices, by slot
  float XT[G][4][N];             // reflection, expansion, outside/inside contraction
  float F[G][kNV];               // vertex values, by slot
  float FT[G][kNT];              // trial values
  unsigned char ord[G][kNV + 1]; // ord[r] = slot of rank r
  unsigned char turn[G];         // turn[k] = k-th simplex of the pending wave
  int active[G];
  int iters[G];
  int nsim;     // simplices of this group (0: empty group)
  int nvalid;   // candidates of the pending wave
  int kind;     // pending wave: 0 initial vertices, 1 trial points
  int state;    // kPending (a wave is ordered) or kDone; written by the deciding warp only
  int it;       // trial waves evaluated in this launch
  int evals;    // candidate evaluations of this group
  int pe;       // of those, candidates whose pulse ends inside the window
  int pub;      // published wave: sequence number << 16 | chunks (0 chunks: nothing to take)
  int claim;    // sequence number << 16 | next chunk of 32 candidates (in wave order) to claim
  int done;     // chunks of the published wave evaluated
};

enum : int { kPending = 0, kDone = 2 };

// The staged saccade of a search block.
struct SacStage {
  float pc[kNumParams];          // box centre of the current saccade
  SacConst sc;
  TraceStage st;
};

template <int G, int N, int NG>
struct SearchSmem {
  GroupSmem<G, N> grp[NG];
  SacStage sv;
  int cur_b;
  int unit;
  int abort;                     // a warp's bounded wait gave up: the block leaves
  uint64_t bar;
};

constexpr int kQSlotFloats = (int)(sizeof(Prop2) / sizeof(float));

// Dynamic shared memory: the block state, the raw and shifted traces (lcap
// floats each) and one single-substep propagator slot per thread.
template <int G, int N, int NG>
size_t search_smem_bytes(int lcap) {
  return ((sizeof(SearchSmem<G, N, NG>) + 127) / 128) * 128 + 2 * (size_t)lcap * sizeof(float) +
         (size_t)kQSlotFloats * search_threads<G, N>() * sizeof(float);
}

// Trial point coordinate (Lagarias et al. coefficients rho 1, chi 2, gamma 1/2).
__device__ __forceinline__ float trial_coord(int q, float xb, float w) {
  const float xr = xb + (xb - w);
  switch (q) {
    case 0: return xr;
    case 1: return xb + 2.0f * (xr - xb);
    case 2: return xb + 0.5f * (xr - xb);
    default: return xb - 0.5f * (xb - w);
  }
}

__device__ __forceinline__ float shrink_coord(float x1, float xi) { return x1 + 0.5f * (xi - x1); }

__device__ __forceinline__ void ULinSrc::load(float (&o)[kNumParams]) const {
#pragma unroll
  for (int j = 0; j < kNumParams; ++j) {
    const float u = half ? shrink_coord(a[j], b[j]) : a[j];
    o[j] = pc[j] * __expf(fminf(fmaxf(u, lnlo), lnhi));
  }
}

// Objective through the register-lean walk.
__device__ __forceinline__ float objective_lean(const ULinSrc& src, const SacConst& sc, const float* z,
                                                float sum0, float c0, int* pe = nullptr) {
  {
    float p[kNumParams];
    src.load(p);
    Coef k;
    make_coef(p, k);
    if (refine_shift(k, sc.h) < 0) return INFINITY;
  }
  KahanSink s{z, sum0, c0, 0.0f};
  walk_lean(src, sc, s, pe);
  return s.mean(sc.L);
}

// Objective of search point u; the lanes in `mask` call it together and
// reconverge inside the walk; PACK picks the packed sample update.
template <int N, bool PACK>
__device__ __forceinline__ float eval_u(const float (&u)[N], const float* pc, float lnlo,
                                        float lnhi, const SacConst& sc, const float* z, float sum0,
                                        float c0, float* qs, int qstride, int* pe, unsigned mask) {
  float p[kNumParams];
  u_to_p<N>(u, pc, lnlo, lnhi, p);
  return objective<PACK>(p, sc, z, sum0, c0, qs, qstride, pe, mask);
}

// Rows of trial point q of simplex gi, as u = a + (b - a) / 2 coordinate by
// coordinate: a = b = the deciding warp's XT row for q < 4 (so u = a exactly),
// the best vertex and vertex q - 3 for the shrink points.  One form for every
// lane, so a warp holding both kinds does not diverge.
template <int G, int N>
__device__ __forceinline__ void trial_rows(const GroupSmem<G, N>& g, int gi, int q, const float*& a, const float*& b) {
  const unsigned char* o = g.ord[gi];
  a = q < 4 ? g.XT[gi][q] : g.U[gi][o[0]];
  b = q < 4 ? g.XT[gi][q] : g.U[gi][o[q - 3]];
}

// Stable ranking of 19 values by one thread: rank[r] = #{s : v_s < v_r or
// (v_s == v_r and s < r)}; the slots are written to ord in rank order.  The
// outer loop is kept rolled: this runs on the decision path, and its fully
// unrolled form (19 x 19 compares) crowds the instruction cache that the
// evaluating warps share.
template <int G, int N>
__device__ __forceinline__ void rank_simplex(GroupSmem<G, N>& g, int gi, const int (&sl)[verts<N>()], const float (&fv)[verts<N>()]) {
#pragma unroll 1
  for (int r = 0; r < verts<N>(); ++r) {
    int rank = 0;
#pragma unroll
    for (int t = 0; t < verts<N>(); ++t) rank += (fv[t] < fv[r] || (fv[t] == fv[r] && t < r)) ? 1 : 0;
    g.ord[gi][rank] = (unsigned char)sl[r];
  }
}

// Value spread within tol_f (the other half of the exit test) from the ranked
// values in ord.
template <int G, int N>
__device__ __forceinline__ int value_spread_ok(const GroupSmem<G, N>& g, int gi, float tolf) {
  const float f0 = g.F[gi][g.ord[gi][0]];
  bool ok = true;
#pragma unroll
  for (int r = 1; r < verts<N>(); ++r) ok = ok && (fabsf(g.F[gi][g.ord[gi][r]] - f0) <= tolf);
  return ok ? 1 : 0;
}

// Ranking of freshly evaluated initial simplices, one lane per simplex.
// Returns whether the lane's simplex is active; okf: its values agree within
// tol_f.
template <int G, int N>
__device__ __forceinline__ bool init_rank(GroupSmem<G, N>& g, int lane, float tolf, bool& okf) {
  const bool live = lane < g.nsim;
  okf = false;
  if (live) {
    int sl[verts<N>()];
    float fv[verts<N>()];
#pragma unroll
    for (int r = 0; r < verts<N>(); ++r) {
      sl[r] = r;
      fv[r] = g.F[lane][r];
    }
    rank_simplex<G, N>(g, lane, sl, fv);
    g.active[lane] = 1;
    g.iters[lane] = 0;
    okf = value_spread_ok<G, N>(g, lane, tolf) != 0;
  }
  __syncwarp();
  return live;
}

// Lagarias decision and re-sort of every active simplex of a group after a
// trial wave, one lane per simplex (the slots and values of its vertices in
// registers, in rank order); only a shrink's coordinates, which are rare, are
// spread over all lanes.  Returns whether the lane's simplex is active; okf:
// its values agree within tol_f.
template <int G, int N>
__device__ __forceinline__ bool decide_group(GroupSmem<G, N>& g, int lane, float tolf, bool& okf) {
  const int gi = lane;
  const bool live = lane < g.nsim && g.active[lane] != 0;
  bool shrink = false;
  okf = false;
  if (live) {
    unsigned char* o = g.ord[gi];
    int sl[verts<N>()];
    float fv[verts<N>()];
#pragma unroll
    for (int r = 0; r < verts<N>(); ++r) {
      sl[r] = o[r];
      fv[r] = g.F[gi][sl[r]];
    }
    const float f1 = fv[0], fn = fv[N - 1], fw = fv[N];
    const float fr = g.FT[gi][0], fe = g.FT[gi][1], fco = g.FT[gi][2], fci = g.FT[gi][3];
    int kind;
    float fnew = 0.0f;
    if (fr < f1) {
      if (fe < fr) { kind = 1; fnew = fe; } else { kind = 0; fnew = fr; }
    } else if (fr < fn) {
      kind = 0; fnew = fr;
    } else if (fr < fw) {
      if (fco <= fr) { kind = 2; fnew = fco; } else kind = -1;
    } else {
      if (fci < fw) { kind = 3; fnew = fci; } else kind = -1;
    }
    g.iters[gi] += 1;
    shrink = kind < 0;
    if (!shrink) {
      // replace the worst vertex; the new point goes after every vertex with
      // a value <= its own (ties stay in front of it)
      const int ws = sl[N];
#pragma unroll
      for (int j = 0; j < N; ++j) g.U[gi][ws][j] = g.XT[gi][kind][j];
      g.F[gi][ws] = fnew;
      int pos = 0;
#pragma unroll
      for (int r = 0; r < N; ++r) pos += fv[r] <= fnew ? 1 : 0;
#pragma unroll
      for (int r = N; r >= 1; --r)
        if (r > pos) {
          sl[r] = sl[r - 1];
          fv[r] = fv[r - 1];
        }
#pragma unroll
      for (int r = 0; r < verts<N>(); ++r)
        if (r == pos) {
          sl[r] = ws;
          fv[r] = fnew;
        }
#pragma unroll
      for (int r = 0; r < verts<N>(); ++r) o[r] = (unsigned char)sl[r];
      okf = true;
#pragma unroll
      for (int r = 1; r < verts<N>(); ++r) okf = okf && (fabsf(fv[r] - fv[0]) <= tolf);
    } else {
      // shrink toward the best vertex: the values now, the coordinates below
#pragma unroll
      for (int r = 1; r < verts<N>(); ++r) g.F[gi][sl[r]] = g.FT[gi][4 + r - 1];
    }
  }
  // shrink coordinates: for each shrinking simplex, its N x N (vertex rank
  // >= 1, coordinate) updates over the lanes (the best vertex's row is only read)
  const unsigned smask = __ballot_sync(0xffffffffu, shrink);
  if (smask) {
    for (unsigned m = smask; m; m &= m - 1) {
      const int gs = __ffs(m) - 1;
      const unsigned char* o = g.ord[gs];
      for (int e = lane; e < N * N; e += 32) {
        const int r = e / N + 1, j = e - (r - 1) * N;
        g.U[gs][o[r]][j] = shrink_coord(g.U[gs][o[0]][j], g.U[gs][o[r]][j]);
      }
    }
    __syncwarp();
    // stable re-sort of the shrunk simplices
    if (shrink) {
      int sl[verts<N>()];
      float fv[verts<N>()];
#pragma unroll
      for (int r = 0; r < verts<N>(); ++r) {
        sl[r] = g.ord[gi][r];
        fv[r] = g.F[gi][sl[r]];
      }
      rank_simplex<G, N>(g, gi, sl, fv);
      okf = value_spread_ok<G, N>(g, gi, tolf) != 0;
    }
  }
  __syncwarp();
  return live;
}

// Order of a wave's simplices: turn[] lists the lanes with `live` set by
// increasing pulse width `upw` (the ln-space coordinate, clamped to the box).
// The candidates of one simplex differ little in pulse width, so 32
// consecutive candidates of this order end their pulse at nearly the same
// sample; with the 9-parameter model every candidate has the same width.
// Ordering the simplices (one per lane, ranked by 32 shuffles) takes the
// place of a 512-bin counting sort of all candidates, which cost the deciding
// warp 18 k of a decision's 42 k cycles for the same order to within the
// spread of one simplex.
template <int G, int N>
__device__ __forceinline__ void order_simplices(GroupSmem<G, N>& g, int lane, bool live, float upw, const SearchParams& P) {
  const unsigned lives = __ballot_sync(0xffffffffu, live);
  int rank = 0;
  if constexpr (search_coord<N>(kPw) < 0) {
    rank = __popc(lives & ((1u << lane) - 1u));
  } else {
    const int bits = __float_as_int(fminf(fmaxf(upw, P.lnlo), P.lnhi));
    const int key = live ? (bits ^ ((bits >> 31) & 0x7fffffff)) : 0x7fffffff;   // ordered as the floats are
#pragma unroll 8
    for (int l = 0; l < 32; ++l) {
      const int k = __shfl_sync(0xffffffffu, key, l);
      rank += k < key || (k == key && l < lane) ? 1 : 0;
    }
  }
  if (live) g.turn[rank] = (unsigned char)lane;
}

// A group's first wave, the initial vertices of its simplices (one warp).
template <int G, int N>
__device__ __forceinline__ void first_wave(GroupSmem<G, N>& g, const SearchParams& P, int lane) {
  constexpr int jp = search_coord<N>(kPw) < 0 ? 0 : search_coord<N>(kPw);
  const bool live = lane < g.nsim;
  order_simplices<G, N>(g, lane, live, live ? g.U[lane][0][jp] : 0.0f, P);
  if (lane == 0) g.kind = 0;
  if (lane == 0) g.state = kPending;
  if (lane == 0) g.nvalid = verts<N>() * g.nsim;
  if (lane == 0) g.evals = verts<N>() * g.nsim;
  __syncwarp();
}

// A group's next trial wave (one warp, one lane per simplex; `live`: the
// lane's simplex is active, okf: its values agree within tol_f).  First the
// other half of the exit test (Sec. 3.3: every vertex within tol_x of the
// best in max-norm) for the simplices that pass the first, spread over all
// lanes; a group with no active simplex left, or at its iteration cap, is
// done.  Then each lane sums its simplex's best N vertices row by row (N
// independent sums, two per packed instruction, 8-byte loads) and writes the
// four trial points (reflection, expansion, both contractions); the N shrink
// points are formed by the evaluating threads from the vertices.
// One lane per simplex instead of one per (simplex, coordinate) reads each
// row's slot once instead of N times and keeps the centroid in registers:
// with the ordering by simplex, 13.4 k cycles for 32 simplices among
// evaluating warps, where centroids, trial points, keys and sort took 34 k.
template <int G, int N>
__device__ __forceinline__ void next_wave(GroupSmem<G, N>& g, const SearchParams& P, int lane, int t_run, bool live,
                                          bool okf) {
  constexpr int jp = search_coord<N>(kPw) < 0 ? 0 : search_coord<N>(kPw);
  for (unsigned m = __ballot_sync(0xffffffffu, live && okf); m; m &= m - 1) {
    const int gs = __ffs(m) - 1;
    const unsigned char* o = g.ord[gs];
    bool ok = true;
    for (int e = lane; e < N * N; e += 32) {
      const int r = e / N + 1, j = e - (r - 1) * N;
      ok = ok && (fabsf(g.U[gs][o[r]][j] - g.U[gs][o[0]][j]) <= P.tolx);
    }
    if (__all_sync(0xffffffffu, ok) && lane == gs) {
      live = false;
      g.active[gs] = 0;
    }
  }
  const int nact = __popc(__ballot_sync(0xffffffffu, live));
  if (g.it >= t_run || nact == 0) {
    if (lane == 0) g.state = kDone;
    if (lane == 0) g.nvalid = 0;
    __syncwarp();
    return;
  }
  float upw = 0.0f;
  if (live) {
    const unsigned char* o = g.ord[lane];
    float acc[N];
    if constexpr (N % 2 == 0) {
      float2 a[N / 2];
#pragma unroll
      for (int j = 0; j < N / 2; ++j) a[j] = make_float2(0.0f, 0.0f);
#pragma unroll 3
      for (int r = 0; r < N; ++r) {
        const float2* x = reinterpret_cast<const float2*>(g.U[lane][o[r]]);
#pragma unroll
        for (int j = 0; j < N / 2; ++j) a[j] = __fadd2_rn(a[j], x[j]);
      }
#pragma unroll
      for (int j = 0; j < N / 2; ++j) {
        acc[2 * j] = a[j].x;
        acc[2 * j + 1] = a[j].y;
      }
    } else {
#pragma unroll
      for (int j = 0; j < N; ++j) acc[j] = 0.0f;
#pragma unroll 3
      for (int r = 0; r < N; ++r) {
        const float* x = g.U[lane][o[r]];
#pragma unroll
        for (int j = 0; j < N; ++j) acc[j] += x[j];
      }
    }
    const float* w = g.U[lane][o[N]];
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const float xb = acc[j] / (float)N;
#pragma unroll
      for (int q = 0; q < 4; ++q) g.XT[lane][q][j] = trial_coord(q, xb, w[j]);
      if (j == jp) upw = xb;
    }
  }
  order_simplices<G, N>(g, lane, live, upw, P);
  if (lane == 0) g.kind = 1;
  if (lane == 0) g.state = kPending;
  if (lane == 0) g.nvalid = trials<N>() * nact;
  if (lane == 0) g.evals += trials<N>() * nact;
  __syncwarp();
}

__device__ __forceinline__ int vload(const int& x) { return *reinterpret_cast<const volatile int*>(&x); }

// Make a group's set-up wave (or its end) visible to the block's warps.  The
// wave's data is written before; then the done count and the claim word are
// reset for the next sequence number, then the published word (sequence,
// chunks) is written, with block-scope fences between, so a warp that claims a
// chunk of this sequence sees the wave.  A finished group publishes 0 chunks.
template <int G, int N>
__device__ __forceinline__ void publish_wave(GroupSmem<G, N>& g, int lane) {
  __syncwarp();
  __threadfence_block();
  // every lane computes the words; lane 0 alone stores them (single
  // predicated stores, so the warp never splits around them)
  const int seq = ((vload(g.pub) >> 16) + 1) & 0x7fff;
  const int n = g.state == kDone ? 0 : (g.nvalid + 31) >> 5;
  if (lane == 0) atomicExch(&g.done, 0);
  if (lane == 0) atomicExch(&g.claim, seq << 16);
  __threadfence_block();
  if (lane == 0) atomicExch(&g.pub, (seq << 16) | n);
  __syncwarp();
}

// Claim the next chunk of a group's published wave, by the whole warp with
// uniform control flow: lane 0 alone reads the words and attempts the
// compare-and-swap (single predicated instructions) and every value is
// broadcast, so the warp stays converged.  Returns the chunk index and its
// wave's chunk count, or -1 when the wave has no chunk left, the claim word
// belongs to another sequence (a wave being published), or other warps kept
// winning the race (the caller tries again).
template <int G, int N>
__device__ __forceinline__ int try_claim(GroupSmem<G, N>& g, int lane, int& nchunks) {
  int pub = 0, old = 0;
  if (lane == 0) pub = vload(g.pub);
  pub = __shfl_sync(0xffffffffu, pub, 0);
  const int n = pub & 0xffff;
  if (n == 0) return -1;
  const int want = pub & ~0xffff;
  if (lane == 0) old = vload(g.claim);
  old = __shfl_sync(0xffffffffu, old, 0);
#pragma unroll 1
  for (int t = 0; t < 64; ++t) {
    if ((old & ~0xffff) != want || (old & 0xffff) >= n) return -1;
    int prev = 0;
    if (lane == 0) prev = atomicCAS(&g.claim, old, old + 1);
    prev = __shfl_sync(0xffffffffu, prev, 0);
    if (prev == old) {
      __threadfence_block();
      nchunks = n;
      return old & 0xffff;
    }
    old = prev;
  }
  return -1;
}

// The warp that completed a group's wave: Nelder-Mead decisions on the values
// just computed (ranking of the initial simplices, or the Lagarias step of
// every active simplex), then the group's next wave and its publication.
template <int G, int N>
__device__ __forceinline__ void advance_group(GroupSmem<G, N>& g, const SearchParams& P, int lane, int t_run) {
  bool live, okf;
  if (g.kind == 0) {
    live = init_rank<G, N>(g, lane, P.tolf, okf);
  } else {
    live = decide_group<G, N>(g, lane, P.tolf, okf);
    if (lane == 0) g.it += 1;
    __syncwarp();
  }
  next_wave<G, N>(g, P, lane, t_run, live, okf);
  publish_wave<G, N>(g, lane);
}

// Evaluate the candidate at position pos (wave order) of a group's pending
// wave; qs is the calling thread's propagator slot.  Returns 1 when that
// candidate's pulse ends inside the window (its pulse-end sample was
// integrated substep by substep), else 0 (also for pos past the wave).
template <int G, int N, bool LEAN, bool PACK>
__device__ __forceinline__ int eval_candidate(GroupSmem<G, N>& g, const SacStage& S, const SearchParams& P,
                                              const float* z, float* qs, int pos) {
  constexpr int NT = search_threads<G, N>();
  const unsigned live = __ballot_sync(0xffffffffu, pos < g.nvalid);   // the lanes that walk
  if (pos >= g.nvalid) return 0;
  int pe = 0;
  const SacConst& sc = S.sc;
  const float sum0 = S.st.sum0, c0 = S.st.c0;
  static_assert(!LEAN || N == N, "register-lean walk: 18 coordinates only");
  // both kinds of wave through one walk: a vertex is the row pair (v, v), for
  // which a + (a - a) / 2 = a exactly
  const float* a;
  const float* bb;
  float* out;
  if (g.kind == 0) {
    const int k = pos / verts<N>(), v = pos - k * verts<N>(), gi = g.turn[k];
    a = bb = g.U[gi][v];
    out = &g.F[gi][v];
  } else {
    const int k = pos / trials<N>(), q = pos - k * trials<N>(), gi = g.turn[k];
    trial_rows(g, gi, q, a, bb);
    out = &g.FT[gi][q];
  }
  if constexpr (LEAN) {
    const ULinSrc src{a, bb, true, S.pc, P.lnlo, P.lnhi};
    *out = objective_lean(src, sc, z, sum0, c0, &pe);
  } else {
    float u[N];
#pragma unroll
    for (int j = 0; j < N; ++j) u[j] = shrink_coord(a[j], bb[j]);
    *out = eval_u<N, PACK>(u, S.pc, P.lnlo, P.lnhi, sc, z, sum0, c0, qs, NT, &pe, live);
  }
  return pe;
}

// Group of a unit's simplex sg and its index in that group: group h holds the
// unit's simplices [group_start(h), group_start(h + 1)).
template <int G, int NG>
__device__ __forceinline__ int group_start(int h, int nunit, bool balanced) {
  return balanced ? (nunit * h) / NG : min(nunit, h * G);
}
template <int G, int NG>
__device__ __forceinline__ int group_of(int sg, int nunit, bool balanced, int& gi) {
  int h = 0;
#pragma unroll
  for (int t = 1; t < NG; ++t)
    if (sg >= group_start<G, NG>(t, nunit, balanced)) h = t;
  gi = sg - group_start<G, NG>(h, nunit, balanced);
  return h;
}

template <int G, int N, int NG, int MINB, bool LEAN, bool PACK>
__global__ void __launch_bounds__(search_threads<G, N>(), MINB) k_search(SearchParams P) {
  constexpr int NT = search_threads<G, N>();
  static_assert(NG >= 2 && NG <= kSearchWarps, "one warp sets up each group's first wave");
  extern __shared__ __align__(128) unsigned char smraw[];
  SearchSmem<G, N, NG>& S = *reinterpret_cast<SearchSmem<G, N, NG>*>(smraw);
  float* yraw = reinterpret_cast<float*>(smraw + ((sizeof(SearchSmem<G, N, NG>) + 127) / 128) * 128);
  float* z = yraw + P.lcap;
  float* qslot = z + P.lcap;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  if (tid == 0) {
    mbar_init(&S.bar, 1);
    fence_mbar_init();
    S.cur_b = -1;
    S.abort = 0;
  }
  __syncthreads();
  uint32_t phase = 0;

  for (;;) {
    if (tid == 0) S.unit = atomicAdd(P.counter, 1);
    __syncthreads();
    const int unit = S.unit;
    if (unit >= P.n_units) break;
    const int2 un = P.slot_list ? make_int2(P.slot_list[unit / P.ngroups], unit % P.ngroups) : P.units[unit];
    const int b = un.x, g0 = un.y;
    if (b != S.cur_b) {
      const DevSac d = P.sacs[b];
      if (!stage_trace(d, P.traces, yraw, z, &S.bar, phase, &S.sv.st)) {
        if (tid == 0) raise_error(P.err, kErrWaitTimeout);
        return;
      }
      if (tid < kNumParams) S.sv.pc[tid] = P.pc[(size_t)b * kNumParams + tid];
      if (tid == 0) {
        S.sv.sc = sac_const(d);
        S.cur_b = b;
      }
      __syncthreads();
    }
    // this unit's simplices: units of NG G (the last takes the rest), or, with
    // P.balanced, the saccade's S simplices split evenly over its P.ngroups
    // units; within the unit, groups of G in order, or an even split
    int s0, nunit;
    const bool bal = P.balanced != 0;
    if (bal) {
      s0 = (int)(((long long)g0 * P.S) / P.ngroups);
      nunit = (int)(((long long)(g0 + 1) * P.S) / P.ngroups) - s0;   // <= NG G
    } else {
      s0 = g0 * NG * G;
      nunit = min(NG * G, P.S - s0);
    }
    // resumable mode (serving): iterations already done by this saccade and
    // this launch's share; the simplex state lives in HBM between launches
    const int it0 = P.state ? P.progress[b] : 0;
    const int t_run = P.state ? min(P.round_iters, P.T - it0) : P.T;
    if (tid < NG) {
      GroupSmem<G, N>& g = S.grp[tid];
      g.nsim = group_start<G, NG>(tid + 1, nunit, bal) - group_start<G, NG>(tid, nunit, bal);
      g.it = 0;
      g.evals = 0;
      g.pe = 0;
      g.nvalid = 0;
      g.state = g.nsim > 0 ? kPending : kDone;
      g.pub = 0;
      g.claim = 0;
      g.done = 0;
    }
    if (it0 > 0) {
      // restore the simplices: vertices, values, order, flags
      const float* gstate = P.state + ((size_t)b * P.S + (size_t)s0) * state_floats<N>();
      for (int idx = tid; idx < nunit * state_floats<N>(); idx += NT) {
        const int sg = idx / state_floats<N>(), r = idx - sg * state_floats<N>();
        int gi;
        GroupSmem<G, N>& g = S.grp[group_of<G, NG>(sg, nunit, bal, gi)];
        const float v = gstate[idx];
        if (r < verts<N>() * N) (&g.U[gi][0][0])[r] = v;
        else if (r < verts<N>() * N + verts<N>()) g.F[gi][r - verts<N>() * N] = v;
        else if (r < verts<N>() * N + 2 * verts<N>()) g.ord[gi][r - verts<N>() * N - verts<N>()] = (unsigned char)__float_as_int(v);
        else if (r == state_floats<N>() - 2) g.active[gi] = __float_as_int(v);
        else if (r == state_floats<N>() - 1) g.iters[gi] = __float_as_int(v);
      }
    } else {
      // ---- initial simplices: centre (Philox for starts >= 1) + step e_i
      constexpr int kBlk = (N + 3) / 4;   // Philox blocks of 4 coordinates
      for (int t5 = tid; t5 < kBlk * nunit; t5 += NT) {
        const int sg = t5 / kBlk, blk = t5 - sg * kBlk;
        int gi;
        GroupSmem<G, N>& g = S.grp[group_of<G, NG>(sg, nunit, bal, gi)];
        const int s = s0 + sg;
        uint32_t r[4] = {0u, 0u, 0u, 0u};
        if (s != 0) philox4x32_10((uint32_t)P.sac_index[b], (uint32_t)s, (uint32_t)blk, 0u, P.seed_lo, P.seed_hi, r);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int j = 4 * blk + q;
          if (j < N)
            g.U[gi][0][j] = s == 0 ? 0.0f : P.lnlo + (P.lnhi - P.lnlo) * ((float)(r[q] >> 8) * (1.0f / 16777216.0f));
        }
      }
      __syncthreads();
      for (int idx = tid; idx < nunit * N * N; idx += NT) {
        const int sg = idx / (N * N);
        int gi;
        GroupSmem<G, N>& g = S.grp[group_of<G, NG>(sg, nunit, bal, gi)];
        const int rem = idx - sg * N * N;
        const int v = rem / N + 1, j = rem - (v - 1) * N;
        float x = g.U[gi][0][j];
        if (j == v - 1) x += P.step;
        g.U[gi][v][j] = x;
      }
    }
    __syncthreads();
    // warp h < NG sets up and publishes group h's first wave
    if (warp < NG) {
      GroupSmem<G, N>& g = S.grp[warp];
      if (g.nsim > 0) {
        if (it0 > 0) next_wave<G, N>(g, P, lane, t_run, lane < g.nsim && g.active[lane] != 0, false);
        else first_wave<G, N>(g, P, lane);
        publish_wave<G, N>(g, lane);
      }
    }
    __syncthreads();

    // ---- steps, with no block barrier: each warp claims 32-candidate chunks
    // of any group's published wave (the group it worked on last first, then
    // the following ones in turn), evaluates them and counts them done; the
    // warp that completes a wave takes that group's decisions and publishes
    // its next wave while the other warps work on the other groups' waves.
    // All warps start on group 0, so the groups' waves complete one after
    // another and each group's decisions overlap the evaluation of the
    // others'.  Every decision to leave the loop is taken on lane 0 and
    // broadcast; a warp that finds nothing to claim waits, for at most
    // kMaxIdleCycles, until a wave is published or every group is done.
    int pref = 0;
    long long idle_since = -1;
#pragma unroll 1
    for (;;) {
      int gsel = -1, ch = -1, nch = 0;
#pragma unroll 1
      for (int t = 0; t < NG && ch < 0; ++t) {
        const int h = pref + t < NG ? pref + t : pref + t - NG;
        ch = try_claim<G, N>(S.grp[h], lane, nch);
        if (ch >= 0) gsel = h;
      }
      if (ch >= 0) {
        __syncwarp();   // orders lane 0's acquire of the wave before every lane's reads
        GroupSmem<G, N>& g = S.grp[gsel];
        const int npe = __popc(__ballot_sync(0xffffffffu,
                                             eval_candidate<G, N, LEAN, PACK>(g, S.sv, P, z, qslot + tid, ch * 32 + lane)));
        __syncwarp();
        __threadfence_block();   // the chunk's values before its done count
        if (lane == 0 && npe) atomicAdd(&g.pe, npe);
        int done_before = 0;
        if (lane == 0) done_before = atomicAdd(&g.done, 1);
        done_before = __shfl_sync(0xffffffffu, done_before, 0);
        const bool last = done_before == nch - 1;
        if (last) __threadfence_block();
        __syncwarp();
        if (last) {
          advance_group<G, N>(g, P, lane, t_run);
          pref = gsel + 1 < NG ? gsel + 1 : 0;
        } else {
          pref = gsel;
        }
        idle_since = -1;
        continue;
      }
      // nothing to claim: 1 = every group done or the block aborts, 2 = waited
      // too long; lane 0's view of the words and the clock decides for the warp
      int fin = 0;
      {
        const long long now = clock64();
        if (idle_since < 0) idle_since = now;
        bool all_done = true;
#pragma unroll
        for (int h = 0; h < NG; ++h) all_done = all_done && vload(S.grp[h].state) == kDone;
        fin = (vload(S.abort) || all_done) ? 1 : (now - idle_since > kMaxIdleCycles ? 2 : 0);
      }
      fin = __shfl_sync(0xffffffffu, fin, 0);
      if (fin == 2) {
        if (lane == 0) raise_error(P.err, kErrWaitTimeout);
        if (lane == 0) atomicExch(&S.abort, 1);
        break;
      }
      if (fin) break;
      __nanosleep(128);
    }
    __syncthreads();
    if (S.abort) return;

    if (P.state) {
      // save the simplices for the next launch
      float* gstate = P.state + ((size_t)b * P.S + (size_t)s0) * state_floats<N>();
      for (int idx = tid; idx < nunit * state_floats<N>(); idx += NT) {
        const int sg = idx / state_floats<N>(), r = idx - sg * state_floats<N>();
        int gi;
        const GroupSmem<G, N>& g = S.grp[group_of<G, NG>(sg, nunit, bal, gi)];
        float v;
        if (r < verts<N>() * N) v = (&g.U[gi][0][0])[r];
        else if (r < verts<N>() * N + verts<N>()) v = g.F[gi][r - verts<N>() * N];
        else if (r < verts<N>() * N + 2 * verts<N>()) v = __int_as_float((int)g.ord[gi][r - verts<N>() * N - verts<N>()]);
        else if (r == state_floats<N>() - 2) v = __int_as_float(g.active[gi]);
        else if (r == state_floats<N>() - 1) v = __int_as_float(g.iters[gi]);
        else v = 0.0f;
        gstate[idx] = v;
      }
    }

    // ---- unit result: lowest value, ties to the lowest simplex index
    if (tid < 32) {
      float* rec = P.unit_best + (size_t)(P.slot_list ? b * P.ngroups + g0 : unit) * kUnitRec;
      float f = INFINITY;
      int best = 0x7fffffff;
      for (int sg = lane; sg < nunit; sg += 32) {
        int gi;
        const GroupSmem<G, N>& g = S.grp[group_of<G, NG>(sg, nunit, bal, gi)];
        const float fv = g.F[gi][g.ord[gi][0]];
        if (fv < f || (fv == f && sg < best)) { f = fv; best = sg; }
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const float f2 = __shfl_xor_sync(0xffffffffu, f, o);
        const int b2 = __shfl_xor_sync(0xffffffffu, best, o);
        if (f2 < f || (f2 == f && b2 < best)) { f = f2; best = b2; }
      }
      const int evals_prev = it0 > 0 ? __float_as_int(rec[3]) : 0;
      const int pe_prev = it0 > 0 ? __float_as_int(rec[22]) : 0;
      int evals = 0, pes = 0;
      for (int h = 0; h < NG; ++h) {
        evals += S.grp[h].evals;
        pes += S.grp[h].pe;
      }
      __syncwarp();
      if (best < nunit) {
        int gi;
        const GroupSmem<G, N>& g = S.grp[group_of<G, NG>(best, nunit, bal, gi)];
        if (lane < N) rec[4 + lane] = g.U[gi][g.ord[gi][0]][lane];
        if (lane == 0) {
          rec[0] = f;
          rec[1] = __int_as_float(s0 + best);
          rec[2] = __int_as_float(g.iters[gi]);
          rec[3] = __int_as_float(evals_prev + evals);
          rec[22] = __int_as_float(pe_prev + pes);
        }
      }
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ finalize
// FP64 re-computation of the winner's error (the serial check next to the
// parallel value, as Fig. 4's CPU_check column), one warp per saccade.  The
// same RK4 map is applied in double precision: within one input phase one RK4
// step of e' = A e is e <- e + Q e with Q = hA(I + hA/2(I + hA/3(I + hA/4))),
// raised to one sample interval by squaring; the pulse-end substep is split
// into two RK4 steps.  Independent of the FP32 search formulation (double
// precision, matrix powers instead of substeps, its own equilibria).
//
// The FP64 pipes bound it: a warp instruction holds its sub-partition's for
// about 64 cycles however many lanes it uses, so the count of warp
// instructions is what is kept small and every lane carries work.  Matrices
// keep the plant's block form (a 4x4 mechanical block, a 4x2 coupling, a
// diagonal activation pair: 26 entries) with one entry per lane, five FMAs a
// product; vectors go one row per lane; and a phase's samples go 32 at a
// time, lane l holding the state after sample l + 1: the first 32 states come
// by doubling ((I + P)^c takes states 1 .. c to c + 1 .. 2 c, one row of one
// state per lane), (I + P)^32 moves them on.  One thread per saccade with
// dense 6x6 matrices in local memory took 365 us for one saccade of 150
// samples and 880 us for 2,000 uneven ones.

// Products by entry: entry e of a 32-double matrix is m[e / 4][e % 4] for
// e < 16, c[(e - 16) / 2][(e - 16) % 2] for e < 24, d[e - 24] for e < 26 and
// 0 above.  Entry e of a b is the dot product of a[ia ..] and b[ib + sb ..]
// over four terms plus a[ka] b[kb]; entries past 25 serve as zeros.
struct Lane64 {
  int e, ia, ib, sb, ka, kb;
  double unit;   // entry e of the identity
  __device__ explicit Lane64(int lane) : e(lane) {
    ia = ib = ka = kb = 26;
    sb = 0;
    unit = 0.0;
    if (e < 16) {
      ia = e & ~3;
      ib = e & 3;
      sb = 4;
      unit = (e >> 2) == (e & 3) ? 1.0 : 0.0;
    } else if (e < 24) {
      ia = 4 * ((e - 16) >> 1);
      ib = 16 + (e & 1);
      sb = 2;
      ka = e;
      kb = 24 + (e & 1);
    } else if (e < 26) {
      ka = kb = e;
      unit = 1.0;
    }
  }
  __device__ __forceinline__ double mul(const double* a, const double* b) const {
    double t = a[ka] * b[kb];
#pragma unroll
    for (int k = 0; k < 4; ++k) t = fma(a[ia + k], b[ib + sb * k], t);
    return t;
  }
  // m[e] = v once every lane has read what it needs
  __device__ __forceinline__ void put(double* m, double v) const {
    __syncwarp();
    m[e] = v;
    __syncwarp();
  }
};

struct Warp64 {
  double A[32], Q[32], W[32], B[32], P[6][32];
  double E[32][6];               // states after samples 1 .. 32 of a phase
  double v[6];                   // the walk's current state
  double par[kNumParams], rcp[12];
  float opc[kNumParams];
};

// out = T4(h A) - I by Horner (w: scratch).
__device__ void step_inc64(const Lane64& L, const double* A, double h, double* w, double* out) {
  L.put(w, fma(0.25 * h, A[L.e], L.unit));
  L.put(w, fma(h * (1.0 / 3.0), L.mul(A, w), L.unit));
  L.put(w, fma(0.5 * h, L.mul(A, w), L.unit));
  L.put(out, h * L.mul(A, w));
}

// r = a + b + a b (increment form of (I + a)(I + b)); r may be a or b.
__device__ __forceinline__ void mul_inc64(const Lane64& L, const double* a, const double* b, double* r) {
  L.put(r, a[L.e] + b[L.e] + L.mul(a, b));
}

// out = (I + q)^n - I for n >= 1 (left to right; out is not q).
__device__ void pow_inc64(const Lane64& L, const double* q, int n, double* out) {
  L.put(out, q[L.e]);
  for (int b = 30 - __clz(n); b >= 0; --b) {
    mul_inc64(L, out, out, out);
    if ((n >> b) & 1) mul_inc64(L, out, q, out);
  }
}

// e <- (I + q) e on every lane's own vector.
__device__ __forceinline__ void apply_inc64(const double* q, double (&e)[6]) {
  double n[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    n[i] = fma(q[16 + 2 * i], e[4], e[i]);
    n[i] = fma(q[17 + 2 * i], e[5], n[i]);
#pragma unroll
    for (int k = 0; k < 4; ++k) n[i] = fma(q[4 * i + k], e[k], n[i]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) e[i] = n[i];
  e[4] = fma(q[24], e[4], e[4]);
  e[5] = fma(q[25], e[5], e[5]);
}

// Row i of (I + q) v (the zero entries past 25 pad the activation rows).
__device__ __forceinline__ double row_inc64(const double* q, const double* v, int i) {
  const bool mech = i < 4;
  double t = fma(q[mech ? 16 + 2 * i : i == 4 ? 24 : 26], v[4], v[i]);
  t = fma(q[mech ? 17 + 2 * i : i == 5 ? 25 : 26], v[5], t);
#pragma unroll
  for (int k = 0; k < 4; ++k) t = fma(q[mech ? 4 * i + k : 26], v[k], t);
  return t;
}

// v <- (I + q) v for the warp's vector in shared memory.
__device__ __forceinline__ void apply_vec64(const Lane64& L, const double* q, double* v) {
  const double t = row_inc64(q, v, L.e < 6 ? L.e : 0);
  __syncwarp();
  if (L.e < 6) v[L.e] = t;
  __syncwarp();
}

__device__ __forceinline__ double warp_sum64(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

struct Err64 {
  double s2, s1;   // this lane's share of the squared and absolute errors
  __device__ __forceinline__ void add(double r) {
    s2 = fma(r, r, s2);
    s1 += fabs(r);
  }
};

// n samples of one phase from the state W.v, the first of them sample k0,
// around the equilibrium angle th; leaves the state after the last one in
// W.v.  W.P[0] holds the one-sample propagator.
__device__ void run_phase64(const Lane64& L, Warp64& W, int k0, int n, double th, double sg, const float* y, Err64& err) {
  if (n <= 0) return;
  apply_vec64(L, W.P[0], W.v);
  if (L.e < 6) W.E[0][L.e] = W.v[L.e];
  __syncwarp();
#pragma unroll 1
  for (int b = 0; b < 5 && (1 << b) < n; ++b) {
    // states 1 .. c give c + 1 .. 2 c by P[b], whose square is P[b + 1]
    for (int t = L.e; t < 6 << b; t += 32) {
      const int st = t / 6, i = t - 6 * st;
      W.E[st + (1 << b)][i] = row_inc64(W.P[b], W.E[st], i);
    }
    if ((2 << b) < n) mul_inc64(L, W.P[b], W.P[b], W.P[b + 1]);
    __syncwarp();
  }
  double e[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) e[i] = W.E[L.e][i];   // (lanes past n hold nothing that is used)
#pragma unroll 1
  for (int i = L.e;; i += 32) {
    if (i < n) err.add(sg * (th + e[0]) - (double)y[k0 + i]);
    if (i - L.e + 32 >= n) break;   // warp-uniform
    apply_inc64(W.P[5], e);
  }
  __syncwarp();
  if (L.e == ((n - 1) & 31))
#pragma unroll
    for (int i = 0; i < 6; ++i) W.v[i] = e[i];
  __syncwarp();
}

// Mean squared and mean absolute error of the OPC vector W.opc's trajectory
// against the trace y, FP64, by one warp.
__device__ void errors64(const Lane64& L, Warp64& W, const DevSac& d, const float* y, double* mse, double* mae) {
  if (L.e < kNumParams) W.par[L.e] = (double)W.opc[L.e];
  __syncwarp();
  const double* p = W.par;
  // the reciprocals, one lane each
  enum { iJ, iBa, iBn, iSa, iSn, iSLa, iSLn, iTaA, iTaN, iTdA, iTdN };
  {
    const int idx[7] = {kJ, kBAg, kBAnt, kSeAg, kSeAnt, kSeAg, kSeAnt};
    double den = 1.0, num = 1.0;
    if (L.e < 7) {
      den = p[idx[L.e]] + (L.e == iSLa ? p[kLtAg] : L.e == iSLn ? p[kLtAnt] : 0.0);
    } else if (L.e < 11) {
      den = p[kTacAg + L.e - 7];   // the four time constants, in OPC order
      num = 1000.0;
    }
    const double r = num / den;
    if (L.e < 11) W.rcp[L.e] = r;
    __syncwarp();
  }
  const double* r = W.rcp;
  const double th0 = d.th0, thf = d.thf, sg = d.sign;
  const double ag = p[kSeAg] * r[iSLa], an = p[kSeAnt] * r[iSLn], kp = p[kNcAg] + p[kNcAnt];
  // substeps refined for stiff candidates, the oracle's rule in double
  const double rate = fmax(fmax(r[iTaA], r[iTaN]), fmax(r[iTdA], r[iTdN]));
  const double est = p[kBp] * r[iJ] + (p[kSeAg] + p[kLtAg]) * r[iBa] + (p[kSeAnt] + p[kLtAnt]) * r[iBn] + rate;
  int nsub = d.nsub;
  double h = 1.0 / ((double)d.fs * nsub);
  for (int t = 0; t < kMaxRefine && !(h * est <= 2.5); ++t) {
    h *= 0.5;
    nsub *= 2;
  }
  double tau = p[kPw] * (double)d.fs * (double)nsub / 1000.0;
  if (!(tau >= 0.0)) tau = 0.0;
  if (tau > 1.0e9) tau = 1.0e9;
  const double fl = floor(tau);
  const double frac = tau - fl;
  // equilibria, one lane each: rest at th0, the pulse held, rest at thf
  double s0[6], s1[6], s2[6];
  {
    const double th = L.e == 0 ? th0 : thf;
    const double ta = p[kNcFix] + p[kNcAg] * th, tn = p[kNcFix] - p[kNcAnt] * th;
    double fa = ta * (1.0 + p[kLtAg] * r[iSa]) + p[kLtAg] * th;
    double fn = tn * (1.0 + p[kLtAnt] * r[iSn]) - p[kLtAnt] * th;
    if (L.e == 1) {
      fa = p[kNsacAg];
      fn = p[kNsacAnt];
    }
    const double q = (ag * fa - an * fn) / (kp + ag * p[kLtAg] + an * p[kLtAnt]);
    const double xa = ag * (fa - p[kLtAg] * q), xn = an * (fn + p[kLtAnt] * q);
    const double s[6] = {q, 0.0, q + xa * r[iSa], xn * r[iSn] - q, fa, fn};
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      s0[i] = __shfl_sync(0xffffffffu, s[i], 0);
      s1[i] = __shfl_sync(0xffffffffu, s[i], 1);
      s2[i] = __shfl_sync(0xffffffffu, s[i], 2);
    }
  }
  Err64 err{0.0, 0.0};
  const int kend = d.onset < d.L - 1 ? d.onset : d.L - 1;
  for (int k = L.e; k <= kend; k += 32) err.add(sg * th0 - (double)y[k]);   // at rest up to onset
  const int ntot = d.L - 1 - d.onset;
  if (ntot > 0) {
    // plant matrix of the pulse phase; the step phase differs in entries 24, 25
    {
      double a = 0.0;
      switch (L.e) {
        case 1: a = 1.0; break;
        case 4: a = -(p[kSeAg] + p[kSeAnt] + kp) * r[iJ]; break;
        case 5: a = -p[kBp] * r[iJ]; break;
        case 6: a = p[kSeAg] * r[iJ]; break;
        case 7: a = -p[kSeAnt] * r[iJ]; break;
        case 8: a = p[kSeAg] * r[iBa]; break;
        case 10: a = -(p[kSeAg] + p[kLtAg]) * r[iBa]; break;
        case 12: a = -p[kSeAnt] * r[iBn]; break;
        case 15: a = -(p[kSeAnt] + p[kLtAnt]) * r[iBn]; break;
        case 20: a = r[iBa]; break;
        case 23: a = r[iBn]; break;
        case 24: a = -r[iTaA]; break;
        case 25: a = -r[iTdN]; break;
        default: break;
      }
      L.put(W.A, a);
    }
    int n1, jsw = 0;
    bool sw;
    if (fl >= (double)ntot * nsub) {
      n1 = ntot;
      sw = false;
    } else {
      const int J = (int)fl;
      n1 = J / nsub;
      jsw = J - n1 * nsub;
      sw = true;
    }
    if (L.e == 0)
#pragma unroll
      for (int i = 0; i < 6; ++i) W.v[i] = s0[i] - s1[i];
    step_inc64(L, W.A, h, W.W, W.Q);
    if (n1 > 0) {
      pow_inc64(L, W.Q, nsub, W.P[0]);
      run_phase64(L, W, d.onset + 1, n1, s1[0], sg, y, err);
    }
    if (sw) {
      // the sample that holds the pulse end
      if (jsw > 0) {
        pow_inc64(L, W.Q, jsw, W.B);
        apply_vec64(L, W.B, W.v);
      }
      step_inc64(L, W.A, frac * h, W.W, W.B);
      apply_vec64(L, W.B, W.v);
      if (L.e == 0)
#pragma unroll
        for (int i = 0; i < 6; ++i) W.v[i] += s1[i] - s2[i];
      L.put(W.A, L.e == 24 ? -r[iTdA] : L.e == 25 ? -r[iTaN] : W.A[L.e]);
      step_inc64(L, W.A, h - frac * h, W.W, W.B);
      apply_vec64(L, W.B, W.v);
      step_inc64(L, W.A, h, W.W, W.Q);
      if (jsw + 1 < nsub) {
        pow_inc64(L, W.Q, nsub - 1 - jsw, W.B);
        apply_vec64(L, W.B, W.v);
      }
      const int k = d.onset + 1 + n1;
      if (L.e == 0) err.add(sg * (s2[0] + W.v[0]) - (double)y[k]);
      if (k + 1 < d.L) {
        pow_inc64(L, W.Q, nsub, W.P[0]);
        run_phase64(L, W, k + 1, d.L - 1 - k, s2[0], sg, y, err);
      }
    }
  }
  *mse = warp_sum64(err.s2) / d.L;
  *mae = warp_sum64(err.s1) / d.L;
}

// Result of one saccade per warp (= block): the lowest value over its unit
// records (ties to the lowest simplex), the winner's OPC vector and its FP64
// errors.
template <int N>
__global__ void __launch_bounds__(32) k_finalize(const DevSac* sacs, const float* traces, const float* pc,
                                                 const int* ustart, int ngroups, const float* unit_best, float lnlo,
                                                 float lnhi, int n, opmm_fit_result* out, const int* list) {
  __shared__ Warp64 W;
  const int i = blockIdx.x, lane = threadIdx.x;
  if (i >= n) return;
  const Lane64 L(lane);
  const int b = list ? list[i] : i;
  int w = 0x7fffffff, wsimp = 0x7fffffff, evals = 0, pe = 0;
  float wf = INFINITY;
  const int u0 = ustart ? ustart[b] : b * ngroups;   // slot-major records when no start table
  for (int u = u0 + lane; u < u0 + ngroups; u += 32) {
    const float* rec = unit_best + (size_t)u * kUnitRec;
    const float f = rec[0];
    const int s = __float_as_int(rec[1]);
    evals += __float_as_int(rec[3]);
    pe += __float_as_int(rec[22]);
    if (w == 0x7fffffff || f < wf || (f == wf && s < wsimp)) { w = u; wf = f; wsimp = s; }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const float f2 = __shfl_xor_sync(0xffffffffu, wf, o);
    const int s2 = __shfl_xor_sync(0xffffffffu, wsimp, o), w2 = __shfl_xor_sync(0xffffffffu, w, o);
    evals += __shfl_xor_sync(0xffffffffu, evals, o);
    pe += __shfl_xor_sync(0xffffffffu, pe, o);
    if (f2 < wf || (f2 == wf && (s2 < wsimp || (s2 == wsimp && w2 < w)))) { w = w2; wf = f2; wsimp = s2; }
  }
  const DevSac d = sacs[b];
  const float* rec = unit_best + (size_t)w * kUnitRec;
  if (lane < kNumParams) {
    // as u_to_p, one entry per lane
    const int c = search_coord<N>(lane);
    const float p0 = pc[(size_t)b * kNumParams + lane];
    W.opc[lane] = c < 0 ? p0 : p0 * __expf(fminf(fmaxf(rec[4 + (c < 0 ? 0 : c)], lnlo), lnhi));
  }
  __syncwarp();
  double mse = INFINITY, mae = INFINITY;
  const bool ok = isfinite(wf);
  if (ok) errors64(L, W, d, traces + d.off, &mse, &mae);
  opmm_fit_result& r = out[i];
  if (lane < kNumParams) r.opc[lane] = W.opc[lane];
  if (lane == 0) {
    r.f = wf;
    r.iterations_run = __float_as_int(rec[2]);
    r.winner = wsimp;
    r.evaluations = evals;
    r.pulse_end_evals = pe;
    r.reserved = 0;
    r.source = OPMM_SOURCE_PLAIN;
    r.rms_deg = ok ? sqrt(mse) : INFINITY;
    r.l1_deg = mae;
    r.status = ok ? 0 : 1;
  }
}

// ------------------------------------------------------------------ refinement
// Gradient-based refinement after the search (Sec. 5 proposes gradient
// methods as the alternative to Nelder-Mead): Levenberg-Marquardt on the
// residual vector r_k = theta_k(u) - y_k of one saccade per block, in the
// search's ln coordinates, box and clamp.  One iteration: at a new point the
// Jacobian by central differences of step delta (2N trajectories, one per
// thread; a column whose two points are too stiff is zero), A = J^T J and
// g = J^T r (FP32 products, compensated sums); (A + lambda D) du = -g with
// D = diag(max(A_jj, 1e-9
// max_i A_ii)) solved by Cholesky in FP64; u' = clamp(u + du); accept when
// f(u') < f(u) (lambda / 10, floor 1e-12, new Jacobian), else lambda * 10
// (ceiling 1e12).  f = sum_k r_k^2 / L over every sample.  Stops early when
// A is zero or the system is not positive definite.
constexpr int kRefineThreads = 64;

// Floats between trajectory rows: an odd number, so that threads that write
// one row each, sample by sample, and dot products that read the same sample
// of many rows, stay on distinct shared-memory banks.
__host__ __device__ constexpr int refine_pitch(int lcap) { return lcap + 1; }   // lcap is a multiple of 4

struct RowSink {
  float* out;
  __device__ __forceinline__ void emit(int k, float dth) { out[k] = dth; }
  __device__ __forceinline__ void block_end() {}
};

// theta_k - thf (positive frame) for every sample of the window into row;
// false (row untouched past onset) when the candidate is too stiff.
// qs: the calling thread's propagator slot in shared memory (stride
// kRefineThreads), so that the powering runs in place as in the search.
__device__ bool refine_row(const float (&p)[kNumParams], const SacConst& sc, float* row, int* pe, float* qs) {
  const int kend = min(sc.onset, sc.L - 1);
  for (int k = 0; k <= kend; ++k) row[k] = sc.th0 - sc.thf;
  RowSink s{row};
  return walk<RowSink, false, true>(p, sc, s, qs, kRefineThreads, true, pe) >= 0;
}

template <int N>
struct RefineSmem {
  double A[N * N];
  double M[N * N];   // damped system, factored in place
  double du[N];
  double inv[N];     // reciprocals of the factor's diagonal
  double g[N];
  double red[kRefineThreads];
  float u[N], ut[N];
  float pc[kNumParams];
  double f, ft, lambda;
  int bad[2 * N];
  int need_jac, go, trial_ok, cur, acc, evals, pe;
  SacConst sc;
  TraceStage st;
  uint64_t bar;
};

// Block sum of per-thread FP64 partials (all threads call it).
template <int N>
__device__ double refine_sum(RefineSmem<N>& S, double v) {
  S.red[threadIdx.x] = v;
  __syncthreads();
  for (int o = kRefineThreads / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) S.red[threadIdx.x] += S.red[threadIdx.x + o];
    __syncthreads();
  }
  const double r = S.red[0];
  __syncthreads();
  return r;
}

// f of a stored trajectory row against the staged trace (all threads).
template <int N>
__device__ double refine_f(RefineSmem<N>& S, const float* row, const float* z, int L) {
  double acc = 0.0;
  for (int k = threadIdx.x; k < L; k += kRefineThreads) {
    const double e = (double)row[k] - (double)z[k];
    acc += e * e;
  }
  return refine_sum<N>(S, acc) / (double)L;
}

// SMEM: the N + 2 rows that the dot products of J^T J read (the
// Jacobian's columns, formed in place of the trajectories at u + delta, and
// the current and the trial point's trajectory) live in dynamic shared memory
// after the staged trace (short windows), else in the per-block global scratch
// area, where the N trajectories at u - delta always go: they are written and
// read once per Jacobian, and without them four blocks fit on an SM instead of
// two (windows of 400 samples), which is what hides the FP64 factorisation of
// one block (40 k of an iteration's 107 k cycles, on one warp) behind the
// others.
template <int N, bool SMEM>
__global__ void __launch_bounds__(kRefineThreads) k_refine(const DevSac* sacs, const float* traces, const float* pcs,
                                                            const float* start, int K, float lnlo, float lnhi,
                                                            float delta, float lambda0, int lcap, float* scratch,
                                                            opmm_fit_result* out, unsigned* err) {
  __shared__ RefineSmem<N> S;
  extern __shared__ __align__(128) unsigned char smraw[];
  float* yraw = reinterpret_cast<float*>(smraw);
  float* z = yraw + lcap;
  float* qslot = z + lcap;                                  // kQSlotFloats x kRefineThreads
  const int b = blockIdx.x, tid = threadIdx.x;
  const DevSac d = sacs[b];
  const int pitch = refine_pitch(lcap);
  float* minus = scratch + (size_t)b * (SMEM ? N : 2 * N + 2) * (size_t)pitch;
  float* rows = SMEM ? qslot + kQSlotFloats * kRefineThreads : minus + (size_t)N * pitch;
  if (tid == 0) {
    mbar_init(&S.bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  uint32_t phase = 0;
  if (!stage_trace(d, traces, yraw, z, &S.bar, phase, &S.st)) {
    if (tid == 0) raise_error(err, kErrWaitTimeout);
    return;
  }
  if (tid < kNumParams) S.pc[tid] = pcs[(size_t)b * kNumParams + tid];
  if (tid == 0) {
    S.sc = sac_const(d);
    S.lambda = lambda0;
    S.need_jac = 1;
    S.cur = 0;
    S.acc = 0;
    S.evals = 1;
    S.pe = 0;
  }
  __syncthreads();
  // start point: the coordinate of the first OPC entry each one scales
  if (tid < N) {
    int j0 = 0;
    for (int j = kNumParams - 1; j >= 0; --j)
      if (search_coord<N>(j) == tid) j0 = j;
    const float u = logf(start[(size_t)b * kNumParams + j0] / S.pc[j0]);
    S.u[tid] = fminf(fmaxf(u, lnlo), lnhi);
  }
  __syncthreads();
  const SacConst sc = S.sc;
  float* rcur[2] = {rows + (size_t)N * pitch, rows + (size_t)(N + 1) * pitch};
  if (tid == 0) {
    float p[kNumParams];
    u_to_p<N>(S.u, S.pc, lnlo, lnhi, p);
    int pe = 0;
    S.trial_ok = refine_row(p, sc, rcur[0], &pe, qslot + tid) ? 1 : 0;
    S.pe += pe;
  }
  __syncthreads();
  {
    const double f = refine_f<N>(S, rcur[0], z, sc.L);
    if (tid == 0) S.f = S.trial_ok && isfinite(f) ? f : INFINITY;
  }
  __syncthreads();
#pragma unroll 1
  for (int it = 0; it < K; ++it) {
    if (!isfinite(S.f)) break;
    const float* r0 = rcur[S.cur];
    if (S.need_jac) {
      if (tid < 2 * N) {
        const int j = tid >> 1;
        float ut[N];
#pragma unroll
        for (int c = 0; c < N; ++c) ut[c] = S.u[c];
        ut[j] += (tid & 1) ? -delta : delta;
        float p[kNumParams];
        u_to_p<N>(ut, S.pc, lnlo, lnhi, p);
        int pe = 0;
        S.bad[tid] = refine_row(p, sc, ((tid & 1) ? minus : rows) + (size_t)j * pitch, &pe, qslot + tid) ? 0 : 1;
        if (pe) atomicAdd(&S.pe, 1);
      }
      __syncthreads();
      // J columns in place of the plus rows (FP32); the products below sum
      // with compensation in FP32 (the GPU's FP64 rate is a small fraction of
      // its FP32 rate) and enter the FP64 solve
      const float inv2d = 1.0f / (2.0f * delta);
      for (int k = tid; k < sc.L; k += kRefineThreads) {
#pragma unroll 6
        for (int j = 0; j < N; ++j) {
          float* jp = rows + (size_t)j * pitch + k;
          *jp = (*jp - minus[(size_t)j * pitch + k]) * inv2d;
        }
      }
      __syncthreads();
      // A (lower triangle) and g: one compensated dot product per entry.  A
      // thread runs its kTasksPer entries side by side: each sum is a chain of
      // four dependent additions per sample, so one alone leaves the SM idle.
      constexpr int kTasks = N * (N + 1) / 2 + N;
      constexpr int kTasksPer = (kTasks + kRefineThreads - 1) / kRefineThreads;
      const float* ja[kTasksPer];
      const float* jb[kTasksPer];
      int ea[kTasksPer], eb[kTasksPer];   // entry (a, b); b = -1: g[a]; a = -1: none
      float sum[kTasksPer], c[kTasksPer];
#pragma unroll
      for (int q = 0; q < kTasksPer; ++q) {
        const int t = tid + q * kRefineThreads;
        int a = -1, bb = -1;
        if (t >= N * (N + 1) / 2) {
          a = t < kTasks ? t - N * (N + 1) / 2 : -1;
        } else {
          a = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
          while ((a + 1) * (a + 2) / 2 <= t) ++a;
          while (a * (a + 1) / 2 > t) --a;
          bb = t - a * (a + 1) / 2;
        }
        ea[q] = a;
        eb[q] = bb;
        ja[q] = rows + (size_t)(a < 0 ? 0 : a) * pitch;
        jb[q] = bb < 0 ? r0 : rows + (size_t)bb * pitch;
        sum[q] = c[q] = 0.0f;
      }
#pragma unroll 4
      for (int k = 0; k < sc.L; ++k) {
        const float zk = z[k];
#pragma unroll
        for (int q = 0; q < kTasksPer; ++q) {
          const float bk = jb[q][k];
          const float y = fmaf(ja[q][k], eb[q] < 0 ? bk - zk : bk, -c[q]);
          const float tt = sum[q] + y;
          c[q] = (tt - sum[q]) - y;
          sum[q] = tt;
        }
      }
#pragma unroll
      for (int q = 0; q < kTasksPer; ++q) {
        const int a = ea[q], bb = eb[q];
        if (a < 0) continue;
        const bool za = S.bad[2 * a] || S.bad[2 * a + 1];
        const bool zb = bb >= 0 && (S.bad[2 * bb] || S.bad[2 * bb + 1]);
        const double acc = za || zb ? 0.0 : (double)sum[q] - (double)c[q];
        if (bb < 0) S.g[a] = acc;
        else S.A[a * N + bb] = S.A[bb * N + a] = acc;
      }
      __syncthreads();
      if (tid == 0) {
        S.need_jac = 0;
        S.evals += 2 * N;
      }
    }
    // damped normal equations in FP64 by warp 0: the Cholesky factor column by
    // column, each column's products leaving the trailing matrix at once,
    // spread over the lanes (every entry subtracts them in column order, as a
    // row-by-row factorisation does, without its chain of up to N dependent
    // FP64 operations per column); forward substitution one row per lane; then
    // lane 0 substitutes back and simulates the trial point
    if (tid < 32) {
      double amax = 0.0;
      for (int j = 0; j < N; ++j) amax = S.A[j * N + j] > amax ? S.A[j * N + j] : amax;
      int go = amax > 0.0 ? 1 : 0;
      double* M = S.M;
      double fwd = 0.0;   // lane i: row i of the forward substitution
      if (go) {
        for (int e = tid; e < N * N; e += 32) M[e] = S.A[e];
        __syncwarp();
        if (tid < N) {
          const double dj = S.A[tid * N + tid] > 1e-9 * amax ? S.A[tid * N + tid] : 1e-9 * amax;
          M[tid * N + tid] += S.lambda * dj;
        }
        __syncwarp();
        for (int j = 0; j < N; ++j) {
          const double sjj = M[j * N + j];
          if (!(sjj > 0.0)) {
            go = 0;
            break;
          }
          const double ljj = sqrt(sjj), il = __drcp_rn(ljj);
          __syncwarp();
          if (tid == 0) {
            M[j * N + j] = ljj;
            S.inv[j] = il;
          }
          if (j + 1 + tid < N) M[(j + 1 + tid) * N + j] *= il;
          __syncwarp();
          for (int i0 = j + 1; i0 < N; i0 += 2) {
            const int i = i0 + (tid >> 4);
            if (i < N)
              for (int k = j + 1 + (tid & 15); k <= i; k += 16) M[i * N + k] -= M[i * N + j] * M[k * N + j];
          }
          __syncwarp();
        }
      }
      if (go) {
        double t = tid < N ? -S.g[tid] : 0.0;
        for (int k = 0; k < N; ++k) {
          const double dk = __shfl_sync(0xffffffffu, t * S.inv[tid < N ? tid : 0], k);
          if (tid == k) fwd = dk;
          if (tid > k && tid < N) t -= M[tid * N + k] * dk;
        }
        if (tid < N) S.du[tid] = fwd;
        __syncwarp();
      }
      if (go && tid == 0) {
        double du[N];
#pragma unroll
        for (int i = N - 1; i >= 0; --i) {
          double t = S.du[i];
#pragma unroll
          for (int k = i + 1; k < N; ++k) t -= M[k * N + i] * du[k];
          du[i] = t * S.inv[i];
        }
        for (int j = 0; j < N; ++j) {
          const double v = (double)S.u[j] + du[j];
          S.ut[j] = (float)(v < (double)lnlo ? (double)lnlo : (v > (double)lnhi ? (double)lnhi : v));
        }
        float p[kNumParams];
        u_to_p<N>(S.ut, S.pc, lnlo, lnhi, p);
        int pe = 0;
        S.trial_ok = refine_row(p, sc, rcur[S.cur ^ 1], &pe, qslot + tid) ? 1 : 0;
        S.pe += pe;
        S.evals += 1;
      }
      if (tid == 0) S.go = go;
    }
    __syncthreads();
    if (!S.go) break;
    {
      const double ft = refine_f<N>(S, rcur[S.cur ^ 1], z, sc.L);
      if (tid == 0) {
        const double f2 = S.trial_ok && isfinite(ft) ? ft : INFINITY;
        if (f2 < S.f) {
          for (int j = 0; j < N; ++j) S.u[j] = S.ut[j];
          S.f = f2;
          S.cur ^= 1;
          S.acc += 1;
          S.lambda = S.lambda / 10.0 > 1e-12 ? S.lambda / 10.0 : 1e-12;
          S.need_jac = 1;
        } else {
          S.lambda = S.lambda * 10.0 < 1e12 ? S.lambda * 10.0 : 1e12;
        }
      }
    }
    __syncthreads();
  }
  if (tid == 0) {
    opmm_fit_result r;
    float p[kNumParams];
    u_to_p<N>(S.u, S.pc, lnlo, lnhi, p);
    for (int j = 0; j < kNumParams; ++j) r.opc[j] = p[j];
    r.f = (float)S.f;
    r.iterations_run = S.acc;
    r.winner = 0;
    r.evaluations = S.evals;
    r.pulse_end_evals = S.pe;
    r.reserved = 0;
    r.source = OPMM_SOURCE_REFINED;
    // the FP64 check of the refined vector runs in k_refine_check
    r.rms_deg = 0.0;
    r.l1_deg = 0.0;
    r.status = isfinite(S.f) ? 0 : 1;
    out[b] = r;
  }
}

// FP64 re-computation of each refined vector's errors (as k_finalize does for
// the search), one warp per saccade.
__global__ void __launch_bounds__(32) k_refine_check(const DevSac* sacs, const float* traces, int n,
                                                     opmm_fit_result* out) {
  __shared__ Warp64 W;
  const int i = blockIdx.x, lane = threadIdx.x;
  if (i >= n) return;
  opmm_fit_result& r = out[i];
  double mse = INFINITY, mae = INFINITY;
  if (r.status == 0) {
    if (lane < kNumParams) W.opc[lane] = r.opc[lane];
    __syncwarp();
    const DevSac d = sacs[i];
    errors64(Lane64(lane), W, d, traces + d.off, &mse, &mae);
    mse = sqrt(mse);
  }
  if (lane == 0) {
    r.rms_deg = mse;
    r.l1_deg = mae;
  }
}

// Allow kernel k the largest dynamic shared memory the device gives one of its
// blocks (the opt-in maximum less its static shared memory), after checking
// that `smem` fits.  The attribute belongs to the kernel for the whole process,
// so it is only ever raised to that fixed maximum: a call for a smaller size
// never lowers the limit under a launch that another plan, a request loop or a
// captured graph makes with a larger one.
template <class K>
static cudaError_t allow_dynamic_smem(K k, size_t smem) {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, k);
  if (e != cudaSuccess) return e;
  int dev = 0, optin = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  if ((size_t)optin < fa.sharedSizeBytes || smem > (size_t)optin - fa.sharedSizeBytes) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

cudaError_t launch_refine(int dim, const DevSac* sacs, const float* traces, const float* pcs, const float* start,
                          int n, int K, float lnlo, float lnhi, float delta, float lambda0, int lcap, float* scratch,
                          opmm_fit_result* out, unsigned* err, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  // the rows of the dot products go to shared memory when they fit in 96 KB
  // (windows up to about 1,200 samples with 18 coordinates)
  const size_t rows_bytes = ((size_t)dim + 2) * (size_t)refine_pitch(lcap) * sizeof(float);
  const bool in_smem = rows_bytes <= (size_t)96 * 1024;
  const size_t smem = 2 * (size_t)lcap * sizeof(float) + (size_t)kQSlotFloats * kRefineThreads * sizeof(float) +
                      (in_smem ? rows_bytes : 0);
  auto run = [&](auto kernel) -> cudaError_t {
    const cudaError_t e = allow_dynamic_smem(kernel, smem);
    if (e != cudaSuccess) return e;
    kernel<<<n, kRefineThreads, smem, st>>>(sacs, traces, pcs, start, K, lnlo, lnhi, delta, lambda0, lcap, scratch, out,
                                            err);
    return cudaGetLastError();
  };
  cudaError_t e = cudaErrorInvalidValue;
  if (dim == 9) e = in_smem ? run(k_refine<9, true>) : run(k_refine<9, false>);
  else if (dim == kNumParams) e = in_smem ? run(k_refine<kNumParams, true>) : run(k_refine<kNumParams, false>);
  if (e != cudaSuccess) return e;
  k_refine_check<<<n, 32, 0, st>>>(sacs, traces, n, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ serving
// Place newly admitted requests into their slots: descriptor (offset rebased
// to the slot's trace area), trace, box centre; progress reset.
__global__ void k_admit(const DevSac* new_sacs, const float* new_traces, const float* new_pc, const int* slots, int n,
                        DevSac* sacs, float* traces, float* pc, int* progress, int slot_stride) {
  const int i = blockIdx.x;
  if (i >= n) return;
  const int s = slots[i];
  DevSac d = new_sacs[i];
  const long long src = d.off;
  d.off = (long long)s * slot_stride;
  const int lp = (d.L + 3) & ~3;
  for (int k = threadIdx.x; k < lp; k += blockDim.x) traces[d.off + k] = k < d.L ? new_traces[src + k] : 0.0f;
  if (threadIdx.x < kNumParams) pc[(size_t)s * kNumParams + threadIdx.x] = new_pc[(size_t)i * kNumParams + threadIdx.x];
  if (threadIdx.x == 0) {
    sacs[s] = d;
    progress[s] = 0;
  }
}

// Iterations done after a scheduling round.
__global__ void k_advance(const int* slots, int n, int* progress, int iters, int T) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int s = slots[i];
  progress[s] = min(T, progress[s] + iters);
}

cudaError_t launch_admit(const DevSac* new_sacs, const float* new_traces, const float* new_pc, const int* slots, int n,
                         DevSac* sacs, float* traces, float* pc, int* progress, int slot_stride, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_admit<<<n, 128, 0, st>>>(new_sacs, new_traces, new_pc, slots, n, sacs, traces, pc, progress, slot_stride);
  return cudaGetLastError();
}

cudaError_t launch_advance(const int* slots, int n, int* progress, int iters, int T, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_advance<<<(n + 127) / 128, 128, 0, st>>>(slots, n, progress, iters, T);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ launch wrappers
cudaError_t launch_gather(const float* const* src, const DevSac* sacs, float* dst, int n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_gather<<<n, 128, 0, st>>>(src, sacs, dst, n);
  return cudaGetLastError();
}

cudaError_t launch_nominal(const DevSac* sacs, int n, int pulse_mode, const float* init_opc, float* pc,
                           cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int threads = 128;
  const int blocks = (n * 32 + threads - 1) / threads;
  k_nominal<<<blocks, threads, 0, st>>>(sacs, n, pulse_mode, init_opc, pc);
  return cudaGetLastError();
}

cudaError_t launch_simulate(const float* opc, int n, const DevSac* sacs, const int* sac_of,
                            const long long* out_off, float* out, cudaStream_t st, int threads) {
  if (n <= 0) return cudaSuccess;
  // Stores in groups of four bound a block by its walk (a window of 16,384
  // samples 0.49 ms from 1 to 1,000 rows), single ones by the rows it writes
  // (0.42 ms for 33 rows, 0.58 for 64, 1.10 for 128): equal at about 53 rows.
  // 20,000 such windows 1.04 ms against 2.80.
  constexpr int kGroupRows = 48;
  k_simulate<<<(n + threads - 1) / threads, threads, 0, st>>>(opc, n, sacs, sac_of, out_off, out, n >= kGroupRows);
  return cudaGetLastError();
}

cudaError_t launch_score(const float* opc, int m, const DevSac& sac, const float* trace, float* f, int num_sms,
                         cudaStream_t st) {
  if (m <= 0) return cudaSuccess;
  int blocks = (m + kScoreThreads - 1) / kScoreThreads;
  if (blocks > 8 * num_sms) blocks = 8 * num_sms;
  const size_t smem = (size_t)sac.L * sizeof(float);
  // without asking a block gets 48 KB of static and dynamic shared memory
  // together; asking costs four runtime calls, so short windows do without.
  // The static part is TraceStage, at most one alignment of the dynamic part.
  static_assert(sizeof(TraceStage) <= 128, "static shared memory of k_score");
  if (smem + 128 > 48 * 1024) {
    cudaError_t e = allow_dynamic_smem(k_score, smem);
    if (e != cudaSuccess) return e;
  }
  k_score<<<blocks, kScoreThreads, smem, st>>>(opc, m, sac, trace, f);
  return cudaGetLastError();
}

// Launch-shape variants of the search kernel: simplices per group G, groups
// per block NG (a block runs a unit of NG G simplices), the search
// coordinates N (18, or 9 for the 9-parameter model), the minimum resident
// blocks per SM the register allocation is bounded for, and the walk: the
// register-lean walk, or the packed sample update (two row FMAs per packed
// FP32 instruction, the same arithmetic), or neither.  The host sees the unit
// size (simplices per block), N and the walk.  More groups per block keep
// more waves open, so that the warps always find chunks to claim while a
// group's decisions are taken.
struct SearchVariantDesc { int G, N, NG, minb, lean, pack; };
static const SearchVariantDesc kVariants[] = {
    {16, 18, 2, 1, 0, 0}, {16, 18, 2, 1, 1, 0}, {8, 18, 2, 1, 0, 0}, {32, 18, 2, 1, 0, 0}, {27, 9, 2, 1, 0, 0},
    {16, 18, 4, 1, 0, 0}, {27, 9, 4, 1, 0, 0},  {24, 18, 3, 1, 0, 0}, {16, 18, 2, 1, 0, 1}, {32, 18, 2, 1, 0, 1},
    {16, 18, 4, 1, 0, 1}, {24, 18, 3, 1, 0, 1}, {27, 9, 4, 1, 0, 1}};
constexpr int kNumVariants = sizeof(kVariants) / sizeof(kVariants[0]);

static bool variant_ok(int v) { return v >= 0 && v < kNumVariants; }
int search_variant_count() { return kNumVariants; }
int search_variant_g(int v) { return variant_ok(v) ? kVariants[v].NG * kVariants[v].G : 0; }
int search_variant_groups(int v) { return variant_ok(v) ? kVariants[v].NG : 0; }
int search_variant_dim(int v) { return variant_ok(v) ? kVariants[v].N : 0; }
int search_variant_minb(int v) { return variant_ok(v) ? kVariants[v].minb : 0; }
int search_variant_lean(int v) { return variant_ok(v) ? kVariants[v].lean : 0; }
int search_variant_pack(int v) { return variant_ok(v) ? kVariants[v].pack : 0; }
// The packed walk at that unit size when there is one (the same results as the
// scalar walk, a quarter faster), else the first variant.
int search_variant_for(int unit, int dim) {
  int first = -1;
  for (int v = 0; v < kNumVariants; ++v)
    if (kVariants[v].NG * kVariants[v].G == unit && kVariants[v].N == dim) {
      if (kVariants[v].pack) return v;
      if (first < 0) first = v;
    }
  return first;
}
// 2 x 32 packed (9 coordinates: 4 x 27 packed), then the smaller packed shape
// for traces too long to leave it room.
int search_variant_default(int dim, int k) {
  static const int pref18[] = {9, 8, -1}, pref9[] = {12, -1};
  return dim == 9 ? pref9[k] : pref18[k];
}

template <int G, int N, int NG, int MINB, bool LEAN, bool PACK>
static cudaError_t occ_v(int lcap, int* bps) {
  const size_t smem = search_smem_bytes<G, N, NG>(lcap);
  cudaError_t e = allow_dynamic_smem(k_search<G, N, NG, MINB, LEAN, PACK>, smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, k_search<G, N, NG, MINB, LEAN, PACK>, search_threads<G, N>(),
                                                       smem);
}

// The dynamic shared-memory attribute is raised to its maximum by
// search_occupancy_v(), which the host calls for the same variant before any
// launch or graph capture.
template <int G, int N, int NG, int MINB, bool LEAN, bool PACK>
static cudaError_t launch_v(const SearchParams& P, int blocks_per_sm, int num_sms, cudaStream_t st) {
  const size_t smem = search_smem_bytes<G, N, NG>(P.lcap);
  k_search<G, N, NG, MINB, LEAN, PACK><<<blocks_per_sm * num_sms, search_threads<G, N>(), smem, st>>>(P);
  return cudaGetLastError();
}

template <int G, int N, int NG, int MINB, bool LEAN, bool PACK>
static int threads_v() { return search_threads<G, N>(); }

template <int G, int N, int NG, int MINB, bool LEAN, bool PACK>
static size_t smem_v(int lcap) { return search_smem_bytes<G, N, NG>(lcap); }

#define OPMM_VARIANT_SWITCH(v, CALL, BAD)             \
  switch (v) {                                        \
    case 0: return CALL(16, 18, 2, 1, false, false);  \
    case 1: return CALL(16, 18, 2, 1, true, false);   \
    case 2: return CALL(8, 18, 2, 1, false, false);   \
    case 3: return CALL(32, 18, 2, 1, false, false);  \
    case 4: return CALL(27, 9, 2, 1, false, false);   \
    case 5: return CALL(16, 18, 4, 1, false, false);  \
    case 6: return CALL(27, 9, 4, 1, false, false);   \
    case 7: return CALL(24, 18, 3, 1, false, false);  \
    case 8: return CALL(16, 18, 2, 1, false, true);   \
    case 9: return CALL(32, 18, 2, 1, false, true);   \
    case 10: return CALL(16, 18, 4, 1, false, true);  \
    case 11: return CALL(24, 18, 3, 1, false, true);  \
    case 12: return CALL(27, 9, 4, 1, false, true);   \
    default: return BAD;                              \
  }

cudaError_t search_occupancy_v(int v, int lcap, int* blocks_per_sm) {
#define OCC_CALL(G, N, NG, M, L, K) occ_v<G, N, NG, M, L, K>(lcap, blocks_per_sm)
  OPMM_VARIANT_SWITCH(v, OCC_CALL, cudaErrorInvalidValue)
#undef OCC_CALL
}

cudaError_t launch_search_v(int v, const SearchParams& P, int blocks_per_sm, int num_sms, cudaStream_t st) {
#define LAUNCH_CALL(G, N, NG, M, L, K) launch_v<G, N, NG, M, L, K>(P, blocks_per_sm, num_sms, st)
  OPMM_VARIANT_SWITCH(v, LAUNCH_CALL, cudaErrorInvalidValue)
#undef LAUNCH_CALL
}

// Threads and dynamic shared memory of a block of variant v.
int search_variant_threads(int v) {
#define THREADS_CALL(G, N, NG, M, L, K) threads_v<G, N, NG, M, L, K>()
  OPMM_VARIANT_SWITCH(v, THREADS_CALL, 0)
#undef THREADS_CALL
}

size_t search_variant_smem(int v, int lcap) {
#define SMEM_CALL(G, N, NG, M, L, K) smem_v<G, N, NG, M, L, K>(lcap)
  OPMM_VARIANT_SWITCH(v, SMEM_CALL, (size_t)0)
#undef SMEM_CALL
}

// Entry points for a fixed 18-coordinate unit size (static fit).
cudaError_t search_occupancy(int unit, int lcap, int* blocks_per_sm) {
  return search_occupancy_v(search_variant_for(unit, kNumParams), lcap, blocks_per_sm);
}

cudaError_t launch_search(int unit, const SearchParams& P, int blocks_per_sm, int num_sms, cudaStream_t st) {
  return launch_search_v(search_variant_for(unit, kNumParams), P, blocks_per_sm, num_sms, st);
}

cudaError_t launch_finalize(const DevSac* sacs, const float* traces, const float* pc, const int* ustart,
                            int ngroups, const float* unit_best, float lnlo, float lnhi, int n,
                            opmm_fit_result* out, cudaStream_t st, const int* list, int dim) {
  if (n <= 0) return cudaSuccess;
  if (dim == 9)
    k_finalize<9><<<n, 32, 0, st>>>(sacs, traces, pc, ustart, ngroups, unit_best, lnlo, lnhi, n, out, list);
  else if (dim == kNumParams)
    k_finalize<kNumParams><<<n, 32, 0, st>>>(sacs, traces, pc, ustart, ngroups, unit_best, lnlo, lnhi, n, out, list);
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}

}  // namespace opmm
