// Batched evaluation of the stage-centric model of arxiv 2605.04178 (Sec. III-A,
// Eqs. 2-8; Eq. 16 for the memory probes), its hand-written adjoint for
// calibration (Sec. III-D), and the model-driven autotuner (Sec. III-B
// adaptive tile selection, Sec. VI autotuning guidance).
//
// FP32 arithmetic (FP64 for the fit), integer tile counts.  The kernels over
// explicit configurations take a 24-byte record per thread; the autotuner tabulates
// the terms of its tiles or decodes a tile from the thread index, and reads a shape
// for 180 of them.  All of them are bound by ALU issue (FP64: by its units), not by
// memory.
#include <math.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <type_traits>
#include <vector>

#include "pm_internal.cuh"

namespace pm {

// Exact unsigned division by a divisor fixed for the whole launch (the number
// of concurrent CTAs), as one multiply-high, a subtract, an add and two shifts
// instead of the generic division sequence (Granlund and Montgomery,
// "Division by Invariant Integers using Multiplication", PLDI 1994, Sec. 4,
// N = 32).  For 1 <= d <= 2^31 and l = ceil(log2 d):
//   m = floor(2^32 (2^l - d) / d) + 1,   t = floor(m x / 2^32),
//   floor(x / d) = (t + ((x - t) >> min(l, 1))) >> max(l - 1, 0)
// for every 0 <= x < 2^32.
struct UDiv {
  uint32_t d, m;
  int s1, s2;
};

inline UDiv make_udiv(uint32_t d) {
  int l = 0;
  while ((1ull << l) < d) ++l;
  UDiv u;
  u.d = d;
  u.m = (uint32_t)((((1ull << l) - d) << 32) / d + 1);
  u.s1 = l < 1 ? l : 1;
  u.s2 = l > 1 ? l - 1 : 0;
  return u;
}

__device__ __forceinline__ uint32_t udiv(uint32_t x, const UDiv& u) {
  const uint32_t t = __umulhi(u.m, x);
  return (t + ((x - t) >> u.s1)) >> u.s2;
}

// Parameters in the arithmetic type F: FP32 for the batched throughput
// paths, FP64 for the calibration objective (pm_model_grad_f64).
// inv[j] = 1 / v[j], rounded once on the host: the per-configuration model
// multiplies where the equations divide by a parameter.  nc[0] / nc[1]
// divide by the concurrent CTAs of one-SM / paired tiles on nc_nsm SMs
// (nc_nsm = 0: not prepared, the generic division is used).  inv_s[s] =
// 1/s and inv_s1[s] = 1/(s - 1) for the ring depths 2..7, inv_nsm = 1/nc_nsm:
// the per-configuration divisions by small integers become multiplications.
constexpr int NP = PM_NPARAMS;     // model parameters
constexpr int NREC = NP + 1;        // loss + gradient per partial record

template <class F>
struct ThetaT {
  F v[NP];
  F inv[NP];
  int reading;       // PM_READING_LITERAL or PM_READING_MEASURED (see pm_model_set_reading)
  int nc_nsm;
  UDiv nc[2];
  F inv_s[8], inv_s1[8], inv_nsm;
};
using Theta = ThetaT<float>;

template <class F>
inline void set_concurrency(ThetaT<F>& t, int n_sm) {
  for (int s = 0; s < 8; ++s) {
    t.inv_s[s] = s >= 1 ? (F)(1.0 / s) : F(0);
    t.inv_s1[s] = s >= 2 ? (F)(1.0 / (s - 1)) : F(0);
  }
  t.inv_nsm = n_sm >= 1 ? (F)(1.0 / n_sm) : F(0);
  t.nc_nsm = 0;
  if (n_sm >= 2) {
    t.nc[0] = make_udiv((uint32_t)n_sm);
    t.nc[1] = make_udiv((uint32_t)(2 * (n_sm / 2)));
    t.nc_nsm = n_sm;
  }
}

__device__ __forceinline__ float pm_exp(float x) { return expf(x); }
__device__ __forceinline__ double pm_exp(double x) { return exp(x); }
__device__ __forceinline__ float pm_log(float x) { return logf(x); }
__device__ __forceinline__ double pm_log(double x) { return log(x); }
__device__ __forceinline__ float pm_max(float a, float b) { return fmaxf(a, b); }
// The FP32 throughput paths take the hardware approximations (relative error
// of a few 1e-7, far inside their 1e-5 tolerance); FP64 stays exact.
__device__ __forceinline__ float pm_exp_fast(float x) { return __expf(x); }
__device__ __forceinline__ double pm_exp_fast(double x) { return exp(x); }
__device__ __forceinline__ float pm_div_fast(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double pm_div_fast(double a, double b) { return a / b; }
// a + b, not fused with the product that b may be
__device__ __forceinline__ float pm_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double pm_add(double a, double b) { return a + b; }
// x / s and x / (s - 1) for a ring depth s (tabulated reciprocals for 2..7)
template <class F>
__device__ __forceinline__ F div_stages(F x, int s, const ThetaT<F>& th) {
  return (s >= 1 && s < 8) ? x * th.inv_s[s] : x / (F)s;
}
template <class F>
__device__ __forceinline__ F div_stages_m1(F x, int s, const ThetaT<F>& th) {
  return (s >= 2 && s < 8) ? x * th.inv_s1[s] : x / (F)(s - 1);
}
__device__ __forceinline__ double pm_max(double a, double b) { return fmax(a, b); }

// ceil(a / b) for a >= 0, b > 0: a shift when b is a power of two (every tile
// extent of the search space), else 32-bit unsigned division whenever both fit
// (64-bit division is a long software sequence); exact either way.
__device__ __forceinline__ int64_t cdiv(int64_t a, int64_t b) {
  if (((uint64_t)a | (uint64_t)b) < 0x80000000ull) {
    const uint32_t ua = (uint32_t)a, ub = (uint32_t)b;
    if ((ub & (ub - 1u)) == 0u) return (int64_t)((ua + ub - 1u) >> (__ffs((int)ub) - 1));
    return (int64_t)((ua + ub - 1u) / ub);
  }
  return (a + b - 1) / b;
}

// Non-negative count to the arithmetic type, through a 32-bit conversion
// when it fits (64-bit conversions run on the narrow FP64 pipe).
template <class F>
__device__ __forceinline__ F count_to(int64_t v) {
  return (uint64_t)v < 0x80000000ull ? (F)(int32_t)v : (F)v;
}

// Element bytes, tensor passes per K-step (three-pass TF32 for FP32) and
// operand copies loaded per element (FP32: hi and lo).
__device__ __forceinline__ float dt_bytes(int dt) { return dt == PM_FP32 ? 4.f : (dt == PM_BF16 ? 2.f : 1.f); }
__device__ __forceinline__ float dt_passes(int dt) { return dt == PM_FP32 ? 3.f : 1.f; }
__device__ __forceinline__ float dt_loads(int dt) { return dt == PM_FP32 ? 2.f : 1.f; }
__device__ __forceinline__ int dt_rate(int dt) { return dt == PM_FP32 ? 6 : (dt == PM_BF16 ? 7 : 8); }

__constant__ int16_t kBM[3] = {64, 128, 256};
__constant__ int16_t kBN[3] = {64, 128, 256};
__constant__ int16_t kBK[3][2] = {{32, 64}, {64, 128}, {64, 128}};

// Valid tile space of the autotuners (TMEM strategy A): ring of `s` stages
// within 227 KiB - 2 KiB, FP32 accumulator columns ceil(BM/128)*BN within the
// 512 TMEM columns.
__host__ __device__ inline bool tile_valid(int BM, int BN, int BK, int s, int g, int dt) {
  if (!(BM == 64 || BM == 128 || BM == 256) || !(BN == 64 || BN == 128 || BN == 256)) return false;
  if (dt == PM_FP32) {
    if (BK != 32 && BK != 64) return false;
  } else if (dt == PM_BF16 || dt == PM_FP8E4M3) {
    if (BK != 64 && BK != 128) return false;
  } else {
    return false;
  }
  if (s < 2 || s > 6 || (g != 1 && g != 2)) return false;
  const int e = dt == PM_FP32 ? 4 : (dt == PM_BF16 ? 2 : 1);
  const int l = dt == PM_FP32 ? 2 : 1;
  const int64_t stage = (int64_t)l * e * BK * (BM + BN / g);
  if ((int64_t)s * stage > 232448 - 2048) return false;
  if (((BM + 127) / 128) * BN > 512) return false;
  return true;
}

// Whether the GEMM kernel keeps one accumulator buffer only: it holds two when
// twice the accumulator columns of the tile (ceil(BM/128) BN, or BN/2 for a
// 64-row tile on a CTA pair), plus strategy B's A copy per stage, fit in the
// 512 TMEM columns.
__host__ __device__ inline bool single_buffer(int BM, int BN, int BK, int s, int g, int dt, int tmem_a) {
  const int acc = (BM < 128 && g == 2) ? BN / 2 : ((BM + 127) / 128) * BN;
  const int le = dt == PM_FP32 ? 8 : (dt == PM_BF16 ? 2 : 1);    // load planes x element bytes
  const int a_ring = tmem_a ? s * ((BM + 127) / 128) * (le * BK / 4) : 0;
  return 2 * acc + a_ring > 512;
}

// Intermediate values of one GEMM evaluation, kept for the adjoint.
template <class F>
struct GemmFwdT {
  F T, T_stage, T_rl, A_rl, B_rl;
  F T_c, T_io, T_tma, oma, X, XT, R, S, invR, invS, T_step, T_store;   // XT: T_c without T_mgmt/K_tiles
  F D, D_r, D_w, bstep, store_bytes, n_instr;   // D_r, D_w: D with strategy B's reads and writes of A
  F waves, Kt;
  F W, E, rho;          // L2 residency of the TMA loads (measured reading)
  F launch;             // T_launch (+ L_alloc + L_dealloc once per launch, measured reading)
  F T_eq8, T_ring;       // Eq. 8 and the ring bound (measured reading)
  int ri;
  bool oma_free, blend, ring;
  bool drain;           // measured reading, one accumulator buffer: each tile's drain is paid
  F inv_s, inv_s1;      // 1 / stages and 1 / (stages - 1) (gemm_forward_space only)
};
using GemmFwd = GemmFwdT<float>;

// Waves of `tiles` CTA tiles over the concurrent CTAs of cta_group g (pairs on
// fewer than two SMs are rejected by the callers; the guard keeps the division
// defined).
template <class F>
__device__ __forceinline__ int64_t wave_count(int64_t tiles, int g, const ThetaT<F>& th, int n_sm) {
  if (th.nc_nsm == n_sm && (uint64_t)tiles < 0x80000000ull) {
    const UDiv u = g == 1 ? th.nc[0] : th.nc[1];
    return (int64_t)udiv((uint32_t)tiles + (u.d - 1u), u);
  }
  return cdiv(tiles, g == 1 ? n_sm : (n_sm >= 2 ? 2 * (n_sm / 2) : 1));
}

// Stage-centric GEMM time:
//   T_TMEM = (D + D_A,r)/BW_rd + n_instr L_mma + (D + D_A,w)/BW_wr   (Eq. 2)
//            D_A = 0 for TMEM strategy A; strategy B writes the A tile
//            into TMEM (D_A,w = l e BM BK) and every pass reads it back
//            (D_A,r = n_p e BM BK); n_instr = 1 (literal reading) or the
//            tensor-pipe instructions of the K-step incl. strategy B's
//            tcgen05.cp copies (measured reading)
//   T_c    = n_p 2 BM' BN BK / (R S) + T_TMEM + T_mgmt/K_tiles    (Eqs. 3, 6)
//            BM' = BM, except 128 for a one-SM 64-row tile (measured
//            reading: M = 64 instructions take the M = 128 time); the
//            measured reading has no T_mgmt/K_tiles (paid once per launch)
//   T_tma  = L_TMA + b_step / (B_TMA rho), b_step = l e BK (BM + BN/g) (Eq. 4,
//            P = 1); rho = 1 (literal reading) or the L2-residency factor
//            1 + (rho_L2 - 1) exp(-W/w0) over the launch's working set W
//            (measured reading)
//   T_io   = (1 - alpha) T_tma + T_sync, T_sync = 2 L_mbar       (Eq. 7; the
//            measured reading drops this T_sync: one barrier per K-step)
//   T_step = max(T_c, T_io) + T_sync                             (Eq. 8; the
//            measured reading adds the bubble of the s-deep ring as O_misc:
//            T_step = max(Eq. 8, (T_tma + T_c + T_sync) / s))
//   T_stage = launch + waves (K_tiles T_step + T_store)
//   T_hat = max(T_stage, launch + max(FLOPs/(n_SM R S), bytes_min/B_peak))
//            launch = T_launch (literal) or T_launch + L_alloc + L_dealloc
//            (measured: the persistent CTAs allocate TMEM once per launch)
//   T_store = L_TMA + 4 BM BN / B_TMA, plus 4 BM BN / B_drain (measured
//            reading) when the kernel keeps one accumulator buffer only, so
//            the next tile waits for the drain (two buffers overlap it)
// W_launch > 0 overrides the working set (a grouped launch passes its own);
// otherwise W = bytes_min of this GEMM (operands once, C once).  single >= 0
// overrides the buffering (a grouped launch passes the launch's); otherwise
// the tile's own.  SPACE: the launch's parameters are space_params' (measured
// reading, L2 blend on), so the branches on them are settled when compiling:
// 10^6 records outside the search space 16.5 -> 14.2 us, the same bits.
template <bool SPACE = false, class F>
__device__ __forceinline__ void gemm_forward(const pm_cfg& c, const ThetaT<F>& th, int n_sm, GemmFwdT<F>& f,
                                             F W_launch = F(-1), int single = -1) {
  const bool measured = SPACE || th.reading == PM_READING_MEASURED;
  const int dt = c.dtype, g = c.cta_group;
  const F e = dt_bytes(dt), np = dt_passes(dt), l = dt_loads(dt);
  const F bytes_min = l * e * ((F)c.M * c.K + (F)c.N * c.K) + F(4) * (F)c.M * (F)c.N;
  f.ri = dt_rate(dt);
  f.R = th.v[f.ri];
  f.invR = th.inv[f.ri];
  const int64_t Kt = cdiv(c.K, c.BK);
  // CTA tiles: ceil(M/BM) ceil(N/BN) (literal); a pair covers 2 BM x BN (measured)
  const int64_t tiles = measured ? (int64_t)g * cdiv(c.M, (int64_t)g * c.BM) * cdiv(c.N, c.BN)
                                 : cdiv(c.M, c.BM) * cdiv(c.N, c.BN);
  const int64_t waves = wave_count(tiles, g, th, n_sm);
  f.Kt = count_to<F>(Kt);
  f.waves = count_to<F>(waves);
  // tile products in integers (exact: at most 2^25), one conversion each
  f.D = (F)(4 * (int)c.BM * (int)c.BN);
  // L_mma once per K-step (literal) or once per tcgen05.mma the K-step
  // issues, BK/k_instr per 128-row block per pass (measured)
  const int kin = dt == PM_FP32 ? 8 : (dt == PM_BF16 ? 16 : 32);
  f.n_instr = measured ? np * (F)((c.BK / kin) * ((c.BM + 127) / 128)) : F(1);
  f.D_w = f.D + (c.tmem_a ? l * e * c.BM * c.BK : F(0));
  f.D_r = f.D + (c.tmem_a ? np * e * c.BM * c.BK : F(0));
  // measured: strategy B's tcgen05.cp per 128-row x 32-byte A slice, each charged L_mma
  if (c.tmem_a && measured) f.n_instr += l * (F)(c.BK * (int)e / 32) * (F)((c.BM + 127) / 128);
  const F T_tmem = f.D_r * th.inv[10] + f.n_instr * th.v[9] + f.D_w * th.inv[11];
  const F T_mgmt = measured ? F(0) : th.v[13] / f.Kt;
  f.S = g == 1 ? F(1) : th.v[14];
  f.invS = g == 1 ? F(1) : th.inv[14];
  const int rows = (measured && g == 1 && c.BM < 128) ? 128 : (int)c.BM;
  f.X = (np * (F)(2 * rows * (int)c.BN * (int)c.BK)) * (f.invR * f.invS);
  f.XT = f.X + T_tmem;
  f.T_c = f.XT + T_mgmt;
  // BN / g: exact for the one- and two-SM tiles (power-of-two BN)
  const F bn_g = g == 1 ? (F)c.BN : (g == 2 ? F(0.5) * (F)c.BN : (F)c.BN / (F)g);
  f.bstep = g <= 2 ? l * e * (F)((int)c.BK * ((int)c.BM + ((int)c.BN >> (g - 1))))
                   : l * e * c.BK * ((F)c.BM + bn_g);
  // measured: B_TMA x rho(W), rho = 1 + (rho_L2 - 1) exp(-W/w0) (loads that
  // hit in L2 arrive faster, Sec. III-A.2; Eq. 16's blend shape); w0 <= 0
  // switches the blend off
  f.W = W_launch > F(0) ? W_launch : bytes_min;
  f.blend = SPACE || (measured && th.v[3] > F(0));
  f.E = f.blend ? pm_exp_fast(-f.W * th.inv[3]) : F(0);
  f.rho = f.blend ? F(1) + (th.v[16] - F(1)) * f.E : F(1);
  f.T_tma = pm_add(th.v[4], f.blend ? pm_div_fast(f.bstep * th.inv[5], f.rho) : f.bstep * th.inv[5]);   // rho = 1 unblended
  const F T_sync = F(2) * th.v[12];
  // 1 - alpha = clamp(c_alpha / s, 0, 1) (literal) or clamp(c_alpha / (s - 1),
  // 0, 1) (measured: s - 1 loads in flight while one stage is consumed; a
  // single stage hides nothing)
  const F r = measured ? (c.stages > 1 ? div_stages_m1(th.v[15], c.stages, th) : F(1))
                       : div_stages(th.v[15], c.stages, th);
  f.oma_free = r > F(0) && r < F(1);
  f.oma = r <= F(0) ? F(0) : (r >= F(1) ? F(1) : r);
  f.T_io = measured ? f.oma * f.T_tma : f.oma * f.T_tma + T_sync;
  f.T_eq8 = pm_max(f.T_c, f.T_io) + T_sync;
  // measured: each stage cycles through its load, its MMAs and its full and
  // empty barriers, so s stages finish at most one K-step per cycle / s
  f.T_ring = measured ? div_stages(f.T_tma + f.T_c + T_sync, c.stages, th) : F(0);
  f.ring = measured && f.T_ring > f.T_eq8;
  f.T_step = f.ring ? f.T_ring : f.T_eq8;
  f.store_bytes = f.D;
  f.drain = measured && (single >= 0 ? single != 0
                                     : single_buffer(c.BM, c.BN, c.BK, c.stages, c.cta_group, c.dtype, c.tmem_a));
  f.T_store = th.v[4] + f.store_bytes * th.inv[5] + (f.drain ? f.store_bytes * th.inv[17] : F(0));
  f.launch = measured ? th.v[0] + th.v[13] : th.v[0];
  f.T_stage = f.launch + f.waves * (f.Kt * f.T_step + f.T_store);
  const F flops = np * F(2) * (F)c.M * (F)c.N * (F)c.K;
  f.A_rl = SPACE || th.nc_nsm == n_sm ? flops * (f.invR * f.invS) * th.inv_nsm : flops * (f.invR * f.invS) / (F)n_sm;
  f.B_rl = bytes_min * th.inv[2];
  f.T_rl = f.launch + (f.A_rl >= f.B_rl ? f.A_rl : f.B_rl);
  f.T = f.T_stage >= f.T_rl ? f.T_stage : f.T_rl;
}

// Adjoint of one tile's K-steps and writeback, tau = K_tiles T_step + T_store
// scaled by the weights g_step (of T_step) and g_store (of T_store):
// d[j] += dtau/dtheta_j; the tensor-rate and S_2SM slopes go to gR and gS
// (the caller adds them to the right entries).  max() passes the gradient
// to its first argument on ties; the clamp stops it outside (0,1).
// SPACE: f is gemm_forward_space's (measured reading, L2 blend on, 2..6 stages).
template <bool SPACE = false, class F>
__device__ __forceinline__ void step_store_adjoint(const pm_cfg& c, const ThetaT<F>& th, const GemmFwdT<F>& f,
                                                   F g_step, F g_store, F (&d)[NP], F& gR, F& gS) {
  const bool measured = SPACE || th.reading == PM_READING_MEASURED;
  d[4] += g_store;
  d[5] -= g_store * (f.store_bytes * th.inv[5]) * th.inv[5];
  if (f.drain) d[17] -= g_store * (f.store_bytes * th.inv[17]) * th.inv[17];
  // T_step = max(T_eq8, T_ring); ties to Eq. 8
  const F g_eq8 = f.ring ? F(0) : g_step;
  const F g_ring = f.ring ? (SPACE ? g_step * f.inv_s : div_stages(g_step, c.stages, th)) : F(0);   // per term of the ring's cycle
  F g_sync = g_eq8 + g_ring;
  F g_c = g_ring, g_io = F(0);
  if (f.T_c >= f.T_io) g_c += g_eq8; else g_io = g_eq8;
  // T_io = oma * T_tma + T_sync
  if (!measured) g_sync += g_io;
  const F g_tma = g_io * f.oma + g_ring;
  if (f.oma_free)
    d[15] += SPACE ? g_io * f.T_tma * f.inv_s1
                   : (measured ? div_stages_m1(g_io * f.T_tma, c.stages, th) : div_stages(g_io * f.T_tma, c.stages, th));
  d[4] += g_tma;
  const F t_bw = f.blend ? pm_div_fast(f.bstep * th.inv[5], f.rho) : f.bstep * th.inv[5];   // b_step / (B_TMA rho)
  d[5] -= g_tma * t_bw * th.inv[5];
  if (f.blend) {
    // rho = 1 + (rho_L2 - 1) E, E = exp(-W/w0)
    const F g_rho = -pm_div_fast(g_tma * t_bw, f.rho);
    d[16] += g_rho * f.E;
    d[3] += g_rho * (th.v[16] - F(1)) * f.E * (f.W * th.inv[3]) * th.inv[3];
  }
  d[12] += F(2) * g_sync;
  // T_c = X + (D + D_A,r)/BW_rd + n_instr L_mma + (D + D_A,w)/BW_wr + L_mgmt/K_tiles
  gR -= g_c * f.X * f.invR;
  gS -= g_c * f.X * f.invS;
  d[10] -= g_c * (f.D_r * th.inv[10]) * th.inv[10];
  d[9] += g_c * f.n_instr;
  d[11] -= g_c * (f.D_w * th.inv[11]) * th.inv[11];
  if (!measured) d[13] += g_c / f.Kt;
}

// Adds the tensor-rate and S_2SM slopes to their entries of d; static
// indices keep d[] in registers.
template <class F>
__device__ __forceinline__ void rate_adjoint(const pm_cfg& c, const GemmFwdT<F>& f, F gR, F gS, F (&d)[NP]) {
  d[6] += f.ri == 6 ? gR : F(0);
  d[7] += f.ri == 7 ? gR : F(0);
  d[8] += f.ri == 8 ? gR : F(0);
  if (c.cta_group == 2) d[14] += gS;
}

// Adjoint of gemm_forward: d[j] += w * dT_hat/dtheta_j.
template <bool SPACE = false, class F>
__device__ __forceinline__ void gemm_adjoint(const pm_cfg& c, const ThetaT<F>& th, const GemmFwdT<F>& f, F w,
                                             F (&d)[NP]) {
  const bool measured = SPACE || th.reading == PM_READING_MEASURED;
  F g_stage = F(0), g_rl = F(0);
  if (f.T_stage >= f.T_rl) g_stage = w; else g_rl = w;
  F gR = F(0), gS = F(0);
  // the launch term of both branches
  if (measured) d[13] += g_rl + g_stage;
  // roofline branch
  d[0] += g_rl;
  if (g_rl != F(0)) {
    if (f.A_rl >= f.B_rl) {
      gR -= g_rl * f.A_rl * f.invR;
      gS -= g_rl * f.A_rl * f.invS;
    } else {
      d[2] -= g_rl * f.B_rl * th.inv[2];
    }
  }
  // stage branch: launch + waves (K_tiles T_step + T_store)
  d[0] += g_stage;
  step_store_adjoint<SPACE>(c, th, f, g_stage * f.waves * f.Kt, g_stage * f.waves, d, gR, gS);
  rate_adjoint(c, f, gR, gS, d);
}

// The records that the search space and the calibration table are made of take
// a shorter way to the same values: GEMM records under the measured reading with
// BM, BN in {64, 128, 256}, BK in {32, 64, 128}, 2..6 stages and M N below 2^41,
// whose counts fit in 32 bits (at most 2^29 + 2^26 tiles) and whose extents are
// divided by shifts.  What depends on (dtype, cta_group) or on the stages alone
// is looked up in shared memory: kernel parameters indexed by a lane's own value
// are read once per distinct value.  The floating-point operations are
// gemm_forward's, in its order, so the results are the same bits.  Both TMEM
// strategies take it: rows of strategy B scattered over a table (the calibration's)
// would send nearly every warp both ways (10^6 mixed records 19.6 us, 9.7 this way).
// So would extents: half of 10^6 records with M above 2^21 cost 12.9 us the
// general way alone, 19.8 with the limit at 2^20 per extent, 8.8 here.
struct SpaceTables {
  float4 rate[6];       // by 2 dtype + (cta_group - 1): 1 / (R S), l e, n_p, 1 / R
  uint4 conc[2];        // by cta_group - 1: the wave division d - 1, m, s1, s2
  float4 depth[8];      // by stages: 1 - alpha, 1 / s, 1 / (s - 1), 0 < c_alpha / (s - 1) < 1
  float inv_s2sm[2];    // by cta_group - 1: 1 / S
};

// Whether a launch's parameters allow the short way.  Launches that they do not (the
// literal reading, no L2 blend, one SM) have kernels without it: 10^6 records under the
// literal reading 10.8 us, 11.7 in a kernel with both ways.
template <class F>
inline bool space_params(const ThetaT<F>& th, int n_sm) {
  return th.reading == PM_READING_MEASURED && th.nc_nsm == n_sm && th.v[3] > F(0);
}

__device__ __forceinline__ void space_tables(const Theta& th, SpaceTables& t) {
  if (threadIdx.x < 6) {
    const int dt = threadIdx.x >> 1, g = 1 + (threadIdx.x & 1);
    const float invR = th.inv[dt_rate(dt)], invS = g == 1 ? 1.f : th.inv[14];
    t.rate[threadIdx.x] = make_float4(invR * invS, dt_loads(dt) * dt_bytes(dt), dt_passes(dt), invR);
  } else if (threadIdx.x < 8) {
    const int i = threadIdx.x - 6;
    t.conc[i] = make_uint4(th.nc[i].d - 1u, th.nc[i].m, (unsigned)th.nc[i].s1, (unsigned)th.nc[i].s2);
    t.inv_s2sm[i] = i == 0 ? 1.f : th.inv[14];
  } else if (threadIdx.x < 16) {
    const int s = threadIdx.x - 8;
    const float r = th.v[15] * th.inv_s1[s];
    t.depth[s] = make_float4(r <= 0.f ? 0.f : (r >= 1.f ? 1.f : r), th.inv_s[s], th.inv_s1[s],
                             r > 0.f && r < 1.f ? 1.f : 0.f);
  }
  __syncthreads();
}

// All conditions without a branch: the fields of a record share words, what may not
// be set in any of them is collected in one (with early exits 10^6 records take 9.0
// us instead of 8.75).
__device__ __forceinline__ bool in_space(const pm_cfg& c) {
  const unsigned tile = (unsigned)(uint16_t)c.BM | (unsigned)(uint16_t)c.BN << 16;
  const unsigned step = (unsigned)(uint16_t)c.BK | (unsigned)(uint8_t)c.stages << 16 | (unsigned)(uint8_t)c.cta_group << 24;
  const unsigned type = (unsigned)(uint8_t)c.dtype | (unsigned)(uint8_t)c.kind << 8 | (unsigned)(uint8_t)c.tmem_a << 16;
  const unsigned sign = (unsigned)(c.M - 1) | (unsigned)(c.N - 1) | (unsigned)(c.K - 1);
  // 64..256 in each half of tile, 32..128 in BK, 0..7 stages, 0..3 groups and types,
  // kind 0 and tmem_a 0 or 1, extents of at least 1, M N < 2^41
  const unsigned stray = (tile & ~0x01C001C0u) | (step & 0xFCF8FF1Fu) | (type & 0x00FEFFFCu) | (sign >> 31) |
                         (__umulhi((unsigned)c.M, (unsigned)c.N) >> 9);
  // then one bit in each of BM, BN and BK, 2..6 stages, groups 1 and 2, types 0..2
  const unsigned pairs = (tile & (tile - 0x00010001u)) | (step & (step - 1u) & 0xE0u);
  return (stray | pairs) == 0u && (tile & 0xFFFFu) != 0u && (tile >> 16) != 0u && (step & 0xE0u) != 0u &&
         ((0x7Cu >> ((step >> 16) & 7u)) & (6u >> (step >> 24)) & (7u >> (type & 3u)) & 1u) != 0u;
}

// The FP64 way keeps K exact in FP32 (small_f64) and the bytes of the operands below
// 2^51 (large_f64).
__device__ __forceinline__ bool in_space_f64(const pm_cfg& c) {
  return in_space(c) && (unsigned)(c.K - 1) < (1u << 24) &&
         ((uint64_t)((unsigned)c.M + (unsigned)c.N) * (unsigned)c.K) >> 48 == 0ull;
}

// Lanes of the warp that have a record in this turn of a loop over records; i is this lane's.
__device__ __forceinline__ unsigned lanes_with_record(int64_t i, int64_t n) {
  const int64_t left = n - (i - (threadIdx.x & 31));
  return left >= 32 ? 0xffffffffu : (1u << (int)left) - 1u;
}

// The whole numbers of a record of the space: tensor-pipe instructions of a
// K-step, bytes through TMEM (below 2^24), and whether the launch keeps one
// accumulator buffer (single_buffer).
struct SpaceInts {
  int n_instr, d_r, d_w;
  bool single;
};

__device__ __forceinline__ SpaceInts space_ints(const pm_cfg& c) {
  SpaceInts r;
  const int BM = c.BM, BN = c.BN, BK = c.BK, dt = c.dtype, blocks = 1 + (BM >> 8);
  const int passes = dt == PM_FP32 ? 3 : 1, esh = 2 - dt;        // element bytes 4, 2, 1
  r.n_instr = passes * (BK >> (3 + dt)) * blocks;
  r.d_r = r.d_w = 4 * BM * BN;
  if (c.tmem_a) {
    const int a = BM * BK << esh, loads = dt == PM_FP32 ? 2 : 1;
    r.d_r += passes * a;
    r.d_w += loads * a;
    r.n_instr += loads * ((BK << esh) >> 5) * blocks;
    const int acc = (BM < 128 && c.cta_group == 2) ? BN >> 1 : blocks * BN;
    r.single = 2 * acc + c.stages * blocks * (loads * (BK << esh) >> 2) > 512;
  } else {
    r.single = BM == 256 && BN == 256;                           // 512 columns
  }
  return r;
}

__device__ __forceinline__ void gemm_forward_space(const pm_cfg& c, const Theta& th, const SpaceTables& tab, GemmFwd& f) {
  const int gi = c.cta_group - 1, BM = c.BM, BN = c.BN, BK = c.BK;
  const float4 rt = tab.rate[2 * c.dtype + gi], dp = tab.depth[c.stages];
  const uint4 nc = tab.conc[gi];
  const float np = rt.z, le = rt.y, inv_rs = rt.x;
  const float bytes_min = le * ((float)c.M * c.K + (float)c.N * c.K) + 4.f * (float)c.M * (float)c.N;
  f.ri = 6 + c.dtype;
  f.invR = rt.w;
  f.invS = tab.inv_s2sm[gi];
  const int kb = BK >> 6;                                        // 32, 64, 128 -> 0, 1, 2
  const unsigned tm = ((unsigned)c.M + (unsigned)((BM << gi) - 1)) >> (6 + (BM >> 7) + gi);
  const unsigned tn = ((unsigned)c.N + (unsigned)(BN - 1)) >> (6 + (BN >> 7));
  const unsigned x = ((tm * tn) << gi) + nc.x;
  const unsigned q = __umulhi(nc.y, x);
  f.waves = (float)(int)((q + ((x - q) >> nc.z)) >> nc.w);
  f.Kt = (float)(int)(((unsigned)c.K + (unsigned)(BK - 1)) >> (5 + kb));
  f.D = (float)(4 * BM * BN);
  const SpaceInts si = space_ints(c);
  f.n_instr = (float)si.n_instr;
  f.D_r = (float)si.d_r;
  f.D_w = (float)si.d_w;
  const float T_tmem = f.D_r * th.inv[10] + f.n_instr * th.v[9] + f.D_w * th.inv[11];
  const int rows = gi == 0 ? max(BM, 128) : BM;
  f.X = (np * (float)(2 * rows * BN * BK)) * inv_rs;
  f.T_c = f.X + T_tmem;
  f.bstep = le * (float)(BK * (BM + (BN >> gi)));
  f.W = bytes_min;
  f.blend = true;
  f.E = pm_exp_fast(-f.W * th.inv[3]);
  f.rho = 1.f + (th.v[16] - 1.f) * f.E;
  f.T_tma = pm_add(th.v[4], pm_div_fast(f.bstep * th.inv[5], f.rho));
  const float T_sync = 2.f * th.v[12];
  f.oma = dp.x;
  f.inv_s = dp.y;
  f.inv_s1 = dp.z;
  f.oma_free = dp.w != 0.f;
  f.T_io = f.oma * f.T_tma;
  f.T_eq8 = pm_max(f.T_c, f.T_io) + T_sync;
  f.T_ring = (f.T_tma + f.T_c + T_sync) * f.inv_s;
  f.ring = f.T_ring > f.T_eq8;
  f.T_step = f.ring ? f.T_ring : f.T_eq8;
  f.store_bytes = f.D;
  f.drain = si.single;
  f.T_store = th.v[4] + f.store_bytes * th.inv[5] + (f.drain ? f.store_bytes * th.inv[17] : 0.f);
  f.launch = th.v[0] + th.v[13];
  f.T_stage = f.launch + f.waves * (f.Kt * f.T_step + f.T_store);
  const float flops = np * 2.f * (float)c.M * (float)c.N * (float)c.K;
  f.A_rl = flops * inv_rs * th.inv_nsm;
  f.B_rl = bytes_min * th.inv[2];
  f.T_rl = f.launch + (f.A_rl >= f.B_rl ? f.A_rl : f.B_rl);
  f.T = f.T_stage >= f.T_rl ? f.T_stage : f.T_rl;
}

// The same way in FP64, with its adjoint.  An FP64 warp instruction holds its
// scheduler's FP64 unit for 64 cycles on this GPU whatever its active lanes, so
// what counts is their number: whole numbers stay integers (products up to 2^52
// enter FP64 with one subtraction, the small ones through the bits of their exact
// FP32 value with none), what depends on the parameters alone comes from the host,
// and the one division by rho is a reciprocal used three times.  About 90
// instructions for the prediction and its slopes in place of 200.
template <class F>
struct SpaceHost {};
template <>
struct SpaceHost<double> {
  double inv_rs[6], inv_rsn[6], inv_r[6];    // by 2 dtype + (cta_group - 1): 1 / (R S), 1 / (n_SM R S), 1 / R
  double oma[8], inv_s[8], inv_s1[8];        // by stages: 1 - alpha, 1 / s, and 1 / (s - 1) where alpha is free, else 0
  double rho_m1, c3, ni10, ni11, t_sync, launch;   // rho_L2 - 1, its share of w0's slope, -1/BW^2, 2 L_mbar, launch
  uint4 conc[2];                             // as SpaceTables
};

static SpaceHost<double> make_space(const ThetaT<double>& th) {
  SpaceHost<double> k = {};
  for (int i = 0; i < 6; ++i) {
    k.inv_r[i] = th.inv[6 + i / 2];
    k.inv_rs[i] = k.inv_r[i] * (i % 2 ? th.inv[14] : 1.0);
    k.inv_rsn[i] = k.inv_rs[i] * th.inv_nsm;
  }
  for (int s = 0; s < 8; ++s) {
    const double r = th.v[15] * th.inv_s1[s];
    k.oma[s] = r <= 0.0 ? 0.0 : (r >= 1.0 ? 1.0 : r);
    k.inv_s[s] = th.inv_s[s];
    k.inv_s1[s] = r > 0.0 && r < 1.0 ? th.inv_s1[s] : 0.0;
  }
  k.rho_m1 = th.v[16] - 1.0;
  k.c3 = k.rho_m1 * th.inv[3] * th.inv[3];
  k.ni10 = -(th.inv[10] * th.inv[10]);
  k.ni11 = -(th.inv[11] * th.inv[11]);
  k.t_sync = 2.0 * th.v[12];
  k.launch = th.v[0] + th.v[13];
  for (int i = 0; i < 2; ++i)
    k.conc[i] = make_uint4(th.nc[i].d - 1u, th.nc[i].m, (unsigned)th.nc[i].s1, (unsigned)th.nc[i].s2);
  return k;
}
static SpaceHost<float> make_space(const ThetaT<float>&) { return {}; }

// A positive integer that FP32 holds exactly, through FP32's bits.
__device__ __forceinline__ double small_f64(int v) {
  const unsigned b = __float_as_uint((float)v);
  return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}
// An integer in [0, 2^52): the low bits of 2^52 + v.
__device__ __forceinline__ double large_f64(long long v) {
  return __longlong_as_double(0x4330000000000000ll | v) - 4503599627370496.0;
}

// T_hat of a record of the space; its slopes are written to d (all NP entries).
__device__ __forceinline__ double space_row(const pm_cfg& c, const ThetaT<double>& th, const SpaceHost<double>& k,
                                            double (&d)[NP]) {
  const int dt = c.dtype, gi = c.cta_group - 1, BM = c.BM, BN = c.BN, BK = c.BK, idx = 2 * dt + gi, s = c.stages;
  const int passes = dt == PM_FP32 ? 3 : 1, le = dt == PM_FP32 ? 8 : 2 >> (dt - 1);
  const SpaceInts si = space_ints(c);
  const long long mn = (long long)c.M * c.N;
  const double W = large_f64(le * (((long long)c.M + c.N) * c.K) + 4 * mn);
  const unsigned tm = ((unsigned)c.M + (unsigned)((BM << gi) - 1)) >> (6 + (BM >> 7) + gi);
  const unsigned tn = ((unsigned)c.N + (unsigned)(BN - 1)) >> (6 + (BN >> 7));
  const uint4 nc = k.conc[gi];
  const unsigned x = ((tm * tn) << gi) + nc.x, q = __umulhi(nc.y, x);
  const double waves = large_f64((long long)((q + ((x - q) >> nc.z)) >> nc.w));
  const double Kt = small_f64((int)((unsigned)(c.K + BK - 1) >> (5 + (BK >> 6))));
  const double D = small_f64(4 * BM * BN), D_r = small_f64(si.d_r), D_w = small_f64(si.d_w), n_i = small_f64(si.n_instr);
  const double inv_rs = k.inv_rs[idx], inv_s = k.inv_s[s], oma = k.oma[s];
  const double X = small_f64(passes * 2 * (gi == 0 ? max(BM, 128) : BM) * BN * BK) * inv_rs;
  const double E = exp(-W * th.inv[3]);
  const double inv_rho = __drcp_rn(fma(k.rho_m1, E, 1.0));
  const double t_bw = small_f64(le * BK * (BM + (BN >> gi))) * th.inv[5] * inv_rho;
  const double T_tma = th.v[4] + t_bw;
  const double T_c = X + fma(D_w, th.inv[11], fma(n_i, th.v[9], D_r * th.inv[10]));
  const double T_io = oma * T_tma;
  const bool c_first = T_c >= T_io;
  const double T_eq8 = fmax(T_c, T_io) + k.t_sync;
  const double T_ring = (T_tma + T_c + k.t_sync) * inv_s;
  const bool ring = T_ring > T_eq8;
  const double d5 = D * th.inv[5];
  double T_store = th.v[4] + d5, d17 = 0.0;
  if (si.single) {
    d17 = D * th.inv[17];
    T_store += d17;
  }
  const double T_stage = fma(waves, fma(Kt, ring ? T_ring : T_eq8, T_store), k.launch);
  const double A_rl = large_f64(2 * passes * mn) * small_f64(c.K) * k.inv_rsn[idx], B_rl = W * th.inv[2];
  const bool a_first = A_rl >= B_rl;
  const double T_rl = k.launch + (a_first ? A_rl : B_rl);
  const bool stage = T_stage >= T_rl;
  // slopes (step_store_adjoint, gemm_adjoint): the roofline branch has no share
  // in the tiles' terms
  const double g_w = stage ? waves : 0.0, g_step = g_w * Kt, g_ring = g_step * inv_s;
  const double g_c = ring ? g_ring : (c_first ? g_step : 0.0), g_io = ring || c_first ? 0.0 : g_step;
  const double g_tma = ring ? g_ring : g_io * oma, g_bw = g_tma * t_bw, g_E = -(g_bw * inv_rho) * E, g_x = g_c * X;
  double g_R = -(g_x * k.inv_r[idx]), g_S = gi ? -(g_x * th.inv[14]) : 0.0;
  d[2] = 0.0;
  if (!stage) {
    if (a_first) {
      g_R = -(A_rl * k.inv_r[idx]);
      g_S = gi ? -(A_rl * th.inv[14]) : 0.0;
    } else {
      d[2] = -(B_rl * th.inv[2]);
    }
  }
  d[0] = d[13] = 1.0;
  d[1] = 0.0;
  d[3] = g_E * W * k.c3;
  d[4] = g_w + g_tma;
  d[5] = -(fma(g_w, d5, g_bw) * th.inv[5]);
  d[6] = dt == PM_FP32 ? g_R : 0.0;
  d[7] = dt == PM_BF16 ? g_R : 0.0;
  d[8] = dt == PM_FP8E4M3 ? g_R : 0.0;
  d[9] = g_c * n_i;
  d[10] = g_c * D_r * k.ni10;
  d[11] = g_c * D_w * k.ni11;
  d[12] = 2.0 * (ring ? g_ring : g_step);
  d[14] = g_S;
  d[15] = g_io * T_tma * k.inv_s1[s];
  d[16] = g_E;
  d[17] = si.single ? -(g_w * d17 * th.inv[17]) : 0.0;
  return stage ? T_stage : T_rl;
}

// Memory probes.  Copy/triad through Eq. 16 with W = beta bytes moved;
// TMA2D: tile latency plus ceil(tiles/SMs) tile round trips (Eq. 4),
// bounded below by the streaming time of Eq. 16.
template <class F>
struct ProbeFwdT {
  F T, T1, T2, Bw, E, W, beta, moved_tiles;
  bool blend;
};
using ProbeFwd = ProbeFwdT<float>;

template <class F>
__device__ __forceinline__ void probe_forward(const pm_cfg& c, const ThetaT<F>& th, int n_sm, ProbeFwdT<F>& f) {
  F W, t2num;
  if (c.kind == PM_KIND_COPY || c.kind == PM_KIND_TRIAD) {
    f.beta = (c.kind == PM_KIND_COPY ? F(8) : F(12)) * (F)c.M;
    W = f.beta;
    t2num = f.beta;
  } else {
    const F t = F(4) * c.BM * c.BN;
    const int64_t nt = cdiv(c.M, c.BM) * cdiv(c.N, c.BN);
    f.moved_tiles = (F)cdiv(nt, n_sm) * F(2) * t;
    f.beta = F(8) * (F)c.M * (F)c.N;
    W = f.beta;
    t2num = f.moved_tiles;
  }
  f.W = W;
  f.blend = th.v[3] > F(0);
  f.E = f.blend ? pm_exp(-W / th.v[3]) : F(0);
  f.Bw = f.blend ? th.v[1] + (th.v[2] - th.v[1]) * f.E : th.v[1];
  if (c.kind == PM_KIND_COPY || c.kind == PM_KIND_TRIAD) {
    f.T1 = th.v[0] + f.beta / f.Bw;
    f.T2 = th.v[0] + f.beta / th.v[2];
  } else {
    f.T1 = th.v[0] + th.v[4] + t2num / th.v[5];
    f.T2 = th.v[0] + f.beta / f.Bw;
  }
  f.T = f.T1 >= f.T2 ? f.T1 : f.T2;
}

template <class F>
__device__ __forceinline__ void bw_adjoint(const ThetaT<F>& th, const ProbeFwdT<F>& f, F gB, F (&d)[NP]) {
  if (f.blend) {
    d[1] += gB * (F(1) - f.E);
    d[2] += gB * f.E;
    const F gE = gB * (th.v[2] - th.v[1]);
    d[3] += gE * f.E * f.W / (th.v[3] * th.v[3]);
  } else {
    d[1] += gB;
  }
}

template <class F>
__device__ __forceinline__ void probe_adjoint(const pm_cfg& c, const ThetaT<F>& th, const ProbeFwdT<F>& f, F w,
                                              F (&d)[NP]) {
  d[0] += w;
  const bool first = f.T1 >= f.T2;
  if (c.kind == PM_KIND_COPY || c.kind == PM_KIND_TRIAD) {
    if (first) bw_adjoint(th, f, -w * f.beta / (f.Bw * f.Bw), d);
    else d[2] -= w * f.beta / (th.v[2] * th.v[2]);
  } else {
    if (first) {
      d[4] += w;
      d[5] -= w * f.moved_tiles / (th.v[5] * th.v[5]);
    } else {
      bw_adjoint(th, f, -w * f.beta / (f.Bw * f.Bw), d);
    }
  }
}

// probe_forward and probe_adjoint in FP64 with one reciprocal in place of five
// divisions, the three kinds in step: a calibration table's few probe rows share a
// warp with its last GEMM rows, and the slowest warp ends the kernel (1,901 mixed
// records 13.0 -> 11.5 us).
__device__ __forceinline__ double probe_row(const pm_cfg& c, const ThetaT<double>& th, int n_sm, double (&d)[NP]) {
  const bool tma = c.kind == PM_KIND_TMA2D;
  double beta, other;                            // bytes, and the time that Eq. 16 is weighed against
  double other_slope;
  if (tma) {
    const int64_t nt = cdiv(c.M, c.BM) * cdiv(c.N, c.BN);
    beta = 8.0 * c.M * c.N;
    other_slope = (double)cdiv(nt, n_sm) * (8.0 * c.BM * c.BN) * th.inv[5];
    other = th.v[4] + other_slope;
  } else {
    beta = (c.kind == PM_KIND_COPY ? 8.0 : 12.0) * c.M;
    other_slope = other = beta * th.inv[2];
  }
  const bool blend = th.v[3] > 0.0;
  const double x = beta * th.inv[3], E = blend ? exp(-x) : 0.0, dB = th.v[2] - th.v[1];
  const double inv_bw = __drcp_rn(blend ? fma(dB, E, th.v[1]) : th.v[1]);
  const double stream = beta * inv_bw;
  // ties go to the first argument: the stream's time of copy and triad, the tiles' of TMA
  const double T_s = th.v[0] + stream, T_o = th.v[0] + other;
  const bool by_stream = tma ? !(T_o >= T_s) : T_s >= T_o;
#pragma unroll
  for (int j = 0; j < NP; ++j) d[j] = 0.0;
  d[0] = 1.0;
  if (by_stream) {
    const double gB = -(stream * inv_bw);
    if (blend) {
      const double gE = gB * E;
      d[1] = gB - gE;
      d[2] = gE;
      d[3] = gE * dB * x * th.inv[3];
    } else {
      d[1] = gB;
    }
  } else if (tma) {
    d[4] = 1.0;
    d[5] = -(other_slope * th.inv[5]);
  } else {
    d[2] = -(other_slope * th.inv[2]);
  }
  return by_stream ? T_s : T_o;
}

// A record the model can evaluate on n_sm SMs; a CTA pair (cta_group 2)
// needs two SMs (Sec. III-A.4), so on one SM a pair record has no time.
__device__ __forceinline__ bool cfg_sane(const pm_cfg& c, int n_sm) {
  if (c.kind == PM_KIND_GEMM)
    return c.M > 0 && c.N > 0 && c.K > 0 && c.BM > 0 && c.BN > 0 && c.BK > 0 && c.stages > 0 &&
           (c.cta_group == 1 || (c.cta_group == 2 && n_sm >= 2)) && c.dtype >= 0 && c.dtype <= 2 &&
           (c.tmem_a == 0 || c.tmem_a == 1);
  if (c.kind == PM_KIND_COPY || c.kind == PM_KIND_TRIAD) return c.M > 0;
  if (c.kind == PM_KIND_TMA2D) return c.M > 0 && c.N > 0 && c.BM > 0 && c.BN > 0;
  return false;
}

__device__ __forceinline__ pm_cfg load_cfg(const pm_cfg* p) {
  // 24-byte record as three 8-byte loads
  const int2* q = reinterpret_cast<const int2*>(p);
  int2 a = __ldg(q), b = __ldg(q + 1), cc = __ldg(q + 2);
  pm_cfg c;
  int2* o = reinterpret_cast<int2*>(&c);
  o[0] = a; o[1] = b; o[2] = cc;
  return c;
}

// Bound: ALU issue (some 215 warp-instructions per 32 configurations in the search
// space, 377 by the general way; 28 bytes each).  10^6 configurations 12.9 -> 8.8 us,
// 10^7 114 -> 70 us with the short way of gemm_forward_space.  Six blocks per SM
// (40 registers, no spills): 48 warps hide the latency of the dependent FP32
// chain better than 40 or, at 32 registers, 64 (10^6: 11.0 us).
// SPACE: the launch's parameters allow the short way.  Its records do not choose
// together: a vote of the warp costs 0.4 us per 10^6 records, and only tables that
// mix tiles inside and outside the search space pay for both ways (every other
// record outside: 18.7 us, 14.1 by the general way alone).
template <bool SPACE>
__global__ void __launch_bounds__(256, 6) model_predict_kernel(const pm_cfg* __restrict__ cfgs, int64_t n, Theta th,
                                                            int n_sm, float* __restrict__ out) {
  __shared__ SpaceTables tab;
  if constexpr (SPACE) space_tables(th, tab);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const pm_cfg c = load_cfg(cfgs + i);
    float t;
    if (SPACE && in_space(c)) {
      GemmFwd f;
      gemm_forward_space(c, th, tab, f);
      t = f.T;
    } else if (!cfg_sane(c, n_sm)) {
      t = __int_as_float(0x7fc00000);
    } else if (c.kind == PM_KIND_GEMM) {
      GemmFwd f;
      gemm_forward<SPACE>(c, th, n_sm, f);
      t = f.T;
    } else {
      ProbeFwd f;
      probe_forward(c, th, n_sm, f);
      t = f.T;
    }
    out[i] = t;
  }
}

// Loss and gradient: per-thread terms and warp sums in F, warp totals
// combined in FP64 into one partial record of NREC values per block; a
// second kernel adds the records in block order (deterministic).
constexpr int kGradThreads = 256;

template <class T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum_d(double v) { return warp_sum<double>(v); }

// Sums of N values over the warp's lanes by recursive halving: at every step a
// lane hands half of its values to its partner and adds the partner's half to
// the rest, so N = 19 takes 21 shuffles and additions in place of 95.  The tree
// of each sum is warp_sum's.  One lane ends with the total of value `index`
// (index < 0: this lane has none).
template <int C, int O, class T, int N>
__device__ __forceinline__ void sum_halving(T (&v)[N], int& first, int& mine) {
  constexpr int H = (C + 1) / 2;
  const bool up = (threadIdx.x & O) != 0;
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const T hi = i + H < C ? v[i + H < N ? i + H : 0] : T(0);
    const T send = up ? v[i] : hi, keep = up ? hi : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
  }
  first += up ? H : 0;
  mine = up ? mine - H : min(mine, H);
  if constexpr (O > 1) sum_halving<H, O / 2>(v, first, mine);
}

template <class T, int N>
__device__ __forceinline__ T warp_sum_each(T (&v)[N], int& index) {
  static_assert(N <= 32, "one lane per value");
  int first = 0, mine = N;
  sum_halving<N, 16>(v, first, mine);
  index = mine > 0 ? first : -1;
  return v[0];
}

// F = float: per-configuration FP32 terms (throughput path); F = double: the
// whole evaluation in FP64 so the calibration's line searches see a smooth
// objective.  The FP32 kernel is held to four blocks per SM (64 registers,
// 32 warps to hide the dependent-instruction latency; 19 % faster than the
// 78-register build at three); the FP64 one at two (128 registers).
template <class F>
constexpr int grad_min_blocks() { return sizeof(F) == 4 ? 4 : 2; }

// Bound: FP32 ALU issue, FP64 at every size the FP64 units.  With the sums by halving,
// the short way and, in FP64, the clusters and space_row, against one general way with
// a tree per sum; both launches of a call: FP32 10^6 configurations 33.5 -> 18.2 us, 10^7
// 224 -> 131; FP64 1,901 configurations 31.6 -> 13.8, 10^6 494 -> 320.
//
// One partial record per kGradThreads threads, the threads of a record spread
// over a cluster of CL blocks: partials[j * records + r] is component j of
// record r.  CL > 1 for few records, so that they use CL times as many SMs;
// the sums are the same, term by term, whatever CL.
//
// SPACE as in model_predict_kernel.  In FP64 the GEMM records of a warp go one way
// together: one outside the space takes the others with it (every other of 10^6
// records outside: 616 -> 437 us; 495 by the general way alone).
template <class F, int CL, bool SPACE>
__global__ void __launch_bounds__(kGradThreads / CL, CL == 1 ? grad_min_blocks<F>() : 1)
    model_grad_kernel(const pm_cfg* __restrict__ cfgs, int64_t n, const __grid_constant__ ThetaT<F> th,
                      const __grid_constant__ SpaceHost<F> sh, int n_sm, const F* __restrict__ t_meas,
                      double* __restrict__ partials) {
  constexpr int kThreads = kGradThreads / CL;
  grid_dependents_launch();                      // the finish kernel may be set up (it waits for this grid)
  if constexpr (CL > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  const int records = (int)(gridDim.x / CL), rec = (int)(blockIdx.x / CL), part = (int)(blockIdx.x % CL);
  // the short way's tables, in shared memory (lanes index them by their own record)
  __shared__ std::conditional_t<sizeof(F) == 4, SpaceTables, SpaceHost<F>> tab;
  if constexpr (!SPACE) {
  } else if constexpr (sizeof(F) == 4) {
    space_tables(th, tab);
  } else {
    const int* from = reinterpret_cast<const int*>(&sh);
    for (int w = threadIdx.x; w < (int)(sizeof(sh) / 4); w += kThreads) reinterpret_cast<int*>(&tab)[w] = from[w];
    __syncthreads();
  }
  F acc[NREC];                                   // loss, then the gradient
#pragma unroll
  for (int j = 0; j < NREC; ++j) acc[j] = F(0);
  for (int64_t i = (int64_t)rec * kGradThreads + part * kThreads + threadIdx.x; i < n;
       i += (int64_t)records * kGradThreads) {
    const pm_cfg c = load_cfg(cfgs + i);
    const F log_t = pm_log(__ldg(t_meas + i));
    F d[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) d[j] = F(0);
    F T;
    bool space = false;
    if constexpr (SPACE && sizeof(F) == 4) space = in_space(c);
    if constexpr (SPACE && sizeof(F) == 8) {
      space = in_space_f64(c);
      const bool outside = __any_sync(lanes_with_record(i, n), !space && c.kind == PM_KIND_GEMM);
      space = space && !outside;
    }
    if (space) {
      if constexpr (sizeof(F) == 4) {
        GemmFwd f;
        gemm_forward_space(c, th, tab, f);
        T = f.T;
        gemm_adjoint<true>(c, th, f, F(1), d);
      } else {
        T = space_row(c, th, tab, d);
      }
    } else if (!cfg_sane(c, n_sm)) {
      T = (F)__int_as_float(0x7fc00000);
    } else if (c.kind == PM_KIND_GEMM) {
      GemmFwdT<F> f;
      gemm_forward<SPACE>(c, th, n_sm, f);
      T = f.T;
      gemm_adjoint(c, th, f, F(1), d);
    } else if constexpr (sizeof(F) == 4) {
      ProbeFwdT<F> f;
      probe_forward(c, th, n_sm, f);
      T = f.T;
      probe_adjoint(c, th, f, F(1), d);
    } else {
      T = probe_row(c, th, n_sm, d);
    }
    const F r = pm_log(T) - log_t;
    acc[0] = fma(r, r, acc[0]);
    const F w = F(2) * r / T;
#pragma unroll
    for (int j = 0; j < NP; ++j) acc[j + 1] = fma(w, d[j], acc[j + 1]);
  }
  // warp sums in F (FP64 arithmetic is scarce on this GPU), warp totals
  // combined in FP64 by the record's first block
  __shared__ double red[kGradThreads / 32][NREC];
  int j;
  const F v = warp_sum_each<F, NREC>(acc, j);
  const int warp = part * (kThreads / 32) + (threadIdx.x >> 5);
  if constexpr (CL == 1) {
    if (j >= 0) red[warp][j] = (double)v;
    __syncthreads();
  } else {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");       // the first block has started
    if (j >= 0)
      asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(mapa_shared(smem_u32(&red[warp][j]), 0)), "d"((double)v)
                   : "memory");
    __syncwarp();
    cluster_sync();
    if (part != 0) return;
  }
  if (threadIdx.x < NREC) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kGradThreads / 32; ++w) s += red[w][threadIdx.x];
    partials[(int64_t)threadIdx.x * records + rec] = s;
  }
}

// Block j sums component j of the records: lane l adds records l, l+32, ... in
// order, then a fixed butterfly combines the lanes, so the result depends only
// on the number of records (deterministic).  Bound: latency; a block per
// component reading consecutive records, twenty loads of a lane in flight (608
// records on 152 SMs), takes 3.7 us where one block with strided records took
// 8.5, and it is set up while the partial sums are made (programmatic launch:
// 1.2 to 2.5 us less from one call to the next).
__global__ void __launch_bounds__(32) model_grad_finish_kernel(const double* partials, int records, int64_t n,
                                                               double* out) {
  constexpr int kBatch = 20;
  grid_dependency_wait();                        // the records are complete and visible
  const double* p = partials + (int64_t)blockIdx.x * records;
  double s = 0.0;
  for (int b = threadIdx.x; b < records; b += 32 * kBatch) {
    double v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) v[u] = b + 32 * u < records ? p[b + 32 * u] : 0.0;
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      if (b + 32 * u < records) s += v[u];
  }
  s = warp_sum_d(s);
  if (threadIdx.x == 0) out[blockIdx.x] = s / (double)n;
}

// Partial records of a call: one per kGradThreads configurations, one wave at most.
static int grad_blocks(int64_t n) {
  const int64_t want = (n + kGradThreads - 1) / kGradThreads;
  const int cap = std::max(1, sm_count()) * 4;             // one wave: four blocks per SM (launch bound)
  return (int)std::max<int64_t>(1, std::min<int64_t>(want, cap));
}

// Autotuner: the k predicted-fastest valid configurations of each shape over
// the 180-point space in lexicographic (BM, BN, BK, stages, cta_group) order,
// in increasing predicted time, ties to the first.  Two splits of the work with
// the same results, bit for bit:
//
// autotune_table_kernel (many shapes): a block tabulates the terms of Eqs. 2-8
// that depend on the tile only, for the valid tiles of the type, once; then a
// warp takes a shape: its lanes work out the shape's terms (bytes, rho, the
// roofline bounds, one wave count per cta_group, BM and BN) and evaluate up to
// six tiles each from the table with the arithmetic of gemm_forward.  Bound:
// ALU issue; BF16 (121 valid tiles), best tile of 5,556 shapes 17.1 -> 7.3 us and
// of 555,555 shapes 1383 -> 359 us against a whole model evaluation per
// (shape, tile); best eight of 5,556 shapes 46.9 -> 14.3 us.
//
// autotune_shape_kernel (few shapes): a block per shape, thread t evaluates
// tile t.  Bound: latency; it has no table to build before the first shape, so
// it is the faster one while every block is resident at once (launch_autotune).
constexpr int kTuneThreads = 512;
constexpr int kTuneTiles = 180;
constexpr int kTunePerLane = (kTuneTiles + 31) / 32;
constexpr int kMaxTopK = 16;

__device__ __forceinline__ void decode_tile(int t, int dt, int& BM, int& BN, int& BK, int& s, int& g) {
  BM = kBM[t / 60];
  BN = kBN[(t / 20) % 3];
  BK = kBK[dt][(t / 10) % 2];
  s = 2 + (t / 2) % 5;
  g = 1 + t % 2;
}

// The tile's wave-count slot (cta_group, BM, BN) and BK index.
__device__ __forceinline__ int tile_slot(int t) { return (t % 2) * 9 + (t / 60) * 3 + (t / 20) % 3; }
__device__ __forceinline__ int tile_bk(int t) { return (t / 10) % 2; }

// k rounds of warp argmin over (time, index): lane l holds the times of the
// candidates l, l + 32, ... in v (INFINITY where there is none).  Lane r < k gets
// round r's time and index (-1: no candidate left).  A NaN time loses to any
// finite one.
__device__ __forceinline__ void warp_topk(float (&v)[kTunePerLane], int k, float& my_t, int& my_i) {
  const int lane = threadIdx.x & 31;
  my_t = INFINITY;
  my_i = -1;
  for (int r = 0; r < k; ++r) {
    float bv = v[0];
    int bi = lane;
#pragma unroll
    for (int j = 1; j < kTunePerLane; ++j)
      if (v[j] < bv || (bv != bv && v[j] < INFINITY)) { bv = v[j]; bi = lane + 32 * j; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov < bv || (ov == bv && oi < bi) || (bv != bv && ov < INFINITY)) { bv = ov; bi = oi; }
    }
    bv = __shfl_sync(0xffffffffu, bv, 0);
    bi = __shfl_sync(0xffffffffu, bi, 0);
    if (!(bv < INFINITY)) bi = -1;
    if (lane == r) { my_t = bv; my_i = bi; }
#pragma unroll
    for (int j = 0; j < kTunePerLane; ++j)
      if (bi == lane + 32 * j) v[j] = INFINITY;
  }
}

// The record of tile t (t < 0: none, BM = 0) for a shape.
__device__ __forceinline__ pm_cfg tune_pick(int M, int N, int K, int dt, int t) {
  pm_cfg p;
  p.M = M; p.N = N; p.K = K;
  p.dtype = (int8_t)dt; p.kind = PM_KIND_GEMM; p.tmem_a = 0;
  p.BM = p.BN = p.BK = 0; p.stages = p.cta_group = 0;
  if (t >= 0) {
    int BM, BN, BK, s, g;
    decode_tile(t, dt, BM, BN, BK, s, g);
    p.BM = (int16_t)BM; p.BN = (int16_t)BN; p.BK = (int16_t)BK;
    p.stages = (int8_t)s; p.cta_group = (int8_t)g;
  }
  return p;
}

__global__ void __launch_bounds__(kTunePerLane * 32) autotune_shape_kernel(const int32_t* __restrict__ MNK, int64_t n,
                                                                          int dt, Theta th, int n_sm, int k,
                                                                          pm_cfg* __restrict__ picks,
                                                                          float* __restrict__ t_pred) {
  __shared__ float times[kTunePerLane * 32];
  const int t = threadIdx.x, lane = t & 31;
  const int64_t shape = blockIdx.x;
  pm_cfg c;
  c.M = __ldg(MNK + 3 * shape);
  c.N = __ldg(MNK + 3 * shape + 1);
  c.K = __ldg(MNK + 3 * shape + 2);
  int BM, BN, BK, s, g;
  decode_tile(min(t, kTuneTiles - 1), dt, BM, BN, BK, s, g);
  float time = INFINITY;
  if (t < kTuneTiles && tile_valid(BM, BN, BK, s, g, dt) && (g == 1 || n_sm >= 2) && c.M > 0 && c.N > 0 && c.K > 0) {
    c.BM = (int16_t)BM; c.BN = (int16_t)BN; c.BK = (int16_t)BK;
    c.stages = (int8_t)s; c.cta_group = (int8_t)g; c.dtype = (int8_t)dt; c.kind = PM_KIND_GEMM; c.tmem_a = 0;
    GemmFwd f;
    gemm_forward(c, th, n_sm, f);
    time = f.T;
  }
  times[t] = time;
  __syncthreads();
  if (t >= 32) return;
  float v[kTunePerLane], my_t;
  int my_i;
#pragma unroll
  for (int j = 0; j < kTunePerLane; ++j) v[j] = times[lane + 32 * j];
  warp_topk(v, k, my_t, my_i);
  if (lane < k) {
    picks[shape * k + lane] = tune_pick(c.M, c.N, c.K, dt, my_i);
    t_pred[shape * k + lane] = my_t;
  }
}

__global__ void __launch_bounds__(kTuneThreads, 2) autotune_table_kernel(const int32_t* __restrict__ MNK, int64_t n,
                                                                         int dt, Theta th, int n_sm, int k,
                                                                         pm_cfg* __restrict__ picks,
                                                                         float* __restrict__ t_pred) {
  __shared__ float4 row_a[kTuneTiles];           // T_c (without T_mgmt), b_step / B_TMA, T_store, 1 - alpha
  __shared__ float2 row_b[kTuneTiles];           // 1 / stages, code: tile | slot << 8 | BK index << 13
  __shared__ int warp_valid[kTuneThreads / 32];
  const bool measured = th.reading == PM_READING_MEASURED;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int n_tiles = 0;
  {
    const int t = threadIdx.x;
    int BM, BN, BK, s, g;
    decode_tile(min(t, kTuneTiles - 1), dt, BM, BN, BK, s, g);
    const bool valid = t < kTuneTiles && tile_valid(BM, BN, BK, s, g, dt) && (g == 1 || n_sm >= 2);
    const unsigned vote = __ballot_sync(0xffffffffu, valid);
    if (lane == 0) warp_valid[warp] = __popc(vote);
    __syncthreads();
    int at = __popc(vote & ((1u << lane) - 1u));
    for (int w = 0; w < (kTuneTiles + 31) / 32; ++w) {
      if (w < warp) at += warp_valid[w];
      n_tiles += warp_valid[w];
    }
    if (valid) {
      pm_cfg c;
      c.M = c.N = c.K = 64;                      // the tabulated terms do not depend on the shape
      c.BM = (int16_t)BM; c.BN = (int16_t)BN; c.BK = (int16_t)BK;
      c.stages = (int8_t)s; c.cta_group = (int8_t)g; c.dtype = (int8_t)dt; c.kind = PM_KIND_GEMM; c.tmem_a = 0;
      GemmFwd f;
      gemm_forward(c, th, n_sm, f);
      row_a[at] = make_float4(f.XT, f.bstep * th.inv[5], f.T_store, f.oma);
      row_b[at] = make_float2(th.inv_s[s], __int_as_float(t | tile_slot(t) << 8 | tile_bk(t) << 13));
    }
    __syncthreads();
  }
  const float e = dt_bytes(dt), np = dt_passes(dt), l = dt_loads(dt);
  const int ri = dt_rate(dt);
  const float T_sync = 2.f * th.v[12];
  const float launch = measured ? th.v[0] + th.v[13] : th.v[0];
  const bool blend = measured && th.v[3] > 0.f;
  for (int64_t shape = (int64_t)blockIdx.x * (kTuneThreads / 32) + warp; shape < n;
       shape += (int64_t)gridDim.x * (kTuneThreads / 32)) {
    const int M = __ldg(MNK + 3 * shape), N = __ldg(MNK + 3 * shape + 1), K = __ldg(MNK + 3 * shape + 2);
    float v[kTunePerLane];
#pragma unroll
    for (int j = 0; j < kTunePerLane; ++j) v[j] = INFINITY;
    if (M > 0 && N > 0 && K > 0) {
      const float bytes_min = l * e * ((float)M * K + (float)N * K) + 4.f * (float)M * (float)N;
      const float E = blend ? pm_exp_fast(-bytes_min * th.inv[3]) : 0.f;
      const float rho = blend ? 1.f + (th.v[16] - 1.f) * E : 1.f;
      const float flops = np * 2.f * (float)M * (float)N * (float)K;
      const float B_rl = bytes_min * th.inv[2];
      float T_rl[2], Kt[2], mgmt[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float inv_rs = th.inv[ri] * (i == 0 ? 1.f : th.inv[14]);
        const float A_rl = th.nc_nsm == n_sm ? flops * inv_rs * th.inv_nsm : flops * inv_rs / (float)n_sm;
        T_rl[i] = launch + (A_rl >= B_rl ? A_rl : B_rl);
        Kt[i] = count_to<float>(cdiv(K, kBK[dt][i]));
        mgmt[i] = measured ? 0.f : th.v[13] / Kt[i];
      }
      float waves = 0.f;
      if (lane < 18) {
        const int g = 1 + lane / 9, BM = kBM[lane % 9 / 3], BN = kBN[lane % 3];
        const int64_t tiles = measured ? (int64_t)g * cdiv(M, (int64_t)g * BM) * cdiv(N, BN) : cdiv(M, BM) * cdiv(N, BN);
        waves = count_to<float>(wave_count(tiles, g, th, n_sm));
      }
#pragma unroll
      for (int j = 0; j < kTunePerLane; ++j) {
        if (32 * j >= n_tiles) break;
        const int i = min(lane + 32 * j, n_tiles - 1);
        const float4 a = row_a[i];
        const float2 b = row_b[i];
        const int code = __float_as_int(b.y);
        const float wv = __shfl_sync(0xffffffffu, waves, (code >> 8) & 31);
        const bool bk1 = (code >> 13) & 1, pair = code & 1;
        const float T_c = a.x + (bk1 ? mgmt[1] : mgmt[0]);
        const float T_tma = th.v[4] + (blend ? pm_div_fast(a.y, rho) : a.y);
        const float T_io = measured ? a.w * T_tma : a.w * T_tma + T_sync;
        const float T_eq8 = pm_max(T_c, T_io) + T_sync;
        const float T_ring = measured ? (T_tma + T_c + T_sync) * b.x : 0.f;
        const float T_step = measured && T_ring > T_eq8 ? T_ring : T_eq8;
        const float T_stage = launch + wv * ((bk1 ? Kt[1] : Kt[0]) * T_step + a.z);
        const float bound = pair ? T_rl[1] : T_rl[0];
        if (lane + 32 * j < n_tiles) v[j] = T_stage >= bound ? T_stage : bound;
      }
    }
    float my_t;
    int my_i;
    warp_topk(v, k, my_t, my_i);
    if (lane < k) {
      picks[shape * k + lane] = tune_pick(M, N, K, dt, my_i < 0 ? -1 : __float_as_int(row_b[my_i].y) & 255);
      t_pred[shape * k + lane] = my_t;
    }
  }
}

// Grouped launches.  The kernel's static schedule (pm_grouped_gemm_run):
// with several groups the launch lists them largest tile (BM x BN) first,
// ties in the caller's order, and deals the listed tiles to the n_conc
// workers round by round, reversing the worker order on odd rounds; one
// group is dealt plainly round by round.  A group-q tile costs
//   tau_q = K_tiles T_step_q + T_store_q
// with that group's (BM, BN) and the launch's (BK, stages, cta_group), and
// the launch ends with its busiest worker:
//   T_hat = launch + max_w sum_q n_{w,q} tau_q.
constexpr int kGroupThreads = 256;       // one launch's makespan and its gradient
constexpr int kGroupTuneThreads = 1024;  // the tuner: a thread per (group, tile)
constexpr int kMaxGroups = 1024;
constexpr int kGroupClasses = 6;         // tile areas 4096 << 4 .. 4096 << 0, then none

// The launch's schedule.  list[i] = the group at position i of the launch's
// list (pos[q] the position of group q), tau[i] = its tile time, and the first
// position past it,
// off[i + 1] = sum of the listed groups' tiles, kept as off = per * P + rem with
// P the period of the deal (n workers dealt plainly, 2 n when odd rounds are
// reversed): a worker's share of any range of positions is then two compares
// (dealt_before) instead of 64-bit divisions per worker and group.
template <class F>
struct Schedule {
  F tau[kMaxGroups];
  int64_t per[kMaxGroups + 1];
  unsigned rem[kMaxGroups + 1];          // below P < 2^32
  int16_t list[kMaxGroups], pos[kMaxGroups];
  uint8_t key[kMaxGroups];               // class << 5 | rank inside its 32 groups
  int cls[kGroupClasses][32];            // groups per class and 32 groups, then their first positions
  int cls_total[kGroupClasses];
  int64_t part[32];                      // tiles per 32 positions, then their first position
};

// How many of the positions [0, off[i]) are dealt to worker w: position t goes
// to worker t mod n, or with reversed odd rounds to the w with t mod 2n in
// {w, 2n - 1 - w}.
template <class F>
__device__ __forceinline__ int64_t dealt_before(const Schedule<F>& sc, int i, int64_t w, int64_t n, bool rev) {
  const int64_t r = sc.rem[i];
  return rev ? 2 * sc.per[i] + (r > w) + (r > 2 * n - 1 - w) : sc.per[i] + (r > w);
}

// Working set of a grouped launch (every group's A rows, its B and its C),
// for the L2 residency of the TMA loads; called by all threads of a block.
template <class F>
__device__ F grouped_working_set(const int32_t* Mg, int G, int N, int K, int dt) {
  __shared__ unsigned long long sum_m;
  if (threadIdx.x == 0) sum_m = 0ull;
  __syncthreads();
  unsigned long long mine = 0ull;
  for (int q = threadIdx.x; q < G; q += blockDim.x) mine += (unsigned long long)Mg[q];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(&sum_m, mine);
  __syncthreads();
  const F sm = (F)sum_m;
  return (F)dt_loads(dt) * (F)dt_bytes(dt) * (sm * (F)K + (F)G * (F)N * (F)K) + F(4) * sm * (F)N;
}

// Inclusive sum over the warp's lanes.
__device__ __forceinline__ int64_t warp_scan(int64_t v) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t u = __shfl_up_sync(0xffffffffu, v, o);
    if ((int)(threadIdx.x & 31) >= o) v += u;
  }
  return v;
}

// Lists the launch's groups: largest tile area first (area / 4096 = 2^class,
// class 4..0; a group without a valid tile, area 0, last), ties in the caller's
// order: a counting sort over 32-group pieces with warp votes, then a prefix
// sum of the listed tiles.  tiles[q] by group; sc.tau is the caller's to fill.
// Called by all threads (blockDim a multiple of 32, at least six warps).
template <class F>
__device__ void grouped_list(const int16_t* bm, const int16_t* bn, const int64_t* tiles, int G, int64_t n_conc,
                             Schedule<F>& sc) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  const int pieces = (G + 31) >> 5;
  for (int pc = warp; pc < pieces; pc += n_warps) {
    const int q = 32 * pc + lane;
    // 0: area 16 * 4096 .. 4: 4096, 5: no tile (G = 1 is its own order)
    const int c = q < G ? 5 - __ffs(((int)bm[q] * (int)bn[q]) >> 12) : -1;
#pragma unroll
    for (int k = 0; k < kGroupClasses; ++k) {
      const unsigned m = __ballot_sync(0xffffffffu, c == k);
      if (c == k) sc.key[q] = (uint8_t)((k << 5) | __popc(m & ((1u << lane) - 1u)));
      if (lane == 0) sc.cls[k][pc] = __popc(m);
    }
  }
  __syncthreads();
  if (warp < kGroupClasses) {
    const int v = lane < pieces ? sc.cls[warp][lane] : 0;
    const int inc = (int)warp_scan(v);
    if (lane < pieces) sc.cls[warp][lane] = inc - v;
    if (lane == 31) sc.cls_total[warp] = inc;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < G; q += blockDim.x) {
    const int key = sc.key[q], c = key >> 5;
    int i = sc.cls[c][q >> 5] + (key & 31);
    for (int k = 0; k < c; ++k) i += sc.cls_total[k];
    sc.list[i] = (int16_t)q;
    sc.pos[q] = (int16_t)i;
  }
  __syncthreads();
  for (int pc = warp; pc < pieces; pc += n_warps) {
    const int i = 32 * pc + lane;
    const int64_t inc = warp_scan(i < G ? tiles[sc.list[i]] : 0);
    if (i < G) sc.per[i + 1] = inc;
    if (lane == 31) sc.part[pc] = inc;
  }
  __syncthreads();
  if (warp == 0) {
    const int64_t v = lane < pieces ? sc.part[lane] : 0;
    const int64_t inc = warp_scan(v);
    if (lane < pieces) sc.part[lane] = inc - v;
  }
  __syncthreads();
  const int64_t P = G > 1 ? 2 * n_conc : n_conc;
  for (int i = threadIdx.x; i < G; i += blockDim.x) {
    const int64_t off = sc.per[i + 1] + sc.part[i >> 5];
    const int64_t per = P > 0 ? off / P : 0;      // no worker: the caller rejects the launch
    sc.per[i + 1] = per;
    sc.rem[i + 1] = (unsigned)(off - per * P);
  }
  if (threadIdx.x == 0) { sc.per[0] = 0; sc.rem[0] = 0; }
  __syncthreads();
}

// Busiest worker's time and (in *w_star) the first worker that has it;
// busy_w adds n_{w,q} tau_q over the list in order.  Called by all threads;
// the result is valid in every thread.
template <class F>
__device__ F grouped_makespan(const Schedule<F>& sc, int G, int64_t n_conc, int* w_star) {
  __shared__ F red_v[32];
  __shared__ int red_i[32];
  const bool rev = G > 1;
  F mx = F(-1);
  int mi = 0x7fffffff;
  for (int64_t w = threadIdx.x; w < n_conc; w += blockDim.x) {
    F busy = F(0);
    int64_t before = 0;
#pragma unroll 4
    for (int i = 0; i < G; ++i) {
      const int64_t upto = dealt_before(sc, i + 1, w, n_conc, rev);
      const int64_t cnt = upto - before;
      before = upto;
      if (cnt) busy += count_to<F>(cnt) * sc.tau[i];
    }
    if (busy > mx) { mx = busy; mi = (int)w; }
  }
  auto reduce = [&]() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const F ov = __shfl_xor_sync(0xffffffffu, mx, o);
      const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
      if (ov > mx || (ov == mx && oi < mi)) { mx = ov; mi = oi; }
    }
  };
  reduce();
  const int lane = threadIdx.x & 31;
  if (lane == 0) { red_v[threadIdx.x >> 5] = mx; red_i[threadIdx.x >> 5] = mi; }
  __syncthreads();
  mx = lane < (int)(blockDim.x >> 5) ? red_v[lane] : F(-1);
  mi = lane < (int)(blockDim.x >> 5) ? red_i[lane] : 0x7fffffff;
  reduce();
  if (w_star) *w_star = mi;
  return mx;
}

template <class F>
__device__ __forceinline__ int64_t launch_tiles(const ThetaT<F>& th, int M, int N, int BM, int BN, int g) {
  return th.reading == PM_READING_MEASURED ? (int64_t)g * cdiv(M, (int64_t)g * BM) * cdiv(N, BN)
                                           : cdiv(M, BM) * cdiv(N, BN);
}

template <class F>
__device__ __forceinline__ F launch_time(const ThetaT<F>& th) {
  return th.reading == PM_READING_MEASURED ? th.v[0] + th.v[13] : th.v[0];
}

// Grouped autotuner: block b handles launch-level combination b =
// (BK index, stages, cta_group) in lexicographic order; a thread per (group,
// tile) evaluates the model, a thread per group picks the (BM, BN) minimising
// tiles x tau, then the makespan of the launch's schedule is evaluated.  The
// row counts and the results are in the caller's page-locked host memory.
//
// Bound: latency (20 blocks, one wave).  Nine threads per group in place of
// nine evaluations per thread, the counting sort and prefix sum in place of one
// thread's loops, and no division in the worker loop took the kernel from
// 84 to 10.7 us at 64 groups.
__global__ void __launch_bounds__(kGroupTuneThreads) grouped_tune_kernel(const int32_t* __restrict__ Mg, int G, int N,
                                                                         int K, int dt, Theta th, int n_sm,
                                                                         float* __restrict__ out_t,
                                                                         int16_t* __restrict__ out_bm,
                                                                         int16_t* __restrict__ out_bn) {
  __shared__ Schedule<float> sc;
  __shared__ int32_t Ms[kMaxGroups];
  __shared__ float tau[kMaxGroups];
  __shared__ int64_t tiles[kMaxGroups];
  __shared__ int16_t bm_s[kMaxGroups], bn_s[kMaxGroups];
  // the candidates of a pass, in memory that the schedule takes later
  static_assert(sizeof(sc.per) >= 4 * kGroupTuneThreads && sizeof(sc.rem) >= 4 * kGroupTuneThreads, "candidates");
  float* const cand_cost = reinterpret_cast<float*>(sc.per);
  float* const cand_tau = reinterpret_cast<float*>(sc.rem);
  const int combo = blockIdx.x;                 // 0..19
  const int BK = kBK[dt][combo / 10];
  const int s = 2 + (combo / 2) % 5;
  const int g = 1 + combo % 2;
  for (int q = threadIdx.x; q < G; q += blockDim.x) Ms[q] = Mg[q];
  __syncthreads();
  const float W = grouped_working_set<float>(Ms, G, N, K, dt);
  bool any_invalid = false;
  constexpr int kPass = kGroupTuneThreads / 9;  // groups per pass
  for (int q0 = 0; q0 < G; q0 += kPass) {
    const int t = (int)threadIdx.x;
    const int q = q0 + t / 9, a = (t % 9) / 3, b = t % 3;
    if (t < 9 * kPass && q < G) {
      float cost = INFINITY, tq = 0.f;
      const int BM = kBM[a], BN = kBN[b];
      if (tile_valid(BM, BN, BK, s, g, dt)) {
        pm_cfg c;
        c.M = Ms[q]; c.N = N; c.K = K; c.BM = (int16_t)BM; c.BN = (int16_t)BN; c.BK = (int16_t)BK;
        c.stages = (int8_t)s; c.cta_group = (int8_t)g; c.dtype = (int8_t)dt; c.kind = 0; c.tmem_a = 0;
        GemmFwd f;
        gemm_forward(c, th, n_sm, f, W);
        tq = f.Kt * f.T_step + f.T_store;                // one tile of this group
        cost = (float)launch_tiles(th, c.M, N, BM, BN, g) * tq;
      }
      cand_cost[t] = cost;
      cand_tau[t] = tq;
    }
    __syncthreads();
    const int p = q0 + t;
    if (t < kPass && p < G) {
      float best = INFINITY;
      int pick = -1;
#pragma unroll
      for (int k = 0; k < 9; ++k)
        if (cand_cost[9 * t + k] < best) { best = cand_cost[9 * t + k]; pick = k; }
      if (pick < 0) any_invalid = true;
      // each group's own tile decides its buffering here; the launch's rule is
      // applied below
      const int bm = pick < 0 ? 0 : kBM[pick / 3], bn = pick < 0 ? 0 : kBN[pick % 3];
      tau[p] = pick < 0 ? 0.f : cand_tau[9 * t + pick];
      tiles[p] = pick < 0 ? 0 : launch_tiles(th, Ms[p], N, bm, bn, g);
      bm_s[p] = (int16_t)bm;
      bn_s[p] = (int16_t)bn;
      out_bm[combo * G + p] = (int16_t)bm;
      out_bn[combo * G + p] = (int16_t)bn;
    }
    __syncthreads();
  }
  any_invalid = __syncthreads_or(any_invalid);
  // the launch keeps one accumulator buffer if any group's tile needs it
  // (measured reading): every other group's tile then pays its drain too
  bool single = false;
  for (int q = threadIdx.x; q < G; q += blockDim.x)
    single = single || (bm_s[q] > 0 && single_buffer(bm_s[q], bn_s[q], BK, s, g, dt, 0));
  single = __syncthreads_or(single);
  if (single && th.reading == PM_READING_MEASURED)
    for (int q = threadIdx.x; q < G; q += blockDim.x)
      if (bm_s[q] > 0 && !single_buffer(bm_s[q], bn_s[q], BK, s, g, dt, 0))
        tau[q] += 4.0f * (float)bm_s[q] * (float)bn_s[q] * th.inv[17];
  __syncthreads();
  const int64_t n_conc = g == 1 ? n_sm : 2 * (n_sm / 2);
  grouped_list(bm_s, bn_s, tiles, G, n_conc, sc);
  for (int q = threadIdx.x; q < G; q += blockDim.x) sc.tau[sc.pos[q]] = tau[q];
  __syncthreads();
  const float t = grouped_makespan(sc, G, n_conc, nullptr);
  if (threadIdx.x == 0)
    out_t[combo] = (any_invalid || (g != 1 && n_sm < 2)) ? INFINITY : launch_time(th) + t;
}

// Stage-model makespan of one grouped launch with given per-group tiles (the
// schedule of pm_grouped_gemm_run; same terms as the grouped autotuner), in
// F; with grad != nullptr also its gradient in theta (out: T_hat, then NP
// slopes): the busiest worker's tiles through the tile adjoint.
template <class F>
__global__ void __launch_bounds__(kGroupThreads) grouped_predict_kernel(const int32_t* __restrict__ Mg,
                                                                        const int16_t* __restrict__ BMg,
                                                                        const int16_t* __restrict__ BNg, int G, int N,
                                                                        int K, int BK, int s, int g, int dt,
                                                                        ThetaT<F> th, int n_sm, bool grad,
                                                                        F* __restrict__ out) {
  __shared__ Schedule<F> sc;
  __shared__ int64_t tiles[kMaxGroups];
  __shared__ int32_t Ms[kMaxGroups];
  __shared__ int16_t bm_s[kMaxGroups], bn_s[kMaxGroups];
  __shared__ F red_d[kGroupThreads / 32][NP];
  for (int q = threadIdx.x; q < G; q += blockDim.x) {
    Ms[q] = Mg[q];
    bm_s[q] = BMg[q];
    bn_s[q] = BNg[q];
  }
  __syncthreads();
  const F W = grouped_working_set<F>(Ms, G, N, K, dt);
  const int64_t n_conc = g == 1 ? n_sm : 2 * (n_sm / 2);
  // one accumulator buffer for the whole launch if any group's tile needs it
  bool single = false;
  for (int q = threadIdx.x; q < G; q += blockDim.x) {
    single = single || single_buffer(bm_s[q], bn_s[q], BK, s, g, dt, 0);
    tiles[q] = launch_tiles(th, Ms[q], N, bm_s[q], bn_s[q], g);
  }
  const int sb = __syncthreads_or(single) ? 1 : 0;
  grouped_list(bm_s, bn_s, tiles, G, n_conc, sc);
  auto group_cfg = [&](int q) {
    pm_cfg c;
    c.M = Ms[q]; c.N = N; c.K = K; c.BM = bm_s[q]; c.BN = bn_s[q]; c.BK = (int16_t)BK;
    c.stages = (int8_t)s; c.cta_group = (int8_t)g; c.dtype = (int8_t)dt; c.kind = 0; c.tmem_a = 0;
    return c;
  };
  for (int q = threadIdx.x; q < G; q += blockDim.x) {
    GemmFwdT<F> f;
    gemm_forward(group_cfg(q), th, n_sm, f, W, sb);
    sc.tau[sc.pos[q]] = f.Kt * f.T_step + f.T_store;
  }
  __syncthreads();
  int w_star = 0;
  const F t = grouped_makespan(sc, G, n_conc, &w_star);
  const bool none = g != 1 && n_sm < 2;
  if (threadIdx.x == 0) out[0] = none ? (F)__int_as_float(0x7fc00000) : launch_time(th) + t;
  if (!grad) return;
  // d T_hat = d launch + sum_q n_{w*,q} d tau_q
  F d[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) d[j] = F(0);
  for (int q = threadIdx.x; q < G; q += blockDim.x) {
    const int i = sc.pos[q];
    const int64_t cnt = dealt_before(sc, i + 1, w_star, n_conc, G > 1) - dealt_before(sc, i, w_star, n_conc, G > 1);
    if (!cnt) continue;
    const pm_cfg c = group_cfg(q);
    GemmFwdT<F> f;
    gemm_forward(c, th, n_sm, f, W, sb);
    F gR = F(0), gS = F(0);
    step_store_adjoint(c, th, f, (F)cnt * f.Kt, (F)cnt, d, gR, gS);
    rate_adjoint(c, f, gR, gS, d);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    const F v = warp_sum<F>(d[j]);
    if (lane == 0) red_d[warp][j] = v;
  }
  __syncthreads();
  if (threadIdx.x < NP) {
    F v = F(0);
    for (int w = 0; w < kGroupThreads / 32; ++w) v += red_d[w][threadIdx.x];
    if (threadIdx.x == 0) v += F(1);                                           // T_launch
    if (threadIdx.x == 13 && th.reading == PM_READING_MEASURED) v += F(1);     // L_alloc + L_dealloc
    out[1 + threadIdx.x] = none ? (F)__int_as_float(0x7fc00000) : v;
  }
}

static std::atomic<int> g_reading{PM_READING_MEASURED};

static Theta to_theta(const pm_params* p, int n_sm) {
  Theta t;
  for (int j = 0; j < NP; ++j) {
    t.v[j] = p->v[j];
    t.inv[j] = (float)(1.0 / (double)p->v[j]);
  }
  t.reading = g_reading.load();
  set_concurrency(t, n_sm);
  return t;
}

}  // namespace pm

using namespace pm;

extern "C" pm_status pm_model_predict(const pm_cfg* cfgs_dev, int64_t n, const pm_params* theta_host, int32_t n_sm,
                                      float* t_out_dev, void* stream) {
  PM_REQUIRE(n >= 0, PM_EINVAL, "n < 0");
  if (n == 0) return PM_OK;
  PM_REQUIRE(cfgs_dev && theta_host && t_out_dev && n_sm > 0, PM_EINVAL, "null pointer or n_sm <= 0");
  PM_REQUIRE(((uintptr_t)cfgs_dev & 7) == 0, PM_EINVAL, "cfgs_dev must be 8-byte aligned");
  const int64_t want = (n + 255) / 256;
  const Theta th = to_theta(theta_host, n_sm);
  const bool space = space_params(th, n_sm);
  // with the short way one resident wave that walks the records up to eight rounds (10^6
  // records 8.8 us, 9.9 with 16 blocks per SM); past that, and without it at every
  // size, smaller shares even out the SMs' speeds (10^7: 78.5 us in one wave, 70.2)
  const int64_t resident = (int64_t)std::max(1, sm_count()) * 6;
  const int64_t cap = space && want <= 8 * resident ? resident : (int64_t)std::max(1, sm_count()) * 16;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, cap));
  auto kern = space ? model_predict_kernel<true> : model_predict_kernel<false>;
  kern<<<grid, 256, 0, static_cast<cudaStream_t>(stream)>>>(cfgs_dev, n, th, n_sm, t_out_dev);
  return launch_status("model_predict_kernel");
}

extern "C" pm_status pm_model_grad_workspace(int64_t n, size_t* bytes) {
  PM_REQUIRE(bytes != nullptr && n >= 0, PM_EINVAL, "bad arguments");
  *bytes = (size_t)grad_blocks(std::max<int64_t>(n, 1)) * NREC * sizeof(double);
  return PM_OK;
}

namespace pm {

template <class F>
static pm_status launch_grad(const pm_cfg* cfgs, int64_t n, const ThetaT<F>& th, int n_sm, const F* t_meas,
                             double* partials, int records, double* out, cudaStream_t s) {
  // FP64, few records: a cluster of eight one-warp blocks per record.  Both launches of
  // a call with / without clusters: 1,901 configurations 13.8 / 18.8 us, 20,000 16.2 /
  // 19.0, 25,856 17.5 / 19.1, 30,000 the same, 38,000 28.8 / 19.5 (the clusters no longer fit
  // at once).  The FP32 kernel is bound by one thread's latency and gains nothing.
  constexpr int CL = sizeof(F) == 8 ? 8 : 1;
  const bool space = space_params(th, n_sm);
  const SpaceHost<F> sh = space ? make_space(th) : SpaceHost<F>{};
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  cfg.attrs = attr;
  if (CL > 1 && records <= 2 * sm_count() / 3) {
    cfg.gridDim = dim3((unsigned)records * CL);
    cfg.blockDim = dim3(kGradThreads / CL);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, space ? model_grad_kernel<F, CL, true> : model_grad_kernel<F, CL, false>,
                                       cfgs, n, th, sh, n_sm, t_meas, partials);
    if (e != cudaSuccess) return cuda_fail(e, "cudaLaunchKernelEx(model_grad_kernel)");
  } else {
    auto kern = space ? model_grad_kernel<F, 1, true> : model_grad_kernel<F, 1, false>;
    kern<<<records, kGradThreads, 0, s>>>(cfgs, n, th, sh, n_sm, t_meas, partials);
    pm_status st = launch_status("model_grad_kernel");
    if (st != PM_OK) return st;
  }
  cfg.gridDim = dim3(NREC);
  cfg.blockDim = dim3(32);
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, model_grad_finish_kernel, (const double*)partials, records, n, out);
  if (e != cudaSuccess) return cuda_fail(e, "cudaLaunchKernelEx(model_grad_finish_kernel)");
  return PM_OK;
}

}  // namespace pm

extern "C" pm_status pm_model_grad(const pm_cfg* cfgs_dev, int64_t n, const pm_params* theta_host, int32_t n_sm,
                                   const float* t_meas_dev, void* workspace_dev, size_t workspace_bytes,
                                   double* out_dev, void* stream) {
  PM_REQUIRE(n > 0, PM_EINVAL, "n must be positive");
  PM_REQUIRE(cfgs_dev && theta_host && t_meas_dev && workspace_dev && out_dev && n_sm > 0, PM_EINVAL,
             "null pointer or n_sm <= 0");
  PM_REQUIRE(((uintptr_t)cfgs_dev & 7) == 0 && ((uintptr_t)workspace_dev & 7) == 0, PM_EINVAL,
             "cfgs_dev and workspace_dev must be 8-byte aligned");
  const int blocks = grad_blocks(n);
  PM_REQUIRE(workspace_bytes >= (size_t)blocks * NREC * sizeof(double), PM_ENOMEM,
             "workspace of %zu bytes is smaller than the %zu needed", workspace_bytes,
             (size_t)blocks * NREC * sizeof(double));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return launch_grad(cfgs_dev, n, to_theta(theta_host, n_sm), n_sm, t_meas_dev, static_cast<double*>(workspace_dev), blocks,
                     out_dev, s);
}

extern "C" pm_status pm_model_grad_f64(const pm_cfg* cfgs_dev, int64_t n, const double* theta_host, int32_t n_sm,
                                       const double* t_meas_dev, void* workspace_dev, size_t workspace_bytes,
                                       double* out_dev, void* stream) {
  PM_REQUIRE(n > 0, PM_EINVAL, "n must be positive");
  PM_REQUIRE(cfgs_dev && theta_host && t_meas_dev && workspace_dev && out_dev && n_sm > 0, PM_EINVAL,
             "null pointer or n_sm <= 0");
  PM_REQUIRE(((uintptr_t)cfgs_dev & 7) == 0 && ((uintptr_t)workspace_dev & 7) == 0 && ((uintptr_t)t_meas_dev & 7) == 0,
             PM_EINVAL, "cfgs_dev, t_meas_dev and workspace_dev must be 8-byte aligned");
  const int blocks = grad_blocks(n);
  PM_REQUIRE(workspace_bytes >= (size_t)blocks * NREC * sizeof(double), PM_ENOMEM,
             "workspace of %zu bytes is smaller than the %zu needed", workspace_bytes,
             (size_t)blocks * NREC * sizeof(double));
  ThetaT<double> th;
  for (int j = 0; j < NP; ++j) {
    th.v[j] = theta_host[j];
    th.inv[j] = 1.0 / theta_host[j];
  }
  th.reading = g_reading.load();
  set_concurrency(th, n_sm);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return launch_grad(cfgs_dev, n, th, n_sm, t_meas_dev, static_cast<double*>(workspace_dev), blocks, out_dev, s);
}

extern "C" pm_status pm_model_set_reading(int32_t reading) {
  PM_REQUIRE(reading == PM_READING_LITERAL || reading == PM_READING_MEASURED, PM_EINVAL,
             "reading %d is not a pm_reading", reading);
  g_reading.store(reading);
  return PM_OK;
}

extern "C" int32_t pm_model_reading(void) { return g_reading.load(); }

namespace pm {

static pm_status launch_autotune(const int32_t* MNK, int64_t n, int32_t dtype, const pm_params* theta_host, int32_t n_sm,
                                 int k, pm_cfg* picks, float* t_pred, cudaStream_t s) {
  const Theta th = to_theta(theta_host, n_sm);
  const int64_t sms = std::max(1, sm_count());
  // measured on 152 SMs, table against block per shape: 900 shapes 4.4 / 4.1 us
  // (best eight 7.0 / 6.4), 1,200 shapes 4.5 / 4.9 us (7.0 / 7.6)
  if (n <= 6 * sms) {
    autotune_shape_kernel<<<(int)n, kTunePerLane * 32, 0, s>>>(MNK, n, dtype, th, n_sm, k, picks, t_pred);
  } else {
    constexpr int64_t kWarps = kTuneThreads / 32;
    const int grid = (int)std::min<int64_t>((n + kWarps - 1) / kWarps, sms * 2);
    autotune_table_kernel<<<grid, kTuneThreads, 0, s>>>(MNK, n, dtype, th, n_sm, k, picks, t_pred);
  }
  return launch_status("autotune_kernel");
}

}  // namespace pm

extern "C" pm_status pm_autotune_pick(const int32_t* MNK_dev, int64_t n, int32_t dtype, const pm_params* theta_host,
                                      int32_t n_sm, pm_cfg* picks_dev, float* t_pred_dev, void* stream) {
  PM_REQUIRE(n >= 0, PM_EINVAL, "n < 0");
  if (n == 0) return PM_OK;
  PM_REQUIRE(MNK_dev && theta_host && picks_dev && t_pred_dev && n_sm > 0, PM_EINVAL, "null pointer or n_sm <= 0");
  PM_REQUIRE(dtype >= 0 && dtype <= 2, PM_EINVAL, "dtype %d is not a pm_dtype", dtype);
  return launch_autotune(MNK_dev, n, dtype, theta_host, n_sm, 1, picks_dev, t_pred_dev, static_cast<cudaStream_t>(stream));
}

extern "C" pm_status pm_autotune_topk(const int32_t* MNK_dev, int64_t n, int32_t dtype, const pm_params* theta_host,
                                      int32_t n_sm, int32_t k, pm_cfg* picks_dev, float* t_pred_dev, void* stream) {
  PM_REQUIRE(n >= 0, PM_EINVAL, "n < 0");
  if (n == 0) return PM_OK;
  PM_REQUIRE(MNK_dev && theta_host && picks_dev && t_pred_dev && n_sm > 0, PM_EINVAL, "null pointer or n_sm <= 0");
  PM_REQUIRE(dtype >= 0 && dtype <= 2, PM_EINVAL, "dtype %d is not a pm_dtype", dtype);
  PM_REQUIRE(k >= 1 && k <= kMaxTopK, PM_EINVAL, "k must be in [1, %d]", kMaxTopK);
  return launch_autotune(MNK_dev, n, dtype, theta_host, n_sm, k, picks_dev, t_pred_dev, static_cast<cudaStream_t>(stream));
}

namespace pm {

// Page-locked host memory of the grouped model calls, one block per calling
// thread: the kernels read the row counts and tiles from it and write their
// results to it, so a call is one launch and one wait.  Device scratch from the
// stream's pool and four copies cost about 270 us a call (the pool gives its
// memory back at every wait and maps it again).  A call holds its thread's block
// until it has waited for its kernel and copied the results.  The blocks of all
// threads are in one list, so that pm_shutdown gives every one of them back: a
// device reset frees them, whichever thread prepares it.  A thread's block is
// also given back when the thread ends.
constexpr size_t kGroupScratch = 4 * kMaxGroups + 2 * 2 * 20 * kMaxGroups + 512;

struct GroupScratch;
static std::mutex g_group_list_mu;
static GroupScratch* g_group_list = nullptr;

struct GroupScratch {
  std::mutex mu;                         // held by the thread's call, and to release the block
  char* p = nullptr;
  GroupScratch *prev = nullptr, *next = nullptr;
  GroupScratch() {
    std::lock_guard<std::mutex> lk(g_group_list_mu);
    next = g_group_list;
    if (next) next->prev = this;
    g_group_list = this;
  }
  ~GroupScratch() {
    {
      std::lock_guard<std::mutex> lk(g_group_list_mu);
      if (next) next->prev = prev;
      (prev ? prev->next : g_group_list) = next;
    }
    release();
  }
  void release() {
    std::lock_guard<std::mutex> lk(mu);
    if (p) cudaFreeHost(p);
    p = nullptr;
  }
};
static thread_local GroupScratch g_group_scratch;

void release_group_scratch() {
  std::lock_guard<std::mutex> lk(g_group_list_mu);
  for (GroupScratch* g = g_group_list; g; g = g->next) g->release();
}

// The calling thread's block, held by `hold` until it goes out of scope.
static pm_status group_scratch(char** out, std::unique_lock<std::mutex>& hold) {
  GroupScratch& g = g_group_scratch;
  hold = std::unique_lock<std::mutex>(g.mu);
  if (!g.p) {
    void* p = nullptr;
    PM_CUDA(cudaHostAlloc(&p, kGroupScratch, cudaHostAllocPortable | cudaHostAllocMapped));
    g.p = static_cast<char*>(p);
  }
  *out = g.p;
  return PM_OK;
}

// All 20 launch-level candidates (BK, stages, cta_group) of the grouped
// autotuner: predicted makespan ht[i] and per-group tiles hbm/hbn[i * G + q].
static pm_status grouped_candidates(int32_t G, const int32_t* M_host, int32_t N, int32_t K, int32_t dtype,
                                    const pm_params* theta_host, int32_t n_sm, cudaStream_t s, float* ht,
                                    std::vector<int16_t>& hbm, std::vector<int16_t>& hbn) {
  PM_REQUIRE(G > 0 && G <= kMaxGroups, PM_EINVAL, "G must be in [1, %d]", kMaxGroups);
  PM_REQUIRE(M_host && theta_host && n_sm > 0, PM_EINVAL, "null pointer or n_sm <= 0");
  PM_REQUIRE(N > 0 && K > 0 && dtype >= 0 && dtype <= 2, PM_EINVAL, "bad N, K or dtype");
  for (int q = 0; q < G; ++q) PM_REQUIRE(M_host[q] > 0, PM_EINVAL, "M[%d] <= 0", q);
  char* buf = nullptr;
  std::unique_lock<std::mutex> hold;
  pm_status st = group_scratch(&buf, hold);
  if (st != PM_OK) return st;
  float* pt = reinterpret_cast<float*>(buf);                    // 20 floats
  int32_t* pM = reinterpret_cast<int32_t*>(buf + 128);          // G
  int16_t* pbm = reinterpret_cast<int16_t*>(pM + G);            // 20 x G each
  int16_t* pbn = pbm + 20 * (size_t)G;
  std::copy(M_host, M_host + G, pM);
  grouped_tune_kernel<<<20, kGroupTuneThreads, 0, s>>>(pM, G, N, K, dtype, to_theta(theta_host, n_sm), n_sm, pt, pbm,
                                                       pbn);
  st = launch_status("grouped_tune_kernel");
  if (st != PM_OK) return st;
  PM_CUDA(cudaStreamSynchronize(s));
  std::copy(pt, pt + 20, ht);
  hbm.assign(pbm, pbm + 20 * (size_t)G);
  hbn.assign(pbn, pbn + 20 * (size_t)G);
  return PM_OK;
}

// Launch-level parameters of candidate i: {BK, stages, cta_group}.
static void grouped_launch_of(int i, int dtype, int32_t* launch) {
  launch[0] = (int32_t)(dtype == PM_FP32 ? (i / 10 ? 64 : 32) : (i / 10 ? 128 : 64));
  launch[1] = 2 + (i / 2) % 5;
  launch[2] = 1 + i % 2;
}

}  // namespace pm

namespace pm {

// One grouped launch's makespan on the GPU (one block), in F; with grad also
// its gradient.  out_host: 1 value, or 1 + NP with grad.
template <class F>
static pm_status grouped_eval(int32_t G, const int32_t* M_host, int32_t N, int32_t K, const int16_t* BM_host,
                              const int16_t* BN_host, int32_t BK, int32_t stages, int32_t cta_group, int32_t dtype,
                              const ThetaT<F>& th, int32_t n_sm, bool grad, F* out_host, cudaStream_t s) {
  PM_REQUIRE(G > 0 && G <= kMaxGroups, PM_EINVAL, "G must be in [1, %d]", kMaxGroups);
  PM_REQUIRE(M_host && BM_host && BN_host && out_host && n_sm > 0, PM_EINVAL, "null pointer or n_sm <= 0");
  PM_REQUIRE(N > 0 && K > 0 && dtype >= 0 && dtype <= 2, PM_EINVAL, "bad N, K or dtype");
  for (int q = 0; q < G; ++q) {
    PM_REQUIRE(M_host[q] > 0, PM_EINVAL, "M[%d] <= 0", q);
    PM_REQUIRE(tile_valid(BM_host[q], BN_host[q], BK, stages, cta_group, dtype), PM_EUNSUPPORTED,
               "group %d: tile %dx%dx%d stages=%d cta_group=%d outside the valid space", q, BM_host[q], BN_host[q],
               BK, stages, cta_group);
  }
  const int n_out = grad ? 1 + NP : 1;
  char* buf = nullptr;
  std::unique_lock<std::mutex> hold;
  pm_status st = group_scratch(&buf, hold);
  if (st != PM_OK) return st;
  F* pt = reinterpret_cast<F*>(buf);                            // 1 + NP values
  int32_t* pM = reinterpret_cast<int32_t*>(buf + 256);          // G each
  int16_t* pbm = reinterpret_cast<int16_t*>(pM + G);
  int16_t* pbn = pbm + G;
  std::copy(M_host, M_host + G, pM);
  std::copy(BM_host, BM_host + G, pbm);
  std::copy(BN_host, BN_host + G, pbn);
  grouped_predict_kernel<F><<<1, kGroupThreads, 0, s>>>(pM, pbm, pbn, G, N, K, BK, stages, cta_group, dtype, th, n_sm,
                                                         grad, pt);
  st = launch_status("grouped_predict_kernel");
  if (st != PM_OK) return st;
  PM_CUDA(cudaStreamSynchronize(s));
  std::copy(pt, pt + n_out, out_host);
  return PM_OK;
}

}  // namespace pm

extern "C" pm_status pm_grouped_predict(int32_t G, const int32_t* M_host, int32_t N, int32_t K,
                                        const int16_t* BM_host, const int16_t* BN_host, int32_t BK, int32_t stages,
                                        int32_t cta_group, int32_t dtype, const pm_params* theta_host, int32_t n_sm,
                                        float* t_pred_host, void* stream) {
  PM_REQUIRE(theta_host && t_pred_host && n_sm > 0, PM_EINVAL, "null pointer or n_sm <= 0");
  return grouped_eval<float>(G, M_host, N, K, BM_host, BN_host, BK, stages, cta_group, dtype,
                             to_theta(theta_host, n_sm), n_sm, false, t_pred_host, static_cast<cudaStream_t>(stream));
}

extern "C" pm_status pm_grouped_grad(int32_t G, const int32_t* M_host, int32_t N, int32_t K, const int16_t* BM_host,
                                     const int16_t* BN_host, int32_t BK, int32_t stages, int32_t cta_group,
                                     int32_t dtype, const double* theta_host, int32_t n_sm, double* out_host,
                                     void* stream) {
  PM_REQUIRE(theta_host && out_host && n_sm > 0, PM_EINVAL, "null pointer or n_sm <= 0");
  ThetaT<double> th;
  for (int j = 0; j < NP; ++j) {
    th.v[j] = theta_host[j];
    th.inv[j] = 1.0 / theta_host[j];
  }
  th.reading = g_reading.load();
  set_concurrency(th, n_sm);
  return grouped_eval<double>(G, M_host, N, K, BM_host, BN_host, BK, stages, cta_group, dtype, th, n_sm, true,
                              out_host, static_cast<cudaStream_t>(stream));
}

extern "C" pm_status pm_grouped_candidates(int32_t G, const int32_t* M_host, int32_t N, int32_t K, int32_t dtype,
                                           const pm_params* theta_host, int32_t n_sm, float* t_pred_host,
                                           int16_t* BM_host, int16_t* BN_host, int32_t* launch_host, void* stream) {
  PM_REQUIRE(t_pred_host && BM_host && BN_host && launch_host, PM_EINVAL, "null output pointer");
  std::vector<int16_t> hbm, hbn;
  pm_status st = grouped_candidates(G, M_host, N, K, dtype, theta_host, n_sm, static_cast<cudaStream_t>(stream),
                                    t_pred_host, hbm, hbn);
  if (st != PM_OK) return st;
  std::copy(hbm.begin(), hbm.end(), BM_host);
  std::copy(hbn.begin(), hbn.end(), BN_host);
  for (int i = 0; i < 20; ++i) grouped_launch_of(i, dtype, launch_host + 3 * i);
  return PM_OK;
}

extern "C" pm_status pm_grouped_autotune(int32_t G, const int32_t* M_host, int32_t N, int32_t K, int32_t dtype,
                                         const pm_params* theta_host, int32_t n_sm, int16_t* BM_out_host,
                                         int16_t* BN_out_host, int32_t* launch_out_host, float* t_pred_host,
                                         void* stream) {
  PM_REQUIRE(BM_out_host && BN_out_host && launch_out_host && t_pred_host, PM_EINVAL, "null output pointer");
  float ht[20];
  std::vector<int16_t> hbm, hbn;
  pm_status st = grouped_candidates(G, M_host, N, K, dtype, theta_host, n_sm, static_cast<cudaStream_t>(stream), ht,
                                    hbm, hbn);
  if (st != PM_OK) return st;
  int best = 0;                                   // first minimum, as the GPU's pick kernel scans
  for (int i = 1; i < 20; ++i)
    if (ht[i] < ht[best]) best = i;
  PM_REQUIRE(ht[best] < INFINITY, PM_EUNSUPPORTED, "no valid grouped configuration");
  for (int q = 0; q < G; ++q) {
    BM_out_host[q] = hbm[(size_t)best * G + q];
    BN_out_host[q] = hbn[(size_t)best * G + q];
  }
  grouped_launch_of(best, dtype, launch_out_host);
  *t_pred_host = ht[best];
  return PM_OK;
}

extern "C" pm_status pm_grouped_gemm_autotune(int32_t G, const int32_t* M_host, int32_t N, int32_t K,
                                              const pm_params* theta_host, int32_t n_sm, int32_t k,
                                              const void* A_op_dev, const void* B_op_dev, float* C_dev, int warmup,
                                              int reps, void* stream, int16_t* BM_out_host, int16_t* BN_out_host,
                                              int32_t* launch_out_host, float* t_pred_host,
                                              pm_probe_result* pick_time_out) {
  PM_REQUIRE(BM_out_host && BN_out_host && launch_out_host, PM_EINVAL, "null output pointer");
  PM_REQUIRE(k >= 1 && k <= 20, PM_EINVAL, "k must be in [1, 20]");
  PM_REQUIRE(warmup >= 0 && reps >= 1 && reps <= 100000, PM_EINVAL, "warmup >= 0 and 1 <= reps <= 1e5 required");
  PM_REQUIRE(A_op_dev && B_op_dev && C_dev, PM_EINVAL, "null operand or output pointer");
  NvtxRange nvtx("pm_grouped_gemm_autotune");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  float ht[20];
  std::vector<int16_t> hbm, hbn;
  pm_status st = grouped_candidates(G, M_host, N, K, PM_BF16, theta_host, n_sm, s, ht, hbm, hbn);
  if (st != PM_OK) return st;
  // the model's k best launches (stable order), each timed; the fastest wins
  int order[20];
  for (int i = 0; i < 20; ++i) order[i] = i;
  std::stable_sort(order, order + 20, [&](int a, int b) { return ht[a] < ht[b]; });
  cudaEvent_t e0, e1;
  PM_CUDA(cudaEventCreate(&e0));
  PM_CUDA(cudaEventCreate(&e1));
  double best_t = 1e300;
  int best = -1;
  pm_probe_result best_r = {};
  pm_clock c0, c1;
  read_clock(&c0);
  for (int j = 0; j < k && st == PM_OK; ++j) {
    const int i = order[j];
    if (!(ht[i] < INFINITY)) break;
    int32_t L[3];
    grouped_launch_of(i, PM_BF16, L);
    const int16_t* bm = hbm.data() + (size_t)i * G;
    const int16_t* bn = hbn.data() + (size_t)i * G;
    for (int w = 0; w < warmup && st == PM_OK; ++w)
      st = pm_grouped_gemm_run(G, M_host, N, K, bm, bn, L[0], L[1], L[2], A_op_dev, B_op_dev, C_dev, stream);
    std::vector<double> t;
    for (int r = 0; r < reps && st == PM_OK; ++r) {
      cudaEventRecord(e0, s);
      st = pm_grouped_gemm_run(G, M_host, N, K, bm, bn, L[0], L[1], L[2], A_op_dev, B_op_dev, C_dev, stream);
      cudaEventRecord(e1, s);
      cudaError_t ce = cudaEventSynchronize(e1);
      if (ce != cudaSuccess) { st = cuda_fail(ce, "cudaEventSynchronize"); break; }
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      t.push_back(ms * 1e-3);
    }
    if (st != PM_OK) break;
    std::sort(t.begin(), t.end());
    const double med = t.size() % 2 ? t[t.size() / 2] : 0.5 * (t[t.size() / 2 - 1] + t[t.size() / 2]);
    if (med < best_t) {
      best_t = med;
      best = i;
      best_r.median_s = med;
      best_r.p25_s = t[t.size() / 4];
      best_r.p75_s = t[(3 * t.size()) / 4];
      best_r.min_s = t.front();
      best_r.bytes = 0.0;
      best_r.final_index = 0;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  read_clock(&c1);
  clock_record(&best_r, c0, c1);
  if (st != PM_OK) return st;
  PM_REQUIRE(best >= 0, PM_EUNSUPPORTED, "no valid grouped configuration");
  for (int q = 0; q < G; ++q) {
    BM_out_host[q] = hbm[(size_t)best * G + q];
    BN_out_host[q] = hbn[(size_t)best * G + q];
  }
  grouped_launch_of(best, PM_BF16, launch_out_host);
  if (t_pred_host) *t_pred_host = ht[best];
  if (pick_time_out) *pick_time_out = best_r;
  return PM_OK;
}

// ----------------------------------------------------------------------------
// Allocation-free variant of pm_model_grad.
//
// Some callers cannot allocate device memory at the point where they need the
// calibration gradient: a host program that links only this library and owns
// no CUDA allocator, a runtime working inside a fixed device-memory budget, or
// code that must not trigger allocator traffic in its hot loop.  For them the
// per-block partial sums live in a fixed array compiled into this library,
// resident on every GPU that loads it for the life of the process.
//
// Capacity: the call launches the same grid as pm_model_grad (grad_blocks(n):
// at most four blocks per SM, one partial record of NREC doubles each), so its
// partial sums are added in the same order and its output is bit-identical to
// pm_model_grad's.  The array holds kGradStaticRecords records (622,592
// bytes), enough for GPUs of up to 1024 SMs; batches are limited to
// kGradStaticRecords * kGradThreads = 1,048,576 configurations per call.
// Every record a call reads is first written by that call, so nothing has to
// be cleared between calls; two calls whose kernels overlap on a GPU share the
// array and race.
namespace pm {

constexpr int kGradStaticRecords = 4096;
static __device__ __align__(256) double g_grad_scratch[kGradStaticRecords * NREC];

static double* g_grad_scratch_ptr[64];
static std::mutex g_grad_scratch_mu;

// Device address of g_grad_scratch for the current device.  In host code the
// array's name is only a host-side stand-in, so the address is looked up once
// per device with that device current.
// Forgets the cached addresses (pm_shutdown; a device reset reloads the module).
void clear_grad_scratch_cache() {
  std::lock_guard<std::mutex> lk(g_grad_scratch_mu);
  for (auto& p : g_grad_scratch_ptr) p = nullptr;
}

static pm_status grad_scratch_address(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  PM_REQUIRE(dev >= 0 && dev < 64, PM_EINVAL, "device index %d out of range", dev);
  std::lock_guard<std::mutex> lk(g_grad_scratch_mu);
  if (g_grad_scratch_ptr[dev] == nullptr) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_grad_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_grad_scratch)");
    g_grad_scratch_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_grad_scratch_ptr[dev];
  return PM_OK;
}

}  // namespace pm

extern "C" pm_status pm_model_grad_noalloc(const pm_cfg* cfgs_dev, int64_t n, const pm_params* theta_host,
                                           int32_t n_sm, const float* t_meas_dev, double* out_dev, void* stream) {
  PM_REQUIRE(n > 0, PM_EINVAL, "n must be positive");
  PM_REQUIRE(n <= (int64_t)kGradStaticRecords * kGradThreads, PM_ENOMEM,
             "pm_model_grad_noalloc takes at most %lld configurations per call (got %lld); split the batch or "
             "use pm_model_grad with a workspace",
             (long long)kGradStaticRecords * kGradThreads, (long long)n);
  PM_REQUIRE(cfgs_dev && theta_host && t_meas_dev && out_dev && n_sm > 0, PM_EINVAL, "null pointer or n_sm <= 0");
  PM_REQUIRE(((uintptr_t)cfgs_dev & 7) == 0, PM_EINVAL, "cfgs_dev must be 8-byte aligned");
  double* scratch = nullptr;
  pm_status st = grad_scratch_address(&scratch);
  if (st != PM_OK) return st;
  const int blocks = grad_blocks(n);
  PM_REQUIRE(blocks <= kGradStaticRecords, PM_ENOMEM, "%d partial records exceed the %d the array holds", blocks,
             kGradStaticRecords);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return launch_grad(cfgs_dev, n, to_theta(theta_host, n_sm), n_sm, t_meas_dev, scratch, blocks, out_dev, s);
}
