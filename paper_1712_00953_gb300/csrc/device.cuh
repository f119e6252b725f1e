// GB300 (sm_103a) device code of the ROK4E reaction step and the Simpler split
// step: the per-cell kernels as templates, their device functions, and the host
// helpers that size and launch them.  Each heavy kernel instantiation is compiled
// in its own translation unit (k_*.cu, through launchers.cuh) so the build runs
// in parallel; rok4e_kernels.cu holds the small kernels and the C ABI.
//
// Mapping.  A "group" of G consecutive lanes of a warp (G = 32 by default:
// one warp per cell) integrates one cell at a time.  Vector loops over the
// N = Ns + 1 state entries, the Ns species and the Nr reactions are strided by
// G; dot products and norms are butterfly (xor) shuffle reductions, which give
// bit-identical results on every lane so that all lanes of a group take the
// same control-flow decisions.  All per-cell vectors (state, f_n, the Krylov
// basis, the four stage vectors, species and reaction work arrays) live in
// shared memory next to a per-block copy of the mechanism.
//
// Batching.  The integration kernel is persistent: one wave of blocks sized
// to the device.  With carried step sizes the cells are sorted by expected
// cost and dealt to static per-block bins (the most expensive alone on an
// SM), each drained from a shared-memory counter; otherwise each group takes
// the next cell index from a global atomic counter (work stealing).  Either
// way cells needing 1 or 200 substeps share one launch without a tail of
// idle blocks.
//
// Arithmetic.  FP64 accuracy throughout, on two kinds of pipe: a warp's FP64
// instruction holds its sub-partition's FP64 unit for 64 cycles, an integer one
// its pipe for 2 to 4, so what 64-bit integers carry to the last FP64 bit is
// (fx.cuh), and FP64 instructions are kept for the rest.  Restatements that differ
// from a literal transcription of the kinetics while computing the same quantities:
//  * with E_k = exp(g_k/RT) (RT/p_ref) and z_k = C_k E_k, 1/Kc is a product of E
//    over the products divided by one over the reactants and q_j = m_j kappa_j
//    (z_ra z_rb - z_pa z_pb), ln kappa = ln k - ln E_ra - ln E_rb: one exponential
//    per reaction and one per species.  Cells outside its range (reactions_direct)
//    take 1/Kc from an exponential of its own;
//  * w = nu^T q is a gather over a species-major list, for all but the smallest
//    mechanisms in 128-bit fixed point wherever every row keeps FP64's bits there.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <mutex>
#include <string>

#include "exp2_table.h"
#include "fx.cuh"
#include "internal.h"
#include "rok4e.h"

namespace rk {

// ---------------------------------------------------------------- constants
constexpr double R_GAS = 8.314462618;
constexpr double P_REF = 101325.0;
constexpr double PREF_OVER_R = P_REF / R_GAS, INV_R = 1.0 / R_GAS;
constexpr double LN_R_OVER_PREF = -9.408091968961747;  // ln(R / P_ref)
constexpr double GAM = 0.572816062482135;
// Table coeff_rok4e (Sec. 4.2); b3 = 0, bhat4 = 0.
constexpr double G21 = -0.602765307997356;
constexpr double G31 = -1.389195789724843, G32 = 1.072950969011413;
constexpr double G41 = 0.992356412977094, G42 = -1.390032613873701, G43 = -0.440875890223325;
constexpr double A21 = 0.432364435748567;
constexpr double A31 = -0.514211316876170, A32 = 1.382271144617360;
constexpr double B1 = 0.194335256262729, B2 = 0.483167813989227, B3 = 0.0, B4 = 0.322496929748044;
constexpr double BH1 = -0.217819895945721, BH2 = 1.03130847478467, BH3 = 0.186511421161047, BH4 = 0.0;
// PI controller (Sec. 4.3), p = 4
constexpr double PI_ALPHA = 0.7 / 4.0, PI_BETA = 0.4 / 4.0;
constexpr double FAC_MIN = 0.2, FAC_MAX = 5.0, SAFETY = 0.8, ERR_FLOOR = 1e-10;
constexpr double BREAKDOWN_TOL = 1e-12, T_END_TOL = 1e-12, H_MIN_FRAC = 1e-12;
constexpr float LOG2_ERR_FLOOR = -33.219281f;  // log2(1e-10)
constexpr int G_OVERFLOW_HI = 0x40654000;  // high word of 170.0
constexpr int MAXM = RK_MAX_KRYLOV;
// Threads per block of the per-cell kernels: 8 warps, so each thread may hold
// up to 255 registers (one such block fills an SM's register file, which the
// cells' shared-memory slots limit the SM to anyway).
constexpr int MAX_BLOCK_THREADS = 256;
// Cells for each SM from which the integrator's wider blocks are taken: with eight
// or fewer they change nothing (1216 cells on 152 SMs: 24.2 ms on eight warps, 24.9
// on sixteen), with sixteen they gain (2500 cells: 34.8 and 28.1 ms).
constexpr int WIDE_MIN_CELLS_PER_SM = 8;
// the explicit integrator fits 128 registers with one warp per cell
constexpr int POINT_BLOCK_THREADS = 512;
constexpr int rkdp_threads(int G) { return G == 32 ? 512 : MAX_BLOCK_THREADS; }
constexpr int EXP_TAB_BYTES = RK_FX_EXP2_N * 8;  // leads the dynamic shared memory

static __constant__ uint64_t c_exp2_table[RK_FX_EXP2_N] = {RK_FX_EXP2_VALUES};
static __constant__ uint64_t c_fx_inv_c[128] = {RK_FX_INV_C_VALUES};
static __constant__ uint64_t c_fx_log2_c[128] = {RK_FX_LOG2_C_VALUES};
static __constant__ double c_log_inv_c[RK_LOG_TABLE_N] = {RK_LOG_INV_C_VALUES};
static __constant__ double c_log_ln_c[RK_LOG_TABLE_N] = {RK_LOG_LN_C_VALUES};

// ------------------------------------------------- table-driven exponential
// exp(x) by Tang's table-driven method (ACM TOMS 15(2), 1989) on the integer
// pipes (fx::exp_double, 1.2 ulp): no FP64 instruction, where the same method
// in FP64 was nine (576 cycles of the sub-partition's FP64 unit; the ~12
// multiplies and ~30 adds and shifts here take ~100 of the integer pipes).
// |x| >= 708, infinities and NaN take the library exp().
__device__ __forceinline__ double exp_fast(double x, const uint64_t* __restrict__ tab) {
  if ((__double2hiint(x) & 0x7fffffff) >= 0x40862000) return exp(x);
  return fx::exp_double(x, tab);
}

// a < b for doubles with b > 0 by their bits (an FP64 comparison takes the FP64
// unit as long as a multiplication): false for NaN a of either sign, as a < b is.
__device__ __forceinline__ bool below(double a, double b) {
  return __double_as_longlong(a) < __double_as_longlong(b) && (__double2hiint(a) & 0x7ff00000) != 0x7ff00000;
}

// 1/x by Newton's iteration for the reciprocal, r <- r + r (1 - x r), from
// an FP32 estimate: two steps square the estimate's relative error twice
// ((2e-7)^4), leaving the last rounding.  Four FP64 operations instead of a
// full-precision division; only for x whose reciprocal and itself are FP32-normal
// (|x| in [2^-125, 2^125): anything else, 0 and NaN too, wraps to a finite wrong
// value).  The conversions to FP32 (truncated) and back are integer moves: a
// conversion instruction takes the FP64 unit as long as an FP64 operation.
__device__ __forceinline__ double rcp_newton(double x) {
  const int hi = __double2hiint(x), sign = hi & (int)0x80000000;
  const float f = __int_as_float((((hi & 0x7fffffff) - (896 << 20)) << 3) | (int)((unsigned)__double2loint(x) >> 29));
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  const int b = __float_as_int(y);
  double r = __hiloint2double(((b >> 3) + (896 << 20)) | sign, b << 29);
  double e = fma(-x, r, 1.0);
  r = fma(r, e, r);
  e = fma(-x, r, 1.0);
  return fma(r, e, r);
}

// 1/x: rcp_newton where x and its reciprocal are FP32-normal (|x| in
// [2^-125, 2^125)), a full division elsewhere (zero, subnormal, huge,
// infinite, NaN).  Within ~1 ulp of the division.
__device__ __forceinline__ double rcp_any(double x) {
  const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
  return ex - 898u < 250u ? rcp_newton(x) : 1.0 / x;
}

// 1/x for the temperature and the mixture sums of a cell.  What is no state any more
// stays visible: 0 (a cell whose mass fractions are all zero, T = 0), NaN, infinities
// and |x| below 2^-128 give NaN, |x| from 2^128 zero, through rounding conversions;
// one integer test on the main path.
static __device__ __noinline__ double rcp_beyond(double x) {
  double r = (double)__frcp_rn(__double2float_rn(x));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}
__device__ __forceinline__ double rcp_state(double x) {
  const unsigned ex = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
  return ex - 898u < 250u ? rcp_newton(x) : rcp_beyond(x);
}

// 1/sqrt(x) for positive, finite, normal x: FP32 estimate of the significand with
// an even exponent (x = 4^k w, w in [1, 4)), one cubically convergent step
// y += y e (1/2 + 3/8 e), e = 1 - w y^2 (|e| < 5e-7, so the rest is below 1e-19).
__device__ __forceinline__ double rsqrt_newton(double x) {
  const int hi = __double2hiint(x);
  const int k = ((hi >> 20) - 1023) >> 1;
  const double w = __hiloint2double(hi - (k << 21), __double2loint(x));
  const int wh = __double2hiint(w);
  float y0;
  asm("rsqrt.approx.ftz.f32 %0, %1;"
      : "=f"(y0)
      : "f"(__int_as_float(((wh - (896 << 20)) << 3) | (int)((unsigned)__double2loint(w) >> 29))));
  const int b = __float_as_int(y0);
  const double y = __hiloint2double((b >> 3) + (896 << 20), b << 29);
  const double e = fma(-(w * y), y, 1.0);
  const double r = fma(y * e, fma(0.375, e, 0.5), y);
  return __hiloint2double(__double2hiint(r) - (k << 20), __double2loint(r));
}
__device__ __forceinline__ double rsqrt_any(double x) {
  const unsigned ex = (unsigned)__double2hiint(x) >> 20;  // sign and exponent
  return ex - 1u < 2046u ? rsqrt_newton(x) : rsqrt(x);
}

// ------------------------------------------------- table-driven logarithm
// ln x by Tang's table-driven method (ACM TOMS 16(4), 1990): x = 2^e m with
// m in [1, 2); the significand's top 7 bits pick the interval
// [1 + j/128, 1 + (j+1)/128) and its tabulated centre reciprocal inv_c_j
// (rounded) with ln_c_j = -ln(inv_c_j), so ln x = e ln2 + ln_c_j + ln(1 + r),
// r = m inv_c_j - 1 by one fma (|r| <= 2^-8), ln(1 + r) by its Taylor
// polynomial through r^7 (truncation below 1e-20).  11 FP64 operations;
// absolute error ~1.5e-16 max(1, |ln x|) (a few ulp only where ln x is near
// 0, which the intervals below 1 reach through cancellation against e ln2).
// Zero, negative, subnormal, infinite and NaN arguments take the library log().
__device__ __forceinline__ double log_fast(double x) {
  const int hi = __double2hiint(x);
  if ((unsigned)(hi - 0x00100000) >= 0x7fe00000u) return log(x);
  const int j = (hi >> 13) & (RK_LOG_TABLE_N - 1);
  const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));
  // e as a double: 2^52 + biased exponent, less 2^52 + 1023 (exact)
  const double e = __hiloint2double(0x43300000, hi >> 20) - 4503599627371519.0;
  const double r = fma(m, c_log_inv_c[j], -1.0);
  double q = fma(r, 1.0 / 7.0, -1.0 / 6.0);
  q = fma(q, r, 0.2);
  q = fma(q, r, -0.25);
  q = fma(q, r, 1.0 / 3.0);
  q = fma(q, r, -0.5);
  const double p = fma(__dmul_rn(r, r), q, r);
  return fma(e, RK_LN2_HI, c_log_ln_c[j]) + fma(e, RK_LN2_LO, p);
}

// ---- double-float ("df") arithmetic: a value h + l held as two FP32 numbers
// with |l| <= ulp(h)/2, ~44-bit significand, on the FP32 pipe.  Products by
// the error-free FMA split (Dekker's two-product), sums by Knuth's two-sum,
// each renormalised.  FP32 exponent range: callers keep magnitudes inside it.
struct df2 {
  float h, l;
};
__device__ __forceinline__ df2 df_from(double x) {
  const float h = __double2float_rn(x);
  return {h, __double2float_rn(x - (double)h)};
}
__device__ __forceinline__ double df_to(df2 a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ df2 df_norm(float s, float e) {
  const float h = s + e;
  return {h, e - (h - s)};
}
__device__ __forceinline__ df2 df_mul(df2 a, df2 b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  return df_norm(p, e);
}
__device__ __forceinline__ df2 df_add(df2 a, df2 b) {
  const float s = a.h + b.h;
  const float bb = s - a.h;
  const float e = ((a.h - (s - bb)) + (b.h - bb)) + (a.l + b.l);
  return df_norm(s, e);
}
__device__ __forceinline__ df2 df_neg(df2 a) { return {-a.h, -a.l}; }
__device__ __forceinline__ df2 df_scale(float c, df2 a) {  // c * a with the exact product of c and a.h
  const float p = c * a.h;
  const float e = fmaf(c, a.h, -p);
  return df_norm(p, fmaf(c, a.l, e));
}

__device__ inline void load_exp_table(uint64_t* dst) {
  for (int i = threadIdx.x; i < RK_FX_EXP2_N; i += blockDim.x) dst[i] = c_exp2_table[i];
}

// --------------------------------------------------------------- error state
// The library's last error (thread-local; defined in rok4e_kernels.cu).
int set_error(int code, const std::string& msg);
int cuda_error(cudaError_t e, const char* where);

// ------------------------------------------------------------------- views
struct MechView {
  int ns, nr, ntb, ntroe;
  int nx;  // state components after T: 0, or 5 (rho, rho u, rho E) for the auxiliary-temperature system
  const uint64_t* etab;  // 2^(j/256) table in shared memory
  const double *W, *invW, *Tmid, *lo, *hi, *lnA, *bexp, *EaR, *eff, *fo, *csr_nu;
  const uint64_t *fA, *fb, *fE;  // fixed-point Arrhenius coefficients (fx.cuh)
  bool fx;                       // every coefficient fits that form
  double fx_T_lo;                // the form's lowest temperature
  bool seg;                      // the gather's list is in shared memory
  const uint32_t* slots;
  const int32_t *meta, *csr_ptr, *csr_j;
  const int32_t* gcsr_j;  // csr_j in global memory
  const int32_t *piece_ptr, *spec_piece;  // gather pieces of the species-major list
  int npiece;
  const uint16_t* gidx;  // fixed-point gather: [glen][gnpp] reactions, pieces of each species
  const int32_t* gspec;
  int glen, gnpp, ghb, gdeep;
  bool gfix;  // gather in fixed point
  const float *Wf, *invWf, *bf, *EaRf, *efff, *csr_nuf;  // FP32 copies
  const int32_t* perm;  // input index of each packed reaction
  int nst, nrt;         // nu^T tiles (species, reactions) of the tensor-core gather
  const uint4* nuT;     // their A operands, per tile and lane
  const int32_t *role_ptr, *role;  // species-major reaction slots (r << 2 | role)
};

// The view of a block that copied the buffer's first `prefix` bytes to base and
// after them the segment: all of it (fxseg), or its thermo coefficients alone.  Then
// fA, fb, fE, gidx and gspec are not in shared memory, m.fx and m.seg say so, and
// nothing may read them; the rows of the species-major list (csr_ptr, csr_nu,
// gcsr_j), lnA, b and Ea/R are read from the whole buffer in global memory, gbase.
__host__ __device__ inline MechView make_view(const unsigned char* base, const unsigned char* gbase,
                                              const MechLayout& L, int64_t prefix, bool fxseg) {
  const unsigned char* fbase = base + prefix - L.off_lo;  // the segment's arrays sit at fbase + their offset
  MechView m;
  m.ns = L.ns;
  m.nr = L.nr;
  m.ntb = L.ntb;
  m.ntroe = L.ntroe;
  m.nx = 0;
  m.etab = nullptr;
  m.W = reinterpret_cast<const double*>(base + L.off_W);
  m.invW = reinterpret_cast<const double*>(base + L.off_invW);
  m.Tmid = reinterpret_cast<const double*>(base + L.off_Tmid);
  m.lo = reinterpret_cast<const double*>(fbase + L.off_lo);
  m.hi = reinterpret_cast<const double*>(fbase + L.off_hi);
  m.lnA = reinterpret_cast<const double*>(gbase + L.off_lnA);
  m.fA = reinterpret_cast<const uint64_t*>(fbase + L.off_fA);
  m.fb = reinterpret_cast<const uint64_t*>(fbase + L.off_fb);
  m.fE = reinterpret_cast<const uint64_t*>(fbase + L.off_fE);
  m.fx = fxseg && L.fx != 0;
  m.fx_T_lo = L.fx_T_lo;
  m.seg = fxseg && L.nr < 8191;
  m.gcsr_j = reinterpret_cast<const int32_t*>(gbase + L.off_csr_j);
  m.bexp = reinterpret_cast<const double*>(gbase + L.off_b);
  m.EaR = reinterpret_cast<const double*>(gbase + L.off_EaR);
  m.eff = reinterpret_cast<const double*>(base + L.off_eff);
  m.fo = reinterpret_cast<const double*>(base + L.off_fo);
  m.csr_nu = reinterpret_cast<const double*>(gbase + L.off_csr_nu);
  m.slots = reinterpret_cast<const uint32_t*>(base + L.off_slots);
  m.meta = reinterpret_cast<const int32_t*>(base + L.off_meta);
  m.csr_ptr = reinterpret_cast<const int32_t*>(gbase + L.off_csr_ptr);
  m.csr_j = reinterpret_cast<const int32_t*>(base + L.off_csr_j);
  m.piece_ptr = reinterpret_cast<const int32_t*>(base + L.off_piece_ptr);
  m.spec_piece = reinterpret_cast<const int32_t*>(base + L.off_spec_piece);
  m.npiece = L.npiece;
  m.gidx = reinterpret_cast<const uint16_t*>(fbase + L.off_gidx);
  m.gspec = reinterpret_cast<const int32_t*>(fbase + L.off_gspec);
  m.glen = L.glen;
  m.gnpp = L.gnpp;
  m.ghb = L.ghb;
  m.gdeep = 73 - 2 * L.ghb;
  m.gfix = L.gfix != 0;
  m.Wf = reinterpret_cast<const float*>(base + L.off_Wf);
  m.invWf = reinterpret_cast<const float*>(base + L.off_invWf);
  m.bf = reinterpret_cast<const float*>(base + L.off_bf);
  m.EaRf = reinterpret_cast<const float*>(base + L.off_EaRf);
  m.efff = reinterpret_cast<const float*>(base + L.off_efff);
  m.csr_nuf = reinterpret_cast<const float*>(base + L.off_csr_nuf);
  m.perm = reinterpret_cast<const int32_t*>(base + L.off_perm);
  m.nst = L.nst;
  m.nrt = L.nrt;
  m.nuT = reinterpret_cast<const uint4*>(base + L.off_nuT);
  m.role_ptr = reinterpret_cast<const int32_t*>(base + L.off_role_ptr);
  m.role = reinterpret_cast<const int32_t*>(base + L.off_role);
  return m;
}

// Per-cell shared-memory slot (offsets in doubles from the slot base).
struct SlotLayout {
  int N, ns, nr, ntb, M;
  int u, src, fn, arg, fr, F, w, Q, K;        // N-vectors (Q: M of them, K: 4)
  int C, dC, cp, hRT, gRT, E, CE, om;  // species (+1 sentinel entry)
  int q, kc, krc, qT;                         // reactions (qT: d q_j / dT at u_n, for J v)
  int tb;                                     // [ntb][4]: [M], dk/d[M], dlnk/dT, 1/Kc
  int tro;                                    // [11][ntroe]: Troe falloff scratch
  int part;                                   // [npiece]: gather partial sums
  int C2, dC2;                                // species: double-float C and dC (precision 3, else -1)
  int dig;                                    // BF16 digits of q, [8][16 nrt] (precision 4, else -1)
  int fj;   // precision 6: FP32 species factors of the J v, when they do not fit beside the
            // FP32 reaction caches in the kc/krc/qT storage (else -1)
  int H, LU, piv, Bm;                    // small (Bm: I - (I - h gamma H)^-1)
  int fbase;  // FP32 region (mixed precision only), offset in doubles
  int fC, fdC, fh, fcp, fdcp, fom, fq, fkc, fkr, ftb, fQ, fw, fpart;  // offsets in floats from fbase
  int stride;
};

// mixed: the FP32 arrays of precision levels 1 and 2; df: the double-float
// species arrays of precision level 3; src: the slot keeps the cell's source.
// Arrays whose lives do not meet share storage, so that an SM holds more cells
// (a warp each): with 19.2 kB at 53 species / 325 reactions instead of 22.7, and a
// mechanism copy of 22 instead of 48 kB, ten instead of eight.
// SLOT_RHS: one source term, no Jacobian caches or vectors.
enum SlotKind { SLOT_ROK4E, SLOT_RKDP, SLOT_POINT, SLOT_RHS };
inline SlotLayout make_slot(const MechLayout& L, int M, SlotKind kind, bool mixed, int nx, bool df, bool tc,
                            bool f32jv, bool src) {
  SlotLayout s;
  s.N = L.ns + 1 + nx;
  s.ns = L.ns;
  s.nr = L.nr;
  s.ntb = L.ntb;
  s.M = M;
  int o = 0;
  auto take = [&](int n) {
    const int r = o;
    o += (n + 1) & ~1;  // keep 16-byte alignment
    return r;
  };
  const int N = s.N, ns1 = L.ns + 1;
  s.u = take(N);
  s.src = src ? take(N) : -1;
  const bool rhs = kind == SLOT_RHS;
  s.fn = rhs ? s.u : take(N);  // (not used)
  s.arg = take(N);
  // a stage's f may overwrite its argument, except in the auxiliary-temperature
  // system, whose T row reads the argument after the species rows are written
  s.fr = kind != SLOT_RKDP && nx > 0 ? take(N) : s.arg;
  s.F = kind == SLOT_RKDP || kind == SLOT_POINT ? take(N) : -1;  // a stage vector; the point kernel's V
  s.w = rhs ? s.u : take(N);
  const int Nq = (N + 1) & ~1;  // stride between Krylov / stage vectors
  s.Q = rhs ? s.u : take(Nq * M);
  s.CE = take(ns1);
  // C is read beside CE only by third-body sums and the reduced-precision J v
  s.C = L.ntb > 0 || mixed || df || f32jv ? take(ns1) : s.CE;
  s.dC = take(ns1);
  s.cp = take(ns1);
  s.hRT = take(ns1);
  s.gRT = take(ns1);
  s.E = take(ns1);
  s.om = s.gRT;  // w is kept (caching evaluation) when the Gibbs factors are done with
  // reactions, and entry nr: the zero rate that pads the gather's pieces
  s.q = take(L.nr + 1);
  s.kc = rhs ? s.q : take(L.nr + 1);
  s.qT = rhs ? s.q : take(L.nr + 1);
  s.krc = take(L.nr + 1);
  // The stage vectors K live only inside an attempt; the J v caches kc, qT
  // (contiguous) only from the caching right-hand side to the end of the
  // Arnoldi process that precedes the attempts.  K shares their storage when
  // it fits there (not krc's, which holds the low words of the gather's rates).
  const int nr_even = (L.nr + 2) & ~1;
  s.K = rhs || 4 * Nq <= 2 * nr_even ? s.kc : take(4 * Nq);
  s.tb = take(4 * (L.ntb > 0 ? L.ntb : 1));
  s.tro = take(11 * (L.ntroe > 0 ? L.ntroe : 1));
  // the gather's pieces ((hi, lo) words in fixed point); LU and its pivots, used
  // only to form B, share them
  int np = 2 * L.gnpp > L.npiece ? 2 * L.gnpp : L.npiece;
  np = np > (M + 1) * MAXM ? np : (M + 1) * MAXM;
  s.part = take(np);
  s.C2 = df ? take(ns1) : -1;
  s.dC2 = df ? take(ns1) : -1;
  s.dig = tc ? take(2 * 16 * L.nrt) : -1;  // 8 x 16 nrt BF16 = 2 x 16 nrt doubles
  // precision 6 keeps its FP32 reaction caches in the first half of the kc/krc/qT
  // storage and its 6 FP32 species arrays in the second half when they fit there
  s.fj = (f32jv && 6 * ns1 > 3 * nr_even) ? take((6 * ns1 + 1) / 2) : -1;
  // M x M matrices stored with row stride MAXM: M rows
  s.H = take(M * MAXM);
  s.LU = s.part;
  s.piv = s.part + M * MAXM;
  s.Bm = take(M * MAXM);
  s.fbase = o;
  int fo = 0;
  auto ftake = [&](int n) {
    const int r = fo;
    fo += (n + 3) & ~3;  // 16-byte alignment
    return r;
  };
  if (mixed) {
    s.fC = ftake(ns1);
    s.fdC = ftake(ns1);
    s.fh = ftake(ns1);
    s.fcp = ftake(ns1);
    s.fdcp = ftake(ns1);
    s.fom = ftake(ns1);
    s.fq = ftake(L.nr > 0 ? L.nr : 1);
    s.fkc = ftake(L.nr > 0 ? L.nr : 1);
    s.fkr = ftake(L.nr > 0 ? L.nr : 1);
    s.ftb = ftake(4 * (L.ntb > 0 ? L.ntb : 1));
    s.fQ = ftake(Nq * M);
    s.fw = ftake(Nq);
    s.fpart = ftake(L.npiece > 0 ? L.npiece : 1);
  } else {
    s.fC = s.fdC = s.fh = s.fcp = s.fdcp = s.fom = s.fq = s.fkc = s.fkr = s.ftb = s.fQ = s.fw = s.fpart = 0;
  }
  o += (fo + 1) / 2;
  s.stride = (o + 3) & ~3;
  return s;
}

// Float with the value of x truncated, and back, by integer moves (a conversion
// takes the FP64 unit as long as an FP64 operation): below 2^-126 zero, from 2^127
// infinity; x >= 0.
__device__ __forceinline__ float float_bits(double x) {
  const int hi = __double2hiint(x), e = hi >> 20;
  const float f = __int_as_float(((hi - (896 << 20)) << 3) | (int)((unsigned)__double2loint(x) >> 29));
  return e < 897 ? 0.f : (e >= 1150 ? INFINITY : f);
}
__device__ __forceinline__ double double_bits(float f) {  // for normal f > 0
  const int b = __float_as_int(f);
  return __hiloint2double((b >> 3) + (896 << 20), b << 29);
}

// A group of G lanes inside one warp.
template <int G>
struct Grp {
  unsigned mask;
  int lane;
  __device__ Grp() {
    const int l = threadIdx.x & 31;
    lane = l % G;
    mask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << (l - lane));
  }
  __device__ __forceinline__ void sync() const { __syncwarp(mask); }
  template <typename T>
  __device__ __forceinline__ T sum(T v) const {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o, G);
    return v;
  }
  __device__ __forceinline__ unsigned umin(unsigned v) const {
    if constexpr (G == 32) return __reduce_min_sync(0xffffffffu, v);
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v = ::min(v, __shfl_xor_sync(mask, v, o, G));
    return v;
  }
  __device__ __forceinline__ int imax(int v) const {
    if constexpr (G == 32) return __reduce_max_sync(0xffffffffu, v);
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v = ::max(v, __shfl_xor_sync(mask, v, o, G));
    return v;
  }
  __device__ __forceinline__ int any(int v) const {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v |= __shfl_xor_sync(mask, v, o, G);
    return v;
  }
};

// Sum K values (K a power of two, K <= G) across the G lanes of a group; on
// return every lane holds all K sums.  Reduce-scatter: at each of the first
// log2 K butterfly levels a lane keeps half of its values and adds its
// partner's copy of that half, so the adds per lane are K - 1 + log2(G/K)
// instead of K log2 G; the sums are then broadcast from the lanes that hold
// them.  All lanes end with bit-identical values.
template <int G, int K, typename T>
__device__ __forceinline__ void sum_many(const Grp<G>& g, T (&v)[K]) {
  static_assert((K & (K - 1)) == 0 && K <= G, "K must be a power of two <= G");
  constexpr int LG = (G == 32 ? 5 : G == 16 ? 4 : G == 8 ? 3 : G == 4 ? 2 : G == 2 ? 1 : 0);
  constexpr int LK = (K == 8 ? 3 : K == 4 ? 2 : K == 2 ? 1 : 0);
#pragma unroll
  for (int l = 0; l < LK; ++l) {
    const int o = G >> (l + 1);
    const int half = K >> (l + 1);
    const bool hi = (g.lane & o) != 0;
#pragma unroll
    for (int j = 0; j < half; ++j) {
      const T send = hi ? v[j] : v[j + half];
      const T keep = hi ? v[j + half] : v[j];
      v[j] = keep + __shfl_xor_sync(g.mask, send, o, G);
    }
  }
#pragma unroll
  for (int o = G >> (LK + 1); o > 0; o >>= 1) v[0] += __shfl_xor_sync(g.mask, v[0], o, G);
  const T mine = v[0];
#pragma unroll
  for (int t = 0; t < K; ++t) v[t] = __shfl_sync(g.mask, mine, t << (LG - LK), G);
}

// Sum the first n (<= MAXM) entries of v across the group (entries past n
// must be zero); dispatches on n to the smallest power-of-two reduction.
template <int G, typename T>
__device__ __forceinline__ void sum_first(const Grp<G>& g, T (&v)[MAXM], int n) {
  static_assert(G >= MAXM, "a group needs at least MAXM lanes");
  if (n <= 1) {
    v[0] = g.sum(v[0]);
  } else if (n <= 2) {
    T t[2] = {v[0], v[1]};
    sum_many<G, 2>(g, t);
    v[0] = t[0];
    v[1] = t[1];
  } else if (n <= 4) {
    T t[4] = {v[0], v[1], v[2], v[3]};
    sum_many<G, 4>(g, t);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = t[i];
  } else {
    sum_many<G, MAXM>(g, v);
  }
}

// Scalars of the last right-hand-side evaluation that the analytic
// Jacobian-vector product needs (uniform across the group).
struct CellScalars {
  double T, invT, lnT, S, invS, rho, invrho, cb, invcb, Sh;
  double TSh, irc;  // T Sh, 1 / (rho cb)
  double Hs, Ds;    // sum (cp_k/R - h_k/RT) w_k / T, sum Y_k d(cp_k/R)/dT / W_k
  double pinv;  // 1 / p (constant pressure) or 1 / rho (constant volume): set by the caller
  int prec;     // precision level (3: double-float J v core, 6: FP32 J v): set by the caller
  // auxiliary-temperature system: sum_k (cp_k/R - 1) F_k / W_k, the T row
  // without its own source, 1 / rho and the velocity
  double B, fT, irho_c, vel[3];
  bool cv;
  bool zf;  // the caches are those of the scaled form (reactions_scaled), read by jvp_eval
};

struct SlotPtrs {
  double *u, *src, *fn, *arg, *fr, *F, *w, *Q, *K;
  double *C, *dC, *cp, *hRT, *gRT, *E, *CE, *om, *q, *kc, *krc, *qT, *tb, *tro, *part;
  df2 *C2, *dC2;
  uint16_t* dig;
  // precision 6: FP32 J v caches in the kc/krc/qT storage -- per reaction k, k/Kc, dq/dT;
  // per species C, rho/W, W/rho, w, h/RT - esh, cp / W
  float *xk, *xkr, *xqT, *xC, *xE, *xEinv, *xom, *xg, *xcp;
  double *H, *LU, *piv, *Bm;
  float *fC, *fdC, *fh, *fcp, *fdcp, *fom, *fq, *fkc, *fkr, *ftb, *fQ, *fw, *fpart;  // mixed precision
  int Nq;  // stride between Krylov / stage vectors
};

__device__ inline SlotPtrs slot_ptrs(double* b, const SlotLayout& s) {
  SlotPtrs p;
  p.u = b + s.u;
  p.src = b + (s.src >= 0 ? s.src : 0);  // not read where the slot has none
  p.fn = b + s.fn;
  p.arg = b + s.arg;
  p.fr = b + s.fr;
  p.F = b + (s.F >= 0 ? s.F : 0);  // not read where the slot has none
  p.w = b + s.w;
  p.Q = b + s.Q;
  p.K = b + s.K;
  p.C = b + s.C;
  p.dC = b + s.dC;
  p.cp = b + s.cp;
  p.hRT = b + s.hRT;
  p.gRT = b + s.gRT;
  p.E = b + s.E;
  p.CE = b + s.CE;
  p.om = b + s.om;
  p.q = b + s.q;
  p.kc = b + s.kc;
  p.krc = b + s.krc;
  p.qT = b + s.qT;
  p.tro = b + s.tro;
  p.part = b + s.part;
  p.C2 = s.C2 >= 0 ? reinterpret_cast<df2*>(b + s.C2) : nullptr;
  p.dC2 = s.dC2 >= 0 ? reinterpret_cast<df2*>(b + s.dC2) : nullptr;
  p.dig = s.dig >= 0 ? reinterpret_cast<uint16_t*>(b + s.dig) : nullptr;
  {
    const int nr_even = (s.nr + 2) & ~1, ns1 = s.ns + 1;
    float* R = reinterpret_cast<float*>(b + s.kc);  // 3 nr_even doubles = 6 nr_even floats
    p.xk = R;
    p.xkr = R + nr_even;
    p.xqT = R + 2 * nr_even;
    float* X = s.fj >= 0 ? reinterpret_cast<float*>(b + s.fj) : R + 3 * nr_even;
    p.xC = X;
    p.xE = X + ns1;
    p.xEinv = X + 2 * ns1;
    p.xom = X + 3 * ns1;
    p.xg = X + 4 * ns1;
    p.xcp = X + 5 * ns1;
  }
  p.tb = b + s.tb;
  p.H = b + s.H;
  p.LU = b + s.LU;
  p.piv = b + s.piv;
  p.Bm = b + s.Bm;
  float* f = reinterpret_cast<float*>(b + s.fbase);
  p.fC = f + s.fC;
  p.fdC = f + s.fdC;
  p.fh = f + s.fh;
  p.fcp = f + s.fcp;
  p.fdcp = f + s.fdcp;
  p.fom = f + s.fom;
  p.fq = f + s.fq;
  p.fkc = f + s.fkc;
  p.fkr = f + s.fkr;
  p.ftb = f + s.ftb;
  p.fQ = f + s.fQ;
  p.fw = f + s.fw;
  p.fpart = f + s.fpart;
  p.Nq = (s.N + 1) & ~1;
  return p;
}

// Where a gather left w = nu^T q: nowhere yet; pieces, or a species' sum each, in
// part; a species' sum each in the rates' place.
enum Gathered { NOT_GATHERED, PIECES_IN_PART, ROWS_IN_PART, ROWS_IN_Q };
// w = nu^T q by rows of the species-major list in FP64, into part[0..ns), for
// mechanisms whose gather list does not fit in shared memory.
template <int G>
__device__ __noinline__ Gathered gather_rows(const MechView& m, const SlotPtrs& s) {
  const Grp<G> g;
  for (int k = g.lane; k < m.ns; k += G) {
    double acc = 0.0;
    for (int e = m.csr_ptr[k]; e < m.csr_ptr[k + 1]; ++e) acc = fma(m.csr_nu[e], s.q[m.gcsr_j[e]], acc);
    s.part[k] = acc;
  }
  g.sync();
  return ROWS_IN_PART;
}
// The same in FP32 (the J v of precision 6).
template <int G>
__device__ __noinline__ void gather_rows_f32(const MechView& m, const float* q, float* part) {
  const Grp<G> g;
  for (int k = g.lane; k < m.ns; k += G) {
    float acc = 0.f;
    for (int e = m.csr_ptr[k]; e < m.csr_ptr[k + 1]; ++e)
      acc = fmaf(__double2float_rn(m.csr_nu[e]), q[m.gcsr_j[e]], acc);
    part[k] = acc;
  }
  g.sync();
}
// High words without signs of a lane's rates (their last bit set where the low word is
// not zero: only a zero gives 0): the largest, and the smallest that is not zero, less
// one (a zero wraps to the top).
struct RateRange {
  uint32_t top = 0u, low = 0xffffffffu;
  __device__ __forceinline__ void take(double q) {
    const uint32_t w = ((uint32_t)__double2hiint(q) & 0x7fffffffu) | (__double2loint(q) != 0 ? 1u : 0u);
    top = ::max(top, w);
    low = ::min(low, w - 1u);
  }
};
constexpr int DEPTH_FP64 = 80;
// The gather in 128-bit fixed point (fx.cuh): the rates in s.q go onto one grid
// below their largest (high words in place, low words in krc's storage), each lane
// adds up whole pieces with integer adds, and a species adds and subtracts its
// pieces and rounds once.  The sums do not depend on their order, so the pieces'
// entries are ordered to meet no shared-memory bank conflicts and no coefficient is
// loaded or multiplied.  An FP64 term took 64 cycles of the FP64 unit, here ~20 of
// the integer pipes and ~5 shared-memory wavefronts.
// The grid ends 2^-(126 - ghb) below the cell's largest rate, and a row of up to
// 2^(ghb - 1) terms may lose a unit with each: a row whose sum is 2^(53 + ghb) units or
// more, 2^-gdeep of the largest, keeps it to 2^-54, half a rounding of FP64.  Where some
// rate that is not zero lies below that and a row's sum too (a cold mixture with few
// species present: the first radicals' rates are tens of orders of magnitude below the
// others'), the caller forms the rates again and sums them in FP64.  Where the rates
// reach down 2^-80 that is likely (53 species, 300 to 2000 K: 5 % of the cells at 2^-60
// to 2^-70, 71 % at 2^-80 to 2^-90) and FP64 is taken at once: its gather costs a
// right-hand side a tenth more, forming the rates again two thirds.
// NOT_GATHERED, with nothing done, for these, when a rate is infinite or NaN and when a
// sum might leave FP64's normal range (from_grid knows no infinity and no subnormals:
// a unit of 2^-1022 or more excludes the latter);
// *again: a row out of reach.
template <int G>
__device__ __forceinline__ Gathered gather_fixed(const MechView& m, const SlotPtrs& s, const RateRange& lane_range,
                                                 bool* again) {
  const Grp<G> g;
  const int top = g.imax((int)lane_range.top), em = top >> 20;
  const uint32_t least = g.umin(lane_range.low);
  const int depth = least == 0xffffffffu ? 0 : em - (int)((least + 1u) >> 20);
  if (em + m.ghb >= 0x7ff || depth > DEPTH_FP64 || (em + m.ghb < 127 && top != 0)) return NOT_GATHERED;
  uint64_t* qh = reinterpret_cast<uint64_t*>(s.q);
  uint64_t* ql = reinterpret_cast<uint64_t*>(s.krc);
  constexpr int U = 4;
  for (int j0 = g.lane; j0 < m.nr; j0 += U * G) {
    fx::Wide w[U];
#pragma unroll
    for (int u = 0; u < U; ++u) w[u] = fx::to_grid(s.q[min(j0 + u * G, m.nr - 1)], em, m.ghb);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (j0 + u * G < m.nr) {
        qh[j0 + u * G] = w[u].hi;
        ql[j0 + u * G] = w[u].lo;
      }
  }
  if (g.lane == 0) qh[m.nr] = ql[m.nr] = 0ull;
  g.sync();
  uint64_t* part = reinterpret_cast<uint64_t*>(s.part);
  const uint4* ix = reinterpret_cast<const uint4*>(m.gidx);
  const char* bh = reinterpret_cast<const char*>(qh);
  const char* bl = reinterpret_cast<const char*>(ql);
  for (int p = g.lane; p < m.gnpp; p += G) {
    fx::Wide a = {0ull, 0ull};
    for (int i = 0; i < m.glen; i += 8) {
      const uint4 v = ix[(i >> 3) * m.gnpp + p];
      const uint32_t o[8] = {v.x & 0xffffu, v.x >> 16, v.y & 0xffffu, v.y >> 16,
                             v.z & 0xffffu, v.z >> 16, v.w & 0xffffu, v.w >> 16};
      uint64_t h[8], l[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        h[t] = *reinterpret_cast<const uint64_t*>(bh + o[t]);
        l[t] = *reinterpret_cast<const uint64_t*>(bl + o[t]);
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) fx::add(a, h[t], l[t]);
    }
    part[p] = a.hi;
    part[m.gnpp + p] = a.lo;
  }
  g.sync();
  bool out = false;
  for (int k = g.lane; k < m.ns; k += G) {
    const int p0 = m.gspec[2 * k], p1 = m.gspec[2 * k + 1], p2 = m.gspec[2 * k + 2];
    int p = p0;
    fx::Wide a = {0ull, 0ull};
#pragma unroll 2
    for (; p < p1; ++p) fx::add(a, part[p], part[m.gnpp + p]);
#pragma unroll 2
    for (; p < p2; ++p) fx::sub(a, part[p], part[m.gnpp + p]);
    const double r = fx::from_grid(a, em, m.ghb);
    s.q[k] = r;
    out |= p0 != p2 && ((__double2hiint(r) >> 20) & 0x7ff) + m.gdeep < em;
  }
  *again = depth > m.gdeep && g.any(out);
  return ROWS_IN_Q;
}
// The same pieces in FP64, for mechanisms of few entries (gfix false), where the
// conversions to the grid and back would cost more than the additions they save.
template <int G>
__device__ __forceinline__ Gathered gather_listed(const MechView& m, const SlotPtrs& s) {
  const Grp<G> g;
  if (g.lane == 0) s.q[m.nr] = 0.0;
  g.sync();
  const char* q = reinterpret_cast<const char*>(s.q);
  for (int p = g.lane; p < m.gnpp; p += G) {
    double a = 0.0;
    for (int i = 0; i < m.glen; ++i) {
      const double x = *reinterpret_cast<const double*>(q + m.gidx[((i >> 3) * m.gnpp + p) * 8 + (i & 7)]);
      a = i == 0 ? x : a + x;
    }
    s.part[p] = a;
  }
  g.sync();
  return PIECES_IN_PART;
}
// (for cells in the direct form, and rates that are not finite: their rows alone
// become so)
template <int G>
__device__ __noinline__ Gathered gather_listed_call(const MechView& m, const SlotPtrs& s) {
  return gather_listed<G>(m, s);
}
// nu^T q of species k after gather_fixed, gather_listed or gather_rows
__device__ __forceinline__ double gathered_row(const MechView& m, const SlotPtrs& s, int k,
                                               Gathered how) {
  if (how == ROWS_IN_Q) return s.q[k];
  if (how == ROWS_IN_PART) return s.part[k];
  const int p1 = m.gspec[2 * k + 1], p2 = m.gspec[2 * k + 2];
  int p = m.gspec[2 * k];
  double a = 0.0, b = 0.0;
  if (p < p1) a = s.part[p++];
  for (; p < p1; ++p) a += s.part[p];
  if (p < p2) b = s.part[p++];
  for (; p < p2; ++p) b += s.part[p];
  return a - b;
}

// The gather in double-float (FP32 pairs, ~44-bit significands, on the FP32
// pipe): the species-major list is cut into pieces of near-equal length (chosen
// when the mechanism is packed), each lane sums whole pieces into part[] and
// piece_sum_df adds a species' pieces in order.  The net coefficients are small integers, exact in FP32, so each
// product nu_e q_j is formed with the pair's precision and summed by two-sums.
template <int G>
__device__ __forceinline__ void gather_pieces_df(const MechView& m, int lane, const df2* __restrict__ q,
                                                 df2* part) {
  for (int p = lane; p < m.npiece; p += G) {
    df2 acc = {0.0f, 0.0f};
    const int e1 = m.piece_ptr[p + 1];
    for (int e = m.piece_ptr[p]; e < e1; ++e) acc = df_add(acc, df_scale(m.csr_nuf[e], q[m.csr_j[e]]));
    part[p] = acc;
  }
}
__device__ __forceinline__ double piece_sum_df(const MechView& m, const df2* part, int k) {
  const int p1 = m.spec_piece[k + 1];
  int p = m.spec_piece[k];
  df2 acc = part[p];
  for (++p; p < p1; ++p) acc = df_add(acc, part[p]);
  return df_to(acc);
}

// ---- w = nu^T q on the tensor cores (precision level 4), exact to FP64 level.
// Each q_j is cut, relative to 2^Es with Es above the cell's largest |q_j|,
// into seven signed 8-bit digits (56 bits below 2^Es; what lies below
// 2^(Es - 56) is dropped, at most 2^-55 of the largest rate); the digits and
// the small-integer net coefficients are exact in BF16, each product is exact
// in FP32 and so is every sum the mma accumulates (|sum| <= 2 x 255 x Nr <
// 2^24), so the FP32 accumulators hold the digit columns of nu^T q exactly.
// mma.m16n8k16: A = a 16 x 16 tile of nu^T (species x reactions, prepacked
// per lane), B = the 16 x 8 tile of digits (reactions x digit 0..6, column 7
// zero), D = 16 species x 8 digit sums; FP64 then adds the seven scaled digit
// sums of each species (rounding once per addition, like a sum of terms).
__device__ __forceinline__ void mma_bf16_m16n8k16(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// A signed integer |v| <= 256 as BF16 (exact: its float's upper half).
__device__ __forceinline__ uint16_t bf16_of_small_int(int v) {
  return (uint16_t)(__float_as_uint((float)v) >> 16);
}

// x * 2^e for a double x holding an integer of magnitude below 2^53 and an
// exponent that keeps the result normal: an integer add to the exponent field.
__device__ __forceinline__ double scale_pow2(double x, int e) {
  return x == 0.0 ? 0.0 : __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x));
}

// out[k] = sum_j nu_jk q_j for the cell (q: Nr doubles in shared memory).
// Returns false, writing nothing, when every |q_j| < 2^-920 (the digit
// weights would leave the normal range): the caller then gathers in FP64.
template <int G>
__device__ bool gather_tc(const MechView& m, const SlotPtrs& s, const double* __restrict__ q,
                          double* __restrict__ out) {
  static_assert(G == 32, "the tensor-core gather runs one cell per warp");
  const Grp<G> g;
  const int lane = g.lane;
  const int nrp = 16 * m.nrt;
  // the scale: 2^(Eb - 1023) above every |q_j| (Eb one above the largest biased exponent)
  int emax = 0;
  for (int j = lane; j < m.nr; j += G) emax = max(emax, (__double2hiint(q[j]) >> 20) & 0x7ff);
  const int Eb = g.imax(emax) + 1;
  if (Eb < 104) return false;
  // digits of |q_j| 2^(56 - Es), most significant first, with q_j's sign
  for (int j = lane; j < m.nr; j += G) {
    const long long bits = __double_as_longlong(q[j]);
    const int e = (int)((bits >> 52) & 0x7ff);
    unsigned long long V = 0ull;
    if (e != 0) {  // zero and subnormal rates (below 2^-1022) drop out
      const unsigned long long mant = ((unsigned long long)bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
      const int sh = e + 4 - Eb;  // V = mant 2^sh < 2^56
      V = sh >= 0 ? (mant << sh) : (sh > -64 ? (mant >> (-sh)) : 0ull);
    }
    const bool neg = bits < 0;
#pragma unroll
    for (int n = 0; n < 7; ++n) {
      const int dn = (int)((V >> (48 - 8 * n)) & 255ull);
      s.dig[n * nrp + j] = bf16_of_small_int(neg ? -dn : dn);
    }
  }
  g.sync();
  const int grp = lane >> 2, tq = lane & 3;
  const uint32_t* drow = reinterpret_cast<const uint32_t*>(s.dig + grp * nrp);
  // digit n weighs 2^(Es - 8 (n + 1)), Es = Eb - 1023
  const int w0 = Eb - 1023 - 8 * (2 * tq + 1), w1 = w0 - 8;
  for (int st = 0; st < m.nst; ++st) {
    float d[4] = {0.f, 0.f, 0.f, 0.f};
    for (int rt = 0; rt < m.nrt; ++rt) {
      const uint4 a = m.nuT[(st * m.nrt + rt) * 32 + lane];
      mma_bf16_m16n8k16(d, a, drow[8 * rt + tq], drow[8 * rt + tq + 4]);
    }
    // this lane: digits 2tq and 2tq+1 of species rows grp (d0, d1) and grp + 8 (d2, d3)
    double r0 = scale_pow2((double)d[1], w1) + scale_pow2((double)d[0], w0);
    double r1 = scale_pow2((double)d[3], w1) + scale_pow2((double)d[2], w0);
    // add the four lanes of the group, least significant digits first
    r0 = __shfl_xor_sync(g.mask, r0, 1) + r0;
    r1 = __shfl_xor_sync(g.mask, r1, 1) + r1;
    r0 = __shfl_xor_sync(g.mask, r0, 2) + r0;
    r1 = __shfl_xor_sync(g.mask, r1, 2) + r1;
    if (tq == 0) {
      const int k0 = 16 * st + grp, k1 = k0 + 8;
      if (k0 < m.ns) out[k0] = r0;
      if (k1 < m.ns) out[k1] = r1;
    }
  }
  g.sync();
  return true;
}

// Cached values of a pressure-dependent reaction for the Jacobian-vector
// product: [M], dk/d[M], d ln k/dT and 1/Kc (and their FP32 copies, MIXED).
template <bool MIXED>
__device__ __forceinline__ void cache_pressure(const SlotPtrs& s, int slot, double Mc, double dkdM, double dlnk,
                                               double rfac) {
  double* t = s.tb + 4 * slot;
  t[0] = Mc;
  t[1] = dkdM;
  t[2] = dlnk;
  t[3] = rfac;
  if (MIXED) {
    float* tf = s.ftb + 4 * slot;
    tf[0] = __double2float_rn(Mc);
    tf[1] = __double2float_rn(dkdM);
    tf[2] = __double2float_rn(dlnk);
    tf[3] = __double2float_rn(rfac);
  }
}
template <int G>
__device__ __forceinline__ double third_body_conc(const MechView& m, const SlotPtrs& s, int slot, bool coop_tb) {
  if (coop_tb) return s.tb[4 * slot];
  const double* e = m.eff + (size_t)slot * m.ns;
  double Mc = 0.0;
  for (int q = 0; q < m.ns; ++q) Mc = fma(e[q], s.C[q], Mc);
  return Mc;
}
// The caches of one reaction that the selected Jacobian-vector product reads.
template <bool MIXED>
__device__ __forceinline__ void cache_reaction(const SlotPtrs& s, const CellScalars* cs, int j, double k, double kr,
                                               double qT) {
  if (cs->prec == 3) {  // double-float copies for the J v core, in the same storage
    reinterpret_cast<df2*>(s.qT)[j] = df_from(qT);
    reinterpret_cast<df2*>(s.kc)[j] = df_from(k);
    reinterpret_cast<df2*>(s.krc)[j] = df_from(kr);
  } else if (cs->prec == 6) {  // FP32 copies for the FP32 J v, in the same storage
    s.xk[j] = __double2float_rn(k);
    s.xkr[j] = __double2float_rn(kr);
    s.xqT[j] = __double2float_rn(qT);
  } else {
    s.qT[j] = qT;
    s.kc[j] = k;
    s.krc[j] = kr;
  }
  if (MIXED) {
    s.fkc[j] = __double2float_rn(k);
    s.fkr[j] = __double2float_rn(kr);
  }
}

// The reactions in the scaled form.  With E_s = e^{g_s/RT} (RT/p_ref) per species
// (1/Kc = prod E'' / prod E') and z = C E,
//   q = k prod C^nu' - k/Kc prod C^nu'' = kappa (z_ra z_rb - z_pa z_pb),
//   ln kappa = ln k - ln E_ra - ln E_rb:
// one exponential whose argument takes both Gibbs factors as additions.  The
// argument is formed in fixed point from the mechanism's coefficients, the
// exponential and the product with kappa stay on the integer pipes (fx.cuh),
// and two FP64 instructions are left, the difference of the two products; the
// form with k, E and 1/E in FP64 took sixteen (28 with the caches, now 11).
struct ScaledRate {
  uint64_t lg, ks;  // log2 kappa in fixed point; kappa = ks 2^(kn - 63)
  int kn;
  double D, zr, zs;  // z_ra z_rb - z_pa z_pb (its first product alone when irreversible), z_pa, z_pb
};
__device__ __forceinline__ ScaledRate scaled_rate(const MechView& m, const SlotPtrs& s, const fx::Temp& ft, int j,
                                                  uint32_t sl, bool rev) {
  const uint64_t* A = reinterpret_cast<const uint64_t*>(s.gRT);
  const int ra = sl & 255, rb = (sl >> 8) & 255, pa = (sl >> 16) & 255, pb = sl >> 24;
  ScaledRate r;
  r.zr = s.CE[pa];
  r.zs = s.CE[pb];
  const double D0 = __dmul_rn(s.CE[ra], s.CE[rb]);
  const double D1 = fma(-r.zr, r.zs, D0);
  r.D = rev ? D1 : D0;
  r.lg = fx::arrhenius(ft, m.fA[j], m.fb[j], m.fE[j]) - A[ra] - A[rb];
  r.ks = fx::exp2_sig(r.lg, m.etab);
  r.kn = fx::exponent(r.lg);
  return r;
}
// What the caching right-hand side at u_n keeps of one reaction.
template <bool MIXED>
__device__ __forceinline__ void cache_scaled(const MechView& m, const SlotPtrs& s, double T, double invT, CellScalars* cs, int j,
                                             uint32_t sl, int kind, bool rev, int slot, double Mc, double mult,
                                             const ScaledRate& r) {
  const int ra = sl & 255, rb = (sl >> 8) & 255, pa = (sl >> 16) & 255, pb = sl >> 24;
  const uint64_t* A = reinterpret_cast<const uint64_t*>(s.gRT);
  const int nt = m.ntroe;
  const double kap0 = fx::pack(r.ks, r.kn);
  const double kap = kind == 2 ? kap0 * mult : kap0;
  double dlnk = fma(m.EaR[j], invT, m.bexp[j]);  // T d ln k / dT
  if (kind == 2) dlnk = s.tro[7 * nt + slot] * T;
  // T d q_j / dT at fixed concentrations (without the third-body factor; the J v
  // multiplies it by vT / T): T d ln k/dT q + T d ln Kc/dT k prod C^nu''/Kc, with
  // T d ln Kc/dT = sum_products h/RT - sum_reactants h/RT - dnu summed from the
  // per-species h/RT - 1
  const double t0 = __dmul_rn(dlnk, r.D);
  const double dlnKc = __dsub_rn(__dadd_rn(s.dC[pa], s.dC[pb]), __dadd_rn(s.dC[ra], s.dC[rb]));
  const double t1 = fma(dlnKc, __dmul_rn(r.zr, r.zs), t0);
  const double qT = __dmul_rn(kap, rev ? t1 : t0);
  if (!MIXED && cs->prec != 3 && cs->prec != 6) {
    // the scaled Jacobian-vector product: kappa, d q/dT and the slot's d kappa/d[M]
    if (kind != 0) cache_pressure<MIXED>(s, slot, Mc, kind == 2 ? kap0 * s.tro[8 * nt + slot] : 0.0, 0.0, 0.0);
    s.kc[j] = kap;
    s.qT[j] = qT;
  } else {
    const double Er = __dmul_rn(s.E[ra], s.E[rb]);
    const double k = __dmul_rn(kap, Er);
    const double kr = rev ? __dmul_rn(kap, __dmul_rn(s.E[pa], s.E[pb])) : 0.0;
    if (kind != 0)
      cache_pressure<MIXED>(s, slot, Mc, kind == 2 ? kap0 * Er * s.tro[8 * nt + slot] : 0.0, dlnk * invT,
                            rev ? fx::exp2_double(A[pa] + A[pb] - A[ra] - A[rb], m.etab) : 0.0);
    cache_reaction<MIXED>(s, cs, j, k, kr, qT);
  }
}
// Reaction j0 + lane (a lane past the last computes the last and stores nothing).
// PRESSURE: the first ones, some of them third-body or falloff.  One reaction at a
// time: two interleaved gained nothing (the warps' chains hide each other) and their
// code cost 4 % through the instruction cache.
template <int G, bool MIXED, bool PRESSURE>
__device__ __forceinline__ void reactions_scaled(const MechView& m, const SlotPtrs& s, const fx::Temp& ft, double T,
                                                 double invT, bool coop_tb, bool cache, CellScalars* cs, int j0,
                                                 int lane, RateRange* range) {
  const int j = min(j0 + lane, m.nr - 1);
  const uint32_t sl = m.slots[j];
  const int meta = m.meta[j], kind = PRESSURE ? meta & 3 : 0;
  const bool rev = (meta >> 2) & 1;
  const ScaledRate r = scaled_rate(m, s, ft, j, sl, rev);
  double Mc = 0.0, mult = 1.0, Dm = r.D;  // Dm: with the third-body or falloff multiplier
  if (kind != 0) {
    Mc = third_body_conc<G>(m, s, meta >> 8, coop_tb);
    mult = kind == 1 ? Mc : s.tro[6 * m.ntroe + (meta >> 8)];
    Dm = __dmul_rn(Dm, mult);
  }
  const double q = fx::mul_sig(r.ks, r.kn, Dm);
  range->take(q);
  if (j0 + lane < m.nr) {
    if (MIXED) reinterpret_cast<df2*>(s.q)[j] = df_from(q);  // double-float copy for the gather
    else s.q[j] = q;
    if (cache) cache_scaled<MIXED>(m, s, T, invT, cs, j, sl, kind, rev, meta >> 8, Mc, mult, r);
  }
}

// The rates again (their caches are kept) and their rows in FP64, for cells with a row
// out of the grid's reach.
template <int G>
__device__ __noinline__ Gathered rates_listed_call(const MechView& m, const SlotPtrs& s, uint64_t lgT, double T,
                                                   double invT, bool coop_tb) {
  const Grp<G> g;
  const fx::Temp ft = fx::temperature(lgT, fx::recip_fixed70(T, invT));
  RateRange range;
  for (int j0 = 0; j0 < m.nr; j0 += G)
    reactions_scaled<G, false, true>(m, s, ft, T, invT, coop_tb, false, nullptr, j0, g.lane, &range);
  g.sync();
  return gather_listed<G>(m, s);
}
// The biased exponents of Y and 1/W and, where E = e^lnE < 1, log2 E, summed and offset
// by 512 (up to two below the exponent of C and of C E with rho's added); all ones for
// Y = 0.  |lnE| by its bits in FP32, of no account from 170.
constexpr unsigned THIN_MIN = 512 + 3 * 1023 - 480;
__device__ __forceinline__ unsigned scaled_exponent(double Y, double invW, double lnE) {
  const unsigned y = (unsigned)__double2hiint(Y) & 0x7fffffffu;
  const int hi = __double2hiint(lnE);
  const float f = ::fminf(float_bits(__hiloint2double(hi & 0x7fffffff, __double2loint(lnE))), 170.f);
  const unsigned low = hi < 0 ? 2u + (unsigned)(f * 1.442696f) : 0u;
  const unsigned e = (y >> 20) + ((unsigned)__double2hiint(invW) >> 20) + 512u - low;
  return y == 0u && __double2loint(Y) == 0 ? 0xffffffffu : e;
}
// Every reaction with 1/Kc from one exponential of its own: the form for cells
// the scaled one does not hold for (a Gibbs factor past e^170, T outside
// [150, 16000) K or below where some rate constant passes 2^-500, coefficients outside
// the fixed-point range, concentrations whose scaled products would not be normal, NaN).
template <int G, bool MIXED>
__device__ __noinline__ void reactions_direct(const MechView& m, const SlotPtrs& s, double T, double invT, double lnT,
                                              double lnRTp, bool coop_tb, bool cache, CellScalars* cs) {
  const Grp<G> g;
  const int ns = m.ns;
  for (int j = g.lane; j < m.nr; j += G) {
    const uint32_t sl = m.slots[j];
    const int ra = sl & 255, rb = (sl >> 8) & 255, pa = (sl >> 16) & 255, pb = sl >> 24;
    const int meta = m.meta[j];
    const int kind = meta & 3;
    const bool rev = (meta >> 2) & 1;
    const double lnk = fma(-m.EaR[j], invT, fma(m.bexp[j], lnT, m.lnA[j]));
    double k = exp_fast(lnk, m.etab);
    const double Pf = __dmul_rn(s.C[ra], s.C[rb]);
    double Rb = 0.0, rfac = 0.0, PfRb = Pf;  // prod C^nu'' / Kc, 1/Kc and Pf - Rb
    if (rev) {
      // ln E with ln(RT/p_ref) in it: its dnu multiples come out of the differences
      rfac = exp_fast((s.gRT[pa] - s.gRT[ra]) + (s.gRT[pb] - s.gRT[rb]), m.etab);
      Rb = __dmul_rn(rfac, __dmul_rn(s.C[pa], s.C[pb]));
      PfRb = __dsub_rn(Pf, Rb);
    }
    double mfac = 1.0;
    double dlnk = 0.0;  // d ln k / dT (cache only)
    if (cache) dlnk = __dmul_rn(fma(m.EaR[j], invT, m.bexp[j]), invT);
    if (kind != 0) {
      const int slot = meta >> 8;
      const double Mc = third_body_conc<G>(m, s, slot, coop_tb);
      double dkdM = 0.0;
      if (kind == 1) {
        mfac = Mc;
      } else {
        // Troe: the multiplier and derivatives from the falloff passes above
        // (Troe reactions hold slots 0..ntroe-1)
        if (cache) {
          dlnk = s.tro[7 * m.ntroe + slot];
          dkdM = k * s.tro[8 * m.ntroe + slot];
        }
        k = k * s.tro[6 * m.ntroe + slot];
      }
      if (cache) cache_pressure<MIXED>(s, slot, Mc, dkdM, dlnk, rfac);
    }
    // q = m k (prod C^nu' - prod C^nu'' / Kc); the third-body factor only where there is one
    const double q0 = __dmul_rn(k, PfRb);
    double qj = q0;
    if (kind == 1) qj = __dmul_rn(mfac, qj);
    if (MIXED) reinterpret_cast<df2*>(s.q)[j] = df_from(qj);  // double-float copy for the gather
    else s.q[j] = qj;
    if (cache) {
      const double kr = __dmul_rn(k, rfac);
      // d q_j / dT at fixed concentrations (without the third-body factor):
      // d ln k/dT q0 + d ln Kc/dT k prod C^nu''/Kc, q0 = k (prod C^nu' - prod C^nu''/Kc),
      // with d ln Kc/dT = (sum_products h/RT - sum_reactants h/RT - dnu) / T
      // summed from the per-species (h/RT - 1)/T
      const double dlnKc = __dsub_rn(__dadd_rn(s.dC[pa], s.dC[pb]), __dadd_rn(s.dC[ra], s.dC[rb]));
      const double qT = fma(dlnk * T, q0, __dmul_rn(dlnKc, __dmul_rn(k, Rb)));  // T d q/dT
      cache_reaction<MIXED>(s, cs, j, k, kr, qT);
    }
  }
}

// ------------------------------------------------------------ chemistry RHS
// out = f(uu) + src (src may be null).  p > 0: constant-pressure reactor at
// pressure p; p < 0: constant-volume reactor of density -p (Eq. cv_reactor with
// internal energies u_k/RT = h_k/RT - 1 and c_v/R = c_p/R - 1 per species).  uu, out: N-vectors in shared memory
// (out may be uu itself, except in the auxiliary-temperature system).  When `cache` is set, the values the analytic
// Jacobian-vector product reuses are kept (rate coefficients, w, d(cp/R)/dT
// and the cell scalars).  Inlined into the 32-lane FP64 integrator and called
// through rhs_eval_call elsewhere; each product that meets a sum is written as
// an explicit fma or __dmul_rn, so no copy can contract it differently,
// chem_rhs and the integrator compute the same bits and R(u) - R(u) is
// exactly zero in a steady-state cell.
template <int G, bool MIXED = false, bool TC = false>
__device__ __forceinline__ void rhs_eval(const MechView& m, const SlotPtrs& s, const double* uu,
                                      const double* src, double p, double* out, bool cache,
                                      CellScalars* cs) {
  const Grp<G> g;
  const int ns = m.ns;
  const double T = uu[ns];
  const double invT = rcp_state(T);
  // log2 T in fixed point gives ln T (0.6 ulp) and the rate constants' T^b
  const bool t_fx = below(T, fx::T_HI) && !below(T, fx::T_LO);
  uint64_t lgT = 0;
  double lnT;
  if (t_fx) {
    lgT = fx::log2_fixed(T, c_fx_inv_c, c_fx_log2_c);
    lnT = fx::from_fixed59(fx::mulhi(lgT, RK_FX_LN2));
  } else {
    lnT = log_fast(T);
  }
  const double lnRTp = LN_R_OVER_PREF + lnT;  // ln(R T / p_ref)
  // species pass 1: thermo, Gibbs factors, sum Y/W
  // T times the factors 2/3, 3/4, 4/5, 3/2, 4/3 of the nested polynomials, one a lane
  // (G >= 8 lanes) and one FP64 multiplication for all
  double th, t21, t23, t34, t45, t32, t43;
  {
    const int l = g.lane & 7;
    const double f = l == 0 ? 2.0 / 3.0 : l == 1 ? 0.75 : l == 2 ? 0.8 : l == 3 ? 1.5 : l == 4 ? 4.0 / 3.0 : 0.5;
    const double t = __dmul_rn(T, f);
    t23 = __shfl_sync(g.mask, t, 0, G);
    t34 = __shfl_sync(g.mask, t, 1, G);
    t45 = __shfl_sync(g.mask, t, 2, G);
    t32 = __shfl_sync(g.mask, t, 3, G);
    t43 = __shfl_sync(g.mask, t, 4, G);
    th = __shfl_sync(g.mask, t, 5, G);
    t21 = cache ? 2.0 * T : 0.0;
  }
  double S = 0.0;
  double Ds = 0.0;  // sum Y_k (dcp_k/R/dT) / W_k (caching only)
  int ghi = 0;  // max over species of the high word of |g/RT + ln(RT/p_ref)| (integer compare)
  unsigned thin = 0xffffffffu;  // min over species present of the exponents of C and C E, less rho's
  for (int k = g.lane; k < ns; k += G) {
    const double* c = below(T, m.Tmid[k]) ? m.lo : m.hi;
    const double a1 = c[k], a2 = c[ns + k], a3 = c[2 * ns + k], a4 = c[3 * ns + k], a5 = c[4 * ns + k];
    // nested with the polynomials' factors in multiples of T: seven coefficients a range
    const double cp = fma(fma(fma(fma(a5, T, a4), T, a3), T, a2), T, a1);
    const double hp = fma(fma(fma(fma(a5, t45, a4), t34, a3), t23, a2), th, a1);
    const double hrt = fma(c[5 * ns + k], invT, hp);
    const double sp = fma(fma(fma(a5, t34, a4), t23, a3), th, a2);
    const double sr = fma(a1, lnT, fma(sp, T, c[6 * ns + k]));
    const double grt = hrt - sr;
    s.cp[k] = cp;
    s.hRT[k] = hrt;
    const double a = grt + lnRTp;  // ln E
    s.gRT[k] = a;
    ghi = max(ghi, __double2hiint(a) & 0x7fffffff);
    thin = ::min(thin, scaled_exponent(uu[k], m.invW[k], a));
    if (cache) {
      const double dcp = fma(fma(fma(a5, t43, a4), t32, a3), t21, a2);
      Ds = fma(__dmul_rn(uu[k], dcp), m.invW[k], Ds);
      // h/RT - 1, whose sum over a reaction's products less its reactants is
      // T d ln Kc/dT; kept in dC, which the J v overwrites later (sentinel entry 0)
      s.dC[k] = hrt - 1.0;
      if (MIXED) {
        s.fh[k] = __double2float_rn(hrt);
        s.fcp[k] = __double2float_rn(cp);
        s.fdcp[k] = __double2float_rn(dcp);
      }
    }
    S = fma(uu[k], m.invW[k], S);
  }
  S = g.sum(S);
  ghi = g.imax(ghi);
  thin = g.umin(thin);
  // auxiliary-temperature system (Eq. chemical_source_balanced): the species
  // components are rho Y_k, so C_k = u_k / W_k and d(rho Y_k)/dt = W_k w_k:
  // the constant-volume arithmetic with unit density
  const bool aux = m.nx > 0;
  const bool cv = __double2hiint(p) < 0 || aux;  // p < 0 (never -0 or NaN)
  const double invS = rcp_state(S);
  // rho = p / (R T S), 1/rho = R T S / p, with 1/p (or 1/rho) from the caller
  const double rho = aux ? 1.0 : (cv ? -p : p * invT * invS * INV_R);
  const double invrho = aux ? 1.0 : (cv ? cs->pinv : R_GAS * T * S * cs->pinv);
  // the scaled form of the reactions holds while every |g/RT + ln(RT/p_ref)| < 170
  // (false for NaN too), T is inside the mechanism's fixed-point range and no C or C E
  // that is not zero lies below 2^-480, so that their products are normal numbers
  const bool zf = m.fx && ghi < G_OVERFLOW_HI && t_fx && __double_as_longlong(T) >= __double_as_longlong(m.fx_T_lo) &&
                  (thin == 0xffffffffu || thin + (((unsigned)__double2hiint(rho) >> 20) & 0x7ffu) >= THIN_MIN);
  // concentrations, Gibbs factors, and (for up to MAXM pressure-dependent
  // reactions) the third-body concentrations [M]_t = sum_k eff_tk C_k
  const bool coop_tb = m.ntb > 0 && m.ntb <= MAXM;
  double mp[MAXM];
#pragma unroll
  for (int t = 0; t < MAXM; ++t) mp[t] = 0.0;
  for (int k = g.lane; k < ns; k += G) {
    const double Ck = rho * uu[k] * m.invW[k];
    s.C[k] = Ck;
    if (MIXED && cache) s.fC[k] = __double2float_rn(Ck);
    if (cache && cs->prec == 3) s.C2[k] = df_from(Ck);
    if (zf) {
      // A = ln E log2 e in fixed point, E = e^{g/RT} (RT/p_ref) = 2^A and z = C E; A
      // replaces ln E.  z and the A of a rate constant come from one rounded A,
      // so its rounding cancels between the two
      const uint64_t A = fx::log2e_fixed(s.gRT[k]);
      const double E = fx::exp2_double(A, m.etab);
      reinterpret_cast<uint64_t*>(s.gRT)[k] = A;
      s.E[k] = E;
      s.CE[k] = __dmul_rn(Ck, E);
    }
    if (coop_tb) {
#pragma unroll
      for (int t = 0; t < MAXM; ++t)
        if (t < m.ntb) mp[t] = fma(m.eff[t * ns + k], Ck, mp[t]);
    }
  }
  if (coop_tb) {
    sum_first<G>(g, mp, m.ntb);
    if (g.lane == 0) {
#pragma unroll
      for (int t = 0; t < MAXM; ++t)
        if (t < m.ntb) s.tb[4 * t] = mp[t];
    }
  }
  g.sync();
  // Troe falloff factors (Sec. 4.4 kinetics; F_cent, Pr, F), spread over the
  // lanes in three passes instead of one lane per reaction running the whole
  // chain: (A) the four exponentials of each reaction, k0/k_inf, e^{-T/T***},
  // e^{-T/T*}, e^{-T**/T}; (B) log10 F_cent and log10 Pr; (C) F, the falloff
  // multiplier Pr/(1+Pr) F and, when caching, d ln k/dT and dk/d[M] / k_inf.
  // Scratch tro (nt = ntroe): [0,4nt) exponentials, [4nt,6nt) logs,
  // [6nt,7nt) multiplier, [7nt,8nt) d ln k/dT, [8nt,9nt) dk/d[M] / k_inf,
  // [9nt,11nt) F_cent and Pr.
  const int nt = m.ntroe;
  if (nt > 0) {
    double* tro = s.tro;
    for (int l = g.lane; l < 4 * nt; l += G) {
      const int i = l >> 2, c = l & 3;
      const double* fo = m.fo + (size_t)i * FO_STRIDE;
      double x;
      if (c == 0) {
        const double lnk_inf = fma(-m.EaR[i], invT, fma(m.bexp[i], lnT, m.lnA[i]));
        x = fma(-fo[2], invT, fma(fo[1], lnT, fo[0])) - lnk_inf;  // ln(k0 / k_inf)
      } else if (c == 1) {
        x = -T * fo[4];
      } else if (c == 2) {
        x = -T * fo[5];
      } else {
        x = fo[6] > 0.0 ? -fo[6] * invT : 0.0;
      }
      const double ex = exp_fast(x, m.etab);
      tro[l] = (c == 3 && !(fo[6] > 0.0)) ? 0.0 : ex;
    }
    g.sync();
    for (int l = g.lane; l < 2 * nt; l += G) {
      const int i = l >> 1;
      const double* fo = m.fo + (size_t)i * FO_STRIDE;
      double y;
      if (l & 1) {
        double Mc;
        if (coop_tb) {
          Mc = s.tb[4 * i];
        } else {
          const double* e = m.eff + (size_t)i * ns;
          Mc = 0.0;
          for (int q = 0; q < ns; ++q) Mc = fma(e[q], s.C[q], Mc);
        }
        y = tro[4 * i] * Mc;  // Pr = [M] k0 / k_inf
        if (!(y > 1e-300)) y = 1e-300;
      } else {
        const double a = fo[3];
        y = fma(1.0 - a, tro[4 * i + 1], fma(a, tro[4 * i + 2], tro[4 * i + 3]));  // F_cent
      }
      tro[9 * nt + l] = y;
      tro[4 * nt + l] = __dmul_rn(log_fast(y), RK_INV_LN10);
    }
    g.sync();
    for (int i = g.lane; i < nt; i += G) {
      const double lFc = tro[4 * nt + 2 * i], lPr = tro[4 * nt + 2 * i + 1];
      const double Fc = tro[9 * nt + 2 * i], Pr = tro[9 * nt + 2 * i + 1];
      const double cc = fma(-0.67, lFc, -0.4);
      const double nn = fma(-1.27, lFc, 0.75);
      const double x = lPr + cc;
      const double D = fma(-0.14, x, nn);
      // one division for 1/(1 + Pr) and 1/(D^2 + x^2):
      //   1/(1 + f1^2) = D^2/(D^2 + x^2) with f1 = x / D
      const double s2 = fma(D, D, x * x);
      const double onePr = 1.0 + Pr;
      const double qd = rcp_any(__dmul_rn(onePr, s2));
      const double iOnePr = s2 * qd;
      const double rr = onePr * qd;  // 1 / (D^2 + x^2)
      const double iden = D * D * rr;
      const double F = exp_fast(lFc * iden * 2.302585092994046, m.etab);  // 10^(lFc / (1 + f1^2))
      tro[6 * nt + i] = Pr * iOnePr * F;
      if (cache) {  // d ln k / dT and d k / d[M] for the analytic J v
        const double* fo = m.fo + (size_t)i * FO_STRIDE;
        const double a = fo[3];
        const double er = tro[4 * i], e3 = tro[4 * i + 1], e1 = tro[4 * i + 2], e2 = tro[4 * i + 3];
        const double dlnk_inf = __dmul_rn(fma(m.EaR[i], invT, m.bexp[i]), invT);
        const double dlnk0 = __dmul_rn(fma(fo[2], invT, fo[1]), invT);
        // d ln F / d log10 Pr = -2 lFc f1 n / (D^2 (1 + f1^2)^2) and
        // d log10 F / d lFc = 1/(1 + f1^2) - 2 lFc f1 (df1/dlFc) / (1 + f1^2)^2,
        // df1/dlFc = (-0.67 D + 1.1762 x) / D^2, written with rr = 1/(D^2 + x^2)
        // (every product that meets a sum is an explicit fma or __dmul_rn, so
        // the compiler cannot contract it differently where this is inlined)
        const double w = __dmul_rn(__dmul_rn(__dmul_rn(__dmul_rn(__dmul_rn(2.0, lFc), x), D), rr), rr);
        const double gg = fma(-w, nn, iOnePr);
        const double dlF_dlFc = fma(-w, fma(-0.67, D, __dmul_rn(1.1762, x)), iden);
        const double e2t = fo[6] > 0.0 ? __dmul_rn(__dmul_rn(__dmul_rn(fo[6], invT), invT), e2) : 0.0;
        const double dFc = fma(-(1.0 - a), __dmul_rn(fo[4], e3), fma(-a, __dmul_rn(fo[5], e1), e2t));
        tro[7 * nt + i] = fma(__dmul_rn(dlF_dlFc, dFc), rcp_any(Fc), fma(gg, dlnk0 - dlnk_inf, dlnk_inf));
        tro[8 * nt + i] = er * F * iOnePr * gg;  // (dk/d[M]) / k_inf
      }
    }
    g.sync();
  }
  // reactions: rate coefficients and rates of progress
  RateRange range;
  if (zf) {
    const fx::Temp ft = fx::temperature(lgT, fx::recip_fixed70(T, invT));
    int j0 = 0;
    for (; j0 < m.ntb; j0 += G)
      reactions_scaled<G, MIXED, true>(m, s, ft, T, invT, coop_tb, cache, cs, j0, g.lane, &range);
    for (; j0 < m.nr; j0 += G)
      reactions_scaled<G, MIXED, false>(m, s, ft, T, invT, coop_tb, cache, cs, j0, g.lane, &range);
  } else {
    reactions_direct<G, MIXED>(m, s, T, invT, lnT, lnRTp, coop_tb, cache, cs);
  }
  g.sync();
  // species pass 2: w = nu^T q, dY/dt and the sums of the temperature equation
  double Sh = 0.0, cb = 0.0;
  const bool zjv = zf && !MIXED && cs->prec != 3 && cs->prec != 6;
  double Hs = 0.0;
  double Ax = 0.0, Bx = 0.0;  // auxiliary T: sum (u_k/RT) F_k / W_k and sum (cv_k/R) F_k / W_k
  bool tc_om = false;  // w already in part[0..ns) from the tensor cores
  if constexpr (TC) tc_om = gather_tc<G>(m, s, s.q, s.part);
  // in fixed point, except where krc's storage is taken (by the caches of the
  // direct form and of precision 3), a rate is not finite or a row is out of reach
  Gathered how = ROWS_IN_PART;
  if (MIXED) {
    gather_pieces_df<G>(m, g.lane, reinterpret_cast<const df2*>(s.q), reinterpret_cast<df2*>(s.part));
    g.sync();
  } else if (!tc_om) {
    bool again = false;
    how = NOT_GATHERED;
    if (zf && !(cache && cs->prec == 3)) how = m.gfix ? gather_fixed<G>(m, s, range, &again) : gather_listed<G>(m, s);
    if (again) how = rates_listed_call<G>(m, s, lgT, T, invT, coop_tb);
    if (how == NOT_GATHERED) how = m.seg ? gather_listed_call<G>(m, s) : gather_rows<G>(m, s);
  }
  for (int k = g.lane; k < ns; k += G) {
    double om;
    if (MIXED) {
      om = piece_sum_df(m, reinterpret_cast<const df2*>(s.part), k);
      if (cache) s.fom[k] = __double2float_rn(om);
    } else {
      om = gathered_row(m, s, k, how);
    }
    if (cache) s.om[k] = om;
    const double r = __dmul_rn(__dmul_rn(m.W[k], om), invrho);
    const double Fk = src ? __dadd_rn(r, src[k]) : r;
    double hk = s.hRT[k], ck = s.cp[k];
    const double ufac = uu[k];
    out[k] = Fk;  // (out may be uu)
    if (cv) {  // internal energies and cv (uniform; the subtractions cost 64 cycles each)
      hk -= 1.0;
      ck -= 1.0;
    }
    Sh = fma(hk, om, Sh);
    cb = fma(ufac * ck, m.invW[k], cb);
    if (aux) {
      Ax = fma((s.hRT[k] - 1.0) * Fk, m.invW[k], Ax);
      Bx = fma((s.cp[k] - 1.0) * Fk, m.invW[k], Bx);
    }
    if (cache) {
      // per-species factors of the analytic J v, written over arrays the
      // remaining RHS no longer reads (lane-private entries k):
      //   E: rho/W_k (times E_k for the scaled J v)   hRT: h_k/RT (u_k/RT at fixed volume)
      //   cp: (cp_k/R, or cv_k/R) / W_k
      // and the sum of (cp_k/R - h_k/RT) w_k / T
      Hs = fma((s.cp[k] - s.hRT[k]) * invT, om, Hs);
      const double rW = rho * m.invW[k];
      s.E[k] = zjv ? s.E[k] * rW : rW;
      if (cv) s.hRT[k] = hk;
      s.cp[k] = ck * m.invW[k];
      if (cs->prec == 6) {  // FP32 copies for the FP32 J v
        s.xC[k] = __double2float_rn(s.C[k]);
        s.xE[k] = __double2float_rn(rW);
        s.xEinv[k] = __double2float_rn(m.W[k] * invrho);
        s.xom[k] = __double2float_rn(om);
        s.xg[k] = __double2float_rn(hk);
        s.xcp[k] = __double2float_rn(s.cp[k]);
      }
    }
  }
  if (aux) {
    double t4[4] = {Sh, cb, Ax, Bx};
    sum_many<G, 4>(g, t4);
    Sh = t4[0];
    cb = t4[1];
    Ax = t4[2];
    Bx = t4[3];
    if (cache) {
      double t2[2] = {Hs, Ds};
      sum_many<G, 2>(g, t2);
      Hs = t2[0];
      Ds = t2[1];
    }
  } else if (cache) {
    double t4[4] = {Sh, cb, Hs, Ds};
    sum_many<G, 4>(g, t4);
    Sh = t4[0];
    cb = t4[1];
    Hs = t4[2];
    Ds = t4[3];
  } else {
    double t2[2] = {Sh, cb};
    sum_many<G, 2>(g, t2);
    Sh = t2[0];
    cb = t2[1];
  }
  const double invcb = rcp_state(cb);
  double fT = 0.0;
  if (aux) {
    // Eq. aux_t_equation with specific internal energies e_k = (u_k/RT) R T / W_k
    // and rho c_v = R cb:  w_T = (-R T Ax + |v|^2/2 d(rho)/dt - v . d(rho v)/dt
    //                              + d(rho E)/dt) / (R cb)
    const double irc = 1.0 / uu[ns + 1];
    const double v0 = uu[ns + 2] * irc, v1 = uu[ns + 3] * irc, v2 = uu[ns + 4] * irc;
    double X = 0.0;
    if (src) {
      const double kin = 0.5 * fma(v0, v0, fma(v1, v1, v2 * v2));
      X = fma(kin, src[ns + 1], src[ns + 5]) - fma(v0, src[ns + 2], fma(v1, src[ns + 3], v2 * src[ns + 4]));
    }
    fT = fma(-T, Ax, X * INV_R) * invcb;
    if (cache) {
      cs->B = Bx;
      cs->fT = fT;
      cs->irho_c = irc;
      cs->vel[0] = v0;
      cs->vel[1] = v1;
      cs->vel[2] = v2;
    }
    // d(rho)/dt, d(rho v)/dt, d(rho E)/dt: the balancing constants alone
    for (int e = ns + 1 + g.lane; e < ns + 1 + m.nx; e += G) out[e] = src ? src[e] : 0.0;
  }
  if (g.lane == 0) {
    const double r = aux ? fT : -T * Sh * invrho * invcb;
    out[ns] = src ? __dadd_rn(r, src[ns]) : r;
    if (cache && cs->prec == 6) s.xC[ns] = 1.f;  // the empty reaction slot
  }
  if (cache) {
    cs->T = T;
    cs->invT = invT;
    cs->lnT = lnT;
    cs->S = S;
    cs->invS = invS;
    cs->rho = rho;
    cs->invrho = invrho;
    cs->cb = cb;
    cs->invcb = invcb;
    cs->Sh = Sh;
    cs->TSh = T * Sh;
    cs->Hs = Hs;
    cs->Ds = Ds;
    cs->irc = invrho * invcb;
    cs->cv = cv;
    cs->zf = zjv;
  }
  g.sync();
}

// rhs_eval behind a call, where its size matters more than the call: the
// point kernels, the finite-difference J v, the explicit integrator's first
// evaluation and the 8/16-lane and mixed variants of the integrator (one
// inlined copy per call site would multiply the compile time).  Same bits as
// the inlined copies.
template <int G, bool MIXED = false, bool TC = false>
__device__ __noinline__ void rhs_eval_call(const MechView& m, const SlotPtrs& s, const double* uu,
                                           const double* src, double p, double* out, bool cache,
                                           CellScalars* cs) {
  rhs_eval<G, MIXED, TC>(m, s, uu, src, p, out, cache, cs);
}
template <int G, bool MIXED, bool INL, bool TC = false>
__device__ __forceinline__ void rhs_dispatch(const MechView& m, const SlotPtrs& s, const double* uu,
                                             const double* src, double p, double* out, bool cache,
                                             CellScalars* cs) {
  if constexpr (INL) rhs_eval<G, MIXED, TC>(m, s, uu, src, p, out, cache, cs);
  else rhs_eval_call<G, MIXED, TC>(m, s, uu, src, p, out, cache, cs);
}

// d[M] of a pressure-dependent reaction from dC: summed over the species by the
// whole group (mp), or by the reaction's own lane when there are many slots.
template <int G>
__device__ __forceinline__ double third_body_rate(const MechView& m, const double* dC, int slot, bool coop_tb,
                                                  const double (&mp)[MAXM]) {
  double dM = 0.0;
  if (coop_tb) {
#pragma unroll
    for (int q = 0; q < MAXM; ++q)
      if (q == slot) dM = mp[q];
  } else {
    const double* e = m.eff + (size_t)slot * m.ns;
    for (int q = 0; q < m.ns; ++q) dM = fma(e[q], dC[q], dM);
  }
  return dM;
}

// dq_j = T d q_j/dT vTT + kappa_j d(z_ra z_rb - z_pa z_pb), vTT = vT / T, of reaction
// j0 + lane (as reactions_scaled): six FP64 instructions.
template <int G, bool PRESSURE>
__device__ __forceinline__ void jvp_scaled(const MechView& m, const SlotPtrs& s, double vTT, bool coop_tb,
                                           const double (&mp)[MAXM], int j0, int lane, RateRange* range) {
  const int j = min(j0 + lane, m.nr - 1);
  const uint32_t sl = m.slots[j];
  const int ra = sl & 255, rb = (sl >> 8) & 255, pa = (sl >> 16) & 255, pb = sl >> 24;
  const int meta = m.meta[j];
  const bool rev = (meta >> 2) & 1;
  const double za = s.CE[ra], zb = s.CE[rb], zp = s.CE[pa], zq = s.CE[pb];
  const double dD0 = fma(s.dC[ra], zb, za * s.dC[rb]);
  const double dD1 = fma(-s.dC[pa], zq, fma(-zp, s.dC[pb], dD0));
  const double kap = s.kc[j];
  double dq = fma(s.qT[j], vTT, kap * (rev ? dD1 : dD0));
  if (PRESSURE && (meta & 3) != 0) {
    const int slot = meta >> 8;
    const double* t = s.tb + 4 * slot;
    double D = za * zb;
    if (rev) D = fma(-zp, zq, D);
    const double dM = third_body_rate<G>(m, s.arg, slot, coop_tb, mp);
    dq = (meta & 3) == 1 ? t[0] * dq + dM * (kap * D) : dq + t[1] * dM * D;
  }
  range->take(dq);
  if (j0 + lane < m.nr) s.q[j] = dq;
}

// The same again and their rows in FP64 (as rates_listed_call).
template <int G>
__device__ __noinline__ Gathered products_listed_call(const MechView& m, const SlotPtrs& s, double vTT, bool coop_tb,
                                                      const double (&mp)[MAXM]) {
  const Grp<G> g;
  RateRange range;
  for (int j0 = 0; j0 < m.nr; j0 += G) jvp_scaled<G, true>(m, s, vTT, coop_tb, mp, j0, g.lane, &range);
  g.sync();
  return gather_listed<G>(m, s);
}
// The reaction rates' derivatives from k and k/Kc (caches not in the scaled form).
template <int G, bool DFG>
__device__ __forceinline__ void jvp_reactions(const MechView& m, const SlotPtrs& s, double vTT, bool coop_tb,
                                              const double (&mp)[MAXM]) {
  const Grp<G> g;
  for (int j = g.lane; j < m.nr; j += G) {
    const uint32_t sl = m.slots[j];
    const int ra = sl & 255, rb = (sl >> 8) & 255, pa = (sl >> 16) & 255, pb = sl >> 24;
    const int meta = m.meta[j];
    const int kind = meta & 3;
    const double dPf = fma(s.dC[ra], s.C[rb], s.C[ra] * s.dC[rb]);
    const double dPb = fma(s.dC[pa], s.C[pb], s.C[pa] * s.dC[pb]);
    const double k = s.kc[j], kr = s.krc[j];
    double dq = fma(s.qT[j], vTT, fma(k, dPf, -kr * dPb));
    if (kind != 0) {
      const int slot = meta >> 8;
      const double* t = s.tb + 4 * slot;
      const double Pf = s.C[ra] * s.C[rb];
      const double Pb = s.C[pa] * s.C[pb];
      const double dM = third_body_rate<G>(m, s.dC, slot, coop_tb, mp);
      if (kind == 1) dq = t[0] * dq + dM * (k * Pf - kr * Pb);
      else dq = dq + t[1] * dM * (Pf - t[3] * Pb);
    }
    if (DFG) reinterpret_cast<df2*>(s.q)[j] = df_from(dq);
    else s.q[j] = dq;
  }
}
template <int G>
__device__ __noinline__ void jvp_reactions_call(const MechView& m, const SlotPtrs& s, double vTT, bool coop_tb,
                                                const double (&mp)[MAXM]) {
  jvp_reactions<G, false>(m, s, vTT, coop_tb, mp);
}

// Analytic Jacobian-vector product out = J(u_n) v, using the values cached by
// the last rhs_eval(..., cache = true) at u_n.  v, out: N-vectors.  Inlined
// (unlike rhs_eval, nothing requires two call sites to produce the same bits),
// which saves the call's register save and restore four times per attempt.
template <int G, bool DFG = false, bool TC = false>
__device__ __forceinline__ void jvp_eval(const MechView& m, const SlotPtrs& s, const double* uu,
                                      const CellScalars& cs, const double* v, double* out) {
  const Grp<G> g;
  const int ns = m.ns;
  const double vT = v[ns];
  const double T = cs.T, invT = cs.invT;
  double a = 0.0;
  for (int k = g.lane; k < ns; k += G) a = fma(v[k], m.invW[k], a);
  a = g.sum(a);
  const double vTT = vT * invT;
  const double drr = cs.cv ? 0.0 : -fma(a, cs.invS, vTT);  // d rho / rho (0 at fixed volume)
  const bool coop_tb = m.ntb > 0 && m.ntb <= MAXM;
  const bool zf = !DFG && cs.zf;
  double mp[MAXM];
#pragma unroll
  for (int t = 0; t < MAXM; ++t) mp[t] = 0.0;
  for (int k = g.lane; k < ns; k += G) {
    const double ev = s.E[k] * v[k];  // E: rho / W_k, scaled form: E_k rho / W_k
    // dC, or dz = E dC in the scaled form
    const double d = fma(zf ? s.CE[k] : s.C[k], drr, ev);
    s.dC[k] = d;
    if (m.ntb > 0) {
      const double dCk = zf ? fma(s.C[k], drr, cs.rho * m.invW[k] * v[k]) : d;
      if (zf) s.arg[k] = dCk;
      if (coop_tb) {
#pragma unroll
        for (int t = 0; t < MAXM; ++t)
          if (t < m.ntb) mp[t] = fma(m.eff[t * ns + k], dCk, mp[t]);
      }
    }
  }
  if (coop_tb) sum_first<G>(g, mp, m.ntb);  // d[M]_t, identical on every lane
  g.sync();
  RateRange range;
  if (zf) {
    int j0 = 0;
    for (; j0 < m.ntb; j0 += G) jvp_scaled<G, true>(m, s, vTT, coop_tb, mp, j0, g.lane, &range);
    for (; j0 < m.nr; j0 += G) jvp_scaled<G, false>(m, s, vTT, coop_tb, mp, j0, g.lane, &range);
  } else if constexpr (DFG) {
    jvp_reactions<G, true>(m, s, vTT, coop_tb, mp);
  } else {
    jvp_reactions_call<G>(m, s, vTT, coop_tb, mp);
  }
  g.sync();
  bool tc_om = false;  // d w already in part[0..ns) from the tensor cores
  if constexpr (TC) tc_om = gather_tc<G>(m, s, s.q, s.part);
  Gathered how = ROWS_IN_PART;
  if (DFG) {
    gather_pieces_df<G>(m, g.lane, reinterpret_cast<const df2*>(s.q), reinterpret_cast<df2*>(s.part));
    g.sync();
  } else if (!tc_om) {
    bool again = false;
    how = NOT_GATHERED;
    if (zf) how = m.gfix ? gather_fixed<G>(m, s, range, &again) : gather_listed<G>(m, s);
    if (again) how = products_listed_call<G>(m, s, vTT, coop_tb, mp);
    if (how == NOT_GATHERED) how = m.seg ? gather_listed_call<G>(m, s) : gather_rows<G>(m, s);
  }
  double dSh = 0.0, dcb = 0.0;
  for (int k = g.lane; k < ns; k += G) {
    const double dom = DFG ? piece_sum_df(m, reinterpret_cast<const df2*>(s.part), k)
                           : gathered_row(m, s, k, how);
    out[k] = m.W[k] * cs.invrho * fma(-s.om[k], drr, dom);
    dSh = fma(s.hRT[k], dom, dSh);
    dcb = fma(s.cp[k], v[k], dcb);
  }
  if (m.nx > 0) {
    // auxiliary temperature: d w_T = (-vT B - T sum_k (u_k/RT) dF_k/W_k + dX/R - w_T dcb) / cb,
    // dF_k = W_k dw_k, X = |v|^2/2 S_rho - v . S_m + S_E, dv = (d(rho v) - v d rho) / rho
    double D1 = 0.0;
    for (int k = g.lane; k < ns; k += G) D1 = fma(s.hRT[k], out[k] * m.invW[k], D1);  // hRT: h/RT - 1
    double t2[2] = {D1, dcb};
    sum_many<G, 2>(g, t2);
    D1 = t2[0];
    dcb = fma(cs.Ds, vT, t2[1]);
    if (g.lane == 0) {
      const double irc = cs.irho_c;
      const double dv0 = (v[ns + 2] - cs.vel[0] * v[ns + 1]) * irc;
      const double dv1 = (v[ns + 3] - cs.vel[1] * v[ns + 1]) * irc;
      const double dv2 = (v[ns + 4] - cs.vel[2] * v[ns + 1]) * irc;
      const double* S = s.src;  // the cell's balancing constants
      const double dX = fma(dv0, fma(cs.vel[0], S[ns + 1], -S[ns + 2]),
                            fma(dv1, fma(cs.vel[1], S[ns + 1], -S[ns + 3]), dv2 * fma(cs.vel[2], S[ns + 1], -S[ns + 4])));
      out[ns] = (fma(-vT, cs.B, fma(-T, D1, dX * INV_R)) - cs.fT * dcb) * cs.invcb;
    }
    for (int e = ns + 1 + g.lane; e < ns + 1 + m.nx; e += G) out[e] = 0.0;
    g.sync();
    return;
  }
  {
    double t2[2] = {dSh, dcb};
    sum_many<G, 2>(g, t2);
    dSh = fma(cs.Hs, vT, t2[0]);
    dcb = fma(cs.Ds, vT, t2[1]);
  }
  if (g.lane == 0) {
    out[ns] = fma(cs.TSh, fma(dcb, cs.invcb, drr), -fma(vT, cs.Sh, T * dSh)) * cs.irc;
  }
  g.sync();
}

// Analytic J v with its reaction-level core in double-float (precision 3):
// dP = d(C_a C_b), dq_j = qT_j vT + k_j dPf - kr_j dPb and the gather
// dw = nu^T dq run on the FP32 pipe with ~44-bit significands from the
// double-float copies rhs_eval wrote at u_n; the species and temperature rows
// (and the third-body / falloff corrections) stay FP64.  Same derivative as
// jvp_eval to ~1e-13 relative, so the Krylov basis is that of the FP64 path.
template <int G>
__device__ __forceinline__ void jvp_eval_df(const MechView& m, const SlotPtrs& s, const double* uu,
                                         const CellScalars& cs, const double* v, double* out) {
  const Grp<G> g;
  const int ns = m.ns;
  const double vT = v[ns];
  const double T = cs.T, invT = cs.invT;
  double a = 0.0;
  for (int k = g.lane; k < ns; k += G) a = fma(v[k], m.invW[k], a);
  a = g.sum(a);
  const double drr = cs.cv ? 0.0 : -fma(a, cs.invS, vT * invT);
  const bool coop_tb = m.ntb > 0 && m.ntb <= MAXM;
  double mp[MAXM];
#pragma unroll
  for (int t = 0; t < MAXM; ++t) mp[t] = 0.0;
  for (int k = g.lane; k < ns; k += G) {
    const double dCk = fma(s.C[k], drr, s.E[k] * v[k]);  // E: rho / W_k
    s.dC[k] = dCk;
    s.dC2[k] = df_from(dCk);
    if (coop_tb) {
#pragma unroll
      for (int t = 0; t < MAXM; ++t)
        if (t < m.ntb) mp[t] = fma(m.eff[t * ns + k], dCk, mp[t]);
    }
  }
  if (coop_tb) sum_first<G>(g, mp, m.ntb);
  g.sync();
  const df2 vT2 = df_from(vT * invT);  // qT holds T d q/dT
  const df2* k2 = reinterpret_cast<const df2*>(s.kc);
  const df2* kr2 = reinterpret_cast<const df2*>(s.krc);
  const df2* qT2 = reinterpret_cast<const df2*>(s.qT);
  df2* dq2 = reinterpret_cast<df2*>(s.q);
  for (int j = g.lane; j < m.nr; j += G) {
    const uint32_t sl = m.slots[j];
    const int ra = sl & 255, rb = (sl >> 8) & 255, pa = (sl >> 16) & 255, pb = sl >> 24;
    const int meta = m.meta[j];
    const int kind = meta & 3;
    const df2 dPf = df_add(df_mul(s.dC2[ra], s.C2[rb]), df_mul(s.C2[ra], s.dC2[rb]));
    const df2 dPb = df_add(df_mul(s.dC2[pa], s.C2[pb]), df_mul(s.C2[pa], s.dC2[pb]));
    df2 dq = df_add(df_mul(qT2[j], vT2), df_add(df_mul(k2[j], dPf), df_neg(df_mul(kr2[j], dPb))));
    if (kind != 0) {  // third body / falloff: the [M] terms in FP64
      const int slot = meta >> 8;
      const double* t = s.tb + 4 * slot;
      const double Pf = s.C[ra] * s.C[rb];
      const double Pb = s.C[pa] * s.C[pb];
      double dM = 0.0;
      if (coop_tb) {
#pragma unroll
        for (int q = 0; q < MAXM; ++q)
          if (q == slot) dM = mp[q];
      } else {
        const double* e = m.eff + (size_t)slot * ns;
        for (int q = 0; q < ns; ++q) dM = fma(e[q], s.dC[q], dM);
      }
      const double dqd = df_to(dq);
      double r;
      if (kind == 1) r = t[0] * dqd + dM * (df_to(k2[j]) * Pf - df_to(kr2[j]) * Pb);
      else r = dqd + t[1] * dM * (Pf - t[3] * Pb);
      dq = df_from(r);
    }
    dq2[j] = dq;
  }
  g.sync();
  gather_pieces_df<G>(m, g.lane, dq2, reinterpret_cast<df2*>(s.part));
  g.sync();
  double dSh = 0.0, dcb = 0.0;
  for (int k = g.lane; k < ns; k += G) {
    const double dom = piece_sum_df(m, reinterpret_cast<const df2*>(s.part), k);
    out[k] = m.W[k] * cs.invrho * fma(-s.om[k], drr, dom);
    dSh = fma(s.hRT[k], dom, dSh);
    dcb = fma(s.cp[k], v[k], dcb);
  }
  {
    double t2[2] = {dSh, dcb};
    sum_many<G, 2>(g, t2);
    dSh = fma(cs.Hs, vT, t2[0]);
    dcb = fma(cs.Ds, vT, t2[1]);
  }
  if (g.lane == 0) {
    out[ns] = (-(vT * cs.Sh + T * dSh) + T * cs.Sh * (drr + dcb * cs.invcb)) * (cs.invrho * cs.invcb);
  }
  g.sync();
}

// Reduced-precision analytic J v (mixed mode): the same derivative as
// jvp_eval evaluated in FP32 from the FP32 copies cached by
// rhs_eval<G, true>(..., cache = true).  v and out stay FP64 vectors.
template <int G>
__device__ __noinline__ void jvp_eval_f32(const MechView& m, const SlotPtrs& s, const double* uu,
                                          const CellScalars& cs, const double* v, double* out) {
  const Grp<G> g;
  const int ns = m.ns;
  const float vT = __double2float_rn(v[ns]);
  const float T = __double2float_rn(cs.T), invT = __double2float_rn(cs.invT);
  const float invS = __double2float_rn(cs.invS), rho = __double2float_rn(cs.rho);
  const float invrho = __double2float_rn(cs.invrho), Sh = __double2float_rn(cs.Sh);
  const float invcb = __double2float_rn(cs.invcb);
  float a = 0.f;
  for (int k = g.lane; k < ns; k += G) a = fmaf(__double2float_rn(v[k]), m.invWf[k], a);
  a = g.sum(a);
  const float drr = cs.cv ? 0.f : -fmaf(a, invS, vT * invT);
  const float esh = cs.cv ? 1.f : 0.f;
  const bool coop_tb = m.ntb > 0 && m.ntb <= MAXM;
  float mp[MAXM];
#pragma unroll
  for (int t = 0; t < MAXM; ++t) mp[t] = 0.f;
  for (int k = g.lane; k < ns; k += G) {
    const float dCk = fmaf(s.fC[k], drr, rho * __double2float_rn(v[k]) * m.invWf[k]);
    s.fdC[k] = dCk;
    if (coop_tb) {
#pragma unroll
      for (int t = 0; t < MAXM; ++t)
        if (t < m.ntb) mp[t] = fmaf(m.efff[t * ns + k], dCk, mp[t]);
    }
  }
  if (coop_tb) sum_first<G>(g, mp, m.ntb);
  g.sync();
  for (int j = g.lane; j < m.nr; j += G) {
    const uint32_t sl = m.slots[j];
    const int ra = sl & 255, rb = (sl >> 8) & 255, pa = (sl >> 16) & 255, pb = sl >> 24;
    const int meta = m.meta[j];
    const int kind = meta & 3;
    const int dnu = ((meta >> 4) & 15) - 4;
    const float Pf = s.fC[ra] * s.fC[rb];
    const float Pb = s.fC[pa] * s.fC[pb];
    const float dPf = fmaf(s.fdC[ra], s.fC[rb], s.fC[ra] * s.fdC[rb]);
    const float dPb = fmaf(s.fdC[pa], s.fC[pb], s.fC[pa] * s.fdC[pb]);
    const float k = s.fkc[j], kr = s.fkr[j];
    float dlnk = (m.bf[j] + m.EaRf[j] * invT) * invT;
    const float dnud = dnu > 0 ? 1.f : (dnu < 0 ? -1.f : 0.f);
    const float dlnKc = (s.fh[pa] + s.fh[pb] - s.fh[ra] - s.fh[rb] - dnud) * invT;
    if (kind == 2) dlnk = s.ftb[4 * (meta >> 8) + 2];
    float dq = k * fmaf(dlnk * vT, Pf, dPf) - kr * fmaf((dlnk - dlnKc) * vT, Pb, dPb);
    if (kind != 0) {
      const int slot = meta >> 8;
      const float* t = s.ftb + 4 * slot;
      float dM = 0.f;
      if (coop_tb) {
#pragma unroll
        for (int q = 0; q < MAXM; ++q)
          if (q == slot) dM = mp[q];
      } else {
        const float* e = m.efff + (size_t)slot * ns;
        for (int q = 0; q < ns; ++q) dM = fmaf(e[q], s.fdC[q], dM);
      }
      if (kind == 1) dq = t[0] * dq + dM * (k * Pf - kr * Pb);
      else dq = dq + t[1] * dM * (Pf - t[3] * Pb);
    }
    s.fq[j] = dq;
  }
  g.sync();
  for (int p = g.lane; p < m.npiece; p += G) {
    float acc = 0.f;
    for (int e = m.piece_ptr[p]; e < m.piece_ptr[p + 1]; ++e) acc = fmaf(m.csr_nuf[e], s.fq[m.csr_j[e]], acc);
    s.fpart[p] = acc;
  }
  g.sync();
  float dSh = 0.f, dcb = 0.f;
  for (int k = g.lane; k < ns; k += G) {
    float dom = 0.f;
    for (int p = m.spec_piece[k]; p < m.spec_piece[k + 1]; ++p) dom += s.fpart[p];
    const float om = s.fom[k];
    const float vk = __double2float_rn(v[k]);
    out[k] = (double)(m.Wf[k] * (dom - om * drr) * invrho);
    dSh = fmaf(s.fh[k] - esh, dom, fmaf((s.fcp[k] - s.fh[k]) * invT * vT, om, dSh));
    dcb = fmaf(fmaf(__double2float_rn(uu[k]) * s.fdcp[k], vT, vk * (s.fcp[k] - esh)), m.invWf[k], dcb);
  }
  {
    float t2[2] = {dSh, dcb};
    sum_many<G, 2>(g, t2);
    dSh = t2[0];
    dcb = t2[1];
  }
  if (g.lane == 0) out[ns] = (double)((-(vT * Sh + T * dSh) + T * Sh * (drr + dcb * invcb)) * (invrho * invcb));
  g.sync();
}

// The analytic J v of jvp_eval in FP32 arithmetic (precision level 6): the
// caching right-hand side at u_n left FP32 copies of the per-reaction k, k/Kc,
// dq/dT and of the per-species factors in the spare storage of the FP64 J v
// caches, and the intermediates -- dC, dq and the gather's partial sums -- are
// kept as FP32 in the first half of the FP64 arrays' own storage, so the slot
// layout, the mechanism copy and the occupancy are the FP64 kernel's and the
// product issues almost no FP64 instruction.  FP32's ~1e-7 rounding (amplified
// where k Pf and k/Kc Pb nearly cancel) is what the Krylov basis sees; the
// stages, the error estimate and the state update stay FP64.
template <int G>
__device__ __forceinline__ void jvp_eval_f32x(const MechView& m, const SlotPtrs& s, const double* uu,
                                              const CellScalars& cs, const double* v, double* out) {
  const Grp<G> g;
  const int ns = m.ns;
  float* fdC = reinterpret_cast<float*>(s.dC);
  float* fq = reinterpret_cast<float*>(s.q);
  float* fpart = reinterpret_cast<float*>(s.part);
  auto f = [](double x) { return __double2float_rn(x); };
  const float vT = f(v[ns]);
  const float T = f(cs.T), vTT = f(v[ns] * cs.invT);  // vT / T, rounded once
  float a = 0.f;
  for (int k = g.lane; k < ns; k += G) a = fmaf(f(v[k]), f(m.invW[k]), a);
  a = g.sum(a);
  const float drr = cs.cv ? 0.f : -fmaf(a, f(cs.invS), vTT);
  const bool coop_tb = m.ntb > 0 && m.ntb <= MAXM;
  float mp[MAXM];
#pragma unroll
  for (int t = 0; t < MAXM; ++t) mp[t] = 0.f;
  for (int k = g.lane; k < ns; k += G) {
    const float dCk = fmaf(s.xC[k], drr, s.xE[k] * f(v[k]));  // xE: rho / W_k
    fdC[k] = dCk;
    if (coop_tb) {
#pragma unroll
      for (int t = 0; t < MAXM; ++t)
        if (t < m.ntb) mp[t] = fmaf(f(m.eff[t * ns + k]), dCk, mp[t]);
    }
  }
  if (g.lane == 0) {
    fdC[ns] = 0.f;  // the empty reaction slot (its C = 1 is in xC)
    fq[m.nr] = 0.f;  // the rate that pads the pieces
  }
  if (coop_tb) sum_first<G>(g, mp, m.ntb);
  g.sync();
  for (int j = g.lane; j < m.nr; j += G) {
    const uint32_t sl = m.slots[j];
    const int ra = sl & 255, rb = (sl >> 8) & 255, pa = (sl >> 16) & 255, pb = sl >> 24;
    const int meta = m.meta[j];
    const int kind = meta & 3;
    const float Cra = s.xC[ra], Crb = s.xC[rb], Cpa = s.xC[pa], Cpb = s.xC[pb];
    const float dPf = fmaf(fdC[ra], Crb, Cra * fdC[rb]);
    const float dPb = fmaf(fdC[pa], Cpb, Cpa * fdC[pb]);
    const float k = s.xk[j], kr = s.xkr[j];
    float dq = fmaf(s.xqT[j], vTT, fmaf(k, dPf, -kr * dPb));  // xqT: T d q/dT
    if (kind != 0) {
      const int slot = meta >> 8;
      const double* t = s.tb + 4 * slot;
      const float Pf = Cra * Crb, Pb = Cpa * Cpb;
      float dM = 0.f;
      if (coop_tb) {
#pragma unroll
        for (int q = 0; q < MAXM; ++q)
          if (q == slot) dM = mp[q];
      } else {
        const double* e = m.eff + (size_t)slot * ns;
        for (int q = 0; q < ns; ++q) dM = fmaf(f(e[q]), fdC[q], dM);
      }
      if (kind == 1) dq = f(t[0]) * dq + dM * (k * Pf - kr * Pb);
      else dq = dq + f(t[1]) * dM * (Pf - f(t[3]) * Pb);
    }
    fq[j] = dq;
  }
  g.sync();
  if (m.seg) {  // d w = nu^T dq, in the fixed-point gather's pieces
    for (int p = g.lane; p < m.gnpp; p += G) {
      float acc = 0.f;
      for (int i = 0; i < m.glen; ++i) acc += fq[m.gidx[((i >> 3) * m.gnpp + p) * 8 + (i & 7)] >> 3];
      fpart[p] = acc;
    }
    g.sync();
  } else {
    gather_rows_f32<G>(m, fq, fpart);
  }
  float dSh = 0.f, dcb = 0.f;
  for (int k = g.lane; k < ns; k += G) {
    float dom = 0.f;
    if (m.seg) {
      int p = m.gspec[2 * k];
      for (; p < m.gspec[2 * k + 1]; ++p) dom += fpart[p];
      for (; p < m.gspec[2 * k + 2]; ++p) dom -= fpart[p];
    } else {
      dom = fpart[k];
    }
    out[k] = (double)(s.xEinv[k] * fmaf(-s.xom[k], drr, dom));  // xEinv: W_k / rho
    dSh = fmaf(s.xg[k], dom, dSh);
    dcb = fmaf(s.xcp[k], f(v[k]), dcb);
  }
  {
    float t2[2] = {dSh, dcb};
    sum_many<G, 2>(g, t2);
    dSh = fmaf(f(cs.Hs), vT, t2[0]);
    dcb = fmaf(f(cs.Ds), vT, t2[1]);
  }
  if (g.lane == 0) {
    const float Sh = f(cs.Sh);
    out[ns] = (double)((-(vT * Sh + T * dSh) + T * Sh * (drr + dcb * f(cs.invcb))) * (f(cs.invrho) * f(cs.invcb)));
  }
  g.sync();
}

// ----------------------------------------------------------------- helpers
template <int G>
__device__ inline double group_dot(const Grp<G>& g, const double* a, const double* b, int N) {
  double acc = 0.0;
  for (int e = g.lane; e < N; e += G) acc = fma(a[e], b[e], acc);
  return g.sum(acc);
}

// J v into out: analytic, or forward difference with the oracle's increment.
template <int G, bool MIXED = false, bool TC = false>
__device__ inline void apply_jv(const MechView& m, const SlotPtrs& s, const CellScalars& cs, int jv_mode,
                                double p, double unorm, const double* v, double* out, int* n_rhs,
                                bool fp32_jv = false) {
  const Grp<G> g;
  const int N = m.ns + 1 + m.nx;
  if (jv_mode == 0) {
    if (MIXED && fp32_jv) jvp_eval_f32<G>(m, s, s.u, cs, v, out);
    else if (!MIXED && cs.prec == 3) jvp_eval_df<G>(m, s, s.u, cs, v, out);
    else if (!MIXED && cs.prec == 6) jvp_eval_f32x<G>(m, s, s.u, cs, v, out);
    else jvp_eval<G, MIXED, TC>(m, s, s.u, cs, v, out);
    return;
  }
  const double nv = sqrt(group_dot<G>(g, v, v, N));
  if (nv == 0.0) {
    for (int e = g.lane; e < N; e += G) out[e] = 0.0;
    g.sync();
    return;
  }
  const double d = sqrt(2.220446049250313e-16) * (1.0 + unorm) / nv;
  for (int e = g.lane; e < N; e += G) s.arg[e] = s.u[e] + d * v[e];
  g.sync();
  CellScalars dummy;
  dummy.pinv = cs.pinv;
  dummy.prec = cs.prec;
  rhs_eval_call<G, MIXED, TC>(m, s, s.arg, s.src, p, out, false, &dummy);
  *n_rhs += 1;
  for (int e = g.lane; e < N; e += G) out[e] = (out[e] - s.fn[e]) / d;
  g.sync();
}

template <int G>
__device__ inline float group_dot_f(const Grp<G>& g, const double* a, const double* b, int N) {
  float acc = 0.f;
  for (int e = g.lane; e < N; e += G) acc = fmaf(__double2float_rn(a[e]), __double2float_rn(b[e]), acc);
  return g.sum(acc);
}

// Arnoldi with classical Gram-Schmidt and one reorthogonalisation pass on
// K_M(J_n, f_n) (Sec. 4.1).  Returns the dimension m <= M; Q and H in the slot.
// MIXED: the first Gram-Schmidt pass takes its inner products in FP32 (from
// the FP32 copy of Q); the reorthogonalisation pass, which removes what the
// first pass left behind -- its FP32 rounding included -- and the norms stay
// FP64, so the basis and H keep FP64 quality (mixed-precision "twice is
// enough").
//
// One FP64 Gram-Schmidt pass of w against the basis vectors q_0..q_{n-1}:
// h = Q^T w (one batched reduction), w <- w - Q h; lane i returns h_i (i < n).  J > 0: n = J
// is known at compile time, so no term carries a predicate (a predicated-off
// FP64 instruction still takes its issue and pipe slot); J = 0: n = jn at run
// time guards each of the MAXM terms.  Either way the same operations in the
// same order for the terms that exist.
// WW: w^T w before the pass joins the reduction, into *ww.
template <int G, int J, bool WW = false>
__device__ __forceinline__ double cgs_pass(const SlotPtrs& s, int N, int jn, double* ww = nullptr) {
  const Grp<G> g;
  const int Nq = s.Nq;
  constexpr int LJ = J > 0 ? J : MAXM;
  double hp[MAXM];
#pragma unroll
  for (int i = 0; i < MAXM; ++i) hp[i] = 0.0;
#pragma unroll 1
  for (int e = g.lane; e < N; e += G) {
    const double we = s.w[e];
#pragma unroll
    for (int i = 0; i < LJ; ++i)
      if (J > 0 || i < jn) hp[i] = fma(s.Q[i * Nq + e], we, hp[i]);
    if (WW) hp[LJ] = fma(we, we, hp[LJ]);
  }
  sum_first<G>(g, hp, (J > 0 ? J : jn) + (WW ? 1 : 0));
  if (WW) *ww = hp[LJ];
#pragma unroll 1
  for (int e = g.lane; e < N; e += G) {
    double we = s.w[e];
#pragma unroll
    for (int i = 0; i < LJ; ++i)
      if (J > 0 || i < jn) we = fma(-hp[i], s.Q[i * Nq + e], we);
    s.w[e] = we;
  }
  double mine = hp[0];
#pragma unroll
  for (int i = 1; i < LJ; ++i) mine = g.lane == i ? hp[i] : mine;
  return mine;
}

template <int G, bool MIXED = false, bool TC = false>
__device__ int arnoldi(const MechView& m, const SlotPtrs& s, const CellScalars& cs, int M, int jv_mode,
                       double p, int* n_rhs, bool fp32_jv = false) {
  const Grp<G> g;
  const int N = m.ns + 1 + m.nx;
  const int Nq = s.Nq;
  if (M > N) M = N;
  for (int i = g.lane; i < M * MAXM; i += G) s.H[i] = 0.0;
  // squared norms; 1/||.|| from one reciprocal square root
  const double beta2 = group_dot<G>(g, s.fn, s.fn, N);
  if (M <= 0 || !(beta2 > 0.0) || !isfinite(beta2)) {
    g.sync();
    return 0;
  }
  double unorm = 0.0;
  if (jv_mode != 0) unorm = sqrt(group_dot<G>(g, s.u, s.u, N));
  const double ibeta = rsqrt_any(beta2);
  for (int e = g.lane; e < N; e += G) {
    const double qe = s.fn[e] * ibeta;
    s.Q[e] = qe;
    if (MIXED) s.fQ[e] = __double2float_rn(qe);
  }
  g.sync();
  constexpr double brk2 = BREAKDOWN_TOL * BREAKDOWN_TOL;  // breakdown ||w_after|| <= tol ||w_before||, on squares
  int mdim = M;
  for (int j = 0; j < M; ++j) {
    apply_jv<G, MIXED, TC>(m, s, cs, jv_mode, p, unorm, s.Q + j * Nq, s.w, n_rhs, fp32_jv);
    // (only the breakdown threshold reads ||J q_j||^2: FP32 is enough there)
    double w02 = 0.0;
    if (MIXED) w02 = (double)group_dot_f<G>(g, s.w, s.w, N);
    else if (M > 6) w02 = group_dot<G>(g, s.w, s.w, N);
    double hcol = 0.0;  // lane i: h_ij
    for (int pass = 0; pass < 2; ++pass) {
      double hpass;
      if (MIXED && pass == 0) {
        double hp[MAXM];
        float part[MAXM];
#pragma unroll
        for (int i = 0; i < MAXM; ++i) part[i] = 0.f;
        for (int e = g.lane; e < N; e += G) {
          const float we = __double2float_rn(s.w[e]);
#pragma unroll
          for (int i = 0; i < MAXM; ++i)
            if (i <= j) part[i] = fmaf(s.fQ[i * Nq + e], we, part[i]);
        }
        sum_first<G>(g, part, j + 1);
#pragma unroll
        for (int i = 0; i < MAXM; ++i) hp[i] = (double)part[i];
        for (int e = g.lane; e < N; e += G) {
          double we = s.w[e];
#pragma unroll
          for (int i = 0; i < MAXM; ++i)
            if (i <= j) we = fma(-hp[i], s.Q[i * Nq + e], we);
          s.w[e] = we;
        }
        hpass = hp[0];
#pragma unroll
        for (int i = 1; i < MAXM; ++i) hpass = g.lane == i ? hp[i] : hpass;
      } else if (M <= 6) {
        const bool first = !MIXED && pass == 0 && j + 1 < M;  // (the last column has no breakdown test to feed)
        // the common Krylov dimensions: column j + 1 known at compile time
        switch (j) {
          case 0: hpass = first ? cgs_pass<G, 1, true>(s, N, 1, &w02) : cgs_pass<G, 1>(s, N, 1); break;
          case 1: hpass = first ? cgs_pass<G, 2, true>(s, N, 2, &w02) : cgs_pass<G, 2>(s, N, 2); break;
          case 2: hpass = first ? cgs_pass<G, 3, true>(s, N, 3, &w02) : cgs_pass<G, 3>(s, N, 3); break;
          case 3: hpass = first ? cgs_pass<G, 4, true>(s, N, 4, &w02) : cgs_pass<G, 4>(s, N, 4); break;
          case 4: hpass = first ? cgs_pass<G, 5, true>(s, N, 5, &w02) : cgs_pass<G, 5>(s, N, 5); break;
          default: hpass = cgs_pass<G, 6>(s, N, 6); break;
        }
      } else {
        hpass = cgs_pass<G, 0>(s, N, j + 1);
      }
      hcol = pass == 0 ? hpass : hcol + hpass;
    }
    if (g.lane <= j) s.H[g.lane * MAXM + j] = hcol;
    if (j + 1 == M) break;
    const double hn2 = group_dot<G>(g, s.w, s.w, N);
    if (hn2 <= brk2 * w02 || hn2 == 0.0) {
      mdim = j + 1;
      break;
    }
    const double ihn = rsqrt_any(hn2);
    const double hn = hn2 * ihn;
    if (g.lane == 0) s.H[(j + 1) * MAXM + j] = hn;
    for (int e = g.lane; e < N; e += G) {
      const double qe = s.w[e] * ihn;
      s.Q[(j + 1) * Nq + e] = qe;
      if (MIXED) s.fQ[(j + 1) * Nq + e] = __double2float_rn(qe);
    }
    g.sync();
  }
  g.sync();
  return mdim;
}

// Solve (I - h gamma H) y = z in place (every lane, redundantly; the factor
// stores reciprocal pivots, so the solve has no divisions).
__device__ inline void solve_small(const SlotPtrs& s, int mdim, double* z) {
  for (int c = 0; c < mdim; ++c) {
    const int pr = (int)s.piv[c];
    if (pr != c) {
      const double t = z[c];
      z[c] = z[pr];
      z[pr] = t;
    }
  }
  for (int r = 1; r < mdim; ++r)
    for (int c = 0; c < r; ++c) z[r] = fma(-s.LU[r * MAXM + c], z[c], z[r]);
  for (int r = mdim - 1; r >= 0; --r) {
    for (int c = r + 1; c < mdim; ++c) z[r] = fma(-s.LU[r * MAXM + c], z[c], z[r]);
    z[r] = z[r] * s.LU[r * MAXM + r];
  }
}

// B = I - (I - h gamma H)^-1 for m = 4 by the whole warp: Gauss-Jordan with
// partial pivoting on [I - h gamma H | I], one element a lane (row l / 8, column
// l mod 8), rows and pivots passed by shuffles.  Seven FP64 instructions a pivot
// instead of a serial elimination by lane 0 through shared memory and four
// solves, which took 15,000 cycles of an attempt's 250,000.
__device__ __forceinline__ void factor_four(const SlotPtrs& s, double h) {
  const int lane = threadIdx.x & 31, r = lane >> 3, c = lane & 7;
  const unsigned all = 0xffffffffu;
  double v = c < 4 ? fma(-(h * GAM), s.H[r * MAXM + c], r == c ? 1.0 : 0.0) : (c - 4 == r ? 1.0 : 0.0);
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    double a[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = __shfl_sync(all, v, 8 * i + p);
    int pr = p;
    long long best = __double_as_longlong(a[p]) & 0x7fffffffffffffffll;
    double piv = a[p];
#pragma unroll
    for (int i = p + 1; i < 4; ++i) {
      const long long cand = __double_as_longlong(a[i]) & 0x7fffffffffffffffll;
      if (cand > best) {
        best = cand;
        pr = i;
        piv = a[i];
      }
    }
    const int from = r == p ? pr : (r == pr ? p : r);  // rows p and pr exchanged
    v = __shfl_sync(all, v, 8 * from + c);
    const double f = r == pr ? a[p] : (r == 0 ? a[0] : r == 1 ? a[1] : r == 2 ? a[2] : a[3]);
    const double row = __shfl_sync(all, v, 8 * p + c) * rcp_any(piv);
    v = r == p ? row : fma(-f, row, v);
  }
  if (c >= 4) s.Bm[r * MAXM + c - 4] = (c - 4 == r ? 1.0 : 0.0) - v;
  __syncwarp();
}

// The same for m = 5 and 6, one column of [I - h gamma H | I] a lane (lanes past
// 2 m repeat the last): a pivot column goes round by shuffles and every lane
// eliminates its own column, m + 5 FP64 instructions a pivot.
template <int M>
__device__ __forceinline__ void factor_columns(const SlotPtrs& s, double h) {
  const int lane = threadIdx.x & 31, c = min(lane, 2 * M - 1);
  const unsigned all = 0xffffffffu;
  const double hg = h * GAM;
  double v[M];
#pragma unroll
  for (int r = 0; r < M; ++r) {
    const double a = fma(-hg, s.H[r * MAXM + min(c, M - 1)], r == c ? 1.0 : 0.0);
    v[r] = c < M ? a : (c - M == r ? 1.0 : 0.0);
  }
#pragma unroll
  for (int p = 0; p < M; ++p) {
    double f[M];
#pragma unroll
    for (int r = 0; r < M; ++r) f[r] = __shfl_sync(all, v[r], p);
    int pr = p;
    long long best = __double_as_longlong(f[p]) & 0x7fffffffffffffffll;
#pragma unroll
    for (int r = p + 1; r < M; ++r) {
      const long long cand = __double_as_longlong(f[r]) & 0x7fffffffffffffffll;
      pr = cand > best ? r : pr;
      best = cand > best ? cand : best;
    }
#pragma unroll
    for (int r = p + 1; r < M; ++r) {  // rows p and pr exchanged
      const bool x = pr == r;
      const double fp = f[p], vp = v[p];
      f[p] = x ? f[r] : fp;
      f[r] = x ? fp : f[r];
      v[p] = x ? v[r] : vp;
      v[r] = x ? vp : v[r];
    }
    v[p] *= rcp_any(f[p]);
#pragma unroll
    for (int r = 0; r < M; ++r)
      if (r != p) v[r] = fma(-f[r], v[p], v[r]);
  }
  if (lane >= M && lane < 2 * M) {
#pragma unroll
    for (int r = 0; r < M; ++r) s.Bm[r * MAXM + lane - M] = (r == lane - M ? 1.0 : 0.0) - v[r];
  }
  __syncwarp();
}

// LU factorisation with partial pivoting of I - h gamma H (m x m), by lane 0.
template <int G>
__device__ inline void factor_small(const SlotPtrs& s, int mdim, double h) {
  const Grp<G> g;
  if (g.lane == 0) {
    double* A = s.LU;
    const double hg = h * GAM;
    for (int i = 0; i < mdim; ++i)
      for (int j = 0; j < mdim; ++j) A[i * MAXM + j] = fma(-hg, s.H[i * MAXM + j], i == j ? 1.0 : 0.0);
    for (int c = 0; c < mdim; ++c) {
      // partial pivoting; |a| compared through its bit pattern (the order of
      // non-negative doubles is the order of their bits), an integer compare
      int pr = c;
      long long best = __double_as_longlong(fabs(A[c * MAXM + c]));
      for (int r = c + 1; r < mdim; ++r) {
        const long long cand = __double_as_longlong(fabs(A[r * MAXM + c]));
        if (cand > best) {
          best = cand;
          pr = r;
        }
      }
      s.piv[c] = (double)pr;
      if (pr != c)
        for (int j = 0; j < mdim; ++j) {
          const double t = A[c * MAXM + j];
          A[c * MAXM + j] = A[pr * MAXM + j];
          A[pr * MAXM + j] = t;
        }
      const double inv = rcp_any(A[c * MAXM + c]);
      for (int r = c + 1; r < mdim; ++r) {
        const double l = A[r * MAXM + c] * inv;
        A[r * MAXM + c] = l;
        for (int j = c + 1; j < mdim; ++j) A[r * MAXM + j] = fma(-l, A[c * MAXM + j], A[r * MAXM + j]);
      }
      A[c * MAXM + c] = inv;  // the diagonal is kept as its reciprocal
    }
  }
  g.sync();
  // B = I - (I - h gamma H)^-1, one column per lane (a solve with e_l), so each
  // stage applies the low-rank correction as one matrix-vector product
  if (g.lane < mdim) {
    double x[MAXM];
#pragma unroll
    for (int i = 0; i < MAXM; ++i) x[i] = i == g.lane ? 1.0 : 0.0;
    solve_small(s, mdim, x);
    for (int i = 0; i < mdim; ++i) s.Bm[i * MAXM + g.lane] = (i == g.lane ? 1.0 : 0.0) - x[i];
  }
  g.sync();
}

// One stage of the transformed form (Eq. s_stage_row_transformed) with the
// low-rank inverse (Eq. solve_kry_jac), in two parts.  stage_rhs: F_i = f_i +
// G_i with G_i = sum_{j<i} (gamma_ij / gamma) k_j (G_i left in s.w) and the partial sums of Q^T F_i.  stage_solve: c = (I - (I - h gamma
// H)^-1) Q^T F_i (B = I - (I - h gamma H)^-1 from factor_small) and
// k_i = F_i - Q c - G_i.  I >= 0: the stage known at compile time; MD > 0: the
// basis dimension known at compile time, so no term carries a predicate (a
// predicated-off FP64 instruction still takes its issue and pipe slot);
// I = -1 / MD = 0: from i / mdim at run time, each of the MAXM terms guarded.
// The same operations in the same order either way.
template <int G, int MD, int I>
__device__ __forceinline__ void stage_rhs(const SlotPtrs& s, int N, int i_rt, int mdim_rt, const double* fi,
                                          double (&part)[MAXM]) {
  const Grp<G> g;
  const int Nq = s.Nq;
  const int i = I >= 0 ? I : i_rt;
  const int mdim = MD > 0 ? MD : mdim_rt;
  constexpr int LM = MD > 0 ? MD : MAXM;
  constexpr double g21 = G21 / GAM, g31 = G31 / GAM, g32 = G32 / GAM;
  constexpr double g41 = G41 / GAM, g42 = G42 / GAM, g43 = G43 / GAM;
  const double* K0 = s.K;
  const double* K1 = s.K + Nq;
  const double* K2 = s.K + 2 * Nq;
#pragma unroll
  for (int l = 0; l < MAXM; ++l) part[l] = 0.0;
#pragma unroll 1
  for (int e = g.lane; e < N; e += G) {
    double Ge = 0.0;
    if (i == 1) Ge = g21 * K0[e];
    else if (i == 2) Ge = fma(g32, K1[e], g31 * K0[e]);
    else if (i == 3) Ge = fma(g43, K2[e], fma(g42, K1[e], g41 * K0[e]));
    const double Fe = fi[e] + Ge;
    s.w[e] = Ge;
#pragma unroll
    for (int l = 0; l < LM; ++l)
      if (MD > 0 || l < mdim) part[l] = fma(s.Q[l * Nq + e], Fe, part[l]);
  }
}

template <int G, int MD>
__device__ __forceinline__ void stage_solve(const SlotPtrs& s, int N, int i, int mdim_rt, const double* fi,
                                            double (&part)[MAXM]) {
  const Grp<G> g;
  const int Nq = s.Nq;
  const int mdim = MD > 0 ? MD : mdim_rt;
  constexpr int LM = MD > 0 ? MD : MAXM;
  double* Ki = s.K + i * Nq;
  if (mdim > 0) sum_first<G>(g, part, mdim);
  // lane l < m forms c_l, every lane then reads all
  double cl = 0.0;
  if (g.lane < mdim) {
#pragma unroll
    for (int c = 0; c < LM; ++c)
      if (MD > 0 || c < mdim) cl = fma(s.Bm[g.lane * MAXM + c], part[c], cl);
  }
  double cz[MAXM];
#pragma unroll
  for (int l = 0; l < LM; ++l) cz[l] = __shfl_sync(g.mask, cl, l, G);
#pragma unroll 1
  for (int e = g.lane; e < N; e += G) {
    double acc = 0.0;
#pragma unroll
    for (int l = 0; l < LM; ++l)
      if (MD > 0 || l < mdim) acc = fma(s.Q[l * Nq + e], cz[l], acc);
    const double Ge = s.w[e];
    Ki[e] = ((fi[e] + Ge) - acc) - Ge;  // F_i as in stage_rhs
  }
  g.sync();
}


template <int G, int MD>
__device__ __forceinline__ void stage_of(const SlotPtrs& s, int N, int i, const double* fi, double (&part)[MAXM]) {
  switch (i) {
    case 0: stage_rhs<G, MD, 0>(s, N, 0, MD, fi, part); break;
    case 1: stage_rhs<G, MD, 1>(s, N, 1, MD, fi, part); break;
    case 2: stage_rhs<G, MD, 2>(s, N, 2, MD, fi, part); break;
    default: stage_rhs<G, MD, 3>(s, N, 3, MD, fi, part); break;
  }
  stage_solve<G, MD>(s, N, i, MD, fi, part);
}

// ------------------------------------------------ cost-ordered work queue
// Cells are handed out longest-expected-first: the expected substep count of
// a cell is dt / h with h its carried step (h_cell), binned on a quarter-octave
// log scale; a counting sort (per-block histograms reserved in one atomic per
// bin, then scattered) writes the queue order.  Cells with no carried step or
// h >= dt land in the cheapest bin.
constexpr int ORDER_BINS = 64;
constexpr int ORDER_THREADS = 256;

__device__ __forceinline__ int cost_bin(double h, double dt) {
  if (!(h > 0.0) || !(h < dt)) return 0;
  const float r = __double2float_rn(dt) / __double2float_rn(h);
  const int b = (int)(4.0f * __log2f(r));
  return b < 0 ? 0 : (b >= ORDER_BINS ? ORDER_BINS - 1 : b);
}

// ------------------------------------------------------- integration kernel
struct IntegrateParams {
  const unsigned char* mech;  // packed mechanism (global)
  MechLayout L;
  SlotLayout S;
  double* Y;
  const double* src;
  double* h_cell;
  int64_t ncell;
  double p, dt, rtol, atol, h0, fixed_h;
  int M, jv_mode, max_attempts, trace_cap, precision;
  double* trace;
  int32_t* stats;
  unsigned long long* counter;
  unsigned long long qstride;  // queue position q takes cell (q * qstride) mod ncell
  const int32_t* order;        // or, when set, cell order[q] (longest expected first)
  int subq;                    // > 0: static bins, subq sub-queues per block (queue order 3)
  const unsigned* nhot;        // with static bins: number of hot cells leading the order, or null
  const double* rho_cell;      // constant-volume densities, or null (constant pressure)
  int nx;                      // state components after T (5: auxiliary-temperature system)
  int64_t mech_copy;           // bytes of the mechanism each block copies (a prefix, by precision)
  int64_t fx_copy;             // bytes of the segment copied after that (without its fixed-point part where that does not fit)
  int64_t tc_bytes;            // precision 4: bytes of nu^T tiles copied after both (else 0)
};

template <int G, bool MIXED, bool TC = false>
__device__ void integrate_cell(const MechView& m, const SlotPtrs& s, const IntegrateParams& P, int64_t cell) {
  const Grp<G> g;
  const int ns = m.ns, N = ns + 1 + m.nx, Nq = s.Nq;
  for (int e = g.lane; e < N; e += G) {
    s.u[e] = P.Y[cell * N + e];
    if (P.S.src >= 0) s.src[e] = P.src ? P.src[cell * N + e] : 0.0;
  }
  g.sync();
  const double* srcp = P.src ? s.src : nullptr;
  const bool fixed = P.fixed_h > 0.0;
  const double pr = P.rho_cell ? -P.rho_cell[cell] : P.p;  // negative: constant-volume density
  const bool fp32_jv = P.precision == 2;
  const double dt = P.dt;
  double h = P.h0 > 0.0 ? P.h0 : dt;
  if (P.h_cell) {
    const double hc = P.h_cell[cell];
    if (hc > 0.0) h = hc;
  }
  if (fixed) h = P.fixed_h;
  const long long n_fixed = fixed ? llround(dt / P.fixed_h) : 0;
  double t = 0.0, left = dt, h_last = h;
  const double tol_t = T_END_TOL * dt, inv_N = 1.0 / N;
  float lg_err_prev = 0.f;  // log2 err_n; err_n = 1 before the first step
  int n_acc = 0, n_rej = 0, n_rhs = 0, status = RK_CELL_OK, n_att = 0;
  CellScalars cs;
  cs.pinv = 1.0 / fabs(pr);
  cs.prec = (P.precision == 3 || P.precision >= 5) ? P.precision : (TC ? 4 : 0);
  constexpr bool INL = G == 32 && !MIXED;  // the RHS inlined on the main path
  int mdim = 0;
  bool fresh = true;  // f_n and the Krylov basis are due at u (start, or after an accepted step)
  double* K0 = s.K;
  double* K1 = s.K + Nq;
  double* K2 = s.K + 2 * Nq;
  double* K3 = s.K + 3 * Nq;
  while (true) {
    if (fresh) {
      rhs_dispatch<G, MIXED, INL, TC>(m, s, s.u, srcp, pr, s.fn, true, &cs);
      n_rhs += 1;
      mdim = arnoldi<G, MIXED, TC>(m, s, cs, P.M, P.jv_mode, pr, &n_rhs, fp32_jv);
      fresh = false;
    }
    if (fixed) {
      if (n_acc >= n_fixed) break;
    } else if (__double_as_longlong(left) <= __double_as_longlong(tol_t)) {  // (tol_t > 0; negative bits are below)
      break;
    }
    if (n_att >= P.max_attempts) {
      status = RK_CELL_MAX_ATTEMPTS;
      break;
    }
    if (!fixed && __double_as_longlong(left) < __double_as_longlong(h)) h = left;  // both positive
    if (G == 32 && mdim == 4) factor_four(s, h);
    else if (G == 32 && mdim == 5) factor_columns<5>(s, h);
    else if (G == 32 && mdim == 6) factor_columns<6>(s, h);
    else factor_small<G>(s, mdim, h);
    // ---- four stages (Algorithm 1); f is evaluated at stages 2 and 3 only
    for (int i = 0; i < 4; ++i) {
      const double* fi;
      if (i == 0) {
        fi = s.fn;
      } else if (i == 1 || i == 2) {
        for (int e = g.lane; e < N; e += G) {
          const double acc = (i == 1) ? A21 * K0[e] : fma(A32, K1[e], A31 * K0[e]);
          s.arg[e] = s.u[e] + h * acc;
        }
        g.sync();
        rhs_dispatch<G, MIXED, INL, TC>(m, s, s.arg, srcp, pr, s.fr, false, &cs);
        n_rhs += 1;
        fi = s.fr;
      } else {
        fi = s.fr;  // alpha_4j = alpha_3j: same argument as stage 3
      }
      double part[MAXM];
      if (mdim == 4) {  // the common Krylov dimensions: stage and dimension known at compile time
        stage_of<G, 4>(s, N, i, fi, part);
      } else if (G == 32 && mdim == 5) {
        stage_of<G, 5>(s, N, i, fi, part);
      } else if (G == 32 && mdim == 6) {
        stage_of<G, 6>(s, N, i, fi, part);
      } else {
        stage_rhs<G, 0, -1>(s, N, i, mdim, fi, part);
        stage_solve<G, 0>(s, N, i, mdim, fi, part);
      }
    }
    // ---- solutions, error estimate
    double part = 0.0;
    int bad = 0;
    for (int e = g.lane; e < N; e += G) {
      const double k0 = K0[e], k1 = K1[e], k2 = K2[e], k3 = K3[e];
      const double ue = s.u[e];
      const double us = ue + h * fma(B4, k3, fma(B2, k1, B1 * k0));  // b3 = 0
      const double uh = ue + h * fma(BH3, k2, fma(BH2, k1, BH1 * k0));  // bhat4 = 0
      const double d = (uh - us) * rcp_any(fma(P.rtol, fabs(us), P.atol));
      part = fma(d, d, part);
      bad |= (__double2hiint(us) & 0x7ff00000) == 0x7ff00000;
      s.arg[e] = us;
    }
    const double err2 = g.sum(part) * inv_N;  // err*^2
    bad = g.any(bad);
    const int att = n_att;
    n_att += 1;
    bool accept;
    double hnew;
    float lg_err = 0.f;
    if (fixed) {
      accept = true;
      hnew = h;
    } else {
      // h* = h min(5, max(0.2, 0.8 err_n^beta / err*^alpha)), the factor in
      // FP32 as 2^(beta log2 err_n - alpha log2 err*) (log2 err_n kept from
      // acceptance; the logarithm of the square halved).  err* <= 1 is err*^2 <= 1,
      // compared through the bits
      const bool fin = (__double2hiint(err2) & 0x7ff00000) != 0x7ff00000;
      float fac = (float)FAC_MIN;
      if (fin) {
        lg_err = fmaxf(0.5f * __log2f(float_bits(err2)), LOG2_ERR_FLOOR);
        fac = fminf((float)FAC_MAX,
                    fmaxf((float)FAC_MIN, (float)SAFETY * exp2f((float)PI_BETA * lg_err_prev - (float)PI_ALPHA * lg_err)));
      }
      hnew = h * double_bits(fac);
      accept = fin && __double_as_longlong(err2) <= 0x3ff0000000000000ll;
    }
    if (P.trace && att < P.trace_cap && g.lane == 0) P.trace[cell * P.trace_cap + att] = accept ? h : -h;
    if (accept) {
      if (bad) {
        status = RK_CELL_NONFINITE;
        break;
      }
      for (int e = g.lane; e < N; e += G) s.u[e] = s.arg[e];
      g.sync();
      t += h;
      left = dt - t;
      if (!fixed) lg_err_prev = lg_err;
      n_acc += 1;
      h_last = hnew;
      h = hnew;
      const bool done =
          fixed ? (n_acc >= n_fixed) : __double_as_longlong(left) <= __double_as_longlong(tol_t);
      fresh = !done;
    } else {
      n_rej += 1;
      h = hnew;
      if (h < H_MIN_FRAC * dt) {
        status = RK_CELL_STEP_UNDERFLOW;
        break;
      }
    }
  }
  for (int e = g.lane; e < N; e += G) P.Y[cell * N + e] = s.u[e];
  if (g.lane == 0) {
    if (P.h_cell) P.h_cell[cell] = h_last;
    if (P.stats) {
      P.stats[4 * cell + 0] = n_acc;
      P.stats[4 * cell + 1] = n_rej;
      P.stats[4 * cell + 2] = n_rhs;
      P.stats[4 * cell + 3] = status;
    }
  }
  g.sync();
}

// Copy the packed mechanism into shared memory (16-byte vector copies).
__device__ inline void load_mech(unsigned char* dst, const unsigned char* src, int64_t bytes) {
  const int64_t n16 = bytes / 16;
  const uint4* s4 = reinterpret_cast<const uint4*>(src);
  uint4* d4 = reinterpret_cast<uint4*>(dst);
  for (int64_t i = threadIdx.x; i < n16; i += blockDim.x) d4[i] = s4[i];
}

template <bool MIXED = false>
__device__ inline void init_sentinels(const SlotPtrs& s, int ns, int lane) {
  if (lane == 0) {
    s.C[ns] = 1.0;
    s.dC[ns] = 0.0;
    if (s.C2) {
      s.C2[ns] = {1.0f, 0.0f};
      s.dC2[ns] = {0.0f, 0.0f};
    }
    s.hRT[ns] = 0.0;
    s.gRT[ns] = 0.0;
    s.E[ns] = 1.0;
    s.CE[ns] = 1.0;
    if (MIXED) {
      s.fC[ns] = 1.f;
      s.fdC[ns] = 0.f;
      s.fh[ns] = 0.f;
    }
  }
}

// Hand cells to the warp groups of a persistent launch until the queue is
// empty, calling body(cell) for each.
template <int G, class Body>
__device__ __forceinline__ void drain_queue(const IntegrateParams& P, const Grp<G>& g, int gid, Body&& body) {
  if (P.subq > 0) {
    // Static bins: the queue (longest expected first) is dealt out in snake
    // order over nb = gridDim.x * subq bins, bin k = sub * gridDim.x + block,
    // so every block -- and within a block every group of warps sharing a
    // sub-queue -- receives a near-equal share of the expensive cells.  Round
    // r of bin k holds queue position r * nb + (r even ? k : nb - 1 - k).
    __shared__ unsigned sub_ctr[4];
    if (threadIdx.x < 4) sub_ctr[threadIdx.x] = 0u;
    __syncthreads();
    // The H hot cells that lead the order (when they are few: at most half the
    // blocks and an eighth of the cells) each get a block -- an SM -- of their
    // own: hot cell b runs on sub-queue 0 of block b and that block takes
    // nothing else, so no other cell shares its SM's FP64 units, shared-memory
    // pipe or instruction cache.  The rest are dealt in snake order over the
    // bins of the other blocks.
    const int sub = gid % P.subq;
    const unsigned long long nblk = gridDim.x;
    unsigned long long H = P.nhot ? (unsigned long long)P.nhot[0] : 0ull;
    if (H * 2ull > nblk || H * 8ull > (unsigned long long)P.ncell) H = 0ull;
    if (H > 0ull) {
      // only while the other cells, spread over the other blocks' four
      // sub-partitions, still finish within the hottest cell's expected time
      const float top_cost = __uint_as_float(P.nhot[1]), rest_cost = __uint_as_float(P.nhot[2]);
      if (rest_cost > top_cost * 4.0f * (float)(nblk - H)) H = 0ull;
    }
    const unsigned long long nb = (nblk - H) * (unsigned long long)P.subq;
    const bool hot_block = blockIdx.x < H;
    const unsigned long long k = hot_block ? 0ull : (unsigned long long)sub * (nblk - H) + (blockIdx.x - H);
    while (true) {
      unsigned r = 0u;
      if (g.lane == 0) r = atomicAdd(&sub_ctr[sub], 1u);
      r = __shfl_sync(g.mask, r, 0, G);
      unsigned long long q;
      if (hot_block) {
        q = (sub == 0 && r == 0u) ? (unsigned long long)blockIdx.x : (unsigned long long)P.ncell;
      } else {
        q = H + (unsigned long long)r * nb + ((r & 1u) ? nb - 1ull - k : k);
      }
      if (q >= (unsigned long long)P.ncell) break;
      const unsigned long long cell =
          P.order ? (unsigned long long)P.order[q] : (q * P.qstride) % (unsigned long long)P.ncell;
      body((int64_t)cell);
    }
    return;
  }
  while (true) {
    unsigned long long q = 0;
    if (g.lane == 0) q = atomicAdd(P.counter, 1ull);
    q = __shfl_sync(g.mask, q, 0, G);
    if (q >= (unsigned long long)P.ncell) break;
    // Interleave the queue over the cell index: neighbouring cells (e.g. the
    // hot side of a flame) spread over all SMs instead of filling a few.
    const unsigned long long cell =
        P.order ? (unsigned long long)P.order[q] : (q * P.qstride) % (unsigned long long)P.ncell;
    body((int64_t)cell);
  }
}

template <int G, bool MIXED, bool TC = false, int THREADS = MAX_BLOCK_THREADS>
__global__ void __launch_bounds__(THREADS, 1) rok4e_integrate_kernel(IntegrateParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  load_exp_table(reinterpret_cast<uint64_t*>(smem));
  load_mech(smem + EXP_TAB_BYTES, P.mech, P.mech_copy);
  load_mech(smem + EXP_TAB_BYTES + P.mech_copy, P.mech + P.L.off_lo, P.fx_copy);
  if (TC) load_mech(smem + EXP_TAB_BYTES + P.mech_copy + P.fx_copy, P.mech + P.L.off_nuT, P.tc_bytes);
  __syncthreads();
  MechView m = make_view(smem + EXP_TAB_BYTES, P.mech, P.L, P.mech_copy, P.fx_copy > P.L.off_fA - P.L.off_lo);
  m.etab = reinterpret_cast<const uint64_t*>(smem);
  m.nx = P.nx;
  if (TC) m.nuT = reinterpret_cast<const uint4*>(smem + EXP_TAB_BYTES + P.mech_copy + P.fx_copy);
  const Grp<G> g;
  const int gid = threadIdx.x / G;
  double* base = reinterpret_cast<double*>(smem + EXP_TAB_BYTES + P.mech_copy + P.fx_copy + (TC ? P.tc_bytes : 0)) +
                 (size_t)gid * P.S.stride;
  const SlotPtrs s = slot_ptrs(base, P.S);
  init_sentinels<MIXED>(s, m.ns, g.lane);
  if (TC)  // digit rows: row 7 and the reaction padding stay zero
    for (int i = g.lane; i < 8 * 16 * m.nrt; i += G) s.dig[i] = 0;
  g.sync();
  drain_queue<G>(P, g, gid, [&](int64_t cell) { integrate_cell<G, MIXED, TC>(m, s, P, cell); });
}

// ------------------------------------------- explicit Dormand-Prince 5(4)
// The explicit reference integrator of the efficiency study (Sec. 4.4):
// seven stages, the 5th-order solution propagated, the embedded 4th-order
// one for the error (J. R. Dormand and P. J. Prince, J. Comput. Appl. Math.
// 6 (1980) 19-26), first-same-as-last; the same RMS error norm as ROK4E and
// the elementary controller h* = h min(5, max(0.2, 0.9 err^-1/5)).
namespace dp {
constexpr double A21 = 1.0 / 5.0;
constexpr double A31 = 3.0 / 40.0, A32 = 9.0 / 40.0;
constexpr double A41 = 44.0 / 45.0, A42 = -56.0 / 15.0, A43 = 32.0 / 9.0;
constexpr double A51 = 19372.0 / 6561.0, A52 = -25360.0 / 2187.0, A53 = 64448.0 / 6561.0, A54 = -212.0 / 729.0;
constexpr double A61 = 9017.0 / 3168.0, A62 = -355.0 / 33.0, A63 = 46732.0 / 5247.0, A64 = 49.0 / 176.0,
                 A65 = -5103.0 / 18656.0;
constexpr double B1 = 35.0 / 384.0, B3 = 500.0 / 1113.0, B4 = 125.0 / 192.0, B5 = -2187.0 / 6784.0,
                 B6 = 11.0 / 84.0;
// b - bhat (b2 = bhat2 = 0, b7 = 0)
constexpr double E1 = 35.0 / 384.0 - 5179.0 / 57600.0, E3 = 500.0 / 1113.0 - 7571.0 / 16695.0,
                 E4 = 125.0 / 192.0 - 393.0 / 640.0, E5 = -2187.0 / 6784.0 + 92097.0 / 339200.0,
                 E6 = 11.0 / 84.0 - 187.0 / 2100.0, E7 = -1.0 / 40.0;
constexpr double SAFETY = 0.9;
}  // namespace dp

template <int G>
__device__ void integrate_cell_rkdp(const MechView& m, const SlotPtrs& s, const IntegrateParams& P, int64_t cell) {
  const Grp<G> g;
  const int ns = m.ns, N = ns + 1 + m.nx, Nq = s.Nq;
  for (int e = g.lane; e < N; e += G) {
    s.u[e] = P.Y[cell * N + e];
    if (P.S.src >= 0) s.src[e] = P.src ? P.src[cell * N + e] : 0.0;
  }
  g.sync();
  const double* srcp = P.src ? s.src : nullptr;
  const bool fixed = P.fixed_h > 0.0;
  const double pr = P.rho_cell ? -P.rho_cell[cell] : P.p;
  const double dt = P.dt;
  double h = P.h0 > 0.0 ? P.h0 : dt;
  if (P.h_cell) {
    const double hc = P.h_cell[cell];
    if (hc > 0.0) h = hc;
  }
  if (fixed) h = P.fixed_h;
  const long long n_fixed = fixed ? llround(dt / P.fixed_h) : 0;
  double t = 0.0, h_last = h;
  int n_acc = 0, n_rej = 0, n_rhs = 0, status = RK_CELL_OK, n_att = 0;
  CellScalars cs;
  cs.pinv = 1.0 / fabs(pr);
  cs.prec = 0;
  // stage vectors k1..k7; k1 and k7 swap roles after an accepted step
  double* k1 = s.fn;
  double* k2 = s.K;
  double* k3 = s.K + Nq;
  double* k4 = s.K + 2 * Nq;
  double* k5 = s.K + 3 * Nq;
  double* k6 = s.F;
  double* k7 = s.w;
  rhs_eval_call<G>(m, s, s.u, srcp, pr, k1, false, &cs);
  n_rhs += 1;
  while (true) {
    if (fixed) {
      if (n_acc >= n_fixed) break;
    } else if (dt - t <= T_END_TOL * dt) {
      break;
    }
    if (n_att >= P.max_attempts) {
      status = RK_CELL_MAX_ATTEMPTS;
      break;
    }
    if (!fixed) h = fmin(h, dt - t);
    for (int i = 1; i < 7; ++i) {
      for (int e = g.lane; e < N; e += G) {
        double acc;
        if (i == 1) acc = dp::A21 * k1[e];
        else if (i == 2) acc = fma(dp::A32, k2[e], dp::A31 * k1[e]);
        else if (i == 3) acc = fma(dp::A43, k3[e], fma(dp::A42, k2[e], dp::A41 * k1[e]));
        else if (i == 4) acc = fma(dp::A54, k4[e], fma(dp::A53, k3[e], fma(dp::A52, k2[e], dp::A51 * k1[e])));
        else if (i == 5)
          acc = fma(dp::A65, k5[e], fma(dp::A64, k4[e], fma(dp::A63, k3[e], fma(dp::A62, k2[e], dp::A61 * k1[e]))));
        else  // a_7j = b_j: the last argument is the 5th-order solution
          acc = fma(dp::B6, k6[e], fma(dp::B5, k5[e], fma(dp::B4, k4[e], fma(dp::B3, k3[e], dp::B1 * k1[e]))));
        s.arg[e] = fma(h, acc, s.u[e]);
      }
      g.sync();
      double* out = i == 1 ? k2 : i == 2 ? k3 : i == 3 ? k4 : i == 4 ? k5 : i == 5 ? k6 : k7;
      rhs_dispatch<G, false, G == 32>(m, s, s.arg, srcp, pr, out, false, &cs);
      n_rhs += 1;
    }
    double part = 0.0;
    int bad = 0;
    for (int e = g.lane; e < N; e += G) {
      const double us = s.arg[e];
      const double d = h * fma(dp::E7, k7[e], fma(dp::E6, k6[e], fma(dp::E5, k5[e], fma(dp::E4, k4[e],
                                                                                   fma(dp::E3, k3[e], dp::E1 * k1[e])))));
      const double r = d / fma(P.rtol, fabs(us), P.atol);
      part = fma(r, r, part);
      bad |= (__double2hiint(us) & 0x7ff00000) == 0x7ff00000;
    }
    const double err = sqrt(g.sum(part) * (1.0 / N));
    bad = g.any(bad);
    const int att = n_att;
    n_att += 1;
    bool accept;
    double hnew;
    if (fixed) {
      accept = true;
      hnew = h;
    } else {
      const bool fin = (__double2hiint(err) & 0x7ff00000) != 0x7ff00000;
      float fac = (float)FAC_MIN;  // FP32 factor, as in the ROK4E controller
      if (fin)
        fac = fminf((float)FAC_MAX, fmaxf((float)FAC_MIN, (float)dp::SAFETY *
                                                              exp2f(-0.2f * __log2f(fmaxf(__double2float_rn(err),
                                                                                          (float)ERR_FLOOR)))));
      hnew = h * (double)fac;
      accept = fin && err <= 1.0;
    }
    if (P.trace && att < P.trace_cap && g.lane == 0) P.trace[cell * P.trace_cap + att] = accept ? h : -h;
    if (accept) {
      if (bad) {
        status = RK_CELL_NONFINITE;
        break;
      }
      for (int e = g.lane; e < N; e += G) s.u[e] = s.arg[e];
      g.sync();
      double* tk = k1;  // first same as last: f(u_{n+1}) is k7
      k1 = k7;
      k7 = tk;
      t += h;
      n_acc += 1;
      h_last = hnew;
      h = hnew;
    } else {
      n_rej += 1;
      h = hnew;
      if (h < H_MIN_FRAC * dt) {
        status = RK_CELL_STEP_UNDERFLOW;
        break;
      }
    }
  }
  for (int e = g.lane; e < N; e += G) P.Y[cell * N + e] = s.u[e];
  if (g.lane == 0) {
    if (P.h_cell) P.h_cell[cell] = h_last;
    if (P.stats) {
      P.stats[4 * cell + 0] = n_acc;
      P.stats[4 * cell + 1] = n_rej;
      P.stats[4 * cell + 2] = n_rhs;
      P.stats[4 * cell + 3] = status;
    }
  }
  g.sync();
}

template <int G>
__global__ void __launch_bounds__(rkdp_threads(G), 1) rkdp_integrate_kernel(IntegrateParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  load_exp_table(reinterpret_cast<uint64_t*>(smem));
  load_mech(smem + EXP_TAB_BYTES, P.mech, P.mech_copy);
  load_mech(smem + EXP_TAB_BYTES + P.mech_copy, P.mech + P.L.off_lo, P.fx_copy);
  __syncthreads();
  MechView m = make_view(smem + EXP_TAB_BYTES, P.mech, P.L, P.mech_copy, P.fx_copy > P.L.off_fA - P.L.off_lo);
  m.etab = reinterpret_cast<const uint64_t*>(smem);
  m.nx = P.nx;
  const Grp<G> g;
  const int gid = threadIdx.x / G;
  double* base = reinterpret_cast<double*>(smem + EXP_TAB_BYTES + P.mech_copy + P.fx_copy) + (size_t)gid * P.S.stride;
  const SlotPtrs s = slot_ptrs(base, P.S);
  init_sentinels<false>(s, m.ns, g.lane);
  g.sync();
  drain_queue<G>(P, g, gid, [&](int64_t cell) { integrate_cell_rkdp<G>(m, s, P, cell); });
}

}  // namespace rk

#include "adjoint.cuh"

namespace rk {

// ------------------------------------------------------------ adjoint kernels
struct AdjointParams {
  const unsigned char* mech;
  MechLayout L;
  AdjLayout A;
  const double* ckpt;        // [(nsteps + 1) x ncell x N] states at the start of every step
  const double* ubar_final;  // [ncell x N] dL/du(t_end)
  double* grad_u0;           // [ncell x N] dL/du(0), or null
  double* wsd;
  Dual* wsD;
  int64_t ncell;
  double p, h;
  int nsteps, M;
};

// One group of G lanes per cell (see adjoint.cuh); 128-thread blocks, at most
// as many as are resident at once, the cells dealt to them in turn (cell c to
// block c mod gridDim.x) when there are more cells than slots.
template <int G>
__global__ void __launch_bounds__(128) rok4e_adjoint_kernel(AdjointParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  load_exp_table(reinterpret_cast<uint64_t*>(smem));
  // everything before the integrators' segment
  unsigned char* base = smem + EXP_TAB_BYTES;
  load_mech(base, P.mech, P.L.off_lo);
  __syncthreads();
  MechView m = make_view(base, base, P.L, P.L.off_lo, false);
  m.lo = reinterpret_cast<const double*>(base + P.L.off_lo17);
  m.hi = reinterpret_cast<const double*>(base + P.L.off_hi17);
  m.etab = reinterpret_cast<const uint64_t*>(smem);
  const Grp<G> g;
  const int gpb = blockDim.x / G;
  const int64_t stride = (int64_t)gridDim.x * gpb;
  const int N = m.ns + 1;
  // whole groups take each cell, so a group's lanes agree on every branch
  for (int64_t c = blockIdx.x + (int64_t)gridDim.x * (threadIdx.x / G); c < P.ncell; c += stride) {
    const AdjFrame F = adj_frame(P.wsd, P.wsD, P.A, c);
    for (int e = g.lane; e < N; e += G) F.ubar[e] = P.ubar_final[c * N + e];
    for (int j = g.lane; j < m.nr; j += G) F.theta[j] = 0.0;
    for (int n = P.nsteps - 1; n >= 0; --n) {
      const double* un = P.ckpt + ((int64_t)n * P.ncell + c) * N;
      for (int e = g.lane; e < N; e += G) F.u[e] = un[e];
      adj_step<G>(m, F, P.p, P.h, P.M, P.A.tape0, P.A.tape_len);
    }
    if (P.grad_u0)
      for (int e = g.lane; e < N; e += G) P.grad_u0[c * N + e] = F.ubar[e];
    g.sync();
  }
}

// One group per cell: f(u) + src, or J(u) v.
struct PointParams {
  const unsigned char* mech;
  MechLayout L;
  SlotLayout S;
  const double* Y;
  const double* src;
  const double* V;
  double* out;
  int64_t ncell;
  double p;
  int mode;  // 0 rhs, 1 analytic jvp, 2 finite-difference jvp, 3 mixed rhs, 4 FP32 analytic jvp,
             // 5 analytic jvp with the double-float core, 6 rhs with the tensor-core gather,
             // 7 analytic jvp with the tensor-core gather, 8 FP32 analytic jvp on the FP64 caches
  const double* rho_cell;  // constant-volume densities, or null
  int nx;                  // state components after T (5: auxiliary-temperature system)
  int64_t mech_copy;       // bytes of the mechanism copied to shared memory (a prefix)
  int64_t fx_copy;         // bytes of the segment copied after that (without its fixed-point part where that does not fit)
  int64_t tc_bytes;        // modes 6 and 7: bytes of nu^T tiles copied after both (else 0)
};

template <int G>
__global__ void __launch_bounds__(POINT_BLOCK_THREADS, 1) chem_point_kernel(PointParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  load_exp_table(reinterpret_cast<uint64_t*>(smem));
  load_mech(smem + EXP_TAB_BYTES, P.mech, P.mech_copy);
  load_mech(smem + EXP_TAB_BYTES + P.mech_copy, P.mech + P.L.off_lo, P.fx_copy);
  if (P.tc_bytes) load_mech(smem + EXP_TAB_BYTES + P.mech_copy + P.fx_copy, P.mech + P.L.off_nuT, P.tc_bytes);
  __syncthreads();
  MechView m = make_view(smem + EXP_TAB_BYTES, P.mech, P.L, P.mech_copy, P.fx_copy > P.L.off_fA - P.L.off_lo);
  m.etab = reinterpret_cast<const uint64_t*>(smem);
  m.nx = P.nx;
  if (P.tc_bytes) m.nuT = reinterpret_cast<const uint4*>(smem + EXP_TAB_BYTES + P.mech_copy + P.fx_copy);
  const Grp<G> g;
  const int gid = threadIdx.x / G;
  const int gpb = blockDim.x / G;
  const int64_t cell = (int64_t)blockIdx.x * gpb + gid;
  if (cell >= P.ncell) return;
  double* base = reinterpret_cast<double*>(smem + EXP_TAB_BYTES + P.mech_copy + P.fx_copy + P.tc_bytes) + (size_t)gid * P.S.stride;
  const SlotPtrs s = slot_ptrs(base, P.S);
  if (P.mode >= 3 && P.mode <= 5) init_sentinels<true>(s, m.ns, g.lane);
  else init_sentinels<false>(s, m.ns, g.lane);
  if (P.mode == 6 || P.mode == 7)
    for (int i = g.lane; i < 8 * 16 * m.nrt; i += G) s.dig[i] = 0;
  const int N = m.ns + 1 + m.nx;
  for (int e = g.lane; e < N; e += G) {
    s.u[e] = P.Y[cell * N + e];
    s.src[e] = P.src ? P.src[cell * N + e] : 0.0;
    if (P.V && P.S.F >= 0) s.F[e] = P.V[cell * N + e];
  }
  g.sync();
  const double pr = P.rho_cell ? -P.rho_cell[cell] : P.p;
  CellScalars cs;
  cs.pinv = 1.0 / fabs(pr);
  cs.prec = 0;
  if (P.mode == 8) {
    cs.prec = 6;
    rhs_eval_call<G>(m, s, s.u, nullptr, pr, s.fn, true, &cs);
    jvp_eval_f32x<G>(m, s, s.u, cs, s.F, s.w);
    for (int e = g.lane; e < N; e += G) P.out[cell * N + e] = s.w[e];
    return;
  }
  if (P.mode == 7) {
    cs.prec = 4;
    rhs_eval_call<G, false, true>(m, s, s.u, nullptr, pr, s.fn, true, &cs);
    jvp_eval<G, false, true>(m, s, s.u, cs, s.F, s.w);
    for (int e = g.lane; e < N; e += G) P.out[cell * N + e] = s.w[e];
    return;
  }
  if (P.mode == 0 || P.mode == 3 || P.mode == 6) {
    if (P.mode == 3) rhs_eval_call<G, true>(m, s, s.u, P.src ? s.src : nullptr, pr, s.fr, false, &cs);
    else if (P.mode == 6) rhs_eval_call<G, false, true>(m, s, s.u, P.src ? s.src : nullptr, pr, s.fr, false, &cs);
    else rhs_eval_call<G>(m, s, s.u, P.src ? s.src : nullptr, pr, s.fr, false, &cs);
    for (int e = g.lane; e < N; e += G) P.out[cell * N + e] = s.fr[e];
    return;
  }
  if (P.mode == 4) {
    rhs_eval_call<G, true>(m, s, s.u, nullptr, pr, s.fn, true, &cs);
    jvp_eval_f32<G>(m, s, s.u, cs, s.F, s.w);
    for (int e = g.lane; e < N; e += G) P.out[cell * N + e] = s.w[e];
    return;
  }
  if (P.mode == 5) {
    cs.prec = 3;
    rhs_eval_call<G>(m, s, s.u, nullptr, pr, s.fn, true, &cs);
    jvp_eval_df<G>(m, s, s.u, cs, s.F, s.w);
    for (int e = g.lane; e < N; e += G) P.out[cell * N + e] = s.w[e];
    return;
  }
  // the auxiliary-temperature T row depends on the source; elsewhere s.src is
  // zero here, so the finite difference sees the bare source term
  rhs_eval_call<G>(m, s, s.u, m.nx > 0 ? s.src : nullptr, pr, s.fn, true, &cs);
  int n_rhs = 0;
  double unorm = 0.0;
  if (P.mode == 2) unorm = sqrt(group_dot<G>(g, s.u, s.u, N));
  apply_jv<G>(m, s, cs, P.mode == 1 ? 0 : 1, pr, unorm, s.F, s.w, &n_rhs);
  for (int e = g.lane; e < N; e += G) P.out[cell * N + e] = s.w[e];
}

}  // namespace rk

struct rk_mech {
  rk::HostMech host;
  unsigned char* dev = nullptr;
  int device = 0;
};

namespace rk {

struct LaunchPlan {
  int G = 32;
  int cells_per_block = 1;
  size_t smem = 0;
  int blocks = 1;
};

inline int device_props(int* n_sm, size_t* smem_optin) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
  int v = 0;
  e = cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return cuda_error(e, "cudaDeviceGetAttribute");
  *n_sm = v;
  e = cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return cuda_error(e, "cudaDeviceGetAttribute");
  *smem_optin = (size_t)v;
  return RK_OK;
}

// The bytes of the segment a block copies: all of it, or the thermo coefficients
// alone where it and `rest` (the prefix, one cell's slot, tiles) do not fit in
// shared memory; such a mechanism runs in the direct form.
inline int64_t segment_bytes(const MechLayout& L, int64_t rest) {
  int n_sm = 0;
  size_t smem_max = 0;
  const int64_t seg = L.off_fx_end - L.off_lo;
  if (device_props(&n_sm, &smem_max) != RK_OK) return seg;
  return rest + seg + EXP_TAB_BYTES + 64 <= (int64_t)smem_max ? seg : L.off_fA - L.off_lo;
}

// Shared memory that precision 4 counts beside its tiles when it decides whether
// it can run: the mechanism arrays and one cell's slot of its first layout.  The
// present layout needs less; the limit on the mechanism's size stays where callers
// know it, and what was refused stays refused.
inline int64_t tensor_core_bytes(const MechLayout& L, int M, int nx) {
  auto even = [](int64_t n) { return (n + 1) & ~int64_t(1); };
  auto al = [](int64_t b) { return (b + 15) & ~int64_t(15); };
  const int64_t ns = L.ns, nr = L.nr, nr1 = nr > 0 ? nr : 1, N = ns + 1 + nx, Nq = even(N);
  const int64_t mech = 3 * al(8 * ns) + 2 * al(8 * 17 * ns) + 3 * al(8 * nr) + al(8 * L.ntb * ns) +
                       al(64 * (int64_t)L.ntb) + al(8 * (int64_t)L.nnz) + 2 * al(4 * nr) + 2 * al(4 * (ns + 1)) +
                       al(4 * (int64_t)L.nnz) + al(4 * ((int64_t)L.npiece + 1));
  int64_t d = 7 * Nq + Nq * M + 10 * even(ns + 1) + 4 * even(nr1) + (4 * Nq <= 3 * even(nr1) ? 0 : 4 * Nq) +
              even(4 * (L.ntb > 0 ? L.ntb : 1)) + even(11 * (L.ntroe > 0 ? L.ntroe : 1)) +
              even(L.npiece > 0 ? L.npiece : 1) + 32 * (int64_t)L.nrt + 3 * 8 * M + 12;
  d = (d + 3) & ~int64_t(3);
  return mech + 8 * d + (int64_t)512 * L.nst * L.nrt + EXP_TAB_BYTES;
}

template <int G, typename K>
int plan_for(K kernel, const rk_mech* mech, const SlotLayout& S, int want_cells, int64_t ncell, bool persistent,
             LaunchPlan* plan, int want_blocks_per_sm = 0, bool fill_device = false, int64_t copy_bytes = -1,
             int max_threads = MAX_BLOCK_THREADS) {
  int n_sm = 0;
  size_t smem_max = 0;
  int rc = device_props(&n_sm, &smem_max);
  if (rc) return rc;
  const size_t mech_bytes = (size_t)(copy_bytes >= 0 ? copy_bytes : mech->host.L.bytes) + EXP_TAB_BYTES;
  const size_t slot_bytes = (size_t)S.stride * sizeof(double);
  smem_max -= 64;  // the kernels' static shared memory (queue counters)
  if (mech_bytes + slot_bytes > smem_max)
    return set_error(RK_E_UNSUPPORTED, "mechanism plus one cell's work arrays exceed shared memory");
  int cells = (int)((smem_max - mech_bytes) / slot_bytes);
  cells = cells > max_threads / G ? max_threads / G : cells;
  if (want_cells > 0 && want_cells < cells) cells = want_cells;
  if (!persistent && (int64_t)cells > ncell) cells = (int)(ncell > 0 ? ncell : 1);
  size_t smem = mech_bytes + (size_t)cells * slot_bytes;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute");
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, cells * G, smem);
  if (e != cudaSuccess) return cuda_error(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
  while (per_sm == 0 && cells > 1) {  // registers limit: shrink the block
    cells /= 2;
    smem = mech_bytes + (size_t)cells * slot_bytes;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, cells * G, smem);
    if (e != cudaSuccess) return cuda_error(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
  }
  if (per_sm == 0) return set_error(RK_E_UNSUPPORTED, "integration kernel cannot be resident on an SM");
  if (want_blocks_per_sm > 0 && want_blocks_per_sm < per_sm) per_sm = want_blocks_per_sm;
  plan->G = G;
  plan->cells_per_block = cells;
  plan->smem = smem;
  const int64_t need = (ncell + cells - 1) / cells;
  int64_t blocks = persistent ? (int64_t)per_sm * n_sm : need;
  if (persistent && blocks > need && !fill_device) blocks = need;
  plan->blocks = (int)(blocks > 0 ? blocks : 1);
  return RK_OK;
}

// Launches of the per-cell kernels.  Each instantiation is defined (and its
// kernel compiled) in one translation unit of its own, through launchers.cuh;
// the C ABI calls them through these declarations.
struct IntegrateLaunch {
  IntegrateParams* P;
  const rk_mech* mech;
  int cells_per_block, blocks_per_sm;
  bool static_bins;  // queue order 3: the block's static bins are dealt in sub-queues
  int64_t ncell;
  cudaStream_t stream;
};
template <int G, bool MIXED, bool TC>
int launch_rok4e(const IntegrateLaunch& a);
template <int THREADS>
int launch_rok4e_wide(const IntegrateLaunch& a);  // FP64, one warp per cell, more than eight cells a block
template <int G>
int launch_rkdp(const IntegrateLaunch& a);
template <int G>
int launch_adjoint(const AdjointParams& P, size_t smem, cudaStream_t st);

}  // namespace rk
