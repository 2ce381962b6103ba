// Internal declarations of the GB300 messenger-field Wiener filter library.
// Device data layout (one plan = one HEALPix nside and one lmax):
//   rings      R  = 4 nside - 1, north to south; ring pairs RP = 2 nside
//              (pair k = north ring k and south ring R-1-k; the equator ring
//              2 nside - 1 is a pair of its own, its south slot unused).
//   Fourier    F[m * RP + k] = double4_32a (north re, north im, south re, south im),
//              m = 0 .. lmax, the azimuthal coefficients of ring pair k.
//              FS: synthesis side (from a_lm), FT: analysis side (to a_lm).
//              Native FP64 stages hold doubles; the double-float stages (ring_df,
//              legendre_df, legendre_tab, spin-2) hold each value as its (hi, lo)
//              floats in the same 8 bytes (df_pack), and FT without the last factor
//              of Omega (LegArgs::fomega), which the analysis multiplies its sums by.
//   a_lm       m-major complex doubles, index(l, m) = m (2 lmax + 1 - m) / 2 + l.
//   maps       RING order doubles.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/wf.h"

namespace wfk {

constexpr int kThreads = 256;       // block size of the per-m Legendre kernels
constexpr int kRingThreads = 512;   // block size of the ring (FFT) kernels: one CTA per ring fills
                                    // an SM's shared memory, so its own warps must hide the latency
constexpr int kLB = 16;             // l values per block of the analysis reduction
constexpr int kStartExp = -100;     // Legendre terms below 2^-100 are not evaluated

// Per-ring description (host-built, read by the ring kernel).
struct RingDev {
  long long off;      // first pixel (RING index)
  int n;              // pixels in the ring (nphi)
  int pair;           // ring pair index k
  int side;           // 0 = north slot, 1 = south slot of the pair
  int shifted;        // first pixel at phi = pi / n (else at phi = 0)
  int logM;           // log2 of the FFT size (n itself, or the Bluestein size)
  int blue;           // 1: n is not a power of two, Bluestein convolution of size M
  long long hs_off;   // offset of this ring length's half-shift table e^{i pi q / n}
  long long ch_off;   // offset of this ring length's chirp e^{-i pi j^2 / n} (Bluestein only)
  long long B_off;    // offset of this ring length's Bluestein filter (bit-reversed, / M)
};

// Rings grouped by FFT size for the ring-stage launches: each class is one
// launch whose shared memory is sized for its own largest FFT (instead of the
// plan's largest), so the many rings with small or power-of-two FFTs run more
// CTAs per SM. order[first .. first + count) lists the class's rings, the two
// rings of a pair next to each other so that the halves of each Fourier
// coefficient record are read and written close together in time.
struct RingClass {
  int logM;    // the largest log2 FFT size in the class
  int first;   // offset into the ring order
  int count;   // rings in the class
  int global;  // 1: the class's FFT buffers do not fit shared memory and live in a global
               //    scratch array, 2^logM 16-byte elements per CTA (CTA i of the class at i 2^logM)
};

// Largest dynamic shared memory a ring-stage CTA asks for (of the 227 KB a CTA
// may use on this GPU; the rest is left for static arrays).
constexpr size_t kRingSmemLimit = 200 * 1024;

// Iteration controller state, resident on the device (Sect. 3 schedule).
struct Ctl {
  // configuration
  int mode;             // 0: fixed lambda and lsht for n_fixed iterations; 1: cooling schedule
  int n_fixed;
  int max_iter;
  int cooling, l_iter0, margin, band_limit, min_level_iters, max_level_iters;
  int lmax;
  double tol, plateau_eps, final_dchi2, sigma_chi2, tau, omega;
  // live state
  double lambda;
  int lsht, l_iter, level, level_iters, iter, done, converged, numeric;
  int have_prev;
  double prev_chi2;
  double last_rel;
};

// Record layout of one iteration (mirrors wf_iter_record).
static_assert(sizeof(wf_iter_record) == 6 * 8 + 2 * 4, "record layout");

struct Plan;

// ---------------------------------------------------------------- launches
// ring kernel modes
enum { RING_SYNTH = 0, RING_ANALYSIS = 1, RING_ITER = 2 };
// Legendre kernel modes
enum { LEG_SYNTH = 0, LEG_ANALYSIS = 1, LEG_ITER = 2 };

struct RingArgs {
  const RingDev *rings;
  const int *order;       // ring of CTA i is order[first + i] (nullptr: first + i)
  const int2 *porder;     // double-float ring stage: (north ring, south ring or -1) of CTA i at porder[first + i]
  int first;
  void *scratch;          // global FFT buffers of a class that does not fit shared memory (else nullptr)
  const double2 *tw;      // e^{-2 pi i k / Mmax}, k < Mmax / 2
  int logMmax;
  const double2 *hs, *chirp, *B;
  const double4_32a *FS;      // synthesis input (RING_SYNTH / RING_ITER)
  double4_32a *FT;            // analysis output (RING_ANALYSIS / RING_ITER)
  int RP;
  const double *map_in;   // RING_ANALYSIS input
  double *map_out;        // RING_SYNTH output
  const double *d, *w;    // RING_ITER: data, inverse noise (0 = masked)
  double *ring_part;      // RING_ITER: [R][2] chi2_N, chi2_lambda_N partials
  const Ctl *ctl;         // RING_ITER: lambda, lsht, done
  int lsht;               // standalone modes
  double omega, tau;
  float fscale;           // double-float records FT: the power of two in (Omega / 4, Omega / 2]
  double *gain;           // [npix] cached w / (1 + (lambda - 1) tau w) (double-float ring kernel)
  double *gainlam;        // [R] lambda the cached gains of each ring belong to (-1: none)
  const Ctl *gate;        // RING_SYNTH / RING_ANALYSIS inside a controlled iteration: skip once gate->done
};

struct LegArgs {
  const double *x;        // [RP] cos(theta) of the north ring of each pair
  const double2 *rec;     // [nalm] recurrence coefficients (a_l, b_l)
  const int *ls;          // [(lmax+1) RP] first evaluated l
  const double2 *sv;      // [(lmax+1) RP] (lambda_{ls}, lambda_{ls+1})
  const double *cl;       // [lmax+1]
  const double4_32a *FT;      // analysis input
  double4_32a *FS;            // synthesis output
  double2 *alm;           // state / output a_lm
  const double2 *alm_in;  // LEG_SYNTH input
  double *m_part;         // LEG_ITER: [lmax+1][3] chi2_S, incr2, norm2
  double *part;           // LEG_ITER, table form: [lmax+1][tab_chunks(lmax)][3]
  float4 *coef;           // LEG_ITER, table form: [nalm] the new state in double-float
  const Ctl *ctl;
  const Ctl *gate;        // LEG_SYNTH / LEG_ANALYSIS inside a controlled iteration: skip once gate->done
                          // (nullptr for the standalone transforms)
  int lsht, lmax, RP;
  double omega, tau;
  double fomega;          // double-float stages: Omega / 2 over RingArgs::fscale
};

// Tables of the double-float Legendre kernel (legendre_df.cu).
struct LegDfArgs {
  const float2 *A;        // [nalm] rescaled recurrence coefficient A_l (hi, lo)
  const double *g;        // [nalm] rescaling factor g_l (lambda = g mu)
  const int *ls;          // [(lmax+1) RP] first evaluated l (|lambda| >= 2^-60)
  const float4 *sv;       // [(lmax+1) RP] mu_{ls} (hi, lo), mu_{ls+1} (hi, lo)
  const float4 *tab;      // precomputed lambda (hi, lo) in rows of two l, or nullptr (recurrence)
  const long long *poff;  // [lmax+1] first table row of each m
};

// Legendre stage over the precomputed table (legendre_tab.cu), for up to
// kLegBatchMax maps of one shape, each with its own Fourier arrays, state, C_l,
// tau, partial sums and controller.
constexpr int kLegBatchMax = 2;
constexpr int kTabRows = 96;      // table rows (two l each) of an analysis CTA
struct LegBatchMaps {
  int n;                          // maps in use (the rest are skipped)
  const double4_32a *FT[kLegBatchMax];
  double4_32a *FS[kLegBatchMax];
  double2 *alm[kLegBatchMax];     // state; the standalone transforms' a_lm in (synthesis) or t_l out (analysis)
  const Ctl *ctl[kLegBatchMax];   // controller; standalone transforms: skip the map once done (nullptr: never)
  // an iteration's, nullptr for the standalone transforms
  double *m_part[kLegBatchMax];   // [lmax+1][3] chi2_S, incr2, norm2
  double *part[kLegBatchMax];     // [lmax+1][tab_chunks(lmax)][3] the same by chunk of rows
  float4 *coef[kLegBatchMax];     // [nalm] the new state as double-floats (re hi, re lo, im hi, im lo)
  const double *cl[kLegBatchMax];
  double tau[kLegBatchMax];
};
// chunks of kTabRows rows of the longest column (m = 0)
int tab_chunks(int lmax);
// mode: LEG_ITER (nb independent iterations), LEG_SYNTH or LEG_ANALYSIS; nb = 1 or 2
void launch_legendre_tab(const LegArgs &a, const LegDfArgs &d, const LegBatchMaps &bm, int nb, cudaStream_t s,
                         int mode);

// Double-float copies of the ring-stage tables (ring_df.cu): float4 =
// (re hi, re lo, im hi, im lo).
struct RingDfArgs {
  const float4 *tw, *hs, *chirp, *B;
  const float2 *d, *w;    // [npix] data and inverse noise as double-float (RING_ITER)
  float2 *gain;           // [npix] cached Eq. 3 gains as double-float
  double *gainlam;        // [R] lambda the cached gains of each ring belong to (-1: none)
};
void launch_to_df2(const double *src, float2 *dst, long long n, cudaStream_t s);
// The twiddles laid out by stage (fft.cuh) for FFTs up to 2^logMmax, from tw[k] = e^{-2 pi i k / 2^logMmax}:
// entries, and the kernels that place them (double-float and, from its high parts, FP32)
inline long long twiddles_df(int logMmax) { return logMmax < 2 ? 1 : 3 * ((1LL << (logMmax - 1)) - 1); }
inline long long twiddles_f32(int logMmax) { return 6 * ((1LL << ((logMmax < 4 ? 4 : logMmax) - 3)) - 1); }
void launch_pack_twiddles(const double2 *tw, int logMmax, float4 *df, float2 *f32, cudaStream_t s);
// One map of a double-float ring-stage launch: what a RingArgs and RingDfArgs hold beside the shape's tables.
constexpr int kRingMapsMax = 4;
struct RingMap {
  const double4_32a *FS;
  double4_32a *FT;
  const double *map_in;
  double *map_out;
  const float2 *d, *w;
  const double *w64;
  float2 *gain;
  double *gainlam;
  double *ring_part;
  const Ctl *ctl, *gate;
  double tau;
};
struct RingMaps { RingMap m[kRingMapsMax]; };

// Batched engine (batch_kernels.cu): B slots of one shape in lockstep.
constexpr int kBatchMax = 64;

struct BatchArgs {
  const RingDev *rings;
  const int2 *porder;        // ring pair of ring-stage CTA i: porder[first + i] = (north ring, south ring or -1)
  int first;
  const float4 *hsf, *chf;
  const float2 *tw2, *Bf2;   // FP32 twiddles by stage and Bluestein filter tables (hi parts)
  int logMmax;
  int lmax, RP, R, B;
  long long npix, nalm;
  double omega;
  const double *d, *w, *cl;  // [B][npix], [B][npix], [B][lmax+1]
  float2 *dw32;              // [B][npix] (d, w) in FP32, read by the mixed-precision ring stage
  double2 *s;                // [B][nalm] exported a_lm of finished slots
  float4 *sdf;               // [B][nalm] state, double-float (re hi, re lo, im hi, im lo), in the
                             // order of the analysis table rows: (m, parity of l - m, (l - m) / 2)
  const int *alm_of_row;     // [nalm] a_lm index m (2 lmax + 1 - m) / 2 + l of each state row
  float2 *fdf;               // [lmax+1][B] Eq. 4 filter f_l(lambda_b) of this iteration, double-float
  float *icl;                // [lmax+1][B] 1 / C_l (0 where C_l = 0)
  float4 *FS, *FT;           // [(m RP + k) B + b] (north re, north im, south re, south im)
  Ctl *ctl;                  // [B]
  const int *active;         // [B]
  double *ring_part;         // [B][R][2]
  double *m_part;            // [B][ntiles][3]
  int ntiles;                // analysis tiles (partials per slot)
  const int *bstate;         // [0] largest live band limit, [1] live slots
  wf_iter_record *last;      // [B]
};

// Tensor-core Legendre stage of the batched engine (batch_tc.cu): work lists,
// per-iteration operands and the error flag of the bounded pipeline waits.
struct TcArgs {
  int Nc;                    // GEMM columns: 2 B (re, im of every slot), a multiple of 16
  int RPp, nkc;              // ring pairs padded to a multiple of 32, and RPp / 32
  const int4 *atiles;        // analysis tiles (m, parity, first i, first lamA row of (m, parity))
  int natiles;
  const int2 *stiles;        // synthesis tiles (m, first ring pair)
  int nstiles;
  const int *offTc;          // [2 (lmax+1)] first 32-wide i chunk of (m, parity)
  float *XT, *SPT;           // analysis / synthesis B operands
  int *err;                  // set when a pipeline wait gave up
  // streamed synthesis table: a launch covers synthesis tiles from tile0 and reads the
  // synthesis-ordered rows of chunks from qbase, rebuilt from lamA into a scratch array
  int tile0, qbase;
  const int4 *chunk_info;    // [nchunks] (first lamA row of the chunk, rows in it, m, 0)
  const float *lamA;
  float *lamTs;              // scratch of the streamed synthesis table (nullptr: resident lamT)
  // split tables: lamA and lamT hold th in their first rows and tl from row loA / loT
  int pre;
  int loA, loT;
};

// A band of m whose synthesis table is rebuilt and used in one step: chunks
// [q0, q1) and synthesis tiles [tile0, tile1).
struct SynBand {
  int q0, q1, tile0, tile1;
};

void launch_lam_tc_tables(const double *x, const LegDfArgs &D, int lmax, int RP, int RPp, const int *offTc,
                          float *lamA, float *lamT, bool split, size_t loA, size_t loT, cudaStream_t s);
struct TcMaps;
// groups: slots per ring-stage CTA for each class (0 or nullptr: the default rule)
void launch_batch_iteration(const BatchArgs &a, const TcArgs &t, const TcMaps &maps, const RingClass *cls, int ncls,
                            const int *groups, int *bstate, cudaStream_t s, const SynBand *bands, int nbands);
void launch_batch_ring_class(const BatchArgs &a, const RingClass &c, int G, cudaStream_t s);
bool batch_ring_group_ok(int logM, int G);
void launch_batch_state(const BatchArgs &a, int *bstate, cudaStream_t s);
void launch_batch_zero_slot(const BatchArgs &a, const TcArgs &t, long long nchunks, int b, cudaStream_t s);
void launch_batch_convert_slot(const BatchArgs &a, int b, cudaStream_t s);
void launch_batch_export_slot(const BatchArgs &a, int b, cudaStream_t s);
void launch_hi_table(const float4 *src, float2 *dst, long long n, cudaStream_t s);

void launch_ring(const RingArgs &a, const RingClass *cls, int ncls, cudaStream_t s, int mode);
// nmaps maps of one shape (a[i], t[i]; the tables and the band limit are those of the first) in as few launches as
// kRingMapsMax allows
void launch_ring_df(const RingArgs *a, const RingDfArgs *t, int nmaps, const RingClass *cls, int ncls,
                    cudaStream_t s, int mode);
// ring order and classes of a ring table (host; rings as built for the plan)
void ring_classes(const RingDev *rings, int R, std::vector<int> &order, std::vector<RingClass> &cls);
void launch_to_df(const double2 *src, float4 *dst, long long n, cudaStream_t s);
void launch_legendre(const LegArgs &a, cudaStream_t s, int mode);
void launch_legendre_df(const LegArgs &a, const LegDfArgs &d, cudaStream_t s, int mode);
void launch_posterior_maps(const double *d, const double *w, double *ya, double *wd, long long npix, cudaStream_t s);
void launch_posterior_norms(const double2 *a, const double2 *ta, const double2 *tb, const double *cl, int lmax,
                            double inv_omega, double *part, cudaStream_t s);
// rows of the precomputed double-float lambda table: of one m (two l each), and of all
__host__ __device__ inline int tab_rows(int lmax, int m) { return (lmax - m + 2) / 2; }
size_t lam_table_rows(int lmax);
// Whether the double-float stages of a shape take the finer forms (FINE: df.cuh, fft.cuh) of their sums and products.
// Their roundings show in short sums and short FFTs: without them the transforms' errors at Nside 8 to 32 are up to
// 1.07 (E and B: 1.25, recurrence form: 1.2) times what they are with records and sums over lanes in double, with them
// 0.96 to 1.01 times. From Nside 128 on folding long sums back (dot2_tidy) does more for the error (0.5 to 0.99 times).
// Latency bounds the kernels up to Nside 64, so they cost little: Nside 16 solve 12.97 ms, 12.47 without the FFT's; a
// T + P solve at Nside 128, bound by FP32 issue in these sums, took 68 instead of 62 ms with them.
inline bool fine_steps(int RP) { return RP <= 128; }
// largest dynamic shared memory of the table form's kernels
size_t leg_tab_smem(int lmax, int RP);
void launch_lam_table(const double *x, const double2 *rec, const int *ls64, const double2 *sv64, const int *ls_df,
                      const long long *poff, int lmax, int RP, float4 *tab, cudaStream_t s);
void launch_df_tables(const double *x, const double2 *rec, int lmax, int RP, double *g, float2 *A, int *ls,
                      float4 *sv, cudaStream_t s);
void launch_start_values(const double *x, const double2 *rec, int lmax, int RP, int *ls,
                         double2 *sv, cudaStream_t s);
void launch_bluestein_setup(const RingDev *rings, const int *order, const RingClass *cls, int ncls, void *scratch,
                            const double2 *tw, int logMmax, const double2 *chirp, double2 *B, cudaStream_t s);
// The controllers of n maps, each with its own partial sums ([R][2] and [lmax+1][3]) and records.
constexpr int kCtlMapsMax = 4;
struct CtlMap {
  Ctl *ctl;
  const double *ring_part, *m_part, *cl;
  wf_iter_record *hist;
  int hist_cap;
};
struct CtlMaps { CtlMap m[kCtlMapsMax]; };
void launch_control(const CtlMap *maps, int n, int R, int lmax, cudaStream_t s);

// Raise a kernel's dynamic shared-memory cap to the device's opt-in maximum
// (once per function). The cap is an attribute of the function, read when a
// launch or a captured graph node runs, so launches of one kernel with
// different shared-memory sizes (ring classes, plans of different shapes)
// must never lower it under one another.
void raise_smem_cap(const void *func);

// error plumbing
void set_error(const std::string &msg);
wf_status cuda_status(cudaError_t e, const char *where);

// iters times one() on s as an executable graph. A launch that is refused while a stream is being captured ends neither
// the capture nor the graph, which would then leave that kernel out: its error is looked at here.
template <class F>
wf_status capture_graph(cudaStream_t s, int iters, cudaGraphExec_t *exec, const char *what, F one) {
  cudaGetLastError();   // an error of before is not this graph's
  cudaError_t e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return cuda_status(e, what);
  for (int i = 0; i < iters; ++i) one();
  const cudaError_t launched = cudaGetLastError();
  cudaGraph_t g = nullptr;
  e = cudaStreamEndCapture(s, &g);
  if (e == cudaSuccess) e = launched;
  if (e == cudaSuccess) e = cudaGraphInstantiate(exec, g, 0);
  if (g) cudaGraphDestroy(g);
  return e == cudaSuccess ? WF_OK : cuda_status(e, what);
}

}  // namespace wfk
