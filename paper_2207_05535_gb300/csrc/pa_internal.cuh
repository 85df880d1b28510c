// Internal layout shared by the engine's host code and its kernels.
//
// Device memory layout (one pool per engine, every run at its own offsets):
//   spins[b]  uint32 [sum R_cap wstride]    replica j of a run at word spin_off + j wstride:
//                                           colour plane 0 in words [0, PW), plane 1 in
//                                           [PW, 2 PW); site n = y L + x has colour (x + y) & 1
//                                           and sits in row y of its plane at bit position
//                                           y * pitch + (x >> 1) (rows padded to the pitch,
//                                           padding bits 0); bit 1 = spin +1; buffer b = step & 1
//   E[b], M[b], fam[b]   [sum R_cap]        energy, magnetisation, beta_0 ancestor
//   parent, cnt          [sum R_cap]        parent map of the children, copy numbers r_j
//   rec                  [sum n_beta]       per-temperature records (pa_step_record)
//   qh, qhp, qhw         [sum n_beta (N+1)] overlap histograms over d (shift / pair / Wang)
//   beta, thr                               schedule and Metropolis thresholds per step
//   wt, wtoff                               weight tables exp(-4 n dbeta) shared by every run
//                                           and step with the same (N, dbeta); wtoff[wt_off + i]
//                                           = offset of step i's table in wt.  Runs with
//                                           theta = PA_THETA_INF also keep per step the
//                                           cumulative level weights of P_beta_i over
//                                           u = 0..2N and, in entry 2N + 1, the last level
//                                           with a positive weight (as a double)
//   J                    per run: site-order "J = -1" bits of right / down bonds
//                        (2 wstride words), then per colour plane word the four bond
//                        masks (same, rotated, up, down neighbour) [2][4][PW]
//   scratch              per run: energy and magnetisation histograms (N+1 u32 each),
//                        level CDF or thresholds (N+1 f64 / u64), level fill counters or
//                        floors (N+1 u32), then members (R_cap u32) / per-CTA totals /
//                        per-CTA family statistics
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

#include <sys/mman.h>
#include <unistd.h>

#include "pa.h"

namespace pa {

constexpr uint32_t TAG_INIT = 1u, TAG_SWEEP = 2u, TAG_RESAMPLE = 3u, TAG_MULTINOMIAL = 4u, TAG_DISORDER = 5u,
                   TAG_DOS = 6u, TAG_WANG = 7u;
constexpr uint32_t WANG_IDX_BITS = 13u;  // PA_WANG_MAX_RCAP = 2^13

// status bits in the engine-wide device status word
constexpr uint32_t ST_CAPACITY = 1u << PA_ERR_CAPACITY;
constexpr uint32_t ST_EXTINCT = 1u << PA_ERR_EXTINCT;
constexpr uint32_t ST_TIMEOUT = 1u << PA_ERR_TIMEOUT;

struct RunDev {
    uint32_t L, N, Lh, wstride;  // wstride: words per replica, a multiple of 4
    uint32_t model, R, R_cap, theta;
    uint32_t n_beta, seed, run_id, disorder_id;
    uint32_t resample, overlap;
    int32_t paired;
    uint32_t pitch;  // bits per row in a colour plane (>= L/2; see row_pitch)
    uint32_t pw;     // words per colour plane = ceil(L pitch / 32)
    uint32_t pad0;
    uint64_t rep_off;   // first replica slot (E, M, fam, parent, cnt)
    uint64_t spin_off;  // first spin word (runs of different L have different wstride)
    uint64_t rec_off, qh_off, beta_off, wt_off, thr_off, J_off, scr_off;
    double ln2N;  // N ln 2 = ln Z(beta_0 = 0)
    uint64_t dos_off;  // theta = PA_THETA_INF: step i's energy CDF at wt[dos_off + i (2N + 2)]
};

struct RunState {
    uint32_t step;   // temperature index of the population held
    uint32_t R_cur;  // R_step
    uint32_t R_new;  // population size produced by the resampling in flight
    uint32_t status; // 0 or a pa_status that stopped the run
    double lnQ;      // ln Q of the resampling in flight
    uint32_t ticket;   // CTAs of the run done in the launch in flight (0 between launches)
    int32_t Emin;      // nearest-integer resampling in flight: lowest energy of the population
    uint32_t n_levels; // and its number of energy levels (Emax - Emin) / 4 + 1
    uint32_t pad;
};

// Kernels that split one population over several CTAs give each CTA about
// CTA_REPLICAS replicas, at most MAX_RUN_CTAS CTAs per run.
constexpr uint32_t CTA_REPLICAS = 16384, MAX_RUN_CTAS = 256;
__host__ __device__ inline uint32_t run_ctas(uint32_t R_cap)
{
    const uint32_t c = (R_cap + CTA_REPLICAS - 1) / CTA_REPLICAS;
    return c < 1 ? 1 : (c > MAX_RUN_CTAS ? MAX_RUN_CTAS : c);
}

// CTAs per run, for the largest of a launch's n_runs populations, of the nearest-integer resampling
// and the measurement: run_ctas, or more where the launch leaves SMs idle.  A CTA takes about 7 us and
// 1 us per 1000 replicas, and splitting a population 4 us for the second resampling launch; with two
// CTAs per SM, 304 run at once.  The split is taken where that predicts a gain of 15 %. One run of R =
// 16000: resampling 20.8 -> 15.8 us, measurement 21.8 -> 17.5; of R = 64000: 27.0 -> 15.9, 26.0 ->
// 21.0; 48 of R = 50000: 37 -> 29, 36 -> 30; 100 of R = 9000 19.0 -> 19.8, 21.9 -> 21.6.  A launch
// that fills the GPU gains nothing: 200 runs of R = 20000 take 42 and 42 us with 2 CTAs each.
inline uint32_t split_ctas(uint32_t n_runs, uint32_t max_Rcap)
{
    const uint32_t least = run_ctas(max_Rcap);
    if (max_Rcap <= 4096 || n_runs == 0) return least;
    auto us = [&](uint32_t nc) { return 7.0 + 1e-3 * max_Rcap / nc + (nc > 1 ? 4.0 : 0.0); };
    const uint32_t most = (uint32_t)std::min<uint64_t>({304 / n_runs, MAX_RUN_CTAS, (max_Rcap + 2047ull) / 2048});
    return most > least && us(most) < 0.85 * us(least) ? most : least;
}

// Threads per CTA of the measurement and of the nearest-integer resampling, for the largest population
// and lattice of a launch.  A run of few replicas is a chain of dependent steps that more threads do
// not shorten, and with 128 threads eight runs share an SM instead of two: 2048 runs of R = 100, L =
// 16: measurement 89 -> 37 us a step, resampling 36 -> 15 us.  But the measurement also clears, adds
// and scans N + 1 levels, which 512 threads do faster until their CTAs, two per SM, no longer run at
// once.  Measurement with 128 against 512 threads, R = 50 to 150: L = 20 14.9 / 15.2 us (152 runs), L
// = 32 17.7 / 17.0 (100), 18.4 / 19.6 (200), L = 64 30.9 / 21.7 (152), 33.8 / 26.0 (304), 35.4 / 41.9
// (400), L = 128 98 / 50 (304), 107 / 120 (700), L = 256 342 / 135 (304), 349 / 239 (400).
// Resampling, which scans only the occupied levels: R = 100 8.2 / 8.5 (one run), 8.3 / 12.6 (400), R =
// 700 10.0 / 8.6, 11.3 / 14.6.
constexpr uint32_t FEW_REPLICAS = 1024;  // capacity: R of about 740
inline uint32_t measure_threads(uint32_t n_runs, uint32_t max_Rcap, uint32_t max_N)
{
    const uint32_t at_once = max_N <= 400 ? 0u : max_N <= 1024 ? 152u : max_N <= 4096 ? 304u : max_N <= 16384 ? 608u : ~0u;
    return max_Rcap <= FEW_REPLICAS && n_runs > at_once ? 128u : 512u;
}
inline uint32_t resample_threads(uint32_t n_runs, uint32_t max_Rcap)
{
    return max_Rcap <= FEW_REPLICAS / 2 || (max_Rcap <= FEW_REPLICAS && n_runs > 152) ? 128u : 512u;
}

struct Pool {
    const RunDev *runs;
    RunState *st;
    uint32_t *spins[2];
    int32_t *E[2];
    int32_t *M[2];
    uint32_t *fam[2];
    uint32_t *parent;
    uint32_t *cnt;
    pa_step_record *rec;
    uint32_t *qh;
    uint32_t *qhp;
    uint32_t *qhw;
    const double *beta;
    const double *wt;                  // weight tables exp(-4 n dbeta), (N + 1) doubles each
    const unsigned long long *wtoff;   // per run and step: offset of its table in wt
    const unsigned long long *thr;
    uint32_t *J;
    unsigned long long *scratch;
    uint32_t *status;
};

// Sweep launch shape for one lattice size.
struct SweepCfg {
    uint32_t fast;   // 0: byte planes; 1: bit-sliced (L/2 a power of two); 2: bit-sliced, padded rows;
                     // 3: bit-sliced, rows repacked without padding in shared memory
    uint32_t block;  // threads per CTA
    uint32_t TPR;    // threads per replica (power of two; bit-sliced kernels: words per plane / WPT)
    uint32_t RPC;    // replicas per CTA
    uint32_t G;      // Philox groups per colour = ceil(N / 8)
    uint32_t PS;     // bytes per colour plane = 4 G (byte planes); the row pitch (padded or compact rows)
    uint32_t smem;   // dynamic shared memory bytes
    uint32_t WPT;    // bit-sliced kernels: plane words per thread
    uint32_t NR;     // power-of-two kernel: children per thread, at the same word
    uint32_t TH;     // half-sweeps of shared Philox parts held in shared memory (0: none)
    uint32_t K;      // consecutive tiles one CTA works through (set by launch_sweep)
    uint32_t Lh, pw; // compact rows: L/2 and words of a stored plane
    uint32_t loads;  // the loads (bits 1 << SweepLoad) at which the tuner times it
};

// How far the sweeps of a lattice size fill the GPU, from the CTAs that its first launch shape takes:
// up to two per SM, a few waves of them, or more.  Below two per SM a launch lasts as long as one CTA,
// so one child per thread and small blocks win; from eight per SM on it is the throughput, two
// children and large blocks; between them whole waves decide (theta = 10, us a launch, one / two
// children): L = 30 100 CTAs 28 / 48, 190 59 / 74, 750 172 / 166, 1500 336 / 319; L = 64 200 28 / 33,
// 800 82 / 87, 1600 158 / 153, 13000 1167 / 1124; L = 256 50 64 / 114, 200 181 / 223, 400 356 / 332,
// 1600 1290 / 1203.
enum SweepLoad : uint32_t { LOAD_FEW = 0, LOAD_SOME = 1, LOAD_FULL = 2, LOAD_ANY = 7 /* mask */ };
inline SweepLoad sweep_load(uint64_t ctas) { return ctas < 304 ? LOAD_FEW : ctas < 1216 ? LOAD_SOME : LOAD_FULL; }
// Few sweeps per launch: kernels of their own for the power-of-two sizes (launch_sweep).
inline bool few_sweeps(uint32_t theta_max) { return theta_max <= 4; }
// The shape before (or without) timing: the first one, and of a load that leaves SMs idle the one
// that spreads the replicas over the most CTAs.
inline uint32_t default_shape(const std::vector<SweepCfg> &shapes, SweepLoad load)
{
    uint32_t pick = 0;
    if (load == LOAD_FEW)
        for (uint32_t c = 1; c < shapes.size(); ++c)
            if (shapes[c].RPC <= shapes[pick].RPC) pick = c;  // of two alike the later: L = 12's padded rows
    return pick;
}

// Row pitch of a colour plane: L/2 when that is a power of two; else the
// smallest power of two >= L/2 that makes L * pitch a multiple of 32 (rows then
// tile 32-bit words, so the bit-sliced sweep applies) for L/2 < 32, and L/2
// rounded up to a multiple of 32 beyond.
inline uint32_t row_pitch(uint32_t L)
{
    const uint32_t Lh = L / 2;
    if ((Lh & (Lh - 1)) == 0) return Lh;
    if (Lh < 32)
        for (uint32_t P = 4; P <= 32; P <<= 1)
            if (P >= Lh && (L * P) % 32 == 0) return P;
    return (Lh + 31) / 32 * 32;
}

inline uint32_t plane_words_of(uint32_t L) { return (L * row_pitch(L) + 31) / 32; }

// Scratch of one run, in 64-bit words from scr_off: the energy and the
// magnetisation histograms of the measurement (N + 1 u32 each, left cleared
// between steps), a per-level f64 / u64 table (N + 1), a per-level u32 table
// (N + 1), then a tail used by one kernel at a time: the multinomial member
// list (R_cap u32), or the per-CTA replica totals of the resampling
// (MAX_RUN_CTAS u32), or the measurement's per-CTA family statistics
// (MEASURE_PART_WORDS each; split_ctas cuts pieces of more than 1365 slots, so a
// run on nc CTAs, whatever the launch's largest population, has more than 1365
// (nc - 1) slots, whose member words are far more than the statistics).
constexpr uint64_t MEASURE_PART_WORDS = 4;
__host__ __device__ inline uint64_t scr_hist_words(uint32_t N) { return (uint64_t(N) + 2) / 2; }
__host__ __device__ inline uint64_t scr_mhist_off(uint32_t N) { return scr_hist_words(N); }
__host__ __device__ inline uint64_t scr_table_off(uint32_t N) { return 2 * scr_hist_words(N); }
__host__ __device__ inline uint64_t scr_level_off(uint32_t N) { return scr_table_off(N) + N + 1; }
__host__ __device__ inline uint64_t scr_tail_off(uint32_t N) { return scr_level_off(N) + scr_hist_words(N); }
inline uint64_t scratch_words(uint32_t N, uint32_t R_cap)
{
    const uint64_t members = (uint64_t(R_cap) + 1) / 2;
    const uint64_t totals = MAX_RUN_CTAS / 2, parts = MEASURE_PART_WORDS * run_ctas(R_cap);
    uint64_t tail = members > totals ? members : totals;
    tail = tail > parts ? tail : parts;
    return scr_tail_off(N) + tail + 4;
}

// Small populations annealed by one launch per step (anneal_small_kernel): one
// thread-block cluster per run (small_shape, small_shape_ahead).
constexpr uint32_t SMALL_MAX_RCAP = 8192;
constexpr uint32_t SMALL_MAX_CTAS = 16;  // largest cluster (above 8 by the non-portable opt-in)
inline bool small_eligible(const RunDev &x)
{
    return (x.L == 8 || x.L == 16 || x.L == 32) && x.theta != PA_THETA_INF && x.resample == PA_NEAREST &&
           x.overlap == 0 && x.R_cap <= SMALL_MAX_RCAP;
}
// Lanes that share one colour-plane word in the small-population kernel's
// sweeps (each draws 8 / LPW of the word's Philox groups); the fastest
// measured for 20 runs of a few hundred replicas: 8 at L = 8, 2 at L = 16,
// 1 and 2 alike at L = 32.
#ifndef SMALL_LPW_L8
#define SMALL_LPW_L8 8
#endif
#ifndef SMALL_LPW_L16
#define SMALL_LPW_L16 2
#endif
#ifndef SMALL_LPW_L32
#define SMALL_LPW_L32 2
#endif

// Launch wrappers implemented in pa_kernels.cu (all asynchronous on `s`).
// `runs`: device list of the indices of the runs to process (the two
// initialisation launches also take NULL for runs 0..n_runs-1).
void launch_reset_runs(const Pool &P, const uint32_t *runs, uint32_t n_runs, cudaStream_t s);
void launch_init_couplings(const Pool &P, const uint32_t *runs, uint32_t n_runs, cudaStream_t s);
// Work lists: tile_off = prefix of per-run tile counts (n + 1 entries).
void launch_init_population(const Pool &P, const uint32_t *tile_off, const uint32_t *runs, uint32_t n_runs,
                            uint32_t n_tiles, uint32_t max_pw, cudaStream_t s);
// Resampling of runs with PA_MULTINOMIAL, one CTA per run.  max_Rcap: the
// largest R_cap among the runs (sets the energies staged in shared memory).
void launch_resample_multinomial(const Pool &P, const uint32_t *runs, uint32_t n_runs, uint32_t max_Rcap,
                                 uint32_t max_N, cudaStream_t s);
// Nearest-integer resampling (PA_NEAREST) from the tables the measurement of
// the previous step prepared, split_ctas CTAs per run, in
// resample_nearest_launches(n_runs, max_Rcap) kernel launches (one when every
// population takes one CTA).  Of a full launch: resample_nearest_launches(max_Rcap).
inline uint32_t resample_nearest_launches(uint32_t max_Rcap) { return run_ctas(max_Rcap) == 1 ? 1u : 2u; }
inline uint32_t resample_nearest_launches(uint32_t n_runs, uint32_t max_Rcap)
{
    return split_ctas(n_runs, max_Rcap) == 1 ? 1u : 2u;
}
void launch_resample_nearest(const Pool &P, const uint32_t *runs, uint32_t n_runs, uint32_t max_Rcap, cudaStream_t s);
// Launch shapes to try for lattice size L (first = default); one entry unless
// the bit-sliced kernel applies.
std::vector<SweepCfg> sweep_candidates(uint32_t L, int allow_fast);
// Consecutive tiles one CTA of launch_sweep works through.
uint32_t sweep_tiles_per_cta(const SweepCfg &cfg, uint32_t n_tiles, uint32_t theta_max);
void launch_sweep(const Pool &P, const uint32_t *group_runs, const uint32_t *tile_off, uint32_t n_group_runs,
                  uint32_t n_tiles, const SweepCfg &cfg, int any_glass, uint32_t theta_max, cudaStream_t s);
void launch_overlap(const Pool &P, const uint32_t *q_runs, uint32_t n_q_runs, uint32_t max_Rcap, int init,
                    cudaStream_t s);
// split_ctas CTAs per run (fewer for the smaller populations); also prepares the
// next nearest-integer resampling of each run.
void launch_measure(const Pool &P, const uint32_t *runs, uint32_t n_runs, uint32_t max_Rcap, uint32_t max_N, int init,
                    cudaStream_t s);
// theta = PA_THETA_INF runs: fresh energies from the exact distribution for
// the population of the step in flight (init: the beta_0 population).
void launch_dos_sample(const Pool &P, const uint32_t *runs, uint32_t n_runs, uint32_t max_R, int init,
                       cudaStream_t s);
// Wang et al.'s pairing and its overlaps for the runs in `runs` (init: step 0);
// max_Rcap: the largest R_cap among them (sets the shared memory).
void launch_wang(const Pool &P, const uint32_t *runs, uint32_t n_runs, uint32_t max_Rcap, int init, cudaStream_t s);
size_t wang_smem_bytes(uint32_t max_Rcap);
void launch_wavg_wang(const pa_step_record *recs, const unsigned long long *rec_off, const uint32_t *qh,
                      const uint32_t *qhp, const uint32_t *qhw, const unsigned long long *qh_off, uint32_t n_groups,
                      uint32_t M, uint32_t n_steps, uint32_t N, uint32_t kind, pa_wavg *out, double *w, double *Pq,
                      double *Pqp, double *Pqw, cudaStream_t s);
void launch_wavg(const pa_step_record *recs, const unsigned long long *rec_off, const uint32_t *qh,
                 const uint32_t *qhp, const unsigned long long *qh_off, uint32_t n_groups, uint32_t M,
                 uint32_t n_steps, uint32_t N, uint32_t kind, pa_wavg *out, double *w, double *Pq, double *Pqp,
                 cudaStream_t s);
// Copies the record of each listed run at the temperature it has reached to out[k].
void launch_gather_records(const Pool &P, const uint32_t *runs, uint32_t n_runs, pa_step_record *out,
                           cudaStream_t s);
// Groups t0 .. t0 + count - 1 of four consecutive sites of the replicas at `words` (one run's
// packed planes, counted from the first replica) as int8 +-1 into out (4 count bytes).
void launch_unpack_spins(const uint32_t *words, const RunDev &rd, uint32_t t0, uint32_t count, int8_t *out,
                         cudaStream_t s);
// n_steps temperatures of the small runs `runs` (all of lattice size L), cs
// CTAs (a cluster) per run.
// Launch shape of the small-run kernel: CTAs per cluster (one cluster per run),
// threads per CTA, the compiled variant (0: 512 threads two CTAs per SM; 1 / 2:
// up to 512 / 768 threads one CTA per SM; 3 / 4: the same with 4 lanes per word
// at L = 8), the half-sweeps whose comparison bits are drawn ahead (0: none)
// and the dynamic shared memory they take.
struct SmallShape {
    uint32_t cs, block, variant, H, smem;
};
// The largest clusters to try.  More than 8 CTAs (the non-portable sizes, at most one such cluster per
// GPC) shorten the sweeps and lengthen the chain of cluster barriers, so they pay where the sweeps
// last longer. One temperature per launch, 8 against 16 CTAs (us per temperature, theta = 10; threads
// that 8 CTAs sweep with): L = 16 R = 400 (461) 34.6 / 28.1 for one run, 35.0 / 37.6 for nine; R = 500
// (568) 42.8 / 31.7, 43.7 / 36.6; R = 1000 (1095) 63.3 / 45.2, 66.5 / 66.6; L = 8 R = 400 20.5 / 20.3,
// 22.2 / 23.6; R = 500 24.5 / 21.0, 24.7 / 22.5.
inline uint32_t small_largest_cluster(uint32_t L, uint32_t n_runs, uint32_t threads_of_8)
{
    return L != 32 && threads_of_8 > (n_runs <= 8 ? 384u : 512u) ? SMALL_MAX_CTAS : 8u;
}
// Several temperatures per launch, where the draws overlap CTA 0's measurement: the line is the
// sweeps' work per thread, theta times the warps of a CTA of 8 times a thread's draws (a word of L = 8
// is drawn by 4 lanes, one of L = 16 by one).  8 / 16 CTAs, one run, by theta: L = 16 R = 500 (352
// threads) 12.2 / 13.3 at 3, 13.6 / 13.4 at 4, 28.1 / 20.9 at 10; R = 700 (448) 12.3 / 13.2 at 2, 13.9
// / 13.5 at 3, 35.5 / 21.2 at 10; L = 8 R = 500 12.3 / 13.1 at 10, 20.8 / 15.9 at 20; R = 700 12.6 /
// 13.2 at 8, 14.7 / 13.5 at 10.  Above 512 threads 16 CTAs at every theta (L = 8 R = 1200 12.5 / 12.4
// at 2, 23.8 / 14.2 at 10; L = 16 R = 1000 13.4 / 13.9, 44.7 / 28.2).  Eight or nine runs leave no
// room for 16 CTAs each (L = 16, theta = 10: R = 500 28.0 / 29.4, R = 600 35.3 / 29.4), five do; up to
// 384 threads the line is a little higher (L = 16 R = 300 at 5, 224 threads: 12.4 / 13.1).
inline uint32_t small_largest_cluster_ahead(uint32_t L, uint32_t n_runs, uint32_t threads_of_8, uint32_t theta_max)
{
    const uint32_t block = (threads_of_8 + 31) / 32 * 32;
    if (n_runs > 5 && threads_of_8 <= 384) return 8;
    const uint32_t line = threads_of_8 <= 384 ? 5000 : 4300;
    return block > 512 || (uint64_t)theta_max * block * (L * L / 64) > line ? SMALL_MAX_CTAS : 8u;
}
// A run whose populations fit a cluster only when several temperatures are drawn ahead takes a single
// temperature per launch in several tiles per CTA, which the per-stage kernels beat from this work on
// (us per temperature, cluster / per stage: L = 16 R = 1500 theta = 2 34.6 / 35.7, theta = 10 85.8 /
// 46; L = 8 R = 1500 24.4 / 33.2, 43.0 / 40.5; R = 2000 27.9 / 34.2, 53.1 / 41.6).
inline bool small_steps_per_stage(uint32_t L, uint32_t R_max, uint32_t theta_max)
{
    return (uint64_t)theta_max * R_max * L * L > 800000;
}
SmallShape small_shape(uint32_t L, int any_glass, uint32_t n_runs, uint32_t R_max, uint32_t R_cap_max);
SmallShape small_shape_ahead(uint32_t L, int any_glass, uint32_t n_runs, uint32_t R_max, uint32_t theta_max);
void launch_anneal_small(const Pool &P, const uint32_t *runs, uint32_t n_runs, uint32_t L, const SmallShape &sh,
                         int any_glass, uint32_t n_steps, cudaStream_t s);
cudaError_t prepare_kernels();
// Philox-only calibration loop: blocks x threads threads, iters x 8 calls each.
void launch_philox_calibration(uint32_t *out, uint32_t blocks, uint32_t threads, uint32_t iters, bool wide,
                               cudaStream_t s);

#ifndef MADV_POPULATE_WRITE
#define MADV_POPULATE_WRITE 23  // Linux 5.14
#endif

// Brings the pages of [p, p + bytes) into memory, writable, without writing to them.  Pages that the
// caller may not write, or that are not there, stay as they are: they are the copy's to meet.
inline void populate_pages(void *p, size_t bytes)
{
    const uintptr_t page = (uintptr_t)sysconf(_SC_PAGESIZE);
    const uintptr_t lo = (uintptr_t)p & ~(page - 1), hi = ((uintptr_t)p + bytes + page - 1) & ~(page - 1);
    (void)madvise(reinterpret_cast<void *>(lo), hi - lo, MADV_POPULATE_WRITE);
}

// Enqueues the copy of a result into the caller's memory, whose pages are first populated from the
// host, while the device still works on the result.  A copy into pages that have never been touched
// takes their faults one by one from the device: 20.8 MB into fresh pages 17 ms, 0.8 ms after
// populating them (0.13 ms into pages in use).  Only pageable memory is populated: pinned pages are
// there already.
inline cudaError_t copy_out(void *host, const void *dev, size_t bytes, cudaStream_t s)
{
    if (bytes >= (1u << 20)) {
        cudaPointerAttributes at{};
        if (cudaPointerGetAttributes(&at, host) != cudaSuccess)
            (void)cudaGetLastError();  // of this query alone: the copy says what is wrong with the pointer
        else if (at.type == cudaMemoryTypeUnregistered)
            populate_pages(host, bytes);
    }
    return cudaMemcpyAsync(host, dev, bytes, cudaMemcpyDeviceToHost, s);
}

}  // namespace pa
