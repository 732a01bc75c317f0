// Interface of the covariance form of the FP32 path (beam_corr.cu).
#pragma once

#include <cuda.h>

#include "internal.cuh"

namespace fftbf {

// One array of a launch and how its lattice is cut (filled by corr_make_job).
struct CorrJob {
  CUtensorMap map;      // the voltages (tma)
  BeamArgs a;
  int ny, nyp;          // N-S feeds, and their slots (a multiple of 16, 32 or 64)
  int nant, np, nt;     // feeds, slots, tiles of 256 slots per axis
  int nch;              // stages of kCorrSteps snapshots per window
  int mode;             // epilogue split 0..3: 8-slot groups per run 4x8, 4x4, 2x2, 4x16
  int tma;              // voltages staged by TMA
  int w_exp;            // the weights are held times 2^w_exp
  float rscale;         // and those of the rows times this, for sums in units of V
  float lscale;         // what lies below a unit is kept times this
  int out_exp;          // beams are V's transform times 2^out_exp
  int64_t item0, nitems;
};
struct CorrSizes {      // shared-memory sizes, the largest over the launch's jobs
  int ns, nr;           // operand stages, staged voltage tiles
  int wslots, vlen, stg, tab;
  int cplx;             // some weights are complex
  int tma;              // some jobs' voltages are staged by TMA
};
struct CorrParams {
  CorrJob one;          // the only job, or
  const CorrJob* table; // a device table of njobs
  int njobs;
  int64_t total;        // work items
  int* err;             // error word, or null: those of the jobs' plans
  CorrSizes s;
};

// Fill a job; false where the kernel does not take the lattice.
bool corr_make_job(const BeamArgs& a, CorrJob* J);
bool corr_sizes(const CorrJob* jobs, int n, CorrSizes* out);
int corr_maps(CorrJob* jobs, int n);
int corr_launch(CorrParams& p, int nsm, cudaStream_t st);
constexpr int kCorrSteps = 64;   // snapshots per operand stage
// Whether it beats the transform of every snapshot (split: the split-FP16 kernel).
bool corr_preferred(const BeamArgs& a, bool split = false);
bool batch_cov(const fftbf_batch* bb, int i);   // plan i of the batch goes through it
int launch_beams_corr(const BeamArgs& a, int nsm, cudaStream_t st);
int corr_plan_jobs(std::vector<CorrJob>& jobs, const CorrJob* d_table, int* err,
                   std::vector<CorrParams>* out);

}  // namespace fftbf
