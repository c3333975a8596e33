// Launchers of the MD-step kernels (step_impl.cuh): the prologue for every molecule size
// and the force-interpolation step kernels of the WCA model; the water-like model's kernels
// are instantiated in step_ljrf.cu and the energy-interpolation ones in step_hadress.cu.
#include "step_impl.cuh"

namespace adress {

cudaError_t launch_step_ljrf(const Sys& s, const Bufs& b, int precision, int mode, int energy, cudaStream_t st);
cudaError_t launch_step_hadress(const Sys& s, const Bufs& b, int precision, int mode, int energy, cudaStream_t st);
cudaError_t launch_run_hadress(const Sys& s, const Bufs& b, int precision, int done, int nsteps, int sample_every, cudaStream_t st);

template <class P, int NA>
static void launch_prologue_na(const Sys& s, const Bufs& b, int integrate, cudaStream_t st) {
  const int blocks = ceil_div((long long)s.M * kGroup, s.force_block);
  if (s.nbox > 1) {
    if (integrate) k_prologue<P, NA, true, true><<<blocks, s.force_block, 0, st>>>(s, b);
    else k_prologue<P, NA, false, true><<<blocks, s.force_block, 0, st>>>(s, b);
  } else {
    if (integrate) k_prologue<P, NA, true, false><<<blocks, s.force_block, 0, st>>>(s, b);
    else k_prologue<P, NA, false, false><<<blocks, s.force_block, 0, st>>>(s, b);
  }
}

template <class P>
static void launch_prologue_p(const Sys& s, const Bufs& b, int integrate, cudaStream_t st) {
  switch (s.NA) {
    case 1: launch_prologue_na<P, 1>(s, b, integrate, st); break;
    case 2: launch_prologue_na<P, 2>(s, b, integrate, st); break;
    case 3: launch_prologue_na<P, 3>(s, b, integrate, st); break;
    default: launch_prologue_na<P, 4>(s, b, integrate, st); break;
  }
}

cudaError_t launch_map(const Sys& s, const Bufs& b, int precision, int integrate, cudaStream_t st) {
  if (precision == ADRESS_FP64) launch_prologue_p<P64>(s, b, integrate, st);
  else launch_prologue_p<P32>(s, b, integrate, st);
  return cudaGetLastError();
}

template <class P>
static void launch_step_p(const Sys& s, const Bufs& b, int mode, int energy, cudaStream_t st) {
  switch (s.NA) {
    case 1: launch_step_na<P, 1, 0, false>(s, b, mode, energy, st); break;
    case 2: launch_step_na<P, 2, 0, false>(s, b, mode, energy, st); break;
    case 3: launch_step_na<P, 3, 0, false>(s, b, mode, energy, st); break;
    default: launch_step_na<P, 4, 0, false>(s, b, mode, energy, st); break;
  }
}

cudaError_t launch_step(const Sys& s, const Bufs& b, int precision, int mode, int energy, cudaStream_t st) {
  if (s.scheme == 1) return launch_step_hadress(s, b, precision, mode, energy, st);
  if (s.nb_model == 1) return launch_step_ljrf(s, b, precision, mode, energy, st);
  if (precision == ADRESS_FP64) launch_step_p<P64>(s, b, mode, energy, st);
  else launch_step_p<P32>(s, b, mode, energy, st);
  return cudaGetLastError();
}

template <class P>
static cudaError_t launch_run_p(const Sys& s, const Bufs& b, int done, int nsteps, int sample_every, cudaStream_t st) {
  switch (s.NA) {
    case 1: return launch_run_na<P, 1, 0, false>(s, b, done, nsteps, sample_every, st);
    case 2: return launch_run_na<P, 2, 0, false>(s, b, done, nsteps, sample_every, st);
    case 3: return launch_run_na<P, 3, 0, false>(s, b, done, nsteps, sample_every, st);
    default: return launch_run_na<P, 4, 0, false>(s, b, done, nsteps, sample_every, st);
  }
}

// The run kernel where the device is far from full: there a step is latency, and a grid barrier
// costs less than two launches (us a step, run kernel against launches, FP32: 1000 molecules 8.6
// and 16.6; 12,000: 12.2 and 18.0; 24,000: 18.6 and 19.3; 30,000: 19.0 and 19.9; 35,000: 19.4 and
// 20.5; 40,000: 23.8 and 21.1, its blocks' third round of tiles).  The line lies short of the crossing,
// where the gain has fallen to a twentieth, and leaves that to the launches up to some 38,000.
// Not for the water-like fluid: its long lists make the step itself longer than the launches (2000
// molecules: 33 both ways), nor in FP64 beyond one tile per SM, on which three blocks reside (2000
// molecules 26.3 and 29.4; 4800: 26.7 and 29.9; 7000: 32.8 and 34.3; 10,000: 46.1 and 41.4; 20,000:
// 71.7 and 62.6).
bool run_kernel_pays(const Sys& s) {
  return !s.cg_mode && s.nb_model == 0 && s.M <= (s.fp64 ? 32ll : 160ll) * s.n_sm;
}

cudaError_t launch_run(const Sys& s, const Bufs& b, int precision, int done, int nsteps, int sample_every, cudaStream_t st) {
  if (s.scheme == 1) return launch_run_hadress(s, b, precision, done, nsteps, sample_every, st);
  return precision == ADRESS_FP64 ? launch_run_p<P64>(s, b, done, nsteps, sample_every, st) : launch_run_p<P32>(s, b, done, nsteps, sample_every, st);
}

}  // namespace adress
