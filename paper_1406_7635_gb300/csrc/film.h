// Plan and arguments of the persistent film kernel (film.cuh): host side.
#pragma once
#include "mm_internal.h"

namespace mm {

// grid barrier and step-error maxima, zero between launches
struct FilmSync {
  unsigned int arrived, left;
  unsigned int err[3];   // attempt a uses slot a % 3
};

struct FilmArgs {
  Geom g;
  Terms T;
  Stt S;
  float* m0;
  float* m1;
  float* k[7];
  const float2* tw;       // twiddle table
  const float* kt;        // octant per kx column [hkx][6][hkz][hky]
  const RegionLUT* lut;
  const float* xlut;
  const int* code;
  float2* spec1;          // [3][hx][nz][ny]
  float2* spec2;          // [3][nz][ny][hxs]
  float* halo;            // [3][nz][ny][nx]: the stage input's rows that other blocks' stencils read
  DevState* st;
  double* hist;
  const double* fixed;
  FilmSync* sync;
  double freq, phase_over_pi;
  double t_end;           // (begin)
  long long nsteps;       // (begin)
  int begin, mode;        // begin: start a call of `mode` (launch_begin_mode)
  int k1;                 // evaluate the first stage only
  int attempts;           // most attempts of this launch
  int state_limit;        // the waits take the context's limit, else the default
  int oct_sm;             // the octant columns are kept in shared memory
};

// Work split of a film (film_plan): rows per block, blocks, shared memory and
// what it holds.  rows = 0: the film steps with the stage kernels.
struct FilmPlan {
  int rows = 0, blocks = 0, oct_sm = 0;
  size_t smem = 0;
};
// Plan of a fused grid of one to four layers with open y and z axes and more
// than 8 cells along y, on the current device; false where the kernel does not
// apply (its blocks must all be resident at once).  Sets the kernel's shared-memory limit.
bool film_plan(const Geom& g, FilmPlan* plan);
cudaError_t launch_film(const FilmPlan& plan, const FilmArgs& args, cudaStream_t s);

// one row length: films (film_l*.cu), two to four layers (film3_l*.cu)
template <int LX>
bool film_plan_l(const Geom& g, int ph, FilmPlan* plan);
template <int LX>
cudaError_t launch_film_l(const FilmPlan& plan, int ph, const FilmArgs& args, cudaStream_t s);
template <int LX>
bool film3_plan_l(const Geom& g, int ph, FilmPlan* plan);
template <int LX>
cudaError_t launch_film3_l(const FilmPlan& plan, int ph, const FilmArgs& args, cudaStream_t s);

}  // namespace mm
