// The persistent kernel on thin 3-D grids, x rows of 16 complex values.
#include "film.cuh"

template bool mm::film3_plan_l<16>(const Geom&, int, FilmPlan*);
template cudaError_t mm::launch_film3_l<16>(const FilmPlan&, int, const FilmArgs&, cudaStream_t);
