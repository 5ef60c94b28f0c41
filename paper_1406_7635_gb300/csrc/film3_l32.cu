// The persistent kernel on thin 3-D grids, x rows of 32 complex values.
#include "film.cuh"

template bool mm::film3_plan_l<32>(const Geom&, int, FilmPlan*);
template cudaError_t mm::launch_film3_l<32>(const FilmPlan&, int, const FilmArgs&, cudaStream_t);
