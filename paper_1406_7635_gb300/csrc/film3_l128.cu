// The persistent kernel on thin 3-D grids, x rows of 128 complex values.
#include "film.cuh"

template bool mm::film3_plan_l<128>(const Geom&, int, FilmPlan*);
template cudaError_t mm::launch_film3_l<128>(const FilmPlan&, int, const FilmArgs&, cudaStream_t);
