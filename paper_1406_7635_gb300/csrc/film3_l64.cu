// The persistent kernel on thin 3-D grids, x rows of 64 complex values.
#include "film.cuh"

template bool mm::film3_plan_l<64>(const Geom&, int, FilmPlan*);
template cudaError_t mm::launch_film3_l<64>(const FilmPlan&, int, const FilmArgs&, cudaStream_t);
