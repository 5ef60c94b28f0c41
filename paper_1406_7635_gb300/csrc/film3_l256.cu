// The persistent kernel on thin 3-D grids, x rows of 256 complex values.
#include "film.cuh"

template bool mm::film3_plan_l<256>(const Geom&, int, FilmPlan*);
template cudaError_t mm::launch_film3_l<256>(const FilmPlan&, int, const FilmArgs&, cudaStream_t);
