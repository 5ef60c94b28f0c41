// The persistent film kernel for x rows of 16 complex values.
#include "film.cuh"

template bool mm::film_plan_l<16>(const Geom&, int, FilmPlan*);
template cudaError_t mm::launch_film_l<16>(const FilmPlan&, int, const FilmArgs&, cudaStream_t);
