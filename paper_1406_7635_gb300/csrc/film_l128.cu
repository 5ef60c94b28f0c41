// The persistent film kernel for x rows of 128 complex values.
#include "film.cuh"

template bool mm::film_plan_l<128>(const Geom&, int, FilmPlan*);
template cudaError_t mm::launch_film_l<128>(const FilmPlan&, int, const FilmArgs&, cudaStream_t);
