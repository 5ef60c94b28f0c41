// The persistent film kernel for x rows of 32 complex values.
#include "film.cuh"

template bool mm::film_plan_l<32>(const Geom&, int, FilmPlan*);
template cudaError_t mm::launch_film_l<32>(const FilmPlan&, int, const FilmArgs&, cudaStream_t);
