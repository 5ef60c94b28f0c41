// Dispatch of the persistent film kernel over the x row length.
#include "film.h"

namespace mm {

#define MM_FILM_EXTERN(L)                                        \
  extern template bool film_plan_l<L>(const Geom&, int, FilmPlan*); \
  extern template cudaError_t launch_film_l<L>(const FilmPlan&, int, const FilmArgs&, cudaStream_t);
MM_FILM_EXTERN(16)
MM_FILM_EXTERN(32)
MM_FILM_EXTERN(64)
MM_FILM_EXTERN(128)
MM_FILM_EXTERN(256)
MM_FILM_EXTERN(512)
#undef MM_FILM_EXTERN

bool film_plan(const Geom& g, FilmPlan* p) {
  *p = FilmPlan();
  if (!g.fused || g.nz != 1 || g.pbcy != 0 || g.py < 32) return false;
  const int ph = g.py / 2;
  switch (g.lx) {
    case 16: return film_plan_l<16>(g, ph, p);
    case 32: return film_plan_l<32>(g, ph, p);
    case 64: return film_plan_l<64>(g, ph, p);
    case 128: return film_plan_l<128>(g, ph, p);
    case 256: return film_plan_l<256>(g, ph, p);
    case 512: return film_plan_l<512>(g, ph, p);
    default: return false;
  }
}

cudaError_t launch_film(const FilmPlan& p, const FilmArgs& a, cudaStream_t s) {
  const int ph = a.g.py / 2;
  switch (a.g.lx) {
    case 16: return launch_film_l<16>(p, ph, a, s);
    case 32: return launch_film_l<32>(p, ph, a, s);
    case 64: return launch_film_l<64>(p, ph, a, s);
    case 128: return launch_film_l<128>(p, ph, a, s);
    case 256: return launch_film_l<256>(p, ph, a, s);
    case 512: return launch_film_l<512>(p, ph, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mm
