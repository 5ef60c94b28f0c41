// Dispatch of the persistent film kernel over the x row length.
#include "film.h"

namespace mm {

bool film_plan(const Geom& g, FilmPlan* p) {
  *p = FilmPlan();
  if (!g.fused || g.nz > 4 || g.pbcy != 0 || g.pbcz != 0 || g.py < 32) return false;
  const int ph = g.py / 2;
  if (g.nz == 1) {
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
  switch (g.lx) {
    case 16: return film3_plan_l<16>(g, ph, p);
    case 32: return film3_plan_l<32>(g, ph, p);
    case 64: return film3_plan_l<64>(g, ph, p);
    case 128: return film3_plan_l<128>(g, ph, p);
    case 256: return film3_plan_l<256>(g, ph, p);
    default: return false;
  }
}

cudaError_t launch_film(const FilmPlan& p, const FilmArgs& a, cudaStream_t s) {
  const int ph = a.g.py / 2;
  if (a.g.nz == 1) {
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
  switch (a.g.lx) {
    case 16: return launch_film3_l<16>(p, ph, a, s);
    case 32: return launch_film3_l<32>(p, ph, a, s);
    case 64: return launch_film3_l<64>(p, ph, a, s);
    case 128: return launch_film3_l<128>(p, ph, a, s);
    case 256: return launch_film3_l<256>(p, ph, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mm
