// Persistent RK kernel of 2-D films and stacks of two to four layers: whole
// Runge-Kutta attempts (Sec. IV) in one cooperative launch.
//
// A film's attempt is a chain of small steps that cannot overlap (stage input,
// x transform, y transform and kernel product, inverse x transform, field,
// next stage input), so one kernel per step pays a launch, a cold start
// (state, tables, codes, material tables) and a drain several times per
// stage.  Here the blocks stay resident for as many attempts as the call
// needs: block b owns ROWS film rows and CPB kx columns, keeps its codes,
// couplings, material tables, stage input and (where they fit) its columns'
// kernel octant in shared memory, its m and stage torques in global memory
// (read back by the thread that wrote them), and exchanges only the spectrum
// (through L2) and the rows that the neighbours' stencils read.  Per stage:
//
//   rows:     stage input -> x R2C of the block's rows -> spec1[c][kx][y]
//   -- grid barrier --
//   columns:  y forward, kernel product, y inverse of the block's columns
//             -> spec2[c][y][kx]   (meanwhile the halo rows arrive)
//   -- grid barrier --
//   rows:     x C2R -> B_demag -> field, torque k_s -> next stage input
//
// and after the last stage one more barrier for the maximum step error (13
// per RK45 attempt); the controller then runs redundantly in every block
// (same inputs, same result), block 0 keeps the device state.  Both spectrum
// exchanges write scattered (8 ROWS or 8 CPB bytes) and read contiguous runs.
//
// Bound by latency: a stage is two grid barriers and, on every block, a serial
// chain of short transforms; bandwidth and arithmetic are far from their
// limits.  Share of a step that a block spends at the barriers / in the column
// phase / in the rows' transforms / in the cells, by clock stamps: 64 x 16 film
// (a block without rows) 67 / 16 / 3 / 4 %, 256 x 256 19 / 32 / 25 / 11 %, 500
// x 387 7 / 48 / 26 / 10 %, 96 x 96 x 4 stack 18 / 37 / 23 / 8 % (a wait
// includes the other blocks' work).  What the design buys is that chain without launches and cold
// starts.  Measured, us per RK45 step, stage kernels in a graph -> this
// kernel: 64 x 16 film 81 -> 37, 128 x 128 74 -> 44, 256 x 256 109 -> 65, 500
// x 387 351 -> 174, 96 x 96 x 4 140 -> 64; 256 x 200 periodic 137 -> 56, with
// RK23 and a Zhang-Li torque 73 -> 31.  A block holds most of a
// multiprocessor's registers, so contexts stepped at once from several
// threads take turns: eight films of 256 x 256 take 513 us per step of all,
// 374 with the stage kernels (four: 257 and 212; eight of 500 x 387: 1388 and
// 2162).  Fewer registers for more blocks per multiprocessor took eight 128 x
// 128 films from 201 to 168 us (143 with the stage kernels) and slowed one
// alone by 2 %.
//
// Every wait at a barrier is bounded; a wait that gives up records
// MM_ERR_TIMEOUT, and m, t and dt stay those of the last accepted attempt
// (candidates go to the other buffer; the parity flips only after a barrier
// that all blocks have passed with their candidates written).
#pragma once
#include <algorithm>

#include "fft.cuh"
#include "film.h"
#include "llg_device.cuh"

namespace mm {

namespace {
using namespace mmfft;

// ---------------------------------------------------------------------------
// Transforms.  A pencil of N points lives in its own area of shared memory in
// natural order (element i at pos(i)) and is transformed in place by LANES
// lanes of one warp, without block barriers; only the forward transform
// exists: the inverse is the same transform on values with real and
// imaginary part exchanged on the way in and out, which the code around it
// does for free (one copy of the instructions, executed by few warps once
// per stage: the instruction fetch counts).
//
// N <= 256: 8 values per lane (16 needed half the warps and took about twice
// the time: a warp alone on its scheduler issues every other cycle).  N = 8 G:
// lane j holds x[j + G r] -> 8-point DFT over r -> times W_N^(j k1) ->
// exchange -> G-point DFTs over j.  G <= 8: 8 / G of them per lane.  G = 16,
// 32 (= 8 B): j = j0 + B r2, lane j0 + B k1: 8-point DFT over r2 -> times
// W_G^(j0 k2) -> exchange -> 8 / B B-point DFTs per lane.  The exchanges use
// pitches that keep both sides free of bank conflicts.
// ---------------------------------------------------------------------------
template <int N>
struct FilmFft {
  static constexpr int G = N / 8, LANES = G, B = G > 8 ? G / 8 : 1;
  static constexpr int G2 = G > 8 ? 8 : G;       // radix of the second step
  static constexpr int H = 8 / G2;               // its DFTs per lane (G <= 8)
  // exchange 1: (k1, j) at k1 P1 + j; exchange 2: (j0, k1, k2) at j0 P2 + k1 + 8 k2
  static constexpr int P1 = G == 32 ? 36 : (G == 16 ? 18 : (G == 8 ? 9 : (G == 4 ? 5 : 3)));
  static constexpr int P2 = G == 32 ? 68 : 72;
  // area of a pencil (values): the offset between pencils of one half-warp
  // spreads them over the banks
  static constexpr int AREA = G == 32 ? 288 : (G == 16 ? 144 : (G == 8 ? 72 : (G == 4 ? 52 : 34)));
  // twiddles: W_N^(j k1) at k1 G + j, then W_G^(j0 k2) at N + k2 B + j0
  static constexpr int TAB = N + (B > 1 ? 8 * B : 0);
  __device__ __forceinline__ static int pos(int i) { return i; }
  template <int NT>
  __device__ __forceinline__ static void tables(float2* t, const float2* __restrict__ tw) {
    for (int i = threadIdx.x; i < N; i += NT)
      t[i] = __ldg(&tw[((i % G) * (i / G) * (kTwN / N)) & (kTwN - 1)]);
    if (B > 1)
      for (int i = threadIdx.x; i < 8 * B; i += NT)
        t[N + i] = __ldg(&tw[((i % B) * (i / B) * (kTwN / G)) & (kTwN - 1)]);
  }
  // x[j + G r] is loaded by ld(i, r), i = j + G r
  template <class LD>
  __device__ __forceinline__ static void run(float2* e, const float2* t, int j, LD ld) {
    float2 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = ld(j + G * r, r);
    __syncwarp();   // (in place: the pencil has been read)
    Dft<8, -1>::run(v);
#pragma unroll
    for (int k = 1; k < 8; ++k) v[k] = cmul(v[k], t[k * G + j]);
#pragma unroll
    for (int k = 0; k < 8; ++k) e[k * P1 + j] = v[k];
    __syncwarp();
    if constexpr (B == 1) {
      float2 w[H][G2];
#pragma unroll
      for (int h = 0; h < H; ++h)
#pragma unroll
        for (int q = 0; q < G2; ++q) w[h][q] = e[(j + G * h) * P1 + q];
      __syncwarp();
#pragma unroll
      for (int h = 0; h < H; ++h) {
        Dft<G2, -1>::run(w[h]);
#pragma unroll
        for (int q = 0; q < G2; ++q) e[j + G * h + 8 * q] = w[h][q];
      }
    } else {
      const int j0 = j % B, k1 = j / B;
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] = e[k1 * P1 + j0 + B * r];
      __syncwarp();
      Dft<8, -1>::run(v);
#pragma unroll
      for (int k = 1; k < 8; ++k) v[k] = cmul(v[k], t[N + k * B + j0]);
#pragma unroll
      for (int k = 0; k < 8; ++k) e[j0 * P2 + k1 + 8 * k] = v[k];
      __syncwarp();
      constexpr int HB = 8 / B;
      float2 w[HB][B];
#pragma unroll
      for (int h = 0; h < HB; ++h)
#pragma unroll
        for (int q = 0; q < B; ++q) w[h][q] = e[q * P2 + j + G * h];
      __syncwarp();
#pragma unroll
      for (int h = 0; h < HB; ++h) {
        Dft<B, -1>::run(w[h]);
#pragma unroll
        for (int q = 0; q < B; ++q) e[j + G * h + 64 * q] = w[h][q];
      }
    }
  }
};

// N = 512: 16 values per lane, one warp per pencil.  Lane j holds
// x[j + 32 r] -> 16-point DFT over r -> times W_512^(j k1) -> exchange -> the
// 32-point DFT of one k1 shared by the lanes 2 k1 + p as two 16-point halves
// (even / odd j) combined by a shuffle.  Element i at i + i / 16.
template <>
struct FilmFft<512> {
  static constexpr int N = 512, LANES = 32, AREA = 544, TAB = N;
  __device__ __forceinline__ static int pos(int i) { return i + (i >> 4); }
  template <int NT>
  __device__ __forceinline__ static void tables(float2* t, const float2* __restrict__ tw) {
    for (int i = threadIdx.x; i < N; i += NT) t[i] = __ldg(&tw[((i % 32) * (i / 32) * (kTwN / N)) & (kTwN - 1)]);
  }
  template <class LD>
  __device__ __forceinline__ static void run(float2* e, const float2* t, int j, LD ld) {
    float2 v[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = ld(j + 32 * r, r);
    __syncwarp();
    Dft<16, -1>::run(v);
#pragma unroll
    for (int k = 1; k < 16; ++k) v[k] = cmul(v[k], t[k * 32 + j]);
#pragma unroll
    for (int k = 0; k < 16; ++k) e[j * 17 + k] = v[k];
    __syncwarp();
    const int p = j & 1, k1 = j >> 1;
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = e[(2 * q + p) * 17 + k1];
    __syncwarp();
    Dft<16, -1>::run(v);
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const float2 m = p ? cmul(v[q], t[32 * q + 16]) : v[q];   // (W_32^q)
      const float2 o = make_float2(__shfl_xor_sync(0xffffffffu, m.x, 1), __shfl_xor_sync(0xffffffffu, m.y, 1));
      e[k1 + 17 * (16 * p + q)] = p ? csub(o, m) : cadd(m, o);
    }
  }
};
__device__ __forceinline__ float2 swapc(float2 a) { return make_float2(a.y, a.x); }

// Work split for rows of LX complex values and PH points per y class: ROWS
// film rows per block, CPB columns per block so that at most kFilmBlocks
// blocks hold the LX + 1 columns, QR of them transformed at a time.
// PZ: 1 for films; the padded z length of thin 3-D grids (two to four
// layers), whose blocks own rows of one layer and whole (y, z) planes of kx.
constexpr int kFilmBlocks = 148;
template <int LX, int PH, int ROWS, int PZ>
struct FilmCfg {
  using FX = FilmFft<LX>;
  using FY = FilmFft<PH>;
  static constexpr int CPB = (LX + 1 + kFilmBlocks - 1) / kFilmBlocks;
  static constexpr int NZ = PZ > 1 ? PZ / 2 : 1;   // most layers
  static constexpr int NTC = ROWS * LX, NTY = 6 * NZ * CPB * FY::LANES;   // one cell, one column lane per thread
  static constexpr int NT0 = ((NTC > NTY ? NTC : NTY) + 31) / 32 * 32;
  static constexpr int NT = NT0 < 64 ? 64 : (NT0 > 512 ? 512 : NT0);
  static constexpr int QR0 = NT / (6 * FY::LANES);
  static constexpr int QR = PZ > 1 || QR0 < 1 ? 1 : (QR0 > CPB ? CPB : QR0);
  // cells per thread: up to four, enough for periodic rows (2 LX cells) except
  // three or more of the longest
  static constexpr int CELLS0 = (2 * NTC + NT - 1) / NT;
  static constexpr int CELLS = CELLS0 > 4 ? 4 : CELLS0;
  static constexpr int LR = PZ > 1 ? 3 * ROWS + 2 : ROWS + 2;   // stencil rows
  static constexpr int ND = PZ > 1 ? 6 : 4;                     // stencil directions
  static constexpr int LANX = (3 * ROWS * FX::LANES + 31) / 32 * 32;
  // column pencils transformed at a time, in rounds of NT lanes
  static constexpr int PPW = 32 / FY::LANES;                    // per warp
  static constexpr int NPEN = (6 * NZ * QR + PPW - 1) / PPW * PPW;
  static_assert(LANX <= NT, "every row pencil has its lanes");
  // pencil areas (whole warps have one, so that idle lanes have a place to work)
  static constexpr int NX = LANX / FX::LANES * FX::AREA, NY = NPEN * FY::AREA;
  static constexpr int FFT = NX > NY ? NX : NY;
  static constexpr int TAB = FX::TAB + (LX + 1) + FY::TAB + PH;
  // octant values per column: xx, yy, zz, xy (one layer: Kxz and Kyz are odd
  // in z and vanish at kz = 0), or all six at PZ / 2 + 1 frequencies
  static constexpr int OCOL = (PZ > 1 ? 6 * (PZ / 2 + 1) : 4) * (PH + 1);
  static constexpr int OCT = CPB * OCOL;
  // stage rows: films keep two buffers (the next input is written while the
  // stencil reads this one); 3-D grids one, refilled from global memory
  static constexpr int STG = PZ > 1 ? 1 : 2;
};

__device__ __forceinline__ void red_release(unsigned int* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(p) : "memory");
}
__device__ __forceinline__ unsigned int ld_acquire(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Stage coefficients h a_sj (entries 0..41, row s) and h e_j (42..48), two
// entries per lane of one warp: the tableau values stay in the lane's
// registers (a constant array indexed by the lane would be read one lane at a
// time), the products are those of prepare_attempt.
__device__ __forceinline__ double film_tableau(int method, int e) {
  if (e >= 49) return 0.0;
  if (e < 42) {
    const int s = e / 6, j = e % 6;
    if (method != 1) return kA[s][j];
    const int rs = s == 6 ? 3 : s;   // slots 0, 1, 2, 6 hold the stages 0..3
    return (s < 3 || s == 6) && j < rs ? kA23[rs][j] : 0.0;
  }
  const int j = e - 42;
  if (method != 1) return kE[j];
  return j < 3 || j == 6 ? kE23[j == 6 ? 3 : j] : 0.0;
}
__device__ __forceinline__ void film_coefs(StageCoef* sc, double h, double a0, double a1, int lane) {
  float* c = reinterpret_cast<float*>(sc);   // ah[7][6], eh[7]
  c[lane] = (float)(a0 * h);
  if (lane < 17) c[lane + 32] = (float)(a1 * h);
}
// time of a stage slot
__device__ __forceinline__ double film_stage_time(double t, double h, int method, int s) {
  if (method != 1) return t + kC[s] * h;
  return s < 3 || s == 6 ? t + kC23[s == 6 ? 3 : s] * h : t;
}

template <int LX, int PH, int ROWS, int PZ>
__global__ void __launch_bounds__(FilmCfg<LX, PH, ROWS, PZ>::NT, 1) k_film(const __grid_constant__ FilmArgs a) {
  using F = FilmCfg<LX, PH, ROWS, PZ>;
  using FX = typename F::FX;
  using FY = typename F::FY;
  constexpr int NT = F::NT, CPB = F::CPB, QR = F::QR, LR = F::LR, CELLS = F::CELLS;
  constexpr int ND = F::ND;
  constexpr bool D3 = PZ > 1;
  const Geom& g = a.g;
  const int nx = g.nx, ny = g.ny, n = (int)g.n, tid = threadIdx.x, lane = tid & 31;
  constexpr int hx = LX + 1;
  // rows y0 .. of layer z
  const int nz = D3 ? g.nz : 1, nch = (ny + ROWS - 1) / ROWS;
  const int z = D3 ? blockIdx.x / nch : 0, y0 = (D3 ? blockIdx.x % nch : blockIdx.x) * ROWS;
  const int kx0 = blockIdx.x * CPB;
  const int nrow = z < nz ? max(0, min(ROWS, ny - y0)) : 0, ncol = max(0, min(CPB, hx - kx0));
  const int ncell = nrow * nx, D = LR * nx;

  extern __shared__ float4 film_dyn[];
  // (the stage rows first: with nx a multiple of 4 they take 16-byte copies)
  float* sst = reinterpret_cast<float*>(film_dyn);            // stage input, STG buffers [3][LR][nx]
  float2* fb = reinterpret_cast<float2*>(sst + (F::STG * 3 * D + 1) / 2 * 2);   // pencil areas (8-byte aligned)
  float2* tx = fb + F::FFT;                                   // x twiddles
  float2* ty = tx + FX::TAB;                                  // y twiddles
  float2* twc = ty + FY::TAB;                                 // W_2PH^y (class 1)
  float2* tw2 = twc + PH;                                     // W_2LX^k, k <= LX
  RegionLUT* lut = reinterpret_cast<RegionLUT*>(tw2 + LX + 1);
  float* ce = reinterpret_cast<float*>(lut + 1);              // exchange couplings [ND][ROWS nx]
  int* sco = reinterpret_cast<int*>(ce + ND * ROWS * nx);      // codes [LR][nx]
  float* soct = reinterpret_cast<float*>(sco + LR * nx);      // octant [CPB][component, kz][PH + 1]
  __shared__ DevState S;
  __shared__ StageCoef sc;
  __shared__ float sinv[7];
  __shared__ float wmax[32];
  __shared__ int flag;

  // ---- constants of the launch ----------------------------------------------
  FX::template tables<NT>(tx, a.tw);
  FY::template tables<NT>(ty, a.tw);
  for (int i = tid; i < PH; i += NT) twc[i] = __ldg(&a.tw[i * (kTwN / (2 * PH))]);
  for (int i = tid; i <= LX; i += NT) tw2[i] = __ldg(&a.tw[(i * (kTwN / (2 * LX))) & (kTwN - 1)]);
  for (int i = tid; i < (int)(sizeof(RegionLUT) / 4); i += NT)
    reinterpret_cast<float*>(lut)[i] = __ldg(reinterpret_cast<const float*>(a.lut) + i);
  // stencil row lr: own layer from y0 - 1 (ROWS + 2 rows), then rows y0 .. of
  // the layer below, then of the layer above; -1 outside the grid
  auto stencil_row = [&](int lr) -> int {
    int yy = y0 - 1 + lr, zz = z;
    if (D3 && lr >= ROWS + 2) {
      const int q = lr - (ROWS + 2);
      yy = y0 + q % ROWS;
      zz = q < ROWS ? z - 1 : z + 1;
    }
    return yy >= 0 && yy < ny && zz >= 0 && zz < nz ? zz * ny + yy : -1;
  };
  for (int e = tid; e < LR * nx; e += NT) {
    const int row = stencil_row(e / nx);
    sco[e] = row >= 0 ? a.code[row * nx + e % nx] : kVacuum;
  }
  const int per = g.hky * g.hkz;
  if (a.oct_sm)
    for (int e = tid; e < ncol * F::OCOL; e += NT) {
      const int q = e / F::OCOL, i = e % F::OCOL;
      // (the components of a column are contiguous: films take the first four)
      soct[e] = __ldg(&a.kt[(kx0 + q) * 6 * per + i]);
    }
  for (int i = tid; i < (int)(sizeof(DevState) / 4); i += NT)
    reinterpret_cast<unsigned*>(&S)[i] = __ldcg(reinterpret_cast<const unsigned*>(a.st) + i);
  __syncthreads();
  // cell e of the block: row and column
  auto split = [&](int e, int& r, int& x) {
    r = 0;
    x = e;
#pragma unroll
    for (int q = 1; q < ROWS; ++q)
      if (x >= nx) {
        x -= nx;
        ++r;
      }
  };
  // stencil positions of own cell (r, x): a missing neighbour is the cell
  // itself (one layer: both z neighbours, not visited)
  auto neighbours = [&](int r, int x, int (&nb)[ND]) {
    const int y = y0 + r, C = (r + 1) * nx + x;
    nb[0] = x > 0 ? C - 1 : (g.pbcx ? C + nx - 1 : C);
    nb[1] = x < nx - 1 ? C + 1 : (g.pbcx ? C - (nx - 1) : C);
    nb[2] = y > 0 ? C - nx : C;
    nb[3] = y < ny - 1 ? C + nx : C;
    if constexpr (D3) {
      nb[4] = z > 0 ? (ROWS + 2 + r) * nx + x : C;
      nb[5] = z < nz - 1 ? (2 * ROWS + 2 + r) * nx + x : C;
    }
  };
  // exchange couplings of the own cells, 2 S H(Aex / Msat) / d^2 per direction
  // (with DMI a missing neighbour is a ghost coupled like the cell itself)
  for (int e = tid; e < ncell; e += NT) {
    int r, x, nb[ND];
    split(e, r, x);
    neighbours(r, x, nb);
    const int C = (r + 1) * nx + x, ci = sco[C];
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      const int cj = sco[nb[d]];
      const bool present = (nb[d] != C || (g.pbcx && d < 2)) && cj != kVacuum;
      float c = 0.0f;
      if (ci != kVacuum && (a.T.dmi ? a.T.exch : 1))
        c = __ldg(&a.xlut[ci * kXStride + (a.T.dmi && !present ? ci : cj)]) *
            (d < 2 ? g.idx2 : (d < 4 ? g.idy2 : g.idz2));
      ce[d * ROWS * nx + e] = c;
    }
  }
  double ca0 = 0, ca1 = 0;   // (warp 0) tableau values of film_coefs
  if (tid < 32) {
    ca0 = film_tableau(S.method, lane);
    ca1 = film_tableau(S.method, lane + 32);
    if (a.begin && tid == 0) {
      S.status = 0;
      S.done = 0;
      S.call_attempts = 0;
      S.err_bits = 0;
      S.ticket = 0;
      S.mode = a.mode;
      S.target = S.accepted + a.nsteps;
      S.t_end = a.t_end;
      if (a.mode == 2 && S.fixed_idx >= S.fixed_n) S.done = 1;
      check_done(&S);
      if (a.nsteps <= 0 && a.mode != 1) S.done = 1;
    }
    __syncwarp();
    if (!S.done) {
      const double h = S.mode == 2 ? a.fixed[S.fixed_idx] : (S.mode == 1 ? fmin(S.dt, S.t_end - S.t) : S.dt);
      film_coefs(&sc, h, ca0, ca1, lane);
      if (tid < 7 && a.T.zeeman)
        sinv[tid] = excitation(a.freq, a.phase_over_pi, film_stage_time(S.t, h, S.method, tid));
      __syncwarp();
      if (tid == 0) S.h = h;
    }
    __syncwarp();
    // (other blocks may read the state while block 0 writes the begun one:
    // beginning a begun state gives the same state)
    if (a.begin && blockIdx.x == 0 && tid == 0) *a.st = S;
  }
  __syncthreads();
  const long long limit = a.state_limit ? S.wait_cycles : kWaitCycles;

  // the block's last act: the last block to leave zeroes the barrier
  auto leave = [&]() {
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      if (atomicAdd(&a.sync->left, 1u) == gridDim.x - 1) {
        a.sync->arrived = 0;
        a.sync->left = 0;
        for (int i = 0; i < 3; ++i) a.sync->err[i] = 0;
      }
    }
  };
  if (S.done) {   // (the same in every block)
    leave();
    return;
  }

  // m and the k's stay in the global buffers; a thread reads only what it wrote
  const int own = (z * ny + y0) * nx;   // first own cell
  auto kbuf = [&](int j) -> float* {
    float* p;
    switch (j) {
      case 0: p = a.k[0]; break;
      case 1: p = a.k[1]; break;
      case 2: p = a.k[2]; break;
      case 3: p = a.k[3]; break;
      case 4: p = a.k[4]; break;
      case 5: p = a.k[5]; break;
      default: p = a.k[6]; break;
    }
    return p + own;
  };

  // grid barrier, arrive and wait apart; the wait is false (in every thread
  // of the block) once the limit has passed
  unsigned int nbar = 0;
  auto arrive = [&]() {
    __syncthreads();
    ++nbar;
    if (tid == 0) red_release(&a.sync->arrived);
  };
  auto wait = [&]() -> bool {
    if (tid == 0) {
      const unsigned int want = nbar * gridDim.x;
      const long long t0 = clock64();
      int ok = 1;
      for (;;) {
        if (clock64() - t0 >= limit) {
          ok = 0;
          break;
        }
        if (ld_acquire(&a.sync->arrived) >= want) break;
      }
      flag = ok;
    }
    __syncthreads();
    return flag != 0;
  };
  auto timeout = [&]() {
    if (tid == 0) {
      a.st->status = -6;   // MM_ERR_TIMEOUT
      a.st->done = 1;
    }
    leave();
  };

  float* rowf = reinterpret_cast<float*>(fb);
  // float index of cell x of component c, row r in the row pencils; a cell
  // uses the place rix ^ 1 of the exchanged parts for its B_demag and, written
  // by the same thread after that is read, for its M
  auto rix = [&](int c, int r, int x) { return 2 * ((c * ROWS + r) * FX::AREA + FX::pos(x >> 1)) + (x & 1); };
  // lane roles in the transforms
  const int px = tid / FX::LANES, jx = tid % FX::LANES;   // row pencil c ROWS + r
  const int pc = tid / FY::LANES, jy = tid % FY::LANES;   // column pencil (q 3 + c) 2 + class

  float kn[CELLS][3], mn[CELLS][3];   // the last stage's torque and the candidate m

  // ---- attempts ---------------------------------------------------------------
  bool fresh = false;   // kn, mn are the current k_0 and m
  for (int att = 0; att < a.attempts; ++att) {
    const int par = S.parity;
    const bool rk23 = S.method == 1;
    float* __restrict__ mcur = (par ? a.m1 : a.m0) + own;
    int cur = 0;   // stage buffer in use
    if (blockIdx.x == 0 && tid == 0) a.sync->err[(att + 1) % 3] = 0;
    // a cell's stage input: stage buffer (3-D: filled from the halo array later),
    // rows for the neighbours, M in the row pencils
    auto put = [&](float* st_, int e, int r, int x, int ci, const float (&v)[3]) {
      const float ms = ci != kVacuum ? lut->msat[ci] : 0.f;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (!D3) st_[c * D + (r + 1) * nx + x] = v[c];
        rowf[rix(c, r, x) ^ 1] = ms * v[c];
        if (D3 || r == 0 || r == nrow - 1) a.halo[c * n + own + e] = v[c];
      }
    };
    {   // the input of the second stage (k1: of the first, m itself)
      const float* k0 = kbuf(k_role(0, par));
      const float c0 = sc.ah[1][0];
#pragma unroll
      for (int q = 0; q < CELLS; ++q) {
        const int e = tid + q * NT;
        if (e >= ncell) break;
        int r, x;
        split(e, r, x);
        float v[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float m = fresh ? mn[q][c] : mcur[c * n + e];
          v[c] = a.k1 ? m : fmaf(c0, fresh ? kn[q][c] : k0[c * n + e], m);
        }
        put(sst, e, r, x, sco[(r + 1) * nx + x], v);
      }
    }
    float emax = 0.f;
    for (int s = a.k1 ? 0 : 1;;) {
      const int nxt = rk23 ? (s == 1 ? 2 : 6) : s + 1;   // slot of the next stage (unused after the last)
      float* st_ = sst + cur * 3 * D;
      __syncthreads();
      // ---- rows: x R2C ----
      if (tid < F::LANX && nrow > 0) {
        const int nin = (nx + 1) / 2;
        float2* e = fb + px * FX::AREA;
        FX::run(e, tx, jx, [&](int i, int) {
          float2 v = i < nin ? swapc(e[FX::pos(i)]) : make_float2(0.f, 0.f);
          if ((nx & 1) && i == nin - 1) v.y = 0.f;   // (x = nx is padding)
          return v;
        });
      }
      __syncthreads();
      // X_k = E_k + W_2L^k O_k on the pairs (k, L - k); consecutive threads on
      // the block's rows (a run of 8 ROWS bytes in spec1)
      if (nrow > 0)
        for (int e = tid; e < 3 * ROWS * (LX / 2 + 1); e += NT) {
          const int r = e % ROWS, k = (e / ROWS) % (LX / 2 + 1), c = e / (ROWS * (LX / 2 + 1));
          if (r >= nrow) continue;
          const float2* row = fb + (c * ROWS + r) * FX::AREA;
          const float2 zk = row[FX::pos(k)], zl = k ? row[FX::pos(LX - k)] : zk;
          const int ks = nz * ny;   // stride of kx in spec1
          float2* dst = a.spec1 + c * hx * ks + z * ny + y0 + r;
          {
            const float2 zc = cconj(zl);
            const float2 E = cscale(cadd(zk, zc), 0.5f), d = csub(zk, zc);
            dst[k * ks] = cadd(E, cmul(tw2[k], make_float2(0.5f * d.y, -0.5f * d.x)));
          }
          if (k != LX / 2) {
            const float2 zc = cconj(zk);
            const float2 E = cscale(cadd(zl, zc), 0.5f), d = csub(zl, zc);
            dst[(LX - k) * ks] = cadd(E, cmul(tw2[LX - k], make_float2(0.5f * d.y, -0.5f * d.x)));
          }
        }
      arrive();
      // the earlier-stage part of the next stage input (of the error estimate
      // after the last stage), while the other blocks arrive:
      // m + sum_{j<s} a_j k_j, j ascending
      float av[CELLS][3];
#pragma unroll
      for (int q = 0; q < CELLS; ++q) {
        const int e = tid + q * NT;
        av[q][0] = av[q][1] = av[q][2] = 0.f;
        if (e >= ncell || s == 0) continue;
        float kj[6][3];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          const float w = s < 6 ? (j < s ? sc.ah[nxt][j] : 0.0f) : sc.eh[j];
          kj[j][0] = kj[j][1] = kj[j][2] = 0.f;
          if (w != 0.0f) {
            const float* k = kbuf(k_role(j, par));
#pragma unroll
            for (int c = 0; c < 3; ++c) kj[j][c] = k[c * n + e];
          }
        }
        if (s < 6) {
#pragma unroll
          for (int c = 0; c < 3; ++c) av[q][c] = mcur[c * n + e];
        }
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          const float w = s < 6 ? (j < s ? sc.ah[nxt][j] : 0.0f) : sc.eh[j];
          if (w != 0.0f) {
#pragma unroll
            for (int c = 0; c < 3; ++c) av[q][c] = fmaf(w, kj[j][c], av[q][c]);
          }
        }
      }
      if (!wait()) return timeout();
      // ---- columns: y forward, kernel product, y inverse ----
      // (the stencil rows of other blocks, in 3-D all of them: their owners
      // wrote them before the barrier)
      if (nrow > 0) {
        constexpr int NH = D3 ? LR : 2;   // rows to fetch per component
        const bool vec = (nx & 3) == 0;   // (rows on 16-byte boundaries)
        const int cpr = vec ? nx / 4 : nx;
        for (int e = tid; e < 3 * NH * cpr; e += NT) {
          const int ch = e % cpr, q = e / cpr, c = q / NH, lr = D3 ? q % NH : (q % NH ? nrow + 1 : 0);
          const int row = stencil_row(lr);
          if (row < 0) continue;
          const int w = vec ? 4 * ch : ch;
          const unsigned d = (unsigned)__cvta_generic_to_shared(&st_[c * D + lr * nx + w]);
          const float* src = a.halo + c * n + row * nx + w;
          if (vec) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
          else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
        }
      }
#pragma unroll 1
      for (int q0 = 0; q0 < ncol; q0 += QR) {
        if (q0 > 0) __syncthreads();   // (the previous columns' areas are read)
        const int nq = min(QR, ncol - q0);
        const int npen = 6 * nz * nq;
        // pencil ((q 3 + c) nz + layer) 2 + class
        for (int p = pc; p < (npen + F::PPW - 1) / F::PPW * F::PPW; p += NT / FY::LANES) {
          const int cls = p & 1, layer = D3 ? (p >> 1) % nz : 0, cq = (p >> 1) / nz, c = cq % 3, q = cq / 3;
          const float2* src = a.spec1 + ((c * hx + kx0 + q0 + q) * nz + layer) * ny;
          const bool on = p < npen;
          FY::run(fb + p * FY::AREA, ty, jy, [&](int y, int) {
            const float2 v = on && y < ny ? __ldcg(src + y) : make_float2(0.f, 0.f);
            return cls ? cmul(v, twc[y]) : v;
          });
        }
        __syncthreads();
        // the kernel product at ky = 2 k + class: Kxy is odd in ky, Kxz in kz,
        // Kyz in both; the result's parts are exchanged (the transform that
        // follows is the inverse)
#pragma unroll 1
        for (int e = tid; e < nq * 2 * PH; e += NT) {
          const int k = e % PH, s2 = (e / PH) & 1, q = e / (2 * PH), ky = 2 * k + s2;
          const int iy = ky > PH ? 2 * PH - ky : ky;
          const float sy = ky > PH ? -1.f : 1.f;
          const float* ko = a.oct_sm ? soct + (q0 + q) * F::OCOL + iy : a.kt + (kx0 + q0 + q) * 6 * per + iy;
          float2* p = fb + (q * 6 * nz + s2) * FY::AREA + FY::pos(k);   // component c, layer l at (c nz + l) 2 AREA
          if constexpr (!D3) {
            const float kxx = ko[0], kyy = ko[PH + 1], kzz = ko[2 * (PH + 1)], kxy = sy * ko[3 * (PH + 1)];
            const float2 X = p[0], Y = p[2 * FY::AREA], Z = p[4 * FY::AREA];
            p[0] = make_float2(kxx * X.y + kxy * Y.y, kxx * X.x + kxy * Y.x);
            p[2 * FY::AREA] = make_float2(kxy * X.y + kyy * Y.y, kxy * X.x + kyy * Y.x);
            p[4 * FY::AREA] = make_float2(kzz * Z.y, kzz * Z.x);
          } else {
            // the PZ-point z transforms of the column's layers in registers
            constexpr int HZ = (PZ / 2 + 1) * (PH + 1);   // octant values per component
            float2 v[3][PZ];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
#pragma unroll
              for (int l = 0; l < PZ; ++l)
                v[c][l] = l < F::NZ && l < nz ? p[(c * nz + l) * 2 * FY::AREA] : make_float2(0.f, 0.f);
              Dft<PZ, -1>::run(v[c]);
            }
#pragma unroll
            for (int kz = 0; kz < PZ; ++kz) {
              const float* o = ko + (kz > PZ / 2 ? PZ - kz : kz) * (PH + 1);
              const float sz = kz > PZ / 2 ? -1.f : 1.f;
              const float kxx = o[0], kyy = o[HZ], kzz = o[2 * HZ], kxy = sy * o[3 * HZ], kxz = sz * o[4 * HZ],
                          kyz = sy * sz * o[5 * HZ];
              const float2 X = v[0][kz], Y = v[1][kz], Z = v[2][kz];
              v[0][kz] = make_float2(kxx * X.x + kxy * Y.x + kxz * Z.x, kxx * X.y + kxy * Y.y + kxz * Z.y);
              v[1][kz] = make_float2(kxy * X.x + kyy * Y.x + kyz * Z.x, kxy * X.y + kyy * Y.y + kyz * Z.y);
              v[2][kz] = make_float2(kxz * X.x + kyz * Y.x + kzz * Z.x, kxz * X.y + kyz * Y.y + kzz * Z.y);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              Dft<PZ, 1>::run(v[c]);
#pragma unroll
              for (int l = 0; l < F::NZ; ++l)
                if (l < nz) p[(c * nz + l) * 2 * FY::AREA] = swapc(v[c][l]);
            }
          }
        }
        __syncthreads();
        for (int p = pc; p < (npen + F::PPW - 1) / F::PPW * F::PPW; p += NT / FY::LANES) {
          float2* e = fb + p * FY::AREA;
          FY::run(e, ty, jy, [&](int i, int) { return e[FY::pos(i)]; });
        }
        __syncthreads();
        // x[y] = x_0[y] + conj(W_2PH^y) x_1[y]; consecutive threads on the
        // block's columns (a run of 8 QR bytes in spec2)
        for (int e = tid; e < nq * 3 * nz * ny; e += NT) {
          const int q = e % nq, y = (e / nq) % ny, cl = e / (nq * ny);   // cl = c nz + layer
          const float2* p = fb + 2 * (q * 3 * nz + cl) * FY::AREA + FY::pos(y);
          a.spec2[(cl * ny + y) * g.hxs + kx0 + q0 + q] = cadd(swapc(p[0]), cmul(swapc(p[FY::AREA]), cconj(twc[y])));
        }
      }
      asm volatile("cp.async.wait_all;\n" ::: "memory");
      arrive();
      if (!wait()) return timeout();
      // ---- rows: x C2R, the pair (k, L - k) by one thread ----
      if (nrow > 0) {
        for (int e = tid; e < 3 * ROWS * (LX / 2 + 1); e += NT) {
          const int k = e % (LX / 2 + 1), pen = e / (LX / 2 + 1), r = pen % ROWS, c = pen / ROWS;
          if (r >= nrow) continue;
          const float2* row = a.spec2 + ((c * nz + z) * ny + y0 + r) * g.hxs;
          const float2 xa = __ldcg(row + k), xb = __ldcg(row + LX - k);
          float2 za, zb;
          {
            const float2 E = cscale(cadd(xa, cconj(xb)), 0.5f);
            const float2 O = cmul(cscale(csub(xa, cconj(xb)), 0.5f), cconj(tw2[k]));
            za = make_float2(E.y + O.x, E.x - O.y);   // (exchanged: inverse)
          }
          {
            const float2 E = cscale(cadd(xb, cconj(xa)), 0.5f);
            const float2 O = cmul(cscale(csub(xb, cconj(xa)), 0.5f), cconj(tw2[LX - k]));
            zb = make_float2(E.y + O.x, E.x - O.y);
          }
          fb[pen * FX::AREA + FX::pos(k)] = za;
          if (k != 0 && k != LX / 2) fb[pen * FX::AREA + FX::pos(LX - k)] = zb;
        }
        __syncthreads();
        if (tid < F::LANX) {
          float2* e = fb + px * FX::AREA;
          FX::run(e, tx, jx, [&](int i, int) { return e[FX::pos(i)]; });
        }
        __syncthreads();
      }
      // ---- cells: field, torque, next stage input or error and candidate ----
      const float sinft = a.T.zeeman ? sinv[s] : 0.0f;
      float* ks = kbuf(k_role(s, par));
      float* nst = sst + (D3 ? 0 : (cur ^ 1) * 3 * D);
      const float wn = s < 6 ? sc.ah[nxt][s] : sc.eh[6];
      float* mnew = (par ? a.m0 : a.m1) + own;
#pragma unroll
      for (int q = 0; q < CELLS; ++q) {
        const int e = tid + q * NT;
        if (e >= ncell) break;
        int r, x, nb[ND];
        split(e, r, x);
        neighbours(r, x, nb);
        const int C = (r + 1) * nx + x, ci = sco[C];
        const float3 mi = f3(st_[C], st_[D + C], st_[2 * D + C]);
        float3 tq = f3(0, 0, 0);
        if (ci != kVacuum) {
          FieldParts P;
          P.demag = f3(rowf[rix(0, r, x) ^ 1], rowf[rix(1, r, x) ^ 1], rowf[rix(2, r, x) ^ 1]);   // (exchanged parts)
          P.dmi = f3(0, 0, 0);
          float3 ex = f3(0, 0, 0);
          if (!a.T.dmi) {
            if (a.T.exch) {
#pragma unroll
              for (int d = 0; d < ND; ++d) {
                const float c = ce[d * ROWS * nx + e];
                ex.x += c * (st_[nb[d]] - mi.x);
                ex.y += c * (st_[D + nb[d]] - mi.y);
                ex.z += c * (st_[2 * D + nb[d]] - mi.z);
              }
            }
          } else {
            const float cbc = lut->dbc[ci];
            float3 v[4];
#pragma unroll
            for (int d = 0; d < ND; ++d) {
              const int j = nb[d];
              const bool present = (j != C || (g.pbcx && d < 2)) && sco[j] != kVacuum;
              const float3 mj = present ? f3(st_[j], st_[D + j], st_[2 * D + j]) : dmi_ghost(mi, d, cbc, g.cdx, g.cdy);
              const float c = ce[d * ROWS * nx + e];
              ex.x += c * (mj.x - mi.x);
              ex.y += c * (mj.y - mi.y);
              ex.z += c * (mj.z - mi.z);
              if (d < 4) v[d] = mj;
            }
            P.dmi = dmi_field(lut->dmi[ci], v[0], v[1], v[2], v[3], g.cdx, g.cdy);
          }
          P.exch = ex;
          field_local<LdAny>(lut, a.T, ci, mi, sinft, P);
          tq = llg_torque(mi, total(P), lut->gfac[ci], lut->alpha[ci], S.precession);
          if (a.S.zl || a.S.sl) {
            float3 h = f3(0, 0, 0);
            if (a.S.zl) {
              const float hd[3] = {a.S.hx, a.S.hy, a.S.hz};
#pragma unroll
              for (int ax = 0; ax < ND / 2; ++ax) {
                const int j1 = nb[2 * ax + 1], j0 = nb[2 * ax];
                const float3 v1 = sco[j1] != kVacuum ? f3(st_[j1], st_[D + j1], st_[2 * D + j1]) : mi;
                const float3 v0 = sco[j0] != kVacuum ? f3(st_[j0], st_[D + j0], st_[2 * D + j0]) : mi;
                const float c = __ldg(&a.S.lut->zlu[ax][ci]) * hd[ax];
                h.x += c * (v1.x - v0.x);
                h.y += c * (v1.y - v0.y);
                h.z += c * (v1.z - v0.z);
              }
            }
            const float3 ts = stt_torque(a.S, ci, mi, h);
            tq = f3(tq.x + ts.x, tq.y + ts.y, tq.z + ts.z);
          }
        }
        const float kv[3] = {tq.x, tq.y, tq.z};
#pragma unroll
        for (int c = 0; c < 3; ++c) ks[c * n + e] = kv[c];
        if (s == 0) continue;
        float v[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) v[c] = fmaf(wn, kv[c], av[q][c]);
        if (s < 6) {
          put(nst, e, r, x, ci, v);
        } else {
          float inv = 0.0f;
          if (ci != kVacuum) {
            float err = sqrtf(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
            if (!(err <= FLT_MAX)) err = __int_as_float(0x7f800000);
            emax = fmaxf(emax, err);
            inv = rsqrtf(mi.x * mi.x + mi.y * mi.y + mi.z * mi.z);
          }
          const float m3[3] = {mi.x, mi.y, mi.z};
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            mn[q][c] = ci != kVacuum ? m3[c] * inv : 0.0f;
            kn[q][c] = kv[c];
            mnew[c * n + e] = mn[q][c];
          }
        }
      }
      if (s == 0) {
        leave();
        return;
      }
      if (s == 6) break;
      s = nxt;
      if (!D3) cur ^= 1;
    }
    for (int o = 16; o > 0; o >>= 1) emax = fmaxf(emax, __shfl_xor_sync(0xffffffffu, emax, o));
    if (lane == 0) wmax[tid >> 5] = emax;
    __syncthreads();
    if (tid < 32) {
      float v = tid < NT / 32 ? wmax[tid] : 0.0f;
      for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
      if (tid == 0 && v > 0.0f) atomicMax(&a.sync->err[att % 3], __float_as_uint(v));
    }
    arrive();
    if (!wait()) return timeout();
    // The controller, by one warp, the same in every block.  (With its float64
    // operands read ahead of the wait 10 steps of a 256 x 256 film took 836
    // us, here 825, 20 of a 64 x 16 film 923 both ways.)
    if (tid < 32) {
      const float eps = __uint_as_float(__ldcg(&a.sync->err[att % 3]));
      const StepDecision d = step_decide(S, eps);
      double hn = 0;
      if (!d.done) {
        hn = S.mode == 2 ? a.fixed[d.fixed_idx] : (S.mode == 1 ? fmin(d.dt, S.t_end - d.t) : d.dt);
        film_coefs(&sc, hn, ca0, ca1, lane);
      }
      __syncwarp();
      if (lane == 0) {
        step_apply(&S, d, eps, blockIdx.x == 0 ? a.hist : nullptr);
        if (!d.done) S.h = hn;
      }
    }
    __syncthreads();
    fresh = S.parity != par;
    // off the critical path: the global state (block 0), the next attempt's
    // field amplitudes
    if (tid >= 32 && tid < 64) {
      if (blockIdx.x == 0)
        for (int i = lane; i < (int)(sizeof(DevState) / 4); i += 32)
          reinterpret_cast<unsigned*>(a.st)[i] = reinterpret_cast<const unsigned*>(&S)[i];
      if (lane < 7 && a.T.zeeman && !S.done)
        sinv[lane] = excitation(a.freq, a.phase_over_pi, film_stage_time(S.t, S.h, S.method, lane));
    }
    if (S.done) break;
  }
  leave();
}

}  // namespace

template <int LX, int PH, int ROWS, int PZ>
bool film_plan_one(const Geom& g, FilmPlan* p) {
  using F = FilmCfg<LX, PH, ROWS, PZ>;
  int dev = 0, sms = 0, coop = 0, smem_max = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (!coop) return false;
  const size_t room = smem_max > 2048 ? (size_t)smem_max - 2048 : 0;   // (static: state, coefficients)
  if (ROWS * g.nx > F::CELLS * F::NT) return false;   // (long periodic rows)
  size_t need = sizeof(float2) * (F::FFT + F::TAB + 1) +
                sizeof(float) * ((3 * F::STG + 1) * F::LR + F::ND * ROWS) * g.nx + sizeof(RegionLUT);
  if (need > room) return false;
  const size_t ob = sizeof(float) * F::OCT;
  p->oct_sm = need + ob <= room;
  if (p->oct_sm) need += ob;
  p->rows = ROWS;
  p->blocks = std::max((g.ny + ROWS - 1) / ROWS * g.nz, (LX + F::CPB) / F::CPB);
  p->smem = need;
  // (a function attribute belongs to the device's context; the cap, not this
  // film's need, so that a later film never lowers an earlier one's)
  if (cudaFuncSetAttribute(k_film<LX, PH, ROWS, PZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room) != cudaSuccess) {
    (void)cudaGetLastError();
    p->rows = 0;
    return false;
  }
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_film<LX, PH, ROWS, PZ>, F::NT, need) != cudaSuccess ||
      (long long)per_sm * sms < p->blocks) {
    (void)cudaGetLastError();
    p->rows = 0;
    return false;
  }
  return true;
}

template <int LX, int PH, int ROWS, int PZ>
cudaError_t launch_film_one(const FilmPlan& p, const FilmArgs& args, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.blocks);
  cfg.blockDim = dim3(FilmCfg<LX, PH, ROWS, PZ>::NT);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;   // (the blocks wait for one another)
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_film<LX, PH, ROWS, PZ>, args);
}

// Rows per block: the fewest whose blocks fit kFilmBlocks.
#define MM_FILM_CASES(DO)                                                  \
  if (g.nz == 1) {                                                         \
    switch (ph) {                                                          \
      case 16: return DO(16, 1, 1);                                        \
      case 32: return DO(32, 1, 1);                                        \
      case 64: return DO(64, 1, 1);                                        \
      case 128: return DO(128, 1, 1);                                      \
      case 256: return DO(256, 2, 1);                                      \
      case 512: return g.ny <= 3 * kFilmBlocks ? DO(512, 3, 1) : DO(512, 4, 1); \
      default: break;                                                      \
    }                                                                      \
  }
#define MM_FILM3_CASES(DO)                                                 \
  if (g.pz == 4) {                                                         \
    switch (ph) {                                                          \
      case 16: return DO(16, 1, 4);                                        \
      case 32: return DO(32, 1, 4);                                        \
      case 64: return DO(64, 1, 4);                                        \
      case 128: return DO(128, 2, 4);                                      \
      default: break;                                                      \
    }                                                                      \
  } else if (g.pz == 8) {                                                  \
    switch (ph) {                                                          \
      case 16: return DO(16, 1, 8);                                        \
      case 32: return DO(32, 1, 8);                                        \
      case 64: return DO(64, 2, 8);                                        \
      case 128: return g.ny <= 3 * (kFilmBlocks / 4) ? DO(128, 3, 8) : DO(128, 4, 8); \
      default: break;                                                      \
    }                                                                      \
  }
#define MM_FILM_PLAN(PH, ROWS, PZ) film_plan_one<LX, PH, ROWS, PZ>(g, p)
#define MM_FILM_LAUNCH(PH, ROWS, PZ) launch_film_one<LX, PH, ROWS, PZ>(p, args, s)
template <int LX>
bool film_plan_l(const Geom& g, int ph, FilmPlan* p) {
  MM_FILM_CASES(MM_FILM_PLAN)
  return false;
}
template <int LX>
cudaError_t launch_film_l(const FilmPlan& p, int ph, const FilmArgs& args, cudaStream_t s) {
  const Geom& g = args.g;
  MM_FILM_CASES(MM_FILM_LAUNCH)
  return cudaErrorInvalidValue;
}
// thin 3-D grids (in translation units of their own)
template <int LX>
bool film3_plan_l(const Geom& g, int ph, FilmPlan* p) {
  MM_FILM3_CASES(MM_FILM_PLAN)
  return false;
}
template <int LX>
cudaError_t launch_film3_l(const FilmPlan& p, int ph, const FilmArgs& args, cudaStream_t s) {
  const Geom& g = args.g;
  MM_FILM3_CASES(MM_FILM_LAUNCH)
  return cudaErrorInvalidValue;
}

}  // namespace mm
