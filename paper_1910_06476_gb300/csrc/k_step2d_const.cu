// Dispatch of the 2D shared-operator kernel on the node count and the tile shape (elements per
// CTA, TX x TY, both even).  Each node count has a few compiled shapes, up to 75 KB of dynamic shared
// memory and 1024 threads; index 0 is the default (by mesh size, see default_tile), the others are
// candidates for the autotuner (sl_tune).  Every shape computes each element with the same arithmetic.
#include "sl_internal.h"

namespace sl {
namespace k2c {
template <int NN, int TX, int TY>
void launch(const Mixed2DConstParams& p, const float* tab, const float* in, float* out, unsigned* st, cudaStream_t s);
}

int k2c_tile_count(int n) { return n <= 12 ? 3 : 2; }

void k2c_tile_shape(int n, int tile, int* tx, int* ty) {
  static const int small[3][2] = {{8, 4}, {4, 4}, {8, 2}};     // n <= 9
  static const int mid[3][2] = {{4, 4}, {4, 2}, {2, 2}};       // n = 10..12
  static const int large[2][2] = {{4, 2}, {2, 2}};             // n = 13..17
  if (tile < 0 || tile >= k2c_tile_count(n)) tile = 0;
  const int(*t)[2] = n <= 9 ? small : n <= 12 ? mid : large;
  *tx = t[tile][0];
  *ty = t[tile][1];
}

// The default shape by mesh size: a grid of few CTAs leaves SMs idle and a tile's phases wait on one another, so
// smaller tiles are quicker there, although they stage more halo per element.  Measured, 8 x 4 against 8 x 2 (n <= 9):
// 64 x 56 elements (112 tiles) n = 4 8.6 / 7.1 us, n = 9 13.2 / 11.3; 96 x 84 (252) n = 5 9.2 / 7.7, n = 9 13.9 / 13.2;
// 150 x 132 (627) n = 5 10.5 / 13.6.  4 x 4 against 4 x 2 (n = 10): 64 x 56 (224) 12.7 / 11.1, 96 x 84 (504) 14.5 /
// 13.1, 150 x 132 (1254) 25.3 / 29.0.
static int default_tile(int n, int kx, int ky) {
  int tx, ty;
  k2c_tile_shape(n, 0, &tx, &ty);
  const int64_t tiles = (int64_t)((kx + tx - 1) / tx) * ((ky + ty - 1) / ty);
  if (n <= 9) return tiles <= 2 * sm_count() ? 2 : 0;
  if (n <= 12) return tiles <= 4 * sm_count() ? 1 : 0;
  return 0;
}

#define SL_K2C(N, A, B) k2c::launch<N, A, B>(p, tab, in, out, status, s)
#define SL_K2C_SMALL(N)                        \
  case N:                                      \
    if (tile == 1) SL_K2C(N, 4, 4);            \
    else if (tile == 2) SL_K2C(N, 8, 2);       \
    else SL_K2C(N, 8, 4);                      \
    break;
#define SL_K2C_MID(N)                          \
  case N:                                      \
    if (tile == 1) SL_K2C(N, 4, 2);            \
    else if (tile == 2) SL_K2C(N, 2, 2);       \
    else SL_K2C(N, 4, 4);                      \
    break;
#define SL_K2C_LARGE(N)                        \
  case N:                                      \
    if (tile == 1) SL_K2C(N, 2, 2);            \
    else SL_K2C(N, 4, 2);                      \
    break;

void launch_step2d_const(const Mixed2DConstParams& p, const float* tab, const float* in, float* out, unsigned* status,
                         cudaStream_t s, int tile) {
  if (tile == 0) tile = default_tile(p.n, p.kx, p.ky);
  switch (p.n) {
    SL_K2C_SMALL(2)
    SL_K2C_SMALL(3)
    SL_K2C_SMALL(4)
    SL_K2C_SMALL(5)
    SL_K2C_SMALL(6)
    SL_K2C_SMALL(7)
    SL_K2C_SMALL(8)
    SL_K2C_SMALL(9)
    SL_K2C_MID(10)
    SL_K2C_MID(11)
    SL_K2C_MID(12)
    SL_K2C_LARGE(13)
    SL_K2C_LARGE(14)
    SL_K2C_LARGE(15)
    SL_K2C_LARGE(16)
    SL_K2C_LARGE(17)
    default: break;
  }
}

#undef SL_K2C_SMALL
#undef SL_K2C_MID
#undef SL_K2C_LARGE
#undef SL_K2C

}  // namespace sl
