// In-place Gauss-Jordan inversion of a 32 x 32 block held 2 x 2 elements per thread in the registers of 256
// threads: the step that k_gj_pivot (digit_screen.cu) builds its pivot blocks from. The arithmetic and the
// barriers are parameters, so that the test suite can run the same code on the host with the threads of a warp
// in any order between two barriers (tests/gj_block_check.cpp).
#pragma once
#include "cvt.cuh"

namespace gwi {

// x[a][b]: element (ty + 16 a, tx + 16 b), t = 16 ty + tx; fcol, prow, rowj: 32 elements each in shared memory.
// AR: neg, is_zero, inv, zero, fma2(a, x, y) = a + x y. SYNC: block(), warp().
// Returns the step of a zero pivot (in every thread; x is then undefined), or -1. No pivoting:
// row j <- row j / p (entry j -> 1 / p); other rows r: a_rc -= a_rj a_jc / p, a_rj <- -a_rj / p
template <class AR, class SYNC, class S = typename AR::S>
GW_HD int gj_invert32(S (&x)[2][2], S* fcol, S* prow, S* rowj, int t, const SYNC& sync) {
  const int tx = t & 15, ty = t >> 4;
#pragma unroll
  for (int jb = 0; jb < 2; ++jb)
    for (int jj = 0; jj < 16; ++jj) {
      const int j = 16 * jb + jj;
      if (tx == jj) {
        fcol[ty] = AR::neg(x[0][jb]);
        fcol[ty + 16] = AR::neg(x[1][jb]);
      }
      if (ty == jj) {
        prow[tx] = x[jb][0];
        prow[tx + 16] = x[jb][1];
      }
      sync.block();
      const S p = prow[j];
      if (AR::is_zero(p)) return j;
      if (t < 32) {
        const S ip = AR::inv(p);
        rowj[t] = t == j ? ip : AR::fma2(AR::zero(), prow[t], ip);
      }
      sync.block();
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const S g = rowj[tx + 16 * b];
          S v = x[a][b];
          if (b == jb && tx == jj) v = AR::zero();
          v = AR::fma2(v, fcol[ty + 16 * a], g);
          x[a][b] = a == jb && ty == jj ? g : v;
        }
      // the warp has read fcol before a lane of it writes the next column there (fcol[ty], fcol[ty + 16] belong to
      // the warp of the rows; prow and rowj, which others read, are a block barrier away from their next write)
      sync.warp();
    }
  return -1;
}

}  // namespace gwi
