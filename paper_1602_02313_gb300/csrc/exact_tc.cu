// FP64 contractions of the GW cycle as exact digit products on the tensor cores (digit_gemm.cuh).
//
// polarization, Eq. (irpol): E = Re P + Im P = X Y^T (the real cover of the Hermitian P used by the
//   mixed path), rows of X = (tau, I): [w (re + im) | w (im - re)], rows of Y = I: [re | im]. One
//   GEMM for all tau of a group, split over K; the FP64 partials are summed, P formed from E and E^T.
// self-energy, Eq. (sigc): d_p(tau) = 2 sum_J (re_p Y1 + im_p Y2)[p][J], [Y1 | Y2] = A B^T with
//   A = [re | im] of the pair rows p and B built from the upper triangle of the Hermitian part of
//   W~(tau); the dot with M runs in the epilogue in FP64.
// Measured: P of one q at Nk 27, Nb 32, NI 128, 32 tau 84.5 -> 2.2 ms, Sigma^c of one q at Nk 8, Nb 32,
// NI 128, 32 tau 33.3 -> 0.80 ms against the CUDA-core kernels; faster at every size measured, down to
// Nk 2, Nb 4, NI 32, 16 tau (70 -> 62 us).
#include <algorithm>

#include "digit_gemm.cuh"

namespace gwi {

namespace {

// ------------------------------------------------------------------ what the GEMM does with its tiles
// Polarization: unit = (K split, M tile, N tile), C[split][row][n] = sum over the split's chunks.
struct OpStore {
  static constexpr int LV = 7;
  struct Job {
    const unsigned char *A, *B;  // [M tile][chunk], [N tile][chunk]
    const int *ea, *eb;          // row exponents [rows], [ncols]
    int mt, nt, chunks, nsplit, rows, ncols, sh;
    double* C;
  };
  struct Unit {
    int m, s, n0, n1;
    __device__ Unit(const Job& J, int u) : m((u / J.nt) % J.mt), s(u / (J.nt * J.mt)), n0(u % J.nt), n1(n0 + 1) {}
    __device__ const unsigned char* A(const Job& J, int) const { return J.A + (size_t)m * J.chunks * XA_BYTES; }
    __device__ const unsigned char* B(const Job& J, int n) const { return J.B + (size_t)n * J.chunks * XB_BYTES; }
    __device__ void range(const Job& J, int, int& c0, int& c1) const {
      const int L = (J.chunks + J.nsplit - 1) / J.nsplit;
      c0 = s * L;
      c1 = min(J.chunks, c0 + L);
    }
  };
  int row, part;
  __device__ OpStore(const Job&, const Unit& U, int r, int p) : row(128 * U.m + r), part(p) {}
  __device__ void tile(const Job& J, const Unit& U, int n, const long long (&y)[16]) {
    if (row >= J.rows) return;
    const int ea = J.ea[row], c0 = XN * n + 16 * part;
    double* o = J.C + ((size_t)U.s * J.rows + row) * J.ncols + c0;
#pragma unroll
    for (int e = 0; e < 16; ++e)
      if (c0 + e < J.ncols) o[e] = fix_to_double(y[e], ea + J.eb[c0 + e] - 62 + J.sh);
  }
  __device__ void finish(const Job&, const Unit&, double (&)[3][128], bool) {}
};

// Self-energy: unit = (M tile, tau), all N tiles jt (32 columns J of Y1 beside the same J of Y2) over the
// K chunks I <= J, dotted with M: D[row][tau].
struct OpDot {
  static constexpr int LV = 7;
  struct Job {
    const unsigned char *A, *B;  // [M tile][chunk], [tau][N tile][chunk]
    const int *ea, *eb;          // row exponents [rows], [tau][J]
    int mt, nt, chunks, rows, sh;
    const double2* M;            // M[k][J][p] of the job's first row
    int np, ni, ntau, tau0, ntau_all, tgrp;
    double* D;
  };
  struct Unit {
    int m, b, n0, n1;
    __device__ Unit(const Job& J, int u) : n0(0), n1(J.nt) {
      // tau in groups of tgrp, inside a group the M tiles, inside those the group's tau: the blocks that run
      // at one time share their W~ and M digits in L2
      const int per = J.mt * J.tgrp, g = u / per, r = u % per, gt = min(J.tgrp, J.ntau - g * J.tgrp);
      m = r / gt;
      b = g * J.tgrp + r % gt;
    }
    __device__ const unsigned char* A(const Job& J, int) const { return J.A + (size_t)m * J.chunks * XA_BYTES; }
    __device__ const unsigned char* B(const Job& J, int n) const {
      return J.B + ((size_t)b * J.nt + n) * J.chunks * XB_BYTES;
    }
    __device__ void range(const Job&, int n, int& c0, int& c1) const {
      c0 = 0;
      c1 = 4 * (n + 1);
    }
  };
  int r, part, row;
  double dacc[4] = {0.0, 0.0, 0.0, 0.0};  // short chains: less rounding, and the FP64 latency overlaps
  __device__ OpDot(const Job&, const Unit& U, int r_, int p) : r(r_), part(p), row(128 * U.m + r_) {}
  __device__ void tile(const Job& J, const Unit& U, int n, const long long (&y)[16]) {
    if (row >= J.rows) return;
    const int k = row / J.np, p = row - k * J.np, j0 = 32 * n + 16 * (part & 1);
    const double2* Mr = J.M + ((size_t)k * J.ni + j0) * J.np + p;
    const int* eb = J.eb + (size_t)(J.tau0 + U.b) * J.ni + j0;
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const double2 a = Mr[(size_t)e * J.np];
      dacc[e & 3] = fma(fix_to_double(y[e], eb[e] - 62 + J.sh), part >= 2 ? a.y : a.x, dacc[e & 3]);
    }
  }
  __device__ void finish(const Job& J, const Unit& U, double (&red)[3][128], bool ok) {
    const double d = (dacc[0] + dacc[1]) + (dacc[2] + dacc[3]);
    if (part) red[part - 1][r] = d;
    asm volatile("bar.sync 1, %0;" ::"n"(X_EPI * 32) : "memory");
    if (!part && ok && row < J.rows) {
      const int ea = J.ea[row];
      J.D[(size_t)row * J.ntau_all + J.tau0 + U.b] =
          ea == kBadExp ? __longlong_as_double(0x7FF8000000000000ll)
                        : scalbn(2.0 * ((d + red[0][r]) + (red[1][r] + red[2][r])), ea);
    }
    asm volatile("bar.sync 1, %0;" ::"n"(X_EPI * 32) : "memory");
  }
};

// ------------------------------------------------------------------ polarization: preparation
// FP64 pair weights w[tau][g], g = k np + p, of tau0 .. tau0 + nt - 1, and the largest high word of each tau
__global__ void k_xw(const double* __restrict__ G, const int* __restrict__ kmq, int nk, int nb, int ntau,
                     double* __restrict__ w, uint32_t* __restrict__ wmax) {
  const int it = blockIdx.y, np = nb * nb, n = nk * np;
  uint32_t h = 0;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x) {
    const int k = g / np, p = g - k * np, a = p / nb, b = p - a * nb;
    const double v = -G[((size_t)k * nb + b) * ntau + it] * G[((size_t)kmq[k] * nb + a) * ntau + (ntau - 1 - it)];
    w[(size_t)it * n + g] = v;
    h = max(h, abs_hi(v));
  }
  h = warp_max(h);
  if ((threadIdx.x & 31) == 0) atomicMax(wmax + it, h);
}

// largest high word of |re|, |im| of each row I over all k and p: one warp per (I, k)
__global__ void k_xrow(const double2* __restrict__ M, int nk, int ni, int np, uint32_t* __restrict__ ymax) {
  const int wid = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (wid >= nk * ni) return;
  const double2* m = M + (size_t)wid * np;  // [k][I] is wid
  uint32_t h = 0;
  for (int p = lane; p < np; p += 32) {
    const double2 v = m[p];
    h = max(h, max(abs_hi(v.x), abs_hi(v.y)));
  }
  h = warp_max(h);
  if (lane == 0) atomicMax(ymax + wid % ni, h);
}

// largest |w| (|re| + |im|) of each row (tau, I) as a float that is not smaller, in units of
// 2^(exponent of w at tau + exponent of row I): one warp per (k, 4 I) and 16 tau, so that a weight is
// loaded and normalised once for four rows
__global__ void __launch_bounds__(256) k_xrowx(const double2* __restrict__ M, const double* __restrict__ w,
                                               const uint32_t* __restrict__ wmax, const uint32_t* __restrict__ ymax,
                                               int nk, int ni, int np, int ntau, uint32_t* __restrict__ xmax) {
  const int wid = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (wid >= nk * (ni / 4)) return;
  const int k = wid / (ni / 4), I = 4 * (wid % (ni / 4)), t0 = 16 * blockIdx.y;
  int ey[4], ew[16];
  float acc[16][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) ey[i] = exp_of(ymax[I + i]);
#pragma unroll
  for (int t = 0; t < 16; ++t) {
    ew[t] = exp_of(wmax[min(t0 + t, ntau - 1)]);
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[t][i] = 0.f;
  }
  const double2* m = M + ((size_t)k * ni + I) * np;
  const size_t n = (size_t)nk * np;
  const double* wk = w + (size_t)k * np;
  for (int p = lane; p < np; p += 32) {
    double x[16];
    double2 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = m[(size_t)i * np + p];
#pragma unroll
    for (int t = 0; t < 16; ++t) x[t] = wk[min(t0 + t, ntau - 1) * n + p];  // all loads in flight at once
    float a[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = norm_up(v[i].x, ey[i]) + norm_up(v[i].y, ey[i]);
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const float b = norm_up(x[t], ew[t]);
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[t][i] = fmaxf(acc[t][i], a[i] * b);
    }
  }
#pragma unroll
  for (int t = 0; t < 16; ++t)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t h = warp_max(__float_as_uint(acc[t][i] * 1.000002f));
      if (lane == 0 && t0 + t < ntau) atomicMax(xmax + (size_t)(t0 + t) * ni + I + i, h);
    }
}

// row exponents of Y (I) and X (tau, I) from the maxima
__global__ void k_xexp(const uint32_t* __restrict__ wmax, const uint32_t* __restrict__ ymax,
                       const uint32_t* __restrict__ xmax, int ni, int ntau, int* __restrict__ ey, int* __restrict__ ex) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < ni) ey[e] = exp_of(ymax[e]);
  if (e >= ni * ntau) return;
  const int a = exp_of(wmax[e / ni]), b = exp_of(ymax[e % ni]);
  // xmax < 2^(f - 126), f its exponent field; a row whose products all vanish takes the smallest scale
  const int f = max(1, (int)(xmax[e] >> 23));
  ex[e] = (a == kBadExp || b == kBadExp) ? kBadExp : a + b + f - 126;
}

// Digits of Y and of X for tau0 .. tau0 + nt - 1, chunks c0 .. c0 + nc - 1 of 8 pairs ([8 re | 8 im],
// X with re + im and im - re). One thread per (chunk, I) and tpt tau: M is read once for them; lanes
// run along I, so that the 16-byte digit writes of a warp are contiguous.
__global__ void __launch_bounds__(256) k_xslice_pol(const double2* __restrict__ M, const double* __restrict__ w,
                                                    const int* __restrict__ ey, const int* __restrict__ ex, int nk, int ni,
                                                    int np, int c0, int nc, int tau0, int nt, int tpt, int doy,
                                                    unsigned char* __restrict__ Yi, unsigned char* __restrict__ Xi) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)nc * ni) return;
  const int I = (int)(e % ni), c = (int)(e / ni);
  const int64_t n = (int64_t)nk * np, g0 = (int64_t)(c0 + c) * 8;
  double re[8], im[8];
  int k = (int)(g0 / np), p = (int)(g0 - (int64_t)k * np);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    double2 v = make_double2(0.0, 0.0);
    if (g0 + q < n) v = M[((size_t)k * ni + I) * np + p];
    re[q] = v.x;
    im[q] = v.y;
    if (++p == np) {
      p = 0;
      ++k;
    }
  }
  long long t[8];
  if (doy && blockIdx.y == 0) {
    const int s = ey[I];
    unsigned char* ch = Yi + ((size_t)(I / XN) * nc + c) * XB_BYTES;
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] = to_fix(re[q], s);
    put8<XN>(ch, I % XN, 0, t);
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] = to_fix(im[q], s);
    put8<XN>(ch, I % XN, 1, t);
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const double a = re[q] + im[q];
    im[q] = im[q] - re[q];
    re[q] = a;
  }
  // the products w x as integers: a 64-bit high product and a shift straight to the row's fixed point
  // (an FP64 product per element would fill the FP64 pipe for 0.19 of the 0.33 ms this kernel took at
  // Nk 27, Nb 32, NI 128, 16 tau)
  Fl64 fr[8], fi[8];
  uint32_t sg = 0;  // signs: bit q re + im, bit 8 + q im - re
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    fr[q] = fl64(re[q]);
    fi[q] = fl64(im[q]);
    sg |= (uint32_t)((uint64_t)__double_as_longlong(re[q]) >> 63) << q;
    sg |= (uint32_t)((uint64_t)__double_as_longlong(im[q]) >> 63) << (8 + q);
  }
  const int tb = blockIdx.y * tpt;
  for (int it = tb; it < min(nt, tb + tpt); ++it) {
    const int row = it * ni + I, s = ex[(size_t)(tau0 + it) * ni + I];
    unsigned char* ch = Xi + ((size_t)(row >> 7) * nc + c) * XA_BYTES;
    const double* wr = w + (size_t)(tau0 + it) * n + g0;
    double wq[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) wq[q] = g0 + q < n ? wr[q] : 0.0;
    long long u[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const Fl64 fw = fl64(wq[q]);
      const uint32_t sw = (uint32_t)((uint64_t)__double_as_longlong(wq[q]) >> 63);
      const long long a = (long long)mul_fix(fr[q], fw, s), b = (long long)mul_fix(fi[q], fw, s);
      t[q] = ((sg >> q) ^ sw) & 1 ? -a : a;
      u[q] = ((sg >> (8 + q)) ^ sw) & 1 ? -b : b;
    }
    put8<128>(ch, row & 127, 0, t);
    put8<128>(ch, row & 127, 1, u);
  }
}

// E[tau0 ..] (+)= sum over the K splits
__global__ void k_xsum(const double* __restrict__ C, int64_t n, int nsplit, int add, double* __restrict__ E) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= n) return;
  double s = add ? E[e] : 0.0;
  for (int q = 0; q < nsplit; ++q) s += C[(int64_t)q * n + e];
  E[e] = s;
}

// P_ab = scale ((E_ab + E_ba) / 2 + i (E_ab - E_ba) / 2), one block per (32 x 32 block, tau)
__global__ void __launch_bounds__(256) k_xform(const double* __restrict__ E, int ni, double scale, double2* __restrict__ P) {
  __shared__ double tb[32][33];
  const int bx = blockIdx.x, by = blockIdx.y, it = blockIdx.z;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const double* Et = E + (size_t)it * ni * ni;
#pragma unroll
  for (int r = 0; r < 4; ++r) tb[ty + 8 * r][tx] = Et[(size_t)(bx * 32 + ty + 8 * r) * ni + by * 32 + tx];
  __syncthreads();
  double2* Pt = P + (size_t)it * ni * ni;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int a = by * 32 + ty + 8 * r, b = bx * 32 + tx;
    const double e1 = Et[(size_t)a * ni + b], e2 = tb[tx][ty + 8 * r];
    Pt[(size_t)a * ni + b] = make_double2(0.5 * (e1 + e2) * scale, 0.5 * (e1 - e2) * scale);
  }
}

// ------------------------------------------------------------------ self-energy: preparation
// row exponents of the pair rows g = k np + p (over I), one thread per row
__global__ void k_xrow_pair(const double2* __restrict__ M, int nk, int ni, int np, int* __restrict__ ea) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= (int64_t)nk * np) return;
  const int k = (int)(g / np), p = (int)(g - (int64_t)k * np);
  const double2* m = M + (size_t)k * ni * np + p;
  uint32_t h = 0;
#pragma unroll 8
  for (int I = 0; I < ni; ++I) {
    const double2 v = m[(size_t)I * np];
    h = max(h, max(abs_hi(v.x), abs_hi(v.y)));
  }
  ea[g] = exp_of(h);
}

// digits of the pair rows: chunk 2 ic holds re, 2 ic + 1 im of I in [16 ic, 16 ic + 16); one thread per
// (row, 8 I), lanes along rows (coalesced reads and writes)
__global__ void __launch_bounds__(256) k_xslice_pair(const double2* __restrict__ M, const int* __restrict__ ea, int rows,
                                                     int ni, int np, unsigned char* __restrict__ Ai) {
  const int g = blockIdx.x * 32 + threadIdx.x, I0 = 8 * (blockIdx.y * 8 + threadIdx.y);
  if (g >= rows || I0 >= ni) return;
  const int k = g / np, p = g - k * np;
  const double2* m = M + ((size_t)k * ni + I0) * np + p;
  double2 v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = m[(size_t)q * np];
  const int s = ea[g];
  unsigned char* ch = Ai + ((size_t)(g >> 7) * (ni / 8) + 2 * (I0 / 16)) * XA_BYTES;
  long long t[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) t[q] = to_fix(v[q].x, s);
  put8<128>(ch, g & 127, (I0 >> 3) & 1, t);
#pragma unroll
  for (int q = 0; q < 8; ++q) t[q] = to_fix(v[q].y, s);
  put8<128>(ch + XA_BYTES, g & 127, (I0 >> 3) & 1, t);
}

// U_IJ + i V_IJ, I <= J: the Hermitian part of W~ (U halved on the diagonal, V zero there)
__device__ __forceinline__ double2 w_upper(const double2* W, int ni, int I, int J) {
  if (I > J) return make_double2(0.0, 0.0);
  const double2 a = W[(size_t)I * ni + J];
  if (I == J) return make_double2(0.5 * a.x, 0.0);
  const double2 b = W[(size_t)J * ni + I];
  return make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
}

// exponents of the columns J of W~(tau) over I <= J: block (32 J x 8), tau = blockIdx.y
__global__ void __launch_bounds__(256) k_xrow_w(const double2* __restrict__ W, int ni, int* __restrict__ ew) {
  __shared__ uint32_t sh[8][32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, J = blockIdx.x * 32 + tx;
  const double2* Wt = W + (size_t)blockIdx.y * ni * ni;
  uint32_t h = 0;
  for (int I = ty; I < ni; I += 8) {
    if (I > J) break;
    const double2 v = w_upper(Wt, ni, I, J);
    h = max(h, max(abs_hi(v.x), abs_hi(v.y)));
  }
  sh[ty][tx] = h;
  __syncthreads();
  if (ty == 0) {
    for (int q = 1; q < 8; ++q) h = max(h, sh[q][tx]);
    ew[(size_t)blockIdx.y * ni + J] = exp_of(h);
  }
}

// digits of W~: N tile jt holds rows Y1 (J = 32 jt + r) and Y2 (r + 32); chunk 2 i multiplies re, chunk
// 2 i + 1 im of 16 I: Y1 rows U, V; Y2 rows -V, U. Block = (jt, ic <= jt, tau), one thread per (J, 8 I).
__global__ void __launch_bounds__(128) k_xslice_w(const double2* __restrict__ W, const int* __restrict__ ew, int ni,
                                                  unsigned char* __restrict__ Bi) {
  const int jt = blockIdx.x, ic = blockIdx.y, it = blockIdx.z;
  if (ic > jt) return;
  const int r = threadIdx.x & 31, q8 = threadIdx.x >> 5, J = 32 * jt + r, I0 = 32 * ic + 8 * q8;
  const double2* Wt = W + (size_t)it * ni * ni;
  const int s = ew[(size_t)it * ni + J];
  long long u[8], v[8], mv[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const double2 x = w_upper(Wt, ni, I0 + q, J);
    u[q] = to_fix(x.x, s);
    v[q] = to_fix(x.y, s);
    mv[q] = -v[q];
  }
  unsigned char* ch = Bi + (((size_t)it * (ni / 32) + jt) * (ni / 8) + 2 * (I0 / 16)) * XB_BYTES;
  put8<XN>(ch, r, q8 & 1, u);
  put8<XN>(ch, r + 32, q8 & 1, mv);
  put8<XN>(ch + XB_BYTES, r, q8 & 1, v);
  put8<XN>(ch + XB_BYTES, r + 32, q8 & 1, u);
}

// Sigc_n(k|tau) += pref sum_a G_a(k-q|tau) d_(a,n)(tau) of the k points k0 .. k0 + nk - 1
__global__ void k_xsig_sum(const double* __restrict__ D, const double* __restrict__ G, const int* __restrict__ kmq, int k0,
                           int nk, int nb, int ntau, double pref, double* __restrict__ S) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)nk * nb * ntau) return;
  const int it = (int)(e % ntau), n = (int)((e / ntau) % nb), k = (int)(e / ((int64_t)ntau * nb));
  const int km = kmq[k0 + k];
  double s = 0.0;
  for (int a = 0; a < nb; ++a)
    s = fma(G[((size_t)km * nb + a) * ntau + it], D[((size_t)k * nb * nb + a * nb + n) * ntau + it], s);
  S[(int64_t)k0 * nb * ntau + e] += pref * s;
}

// ------------------------------------------------------------------ host side
constexpr size_t kXBudget = 2ull << 30;  // bytes of one operand's digits held at once

}  // namespace

// P(tau) of one q in FP64. Returns GW_EUNSUPPORTED when the workspace cannot be had (see x_workspace).
gw_status launch_pol_exact(gw_ctx* c, int iq, const double* G, double* P) {
  const int nk = c->nk, ni = c->ni, np = c->nb * c->nb, ntau = c->ntau;
  const int64_t n = (int64_t)nk * np;
  const int kc = (int)((n + 7) / 8), nt = (ni + XN - 1) / XN;
  // chunks of 8 pairs per K pass and tau per group: the digits of Y and of X within kXBudget each
  const size_t ych = (size_t)nt * XB_BYTES, x1ch = (size_t)((ni + 127) / 128) * XA_BYTES;
  int nc = (int)std::min<int64_t>(kc, std::max<size_t>(X_BLK, kXBudget / std::max(ych, x1ch)));
  int tg = ntau;
  auto mtiles = [&](int t) { return (t * ni + 127) / 128; };
  while (tg > 1 && (size_t)mtiles(tg) * XA_BYTES * nc > kXBudget) --tg;
  tg = (ntau + (ntau + tg - 1) / tg - 1) / ((ntau + tg - 1) / tg);  // groups of equal size
  const int mt = mtiles(tg);
  // K splits: whole accumulation blocks, as many as give the least waves x (chunks + a unit's fixed cost)
  const int sms = num_sms(c);
  int nsplit = 1;
  double best = 1e300;
  for (int s = 1; s <= std::min(64, (nc + X_BLK - 1) / X_BLK); ++s) {
    const int L = (nc + s - 1) / s, units = mt * nt * s;
    const double t = (double)((units + sms - 1) / sms) * (L + 8.0);
    if (t < best * 0.98) {
      best = t;
      nsplit = s;
    }
  }
  const size_t b_w = align256(sizeof(double) * (size_t)ntau * n), b_max = align256(4 * ((size_t)ntau + ni + (size_t)ntau * ni)),
               b_exp = align256(4 * ((size_t)ni + (size_t)ntau * ni)), b_y = align256(ych * nc),
               b_x = align256((size_t)mt * XA_BYTES * nc), b_c = align256(sizeof(double) * (size_t)nsplit * tg * ni * ni),
               b_e = align256(sizeof(double) * (size_t)ntau * ni * ni);
  if (!x_workspace(c, XW_POL, b_w + b_max + b_exp + b_y + b_x + b_c + b_e)) return GW_EUNSUPPORTED;
  char* q = (char*)c->x_ws[XW_POL];
  double* w = (double*)q;
  uint32_t* wmax = (uint32_t*)(q += b_w);
  uint32_t *ymax = wmax + ntau, *xmax = ymax + ni;
  int* ey = (int*)(q += b_max);
  int* ex = ey + ni;
  unsigned char* Yi = (unsigned char*)(q += b_exp);
  unsigned char* Xi = (unsigned char*)(q += b_y);
  double* C = (double*)(q += b_x);
  double* E = (double*)(q += b_c);
  const double2* M = (const double2*)m_block(c, iq);
  if (!M) return GW_ECUDA;
  gw_status st;
  cudaMemsetAsync(wmax, 0, b_max, c->stream);
  k_xw<<<dim3((unsigned)std::min<int64_t>((n + 255) / 256, 1024), ntau), 256, 0, c->stream>>>(
      G, c->d_kmq + (size_t)iq * nk, nk, c->nb, ntau, w, wmax);
  if ((st = check_launch(c, "exact pol weights")) != GW_OK) return st;
  const unsigned rw = (unsigned)(((int64_t)nk * ni * 32 + 255) / 256);
  k_xrow<<<rw, 256, 0, c->stream>>>(M, nk, ni, np, ymax);
  if ((st = check_launch(c, "exact pol rows")) != GW_OK) return st;
  k_xrowx<<<dim3((rw + 3) / 4, (ntau + 15) / 16), 256, 0, c->stream>>>(M, w, wmax, ymax, nk, ni, np, ntau, xmax);
  if ((st = check_launch(c, "exact pol rows")) != GW_OK) return st;
  k_xexp<<<(ni * ntau + 255) / 256, 256, 0, c->stream>>>(wmax, ymax, xmax, ni, ntau, ey, ex);
  if ((st = check_launch(c, "exact pol exponents")) != GW_OK) return st;
  for (int c0 = 0; c0 < kc; c0 += nc) {
    const int cn = std::min(nc, kc - c0);
    for (int t0 = 0; t0 < ntau; t0 += tg) {
      const int tn = std::min(tg, ntau - t0);
      const int64_t ns = ((int64_t)cn * ni + 255) / 256;  // blocks; several tau per thread once they fill the GPU
      const int tpt = (int)std::max<int64_t>(1, std::min<int64_t>(tn, ns * tn / (8 * sms)));
      k_xslice_pol<<<dim3((unsigned)ns, (tn + tpt - 1) / tpt), 256, 0, c->stream>>>(M, w, ey, ex, nk, ni, np, c0, cn, t0, tn,
                                                                                  tpt, t0 == 0, Yi, Xi);
      if ((st = check_launch(c, "exact pol digits")) != GW_OK) return st;
      const int sp = std::min(nsplit, (cn + X_BLK - 1) / X_BLK);
      OpStore::Job J{};
      J.A = Xi;
      J.B = Yi;
      J.ea = ex + (size_t)t0 * ni;
      J.eb = ey;
      J.mt = mtiles(tn);
      J.nt = nt;
      J.chunks = cn;
      J.nsplit = sp;
      J.rows = tn * ni;
      J.ncols = ni;
      J.sh = drop_bits((int64_t)XK * ((cn + sp - 1) / sp));
      J.C = C;
      if ((st = run_gemm<OpStore>(c, J, J.mt * nt * sp, "exact pol gemm")) != GW_OK) return st;
      const int64_t ne = (int64_t)tn * ni * ni;
      k_xsum<<<(unsigned)((ne + 255) / 256), 256, 0, c->stream>>>(C, ne, sp, c0 > 0, E + (size_t)t0 * ni * ni);
      if ((st = check_launch(c, "exact pol sum")) != GW_OK) return st;
    }
  }
  k_xform<<<dim3(ni / 32, ni / 32, ntau), 256, 0, c->stream>>>(E, ni, 1.0 / (c->omega * nk), (double2*)P);
  return check_launch(c, "exact pol form");
}

// Sigma^c of one q in FP64, accumulated. GW_EUNSUPPORTED as above.
gw_status launch_sigma_exact(gw_ctx* c, int iq, const double* G, const double* W, double* Sg) {
  const int nk = c->nk, ni = c->ni, np = c->nb * c->nb, ntau = c->ntau, ch = ni / 8, nt = ni / 32;
  auto mtiles = [&](int k) { return (int)(((int64_t)k * np + 127) / 128); };
  int kg = nk;  // k points per pass, tau per group: digits within kXBudget
  while (kg > 1 && (size_t)mtiles(kg) * ch * XA_BYTES > kXBudget) --kg;
  const size_t b1 = (size_t)nt * ch * XB_BYTES;
  const int tg = (int)std::min<size_t>(ntau, std::max<size_t>(1, kXBudget / b1));
  const size_t b_ea = align256(sizeof(int) * (size_t)nk * np), b_ew = align256(sizeof(int) * (size_t)ntau * ni),
               b_a = align256((size_t)mtiles(kg) * ch * XA_BYTES), b_b = align256(b1 * tg),
               b_d = align256(sizeof(double) * (size_t)kg * np * ntau);
  if (!x_workspace(c, XW_SIGMA, b_ea + b_ew + b_a + b_b + b_d)) return GW_EUNSUPPORTED;
  char* q = (char*)c->x_ws[XW_SIGMA];
  int* ea = (int*)q;
  int* ew = (int*)(q += b_ea);
  unsigned char* Ai = (unsigned char*)(q += b_ew);
  unsigned char* Bi = (unsigned char*)(q += b_a);
  double* D = (double*)(q += b_b);
  const double2* M = (const double2*)m_block(c, iq);
  if (!M) return GW_ECUDA;
  gw_status st;
  k_xrow_pair<<<(unsigned)(((int64_t)nk * np + 127) / 128), 128, 0, c->stream>>>(M, nk, ni, np, ea);
  if ((st = check_launch(c, "exact sigma rows")) != GW_OK) return st;
  k_xrow_w<<<dim3(ni / 32, ntau), 256, 0, c->stream>>>((const double2*)W, ni, ew);
  if ((st = check_launch(c, "exact sigma rows")) != GW_OK) return st;
  for (int k0 = 0; k0 < nk; k0 += kg) {
    const int kn = std::min(kg, nk - k0), rows = kn * np;
    const double2* Mk = M + (size_t)k0 * ni * np;
    k_xslice_pair<<<dim3((rows + 31) / 32, (ni + 63) / 64), dim3(32, 8), 0, c->stream>>>(Mk, ea + (size_t)k0 * np, rows, ni,
                                                                                        np, Ai);
    if ((st = check_launch(c, "exact sigma digits")) != GW_OK) return st;
    for (int t0 = 0; t0 < ntau; t0 += tg) {
      const int tn = std::min(tg, ntau - t0);
      if (k0 == 0 || tg < ntau) {
        k_xslice_w<<<dim3(nt, nt, tn), 128, 0, c->stream>>>((const double2*)W + (size_t)t0 * ni * ni, ew + (size_t)t0 * ni,
                                                            ni, Bi);
        if ((st = check_launch(c, "exact sigma digits")) != GW_OK) return st;
      }
      OpDot::Job J{};
      J.A = Ai;
      J.B = Bi;
      J.ea = ea + (size_t)k0 * np;
      J.eb = ew;
      J.mt = mtiles(kn);
      J.nt = nt;
      J.chunks = ch;
      J.rows = rows;
      J.M = Mk;
      J.np = np;
      J.ni = ni;
      J.ntau = tn;
      J.tau0 = t0;
      J.ntau_all = ntau;
      J.sh = drop_bits(2 * ni);
      J.tgrp = 8;
      J.D = D;
      if ((st = run_gemm<OpDot>(c, J, J.mt * tn, "exact sigma gemm")) != GW_OK) return st;
    }
    const int64_t ne = (int64_t)kn * c->nb * ntau;
    k_xsig_sum<<<(unsigned)((ne + 127) / 128), 128, 0, c->stream>>>(D, G, c->d_kmq + (size_t)iq * nk, k0, kn, c->nb, ntau,
                                                                   -1.0 / (c->omega * nk), Sg);
    if ((st = check_launch(c, "exact sigma sum")) != GW_OK) return st;
  }
  return GW_OK;
}

}  // namespace gwi
