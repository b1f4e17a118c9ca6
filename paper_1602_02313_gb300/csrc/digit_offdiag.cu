// Off-diagonal self-energy (gw_selfenergy_offdiag) as exact digit products on the tensor cores
// (digit_gemm.cuh). With a_jm the pair rows of M[k] (band j at k - q, band m at k):
//   GEMM 1   Z_jm(tau) = G_j(tau) W~(tau) a_jm            rows (k, j, m), columns I (Re, Im), K = J
//   GEMM 2   Sigma_nm(k|tau) = pref sum_jI conj(a_jn^I) Z_jm^I(tau)   rows (tau, m) of a k, columns n, K = (j, I)
// and Sigma^x as one more "tau" of GEMM 2 with Z_jm^I = occ_j v_I a_jm^I. Z is FP64 in between. k points and
// tau go in groups whose operands and Z fit 2 GiB.
// Bound: the products' shared-memory operand rate (34 MMAs of 48 clocks per 16 K, digit_gemm.cuh) and, for Z, writing it,
// its digits and reading both (44 bytes per element twice). Measured at Nk 8, Nb 32, NI 128, 16 tau: Sigma^c and Sigma^x
// 29.5 -> 1.0 ms against the CUDA-core kernels of offdiag.cu (GEMM 1 0.61, GEMM 2 0.20, digits of Z 0.11). GEMM 2 has
// short sums where G_j(tau) leaves a few j, so both GEMMs keep eight levels: with seven the error against exact sums
// was up to 1.7 times the CUDA-core kernels', with eight it is 0.2 to 0.6 of theirs (Nb 4 .. 33, NI 32 .. 128).
#include <algorithm>

#include "digit_gemm.cuh"

namespace gwi {

namespace {

constexpr size_t kOdBudget = 2ull << 30;

// ------------------------------------------------------------------ digits of W~ and M
// exponents of the rows I of W~(tau) over J: one warp per (tau, I)
__global__ void k_od_wmax(const double2* __restrict__ W, int ni, int n, int* __restrict__ ew) {
  const int wid = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (wid >= n) return;
  const double2* w = W + (size_t)wid * ni;
  uint32_t h = 0;
  for (int J = lane; J < ni; J += 32) h = max(h, max(abs_hi(w[J].x), abs_hi(w[J].y)));
  h = warp_max(h);
  if (lane == 0) ew[wid] = exp_of(h);
}

// W~ as a B operand: rows 2 I = [Re W | -Im W], 2 I + 1 = [Im W | Re W], chunk 2 jc (2 jc + 1) meets Re (Im) a of 16 J
__global__ void __launch_bounds__(128) k_od_wdig(const double2* __restrict__ W, const int* __restrict__ ew, int ni,
                                                 unsigned char* __restrict__ Bi) {
  const int I = blockIdx.x * 32 + (threadIdx.x & 31), J0 = 8 * (blockIdx.y * 4 + (threadIdx.x >> 5)), it = blockIdx.z;
  const double2* w = W + ((size_t)it * ni + I) * ni + J0;
  const int s = ew[(size_t)it * ni + I], k8 = (J0 >> 3) & 1;
  long long re[8], im[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    re[q] = to_fix(w[q].x, s);
    im[q] = to_fix(w[q].y, s);
  }
  unsigned char* ch = Bi + (((size_t)it * (ni / 32) + I / 32) * (ni / 8) + 2 * (J0 / 16)) * XB_BYTES;
  put8<XN>(ch, 2 * I % XN, k8, re);
  put8<XN>(ch, 2 * I % XN + 1, k8, im);
  put8<XN>(ch + XB_BYTES, 2 * I % XN + 1, k8, re);
#pragma unroll
  for (int q = 0; q < 8; ++q) im[q] = -im[q];
  put8<XN>(ch + XB_BYTES, 2 * I % XN, k8, im);
}

// exponents of the pair rows over I, and the largest high word of |a_jn| over (j, I) of each (k, n): a
// thread per (k, p), 16 I
__global__ void k_od_amax(const double2* __restrict__ M, int ni, int np, int nb, uint32_t* __restrict__ pmax,
                          uint32_t* __restrict__ nmax) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.z;
  if (p >= np) return;
  const double2* m = M + ((size_t)k * ni + 16 * blockIdx.y) * np + p;
  uint32_t h = 0;
#pragma unroll
  for (int I = 0; I < 16; ++I) h = max(h, max(abs_hi(m[(size_t)I * np].x), abs_hi(m[(size_t)I * np].y)));
  atomicMax(pmax + (size_t)k * np + p, h);
  atomicMax(nmax + k * nb + p % nb, h);
}

// pair rows as the A operand of GEMM 1 (chunk 2 ic re, 2 ic + 1 im of 16 I); rows flat over the group's k
__global__ void __launch_bounds__(256) k_od_adig(const double2* __restrict__ M, const uint32_t* __restrict__ pmax, int rows,
                                                 int ni, int np, unsigned char* __restrict__ Ai) {
  const int g = blockIdx.x * 32 + threadIdx.x, I0 = 8 * (blockIdx.y * 8 + threadIdx.y);
  if (g >= rows || I0 >= ni) return;
  const int k = g / np, p = g - k * np, s = exp_of(pmax[g]);
  const double2* m = M + ((size_t)k * ni + I0) * np + p;
  double2 v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = m[(size_t)q * np];
  unsigned char* ch = Ai + ((size_t)(g >> 7) * (ni / 8) + 2 * (I0 / 16)) * XA_BYTES;
  long long t[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) t[q] = to_fix(v[q].x, s);
  put8<128>(ch, g & 127, (I0 >> 3) & 1, t);
#pragma unroll
  for (int q = 0; q < 8; ++q) t[q] = to_fix(v[q].y, s);
  put8<128>(ch + XA_BYTES, g & 127, (I0 >> 3) & 1, t);
}

// conj(a) as the B operand of GEMM 2: chunk (j, 8 I) = [8 Re Z | 8 Im Z]; rows 2 n = [Re a | Im a],
// 2 n + 1 = [-Im a | Re a]. A thread per (k, p = (j, n), 8 I).
__global__ void __launch_bounds__(256) k_od_bdig(const double2* __restrict__ M, const uint32_t* __restrict__ nmax, int ni,
                                                 int np, int nb, int nt2, unsigned char* __restrict__ Bi) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x, ic = blockIdx.y, k = blockIdx.z;
  if (p >= np) return;
  const int j = p / nb, n = p - j * nb, s = exp_of(nmax[k * nb + n]);
  const double2* m = M + ((size_t)k * ni + 8 * ic) * np + p;
  long long re[8], im[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const double2 v = m[(size_t)q * np];
    re[q] = to_fix(v.x, s);
    im[q] = to_fix(v.y, s);
  }
  unsigned char* ch = Bi + (((size_t)k * nt2 + 2 * n / XN) * (nb * (ni / 8)) + j * (ni / 8) + ic) * XB_BYTES;
  put8<XN>(ch, 2 * n % XN, 0, re);
  put8<XN>(ch, 2 * n % XN, 1, im);
  put8<XN>(ch, 2 * n % XN + 1, 1, re);
#pragma unroll
  for (int q = 0; q < 8; ++q) im[q] = -im[q];
  put8<XN>(ch, 2 * n % XN + 1, 0, im);
}

// Z of Sigma^x: the group's last "tau". Z[k][t][j][I][m]
__global__ void __launch_bounds__(256) k_od_x(const double2* __restrict__ M, const double* __restrict__ v,
                                              const double* __restrict__ occ, const int* __restrict__ kmq, int ni, int np,
                                              int nb, int nz, double2* __restrict__ Z, uint32_t* __restrict__ zmax) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x, ic = blockIdx.y, k = blockIdx.z;
  if (p >= np) return;
  const int j = p / nb, m = p - j * nb;
  const double f = occ[(size_t)kmq[k] * nb + j];
  uint32_t h = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int I = 8 * ic + q;
    const double2 a = M[((size_t)k * ni + I) * np + p];
    const double s = f * v[I];
    const double2 z = make_double2(s * a.x, s * a.y);
    Z[((((size_t)k * nz + nz - 1) * nb + j) * ni + I) * nb + m] = z;
    h = max(h, max(abs_hi(z.x), abs_hi(z.y)));
  }
  atomicMax(zmax + ((size_t)k * nz + nz - 1) * nb + m, h);
}

// Z as the A operand of GEMM 2: rows r = (t, m) of a k, chunk (j, 8 I) = [8 re | 8 im]
__global__ void __launch_bounds__(256) k_od_zdig(const double2* __restrict__ Z, const uint32_t* __restrict__ zmax, int ni,
                                                 int nb, int nz, int mt2, unsigned char* __restrict__ Ai) {
  const int r = blockIdx.x * 32 + threadIdx.x, k = blockIdx.z, c = blockIdx.y * 8 + threadIdx.y;  // c = (j, 8 I)
  if (r >= nz * nb || c >= nb * (ni / 8)) return;
  const int t = r / nb, m = r - t * nb, j = c / (ni / 8), I0 = 8 * (c - j * (ni / 8));
  const int s = exp_of(zmax[((size_t)k * nz + t) * nb + m]);
  const double2* z = Z + ((((size_t)k * nz + t) * nb + j) * ni + I0) * nb + m;
  double2 v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = z[(size_t)q * nb];
  unsigned char* ch = Ai + (((size_t)k * mt2 + (r >> 7)) * (nb * (ni / 8)) + c) * XA_BYTES;
  long long d[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) d[q] = to_fix(v[q].x, s);
  put8<128>(ch, r & 127, 0, d);
#pragma unroll
  for (int q = 0; q < 8; ++q) d[q] = to_fix(v[q].y, s);
  put8<128>(ch, r & 127, 1, d);
}

// ------------------------------------------------------------------ the products
// GEMM 1: unit = (M tile of pair rows, tau), all tiles n of 32 columns I
struct OpOdZ {
  static constexpr int LV = 8;
  struct Job {
    const unsigned char *A, *B;
    const uint32_t* pmax;  // [rows]
    const int* ew;         // [tau][I] from tau0
    const double* G;       // [nk][nb][ntau]
    const int* kmq;        // of the group's first k
    double2* Z;            // [k][nz][nb][ni][nb]
    uint32_t* zmax;        // [k][nz][nb]
    int mt, nt, chunks, rows, np, nb, ni, nz, ntg, tau0, ntau;
  };
  struct Unit {
    int m, t, n0, n1;
    __device__ Unit(const Job& J, int u) : n0(0), n1(J.nt) {  // tau in groups of 8 (see OpDot)
      const int per = J.mt * 8, g = u / per, r = u % per, gt = min(8, J.ntg - g * 8);
      m = r / gt;
      t = g * 8 + r % gt;
    }
    __device__ const unsigned char* A(const Job& J, int) const { return J.A + (size_t)m * J.chunks * XA_BYTES; }
    __device__ const unsigned char* B(const Job& J, int n) const {
      return J.B + ((size_t)t * J.nt + n) * J.chunks * XB_BYTES;
    }
    __device__ void range(const Job& J, int, int& c0, int& c1) const {
      c0 = 0;
      c1 = J.chunks;
    }
  };
  int row, part;
  uint32_t h = 0;
  __device__ OpOdZ(const Job&, const Unit& U, int r, int p) : row(128 * U.m + r), part(p) {}
  __device__ void tile(const Job& J, const Unit& U, int n, const long long (&hi)[16], const long long (&lo)[16]) {
    if (row >= J.rows) return;
    const int k = row / J.np, p = row - k * J.np, j = p / J.nb, m = p - j * J.nb, I0 = 32 * n + 8 * part;
    const int ea = exp_of(J.pmax[row]);
    const int* ew = J.ew + (size_t)U.t * J.ni + I0;
    const double g = J.G[((size_t)J.kmq[k] * J.nb + j) * J.ntau + J.tau0 + U.t];
    double2* z = J.Z + ((((size_t)k * J.nz + U.t) * J.nb + j) * J.ni + I0) * J.nb + m;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = ea + ew[q] - 62;
      const double2 v = make_double2(g * fix_to_double(hi[2 * q], lo[2 * q], e), g * fix_to_double(hi[2 * q + 1], lo[2 * q + 1], e));
      z[(size_t)q * J.nb] = v;
      h = max(h, max(abs_hi(v.x), abs_hi(v.y)));
    }
  }
  __device__ void finish(const Job& J, const Unit& U, double (&)[3][128], bool ok) {
    if (!ok || row >= J.rows) return;
    const int k = row / J.np, m = (row - k * J.np) % J.nb;
    atomicMax(J.zmax + ((size_t)k * J.nz + U.t) * J.nb + m, h);
  }
};

// GEMM 2: unit = (K split, k, M tile of rows (t, m), N tile of 32 columns n)
struct OpOdS {
  static constexpr int LV = 8;
  struct Job {
    const unsigned char *A, *B;
    const uint32_t *zmax, *nmax;
    double2* C;  // [split][k][n][m][t]
    int nkg, mt, nt, chunks, nsplit, rows, nb, nz;
  };
  struct Unit {
    int s, k, m, n0, n1;
    __device__ Unit(const Job& J, int u)
        : s(u / (J.nkg * J.mt * J.nt)), k(u / (J.mt * J.nt) % J.nkg), m(u / J.nt % J.mt), n0(u % J.nt), n1(n0 + 1) {}
    __device__ const unsigned char* A(const Job& J, int) const {
      return J.A + ((size_t)k * J.mt + m) * J.chunks * XA_BYTES;
    }
    __device__ const unsigned char* B(const Job& J, int n) const {
      return J.B + ((size_t)k * J.nt + n) * J.chunks * XB_BYTES;
    }
    __device__ void range(const Job& J, int, int& c0, int& c1) const {
      const int L = (J.chunks + J.nsplit - 1) / J.nsplit;
      c0 = s * L;
      c1 = min(J.chunks, c0 + L);
    }
  };
  int row, part;
  __device__ OpOdS(const Job&, const Unit& U, int r, int p) : row(128 * U.m + r), part(p) {}
  __device__ void tile(const Job& J, const Unit& U, int n, const long long (&hi)[16], const long long (&lo)[16]) {
    if (row >= J.rows) return;
    const int t = row / J.nb, m = row - t * J.nb, c0 = 32 * n + 8 * part;
    const int ea = exp_of(J.zmax[((size_t)U.k * J.nz + t) * J.nb + m]);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (c0 + q >= J.nb) break;
      const int e = ea + exp_of(J.nmax[U.k * J.nb + c0 + q]) - 62;
      J.C[((((size_t)U.s * J.nkg + U.k) * J.nb + c0 + q) * J.nb + m) * J.nz + t] =
          make_double2(fix_to_double(hi[2 * q], lo[2 * q], e), fix_to_double(hi[2 * q + 1], lo[2 * q + 1], e));
    }
  }
  __device__ void finish(const Job&, const Unit&, double (&)[3][128], bool) {}
};

// S[k][n][m][tau0 + t] += pref sum over splits, and Sx from the last t when it is Sigma^x's
__global__ void k_od_out(const double2* __restrict__ C, int64_t n, int nsplit, int nz, int ntg, int tau0, int ntau,
                         double pref, double2* __restrict__ S, double2* __restrict__ Sx) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;  // (k, n, m, t)
  if (e >= n) return;
  double2 s = C[e];
  for (int q = 1; q < nsplit; ++q) {
    const double2 c = C[q * n + e];
    s = make_double2(s.x + c.x, s.y + c.y);
  }
  const int t = (int)(e % nz);
  const int64_t knm = e / nz;
  double2* o = t < ntg ? S + knm * ntau + tau0 + t : Sx + knm;
  *o = make_double2(fma(pref, s.x, o->x), fma(pref, s.y, o->y));
}

}  // namespace

// GW_EUNSUPPORTED when the workspace cannot be had (nothing launched)
gw_status launch_offdiag_digits(gw_ctx* c, int iq, const double* G, const double* occ, const double* W, double* S,
                                double* Sx) {
  const int ni = c->ni, nb = c->nb, nk = c->nk, np = nb * nb, ntau = c->ntau, x = Sx ? 1 : 0;
  const int ch1 = ni / 8, nt1 = ni / 32, ch2 = nb * (ni / 8), nt2 = (2 * nb + XN - 1) / XN;
  auto mt1 = [&](int k) { return (int)(((int64_t)k * np + 127) / 128); };
  auto mt2 = [&](int t) { return ((t + x) * nb + 127) / 128; };
  auto bytes_w = [&](int t) { return (size_t)t * nt1 * ch1 * XB_BYTES; };
  auto bytes_k = [&](int t) {  // one k, t tau: M as both operands, Z and its digits
    return (size_t)mt1(1) * ch1 * XA_BYTES + (size_t)nt2 * ch2 * XB_BYTES + sizeof(double2) * (size_t)(t + x) * np * ni +
           (size_t)mt2(t) * ch2 * XA_BYTES;
  };
  int tg = ntau;
  while (tg > 1 && bytes_k(tg) + bytes_w(tg) > kOdBudget) tg = (tg + 1) / 2;
  const size_t left = kOdBudget > bytes_w(tg) ? kOdBudget - bytes_w(tg) : 0;
  const int kg = (int)std::max<size_t>(1, std::min<size_t>(nk, left / bytes_k(tg)));
  const int tiles2 = kg * mt2(tg) * nt2;
  const int nsplit = std::max(1, std::min({2 * num_sms(c) / tiles2, ch2 / (2 * X_BLK), 16}));
  const size_t b_ew = align256(sizeof(int) * (size_t)ntau * ni), b_w = align256(bytes_w(tg)),
               b_max = align256(4 * ((size_t)kg * np + (size_t)kg * nb + (size_t)kg * (tg + x) * nb)),
               b_a = align256((size_t)mt1(kg) * ch1 * XA_BYTES), b_b = align256((size_t)kg * nt2 * ch2 * XB_BYTES),
               b_z = align256(sizeof(double2) * (size_t)kg * (tg + x) * np * ni),
               b_zd = align256((size_t)kg * mt2(tg) * ch2 * XA_BYTES),
               b_c = align256(sizeof(double2) * (size_t)nsplit * kg * np * (tg + x));
  if (!x_workspace(c, XW_OFFDIAG, b_ew + b_w + b_max + b_a + b_b + b_z + b_zd + b_c)) return GW_EUNSUPPORTED;
  char* q = (char*)c->x_ws[XW_OFFDIAG];
  int* ew = (int*)q;
  unsigned char* Wd = (unsigned char*)(q += b_ew);
  uint32_t* pmax = (uint32_t*)(q += b_w);
  uint32_t *nmax = pmax + (size_t)kg * np, *zmax = nmax + (size_t)kg * nb;
  unsigned char* Ad = (unsigned char*)(q += b_max);
  unsigned char* Bd = (unsigned char*)(q += b_a);
  double2* Z = (double2*)(q += b_b);
  unsigned char* Zd = (unsigned char*)(q += b_z);
  double2* C = (double2*)(q += b_zd);
  const double2* M = (const double2*)m_block(c, iq);
  if (!M) return GW_ECUDA;
  const int* kmq = c->d_kmq + (size_t)iq * nk;
  gw_status st;
  k_od_wmax<<<(unsigned)(((int64_t)ntau * ni * 32 + 255) / 256), 256, 0, c->stream>>>((const double2*)W, ni, ntau * ni, ew);
  if ((st = check_launch(c, "offdiag W rows")) != GW_OK) return st;
  for (int t0 = 0; t0 < ntau; t0 += tg) {
    const int tn = std::min(tg, ntau - t0), xs = x && t0 == 0, nz = tn + xs;  // Sigma^x goes with the first tau
    k_od_wdig<<<dim3(ni / 32, ni / 32, tn), 128, 0, c->stream>>>((const double2*)W + (size_t)t0 * ni * ni,
                                                                 ew + (size_t)t0 * ni, ni, Wd);
    if ((st = check_launch(c, "offdiag W digits")) != GW_OK) return st;
    for (int k0 = 0; k0 < nk; k0 += kg) {
      const int kn = std::min(kg, nk - k0), rows = kn * np, m2 = (nz * nb + 127) / 128;
      const double2* Mk = M + (size_t)k0 * ni * np;
      const unsigned pb = (np + 255) / 256;
      cudaMemsetAsync(pmax, 0, b_max, c->stream);
      k_od_amax<<<dim3(pb, ni / 16, kn), 256, 0, c->stream>>>(Mk, ni, np, nb, pmax, nmax);
      if ((st = check_launch(c, "offdiag rows")) != GW_OK) return st;
      k_od_adig<<<dim3((rows + 31) / 32, (ni + 63) / 64), dim3(32, 8), 0, c->stream>>>(Mk, pmax, rows, ni, np, Ad);
      if ((st = check_launch(c, "offdiag digits")) != GW_OK) return st;
      k_od_bdig<<<dim3(pb, ni / 8, kn), 256, 0, c->stream>>>(Mk, nmax, ni, np, nb, nt2, Bd);
      if ((st = check_launch(c, "offdiag digits")) != GW_OK) return st;
      OpOdZ::Job J{};
      J.A = Ad;
      J.B = Wd;
      J.pmax = pmax;
      J.ew = ew + (size_t)t0 * ni;
      J.G = G;
      J.kmq = kmq + k0;
      J.Z = Z;
      J.zmax = zmax;
      J.mt = mt1(kn);
      J.nt = nt1;
      J.chunks = ch1;
      J.rows = rows;
      J.np = np;
      J.nb = nb;
      J.ni = ni;
      J.nz = nz;
      J.ntg = tn;
      J.tau0 = t0;
      J.ntau = ntau;
      if ((st = run_gemm<OpOdZ>(c, J, J.mt * tn, "offdiag gemm")) != GW_OK) return st;
      if (xs) {
        k_od_x<<<dim3(pb, ni / 8, kn), 256, 0, c->stream>>>(Mk, c->d_v + (size_t)iq * ni, occ, kmq + k0, ni, np, nb, nz, Z,
                                                            zmax);
        if ((st = check_launch(c, "offdiag exchange")) != GW_OK) return st;
      }
      k_od_zdig<<<dim3((nz * nb + 31) / 32, (ch2 + 7) / 8, kn), dim3(32, 8), 0, c->stream>>>(Z, zmax, ni, nb, nz, m2, Zd);
      if ((st = check_launch(c, "offdiag Z digits")) != GW_OK) return st;
      OpOdS::Job K{};
      K.A = Zd;
      K.B = Bd;
      K.zmax = zmax;
      K.nmax = nmax;
      K.C = C;
      K.nkg = kn;
      K.mt = m2;
      K.nt = nt2;
      K.chunks = ch2;
      K.nsplit = nsplit;
      K.rows = nz * nb;
      K.nb = nb;
      K.nz = nz;
      if ((st = run_gemm<OpOdS>(c, K, nsplit * kn * m2 * nt2, "offdiag gemm")) != GW_OK) return st;
      const int64_t n = (int64_t)kn * np * nz;
      k_od_out<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(C, n, nsplit, nz, tn, t0, ntau, -1.0 / (c->omega * nk),
                                                                  (double2*)S + (size_t)k0 * np * ntau,
                                                                  (double2*)Sx + (Sx ? (size_t)k0 * np : 0));
      if ((st = check_launch(c, "offdiag sum")) != GW_OK) return st;
    }
  }
  return GW_OK;
}

}  // namespace gwi
