// The dielectric inverse of the mixed chain (gw_screen, GW_F32X2) as exact digit products on the tensor
// cores (digit_gemm.cuh): X = (1 - Pi)^-1 - 1 by blocked in-place Gauss-Jordan, W~ = v^1/2 X v^1/2.
//
// For each block R of 64 rows (the last one 32 when NI is an odd multiple of 32), over a group of
// systems at once:
//   k_gj_pivot   P = A_RR^-1 in shared memory, float-float (no pivoting: 1 - Pi has Hermitian part >= 1)
//   k_gj_digits  digits of the old rows R (as rows c of A_Rc^T) and of the old columns R (rows i of A_iR)
//   GEMM 1       A_Rc <- P A_Rc (A_RR <- P)
//   k_gj_cols    digits of the new rows R
//   GEMM 2       A_ic <- A_ic - A_iR A_Rc for the rows i outside R (from zero in the columns R)
// A is FP64 throughout; only P carries float-float rounding (2^-44). Systems go in groups of kGroup bytes:
// smaller ones would stay in L2 over the steps, but the pivots need more than 152 systems at once (384
// systems of NI 256: 10.3 ms in groups of 160 MB, 5.2 in groups of 768 MB, 5.0 in one). Blocks of 64 rather
// than 32 rows halve the passes over A and the readouts per MMA.
// Measured: 384 systems of NI 256 17.0 -> 4.6 ms (float-float elimination on the FP32 pipes before), 16
// systems of NI 64 0.46 -> 0.16, of NI 32 0.16 -> 0.06; errors 8.2e-15 against 9.8e-15 at NI 256. Of the 4.6:
// pivots 1.3 (ALU), updates 1.6 (their MMAs 0.9), digits 0.8 and build / output 0.35 (HBM), rows 0.5.
#include <algorithm>

#include "arith.cuh"
#include "digit_gemm.cuh"
#include "gj_block.cuh"

namespace gwi {

namespace {

using arith::Ff32;

constexpr int GJ = 64;              // rows per step
constexpr int GJ_LD = GJ + 1;       // leading dimension of the pivot block in shared memory
constexpr size_t kGroup = 1536ull << 20;  // bytes of the matrices and digits of one group

struct GjJob {
  double2* A;                       // [system][ni][ni]
  double2* P;                       // [system][64][64]: A_RR^-1
  unsigned char *rowd, *cold, *pd, *newd;  // digits: rows c of A_Rc^T, rows i of A_iR, P, columns c of the new rows
  int *erow, *ecol, *ep, *enew;     // their row exponents
  int ni, mt, nt, k0, bw, chunks;   // M tiles of ni rows, N tiles of 2 ni columns, K chunks of 2 bw
  int sh;
  __host__ __device__ size_t row_image() const { return (size_t)mt * (2 * GJ / XK) * XA_BYTES; }
  __host__ __device__ size_t col_image() const { return (size_t)nt * (2 * GJ / XK) * XB_BYTES; }
  __host__ __device__ size_t p_image() const { return (size_t)2 * (2 * GJ / XK) * XB_BYTES; }
};

// A = 1 - v^1/2 P v^1/2, info = 0
__global__ void k_gj_build(const double2* __restrict__ P, const double* __restrict__ sqrtv, int sys0, int nnu, int ni,
                           double2* __restrict__ A, int* __restrict__ info) {
  const int s = blockIdx.y, iqb = (sys0 + s) / nnu;
  const double* sv = sqrtv + (size_t)iqb * ni;
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nn = (int64_t)ni * ni;
  if (e == 0) info[sys0 + s] = 0;
  if (e >= nn) return;
  const int I = (int)(e / ni), J = (int)(e % ni);
  const double q = sv[I] * sv[J];
  const double2 p = P[(sys0 + s) * nn + e];
  A[s * nn + e] = make_double2((I == J ? 1.0 : 0.0) - q * p.x, -q * p.y);
}

// W~ = v^1/2 (A - 1) v^1/2
__global__ void k_gj_out(const double2* __restrict__ A, const double* __restrict__ sqrtv, int sys0, int nnu, int ni,
                         double2* __restrict__ W) {
  const int s = blockIdx.y, iqb = (sys0 + s) / nnu;
  const double* sv = sqrtv + (size_t)iqb * ni;
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nn = (int64_t)ni * ni;
  if (e >= nn) return;
  const int I = (int)(e / ni), J = (int)(e % ni);
  const double q = sv[I] * sv[J];
  const double2 x = A[s * nn + e];
  W[(sys0 + s) * nn + e] = make_double2(q * (x.x - (I == J ? 1.0 : 0.0)), q * x.y);
}

struct BlockSync {
  __device__ __forceinline__ void block() const { __syncthreads(); }
  __device__ __forceinline__ void warp() const { __syncwarp(); }
};

// One system per block: P = A_RR^-1 in float-float, written in FP64 (to P and, when R is the whole matrix,
// to A) and as digits: row 2 r = [Re P_r | -Im P_r], 2 r + 1 = [Im P_r | Re P_r]. In-place Gauss-Jordan by
// two 32-wide blocks H: H's 32 x 32 inverse by elimination with 2 x 2 elements per thread in registers
// (gj_block.cuh; a step moves only its row and column through shared memory), then three 32^3 products for the other half.
// Summing 32 products before one subtraction keeps the error below that of 64 elimination steps (1.2e-14
// against 0.8e-14 for random matrices), and the steps are short: ALU-bound (64^3 complex multiply-adds of
// 48 operations) with two or three blocks per SM.
__global__ void __launch_bounds__(256, 3) k_gj_pivot(GjJob J, int sys0, int* __restrict__ info) {
  using S = Ff32::S;
  extern __shared__ __align__(16) unsigned char gsm[];
  S* B = reinterpret_cast<S*>(gsm);  // [64][65]
  __shared__ S fcol[32], prow[32], rowj[32];
  const int s = blockIdx.x, t = threadIdx.x, bw = J.bw, tx = t & 15, ty = t >> 4;
  if (info[sys0 + s]) return;  // an earlier block had a zero pivot
  double2* A = J.A + (size_t)s * J.ni * J.ni + (size_t)J.k0 * J.ni + J.k0;
  for (int e = t; e < bw * bw; e += 256) {
    const double2 a = A[(size_t)(e / bw) * J.ni + e % bw];
    B[(e / bw) * GJ_LD + e % bw] = Ff32::from(a.x, a.y);
  }
  __syncthreads();
  for (int h0 = 0; h0 < bw; h0 += 32) {
    S* H = B + h0 * GJ_LD + h0;
    S x[2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) x[a][b] = H[(ty + 16 * a) * GJ_LD + tx + 16 * b];
    const int zero = gj_invert32<Ff32>(x, fcol, prow, rowj, t, BlockSync());
    if (zero >= 0) {
      if (t == 0) info[sys0 + s] = J.k0 + h0 + zero + 1;
      return;
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) H[(ty + 16 * a) * GJ_LD + tx + 16 * b] = x[a][b];
    __syncthreads();
    if (bw == 32) break;
    // the other half O: rows H <- H^-1 B_HO, columns H <- -B_OH H^-1, B_OO -= B_OH (new B_HO)
    const int o0 = 32 - h0;
    S *HO = B + h0 * GJ_LD + o0, *OH = B + o0 * GJ_LD + h0, *OO = B + o0 * GJ_LD + o0;
    auto product = [&](const S* L, const S* R, S (&y)[2][2]) {
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) y[a][b] = Ff32::azero();
      for (int k = 0; k < 32; ++k)
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
          for (int b = 0; b < 2; ++b) Ff32::mac(y[a][b], L[(ty + 16 * a) * GJ_LD + k], R[k * GJ_LD + tx + 16 * b]);
    };
    S y[2][2];
    product(H, HO, y);
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) HO[(ty + 16 * a) * GJ_LD + tx + 16 * b] = Ff32::val(y[a][b]);
    product(OH, H, x);
    __syncthreads();
    product(OH, HO, y);
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int o = (ty + 16 * a) * GJ_LD + tx + 16 * b;
        OO[o] = Ff32::sub(OO[o], y[a][b]);
        OH[o] = Ff32::neg(Ff32::val(x[a][b]));
      }
    __syncthreads();
  }
  double2* P = J.P + (size_t)s * GJ * GJ;
  for (int e = t; e < bw * bw; e += 256) {
    const double2 v = Ff32::to(B[(e / bw) * GJ_LD + e % bw]);
    P[(e / bw) * GJ + e % bw] = v;
    if (bw == J.ni) A[(size_t)(e / bw) * J.ni + e % bw] = v;
  }
  if (bw == J.ni) return;
  unsigned char* img = J.pd + s * J.p_image();
  for (int e = t; e < bw * (bw / 8); e += 256) {
    const int r = e % bw, c = e / bw;
    uint32_t h = 0;
    for (int k = 0; k < bw; ++k) {
      const S v = B[r * GJ_LD + k];
      h = max(h, max(__float_as_uint(v.rh) & 0x7FFFFFFFu, __float_as_uint(v.ih) & 0x7FFFFFFFu));
    }
    // |x| < 2^(field - 126) for the high word, one more for the low word's share
    const int ex = h >= 0x7F800000u ? kBadExp : (int)(h >> 23) - 125;
    if (c == 0) J.ep[s * GJ + r] = ex;
    long long re[8], im[8], mi[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const double2 v = Ff32::to(B[r * GJ_LD + 8 * c + q]);
      re[q] = to_fix(v.x, ex);
      im[q] = to_fix(v.y, ex);
      mi[q] = -im[q];
    }
    unsigned char* ch = img + ((size_t)(2 * r / XN) * J.chunks + c) * XB_BYTES;
    put8<XN>(ch, 2 * r % XN, 0, re);
    put8<XN>(ch, 2 * r % XN, 1, mi);
    put8<XN>(ch, 2 * r % XN + 1, 0, im);
    put8<XN>(ch, 2 * r % XN + 1, 1, re);
  }
}

__device__ __forceinline__ uint32_t max_hi(const double2 (&v)[8], uint32_t (&sh)[8][32], int tx, int ty) {
  uint32_t h = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) h = max(h, max(abs_hi(v[q].x), abs_hi(v[q].y)));
  sh[ty][tx] = h;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q) h = max(h, sh[q][tx]);
  return h;
}

// Digits as an A operand, block = 32 rows x 8 chunks (of 8 complex k); blockIdx.y 0: rows c of A_Rc^T,
// 1: rows i of A_iR; blockIdx.z: system
__global__ void __launch_bounds__(256) k_gj_digits(GjJob J) {
  __shared__ uint32_t sh[8][32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, row = blockIdx.x * 32 + tx, s = blockIdx.z;
  const bool cols = blockIdx.y;
  const double2* A = J.A + (size_t)s * J.ni * J.ni;
  double2 v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = J.k0 + 8 * ty + q;
    v[q] = 8 * ty < J.bw ? (cols ? A[(size_t)row * J.ni + k] : A[(size_t)k * J.ni + row]) : make_double2(0.0, 0.0);
  }
  const int ex = exp_of(max_hi(v, sh, tx, ty));
  if (ty == 0) (cols ? J.ecol : J.erow)[s * J.ni + row] = ex;
  if (8 * ty >= J.bw) return;
  unsigned char* ch = (cols ? J.cold : J.rowd) + s * J.row_image() + ((size_t)(row >> 7) * J.chunks + ty) * XA_BYTES;
  long long t[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) t[q] = to_fix(v[q].x, ex);
  put8<128>(ch, row & 127, 0, t);
#pragma unroll
  for (int q = 0; q < 8; ++q) t[q] = to_fix(v[q].y, ex);
  put8<128>(ch, row & 127, 1, t);
}

// Digits of the new rows R as a B operand: columns c, rows 2 c = [Re | -Im], 2 c + 1 = [Im | Re] over k
__global__ void __launch_bounds__(256) k_gj_cols(GjJob J) {
  __shared__ uint32_t sh[8][32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, c = blockIdx.x * 32 + tx, s = blockIdx.z;
  const double2* A = J.A + (size_t)s * J.ni * J.ni;
  double2 v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q)
    v[q] = 8 * ty < J.bw ? A[(size_t)(J.k0 + 8 * ty + q) * J.ni + c] : make_double2(0.0, 0.0);
  const int ex = exp_of(max_hi(v, sh, tx, ty));
  if (ty == 0) J.enew[s * J.ni + c] = ex;
  if (8 * ty >= J.bw) return;
  unsigned char* ch = J.newd + s * J.col_image() + ((size_t)(2 * c / XN) * J.chunks + ty) * XB_BYTES;
  long long re[8], im[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    re[q] = to_fix(v[q].x, ex);
    im[q] = to_fix(v[q].y, ex);
  }
  put8<XN>(ch, 2 * c % XN, 0, re);
  put8<XN>(ch, 2 * c % XN + 1, 0, im);
  put8<XN>(ch, 2 * c % XN + 1, 1, re);
#pragma unroll
  for (int q = 0; q < 8; ++q) im[q] = -im[q];
  put8<XN>(ch, 2 * c % XN, 1, im);
}

// GEMM 1: unit = (system, M tile of columns c), tiles n over the 2 bw columns (Re, Im of row r)
struct OpGjRows {
  static constexpr int LV = 7;
  using Job = GjJob;
  struct Unit {
    int s, m, n0, n1;
    __device__ Unit(const Job& J, int u) : s(u / J.mt), m(u % J.mt), n0(0), n1(2 * J.bw / XN) {}
    __device__ const unsigned char* A(const Job& J, int) const {
      return J.rowd + s * J.row_image() + (size_t)m * J.chunks * XA_BYTES;
    }
    __device__ const unsigned char* B(const Job& J, int n) const {
      return J.pd + s * J.p_image() + (size_t)n * J.chunks * XB_BYTES;
    }
    __device__ void range(const Job& J, int, int& c0, int& c1) const {
      c0 = 0;
      c1 = J.chunks;
    }
  };
  int c, part;
  __device__ OpGjRows(const Job&, const Unit& U, int r, int p) : c(128 * U.m + r), part(p) {}
  __device__ void tile(const Job& J, const Unit& U, int n, const long long (&y)[16]) {
    if (c >= J.ni) return;
    const int r0 = (XN * n + 16 * part) / 2, ea = J.erow[U.s * J.ni + c], cr = c - J.k0;
    const bool inR = cr >= 0 && cr < J.bw;
    double2* A = J.A + (size_t)U.s * J.ni * J.ni + (size_t)(J.k0 + r0) * J.ni + c;
    const double2* P = J.P + ((size_t)U.s * GJ + r0) * GJ + cr;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = ea + J.ep[U.s * GJ + r0 + q] - 62 + J.sh;
      A[(size_t)q * J.ni] =
          inR ? P[q * GJ] : make_double2(fix_to_double(y[2 * q], e), fix_to_double(y[2 * q + 1], e));
    }
  }
  __device__ void finish(const Job&, const Unit&, double (&)[3][128], bool) {}
};

// GEMM 2: unit = (system, M tile of rows i, N tile of 32 columns c)
struct OpGjUpdate {
  static constexpr int LV = 7;
  using Job = GjJob;
  struct Unit {
    int s, m, n0, n1;
    __device__ Unit(const Job& J, int u) : s(u / (J.mt * J.nt)), m(u / J.nt % J.mt), n0(u % J.nt), n1(n0 + 1) {}
    __device__ const unsigned char* A(const Job& J, int) const {
      return J.cold + s * J.row_image() + (size_t)m * J.chunks * XA_BYTES;
    }
    __device__ const unsigned char* B(const Job& J, int n) const {
      return J.newd + s * J.col_image() + (size_t)n * J.chunks * XB_BYTES;
    }
    __device__ void range(const Job& J, int, int& c0, int& c1) const {
      c0 = 0;
      c1 = J.chunks;
    }
  };
  int i, part;
  __device__ OpGjUpdate(const Job&, const Unit& U, int r, int p) : i(128 * U.m + r), part(p) {}
  __device__ void tile(const Job& J, const Unit& U, int n, const long long (&y)[16]) {
    if (i >= J.ni || (i >= J.k0 && i < J.k0 + J.bw)) return;
    const int c0 = 32 * n + 8 * part, ea = J.ecol[U.s * J.ni + i];
    const bool inR = c0 >= J.k0 && c0 < J.k0 + J.bw;  // blocks of 32 columns lie inside R or outside
    double* A = reinterpret_cast<double*>(J.A + ((size_t)U.s * J.ni + i) * J.ni + c0);
    const int* eb = J.enew + U.s * J.ni + c0;
#pragma unroll
    for (int q = 0; q < 8; q += 2) {  // 32 bytes: two complex elements
      double a[4] = {0.0, 0.0, 0.0, 0.0};
      if (!inR)
        asm volatile("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(a[0]), "=d"(a[1]), "=d"(a[2]), "=d"(a[3]) : "l"(A + 2 * q));
#pragma unroll
      for (int h = 0; h < 4; ++h) a[h] -= fix_to_double(y[2 * q + h], ea + eb[q + h / 2] - 62 + J.sh);
      asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(A + 2 * q), "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]) : "memory");
    }
  }
  __device__ void finish(const Job&, const Unit&, double (&)[3][128], bool) {}
};

}  // namespace

// W~ of nqb q points from iq0. GW_EUNSUPPORTED when the workspace cannot be had.
gw_status launch_screen_digits(gw_ctx* c, int iq0, int nqb, const double* P, double* W, int* info, double* aug) {
  const int ni = c->ni, nsys = nqb * c->nnu;
  GjJob J{};
  J.ni = ni;
  J.mt = (ni + 127) / 128;
  J.nt = ni / 32;
  const size_t mat = sizeof(double2) * (size_t)ni * ni, bp = sizeof(double2) * GJ * GJ,
               be = align256(sizeof(int) * (3 * (size_t)ni + GJ)),
               dig = ni > GJ ? 2 * J.row_image() + J.col_image() + J.p_image() : 0;
  const int gs = (int)std::max<size_t>(1, std::min<size_t>(nsys, kGroup / (mat + dig + bp)));
  if (!x_workspace(c, XW_SCREEN, gs * (bp + be + dig))) return GW_EUNSUPPORTED;
  char* q = (char*)c->x_ws[XW_SCREEN];
  J.A = (double2*)aug;
  J.P = (double2*)q;
  J.erow = (int*)(q += gs * bp);
  J.ecol = J.erow + (size_t)gs * ni;
  J.enew = J.ecol + (size_t)gs * ni;
  J.ep = J.enew + (size_t)gs * ni;
  J.rowd = (unsigned char*)(q += gs * be);
  J.cold = J.rowd + gs * J.row_image();
  J.newd = J.cold + gs * J.row_image();
  J.pd = J.newd + gs * J.col_image();
  const double* sv = c->d_sqrtv + (size_t)iq0 * ni;
  const size_t psm = sizeof(Ff32::S) * GJ * GJ_LD;
  cudaFuncSetAttribute(k_gj_pivot, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psm);
  const unsigned nb = (unsigned)(((int64_t)ni * ni + 255) / 256);
  gw_status st = GW_OK;
  kt_begin(c, "k_screen_inv");
  for (int s0 = 0; s0 < nsys && st == GW_OK; s0 += gs) {
    const int sn = std::min(gs, nsys - s0);
    k_gj_build<<<dim3(nb, sn), 256, 0, c->stream>>>((const double2*)P, sv, s0, c->nnu, ni, J.A, info);
    st = check_launch(c, "screen build");
    for (J.k0 = 0; J.k0 < ni && st == GW_OK; J.k0 += J.bw) {
      J.bw = std::min(GJ, ni - J.k0);
      J.chunks = 2 * J.bw / XK;
      J.sh = drop_bits(2 * J.bw);
      k_gj_pivot<<<sn, 256, psm, c->stream>>>(J, s0, info);
      if ((st = check_launch(c, "screen pivot")) != GW_OK || J.bw == ni) break;
      k_gj_digits<<<dim3(ni / 32, 2, sn), 256, 0, c->stream>>>(J);
      if ((st = check_launch(c, "screen digits")) != GW_OK) break;
      if ((st = run_gemm<OpGjRows>(c, J, sn * J.mt, "screen rows")) != GW_OK) break;
      k_gj_cols<<<dim3(ni / 32, 1, sn), 256, 0, c->stream>>>(J);
      if ((st = check_launch(c, "screen digits")) != GW_OK) break;
      st = run_gemm<OpGjUpdate>(c, J, sn * J.mt * J.nt, "screen update");
    }
    if (st != GW_OK) break;
    k_gj_out<<<dim3(nb, sn), 256, 0, c->stream>>>(J.A, sv, s0, c->nnu, ni, (double2*)W);
    st = check_launch(c, "screen out");
  }
  kt_end(c);
  return st;
}

}  // namespace gwi
