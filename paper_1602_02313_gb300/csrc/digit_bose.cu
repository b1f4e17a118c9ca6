// Bosonic transforms tau <-> i nu as exact digit products on the tensor cores (digit_gemm.cuh).
//
// The maps are fixed matrices of at most 256 x 256 applied to NI^2 elements a q: 16 flop per byte, which
// the FP64 pipes (and float-float arithmetic on the FP32 pipes) cannot feed. Forward,
// out[j][b] = sum_i T[j][i] in[i][b]: rows b = [Re in | Im in], columns (Re, Im) of every j. Backward,
// Re W(tau_i) = sum_j A_ij Re g_j + B_ij Im g_j and Im W(tau_i) the same of h, g = (W + W^T) / 2 and
// h = (W - W^T) / 2i: W(tau) is Hermitian, so only I <= J is computed and both halves are written.
// The digits of a piece of rows (at most kPiece bytes, so that they stay in L2) are written by one
// kernel and multiplied by the next. Measured, 8 q, NI 256, 48 tau and frequencies, both directions:
// 1.55 ms against 5.21 ms in float-float on the FP32 pipes, errors 1.1e-13 and 2.4e-15 against 1.7e-12
// and 5.9e-14; NI 32, 16 tau, one q: 45 against 60 us. The GEMMs' bound is 0.45 ms of MMAs; the digits'
// writing takes 0.6 ms, the levels' readout (every 96 k) the rest.
#include <algorithm>

#include "digit_gemm.cuh"

namespace gwi {

namespace {

constexpr size_t kPiece = 112ull << 20;

// ------------------------------------------------------------------ digits of the matrices
// The entries of a column (one tau or frequency) of the maps range over many powers of two, and so do the
// data of different tau: the columns are scaled to one size and the data by the inverse (powers of two,
// exact), so that the digits of a row resolve its contributions to the sums alike.

// ec[i] >= 0: scale exponent of column i, the largest of |T_ji| over j relative to the smallest column's
__global__ void __launch_bounds__(256) k_bcol(const double* __restrict__ T, int nf, int nt, int bwd, int* __restrict__ ec) {
  __shared__ int lo;
  const int n = bwd ? nf : nt;
  if (threadIdx.x == 0) lo = 1 << 20;
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    uint32_t h = 0;
    if (bwd)
      for (int j = 0; j < nt; ++j) h = max(h, max(abs_hi(T[(size_t)j * 2 * nf + i]), abs_hi(T[(size_t)j * 2 * nf + nf + i])));
    else
      for (int j = 0; j < nf; ++j) h = max(h, max(abs_hi(T[2 * ((size_t)j * nt + i)]), abs_hi(T[2 * ((size_t)j * nt + i) + 1])));
    ec[i] = h ? (int)(h >> 20) : -1;
    if (h) atomicMin(&lo, (int)(h >> 20));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) ec[i] = ec[i] < 0 ? 0 : min(ec[i] - lo, 64);
}

// exponent of x 2^-ec, as a running maximum (none: kNone)
constexpr int kNone = -(1 << 20);
__device__ __forceinline__ int exp_at(double x, int ec) {
  const uint32_t h = abs_hi(x);
  return h == 0 && x == 0.0 ? kNone : (int)(h >> 20) - 1022 - ec;
}

// Forward: row 2 j = [Re T_j | -Im T_j], row 2 j + 1 = [Im T_j | Re T_j] over chunks of 8 tau
__global__ void k_bdig_t(const double2* __restrict__ T, const int* __restrict__ ec, int nf, int nt, int chunks, int rows,
                         unsigned char* __restrict__ Bi, int* __restrict__ eb) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= rows * chunks) return;
  const int rr = e % rows, c = e / rows, j = rr >> 1;
  int s = kNone;
  if (j < nf)
    for (int i = 0; i < nt; ++i) {
      const double2 t = T[(size_t)j * nt + i];
      s = max(s, max(exp_at(t.x, ec[i]), exp_at(t.y, ec[i])));
    }
  if (c == 0) eb[rr] = s == kNone ? 0 : s;
  long long a[8], b[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int i = 8 * c + q;
    const bool in = j < nf && i < nt;
    const double2 t = in ? T[(size_t)j * nt + i] : make_double2(0.0, 0.0);
    const int x = s + (in ? ec[i] : 0);
    a[q] = to_fix(rr & 1 ? t.y : t.x, x);
    b[q] = to_fix(rr & 1 ? t.x : -t.y, x);
  }
  unsigned char* ch = Bi + ((size_t)(rr / XN) * chunks + c) * XB_BYTES;
  put8<XN>(ch, rr % XN, 0, a);
  put8<XN>(ch, rr % XN, 1, b);
}

// Backward: row i = [A_i | B_i] (Tb[i][0 .. nf), Tb[i][nf .. 2 nf)) over chunks of 8 frequencies
__global__ void k_bdig_tb(const double* __restrict__ Tb, const int* __restrict__ ec, int nf, int nt, int chunks, int rows,
                          unsigned char* __restrict__ Bi, int* __restrict__ eb) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= rows * chunks) return;
  const int i = e % rows, c = e / rows;
  int s = kNone;
  if (i < nt)
    for (int j = 0; j < 2 * nf; ++j) s = max(s, exp_at(Tb[(size_t)i * 2 * nf + j], ec[j < nf ? j : j - nf]));
  if (c == 0) eb[i] = s == kNone ? 0 : s;
  long long a[8], b[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int j = 8 * c + q;
    const bool in = i < nt && j < nf;
    a[q] = in ? to_fix(Tb[(size_t)i * 2 * nf + j], s + ec[j]) : 0;
    b[q] = in ? to_fix(Tb[(size_t)i * 2 * nf + nf + j], s + ec[j]) : 0;
  }
  unsigned char* ch = Bi + ((size_t)(i / XN) * chunks + c) * XB_BYTES;
  put8<XN>(ch, i % XN, 0, a);
  put8<XN>(ch, i % XN, 1, b);
}

// ------------------------------------------------------------------ digits of the data
// largest high word of x 2^ec, ec in [0, 64] (0xFFFFFFFF: not finite), and the row's exponent from it
__device__ __forceinline__ uint32_t hi_at(double x, int ec) {
  const uint32_t h = abs_hi(x);
  return h >= 0x7FF00000u ? 0xFFFFFFFFu : h + ((uint32_t)ec << 20);
}
// Block = 32 rows x 8 chunk lanes: the maximum over the row's chunk lanes
__device__ __forceinline__ int row_exp(uint32_t h, uint32_t (&sh)[8][32], int tx, int ty) {
  sh[ty][tx] = h;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q) h = max(h, sh[q][tx]);
  return h == 0xFFFFFFFFu ? kBadExp : (int)(h >> 20) - 1022;
}

// Forward: rows R = z batch + b of the piece [R0, R0 + rows)
__global__ void __launch_bounds__(256) k_bdig_fwd(const double2* __restrict__ in, const int* __restrict__ ec, int64_t batch,
                                                  int nt, int chunks, int64_t R0, int rows, unsigned char* __restrict__ Ai,
                                                  int* __restrict__ ea) {
  __shared__ uint32_t sh[8][32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, row = blockIdx.x * 32 + tx;
  const bool live = row < rows;
  const int64_t R = R0 + (live ? row : 0), z = R / batch, b = R - z * batch;
  const double2* x = in + (size_t)z * nt * batch + b;
  auto load = [&](int c, double2 (&v)[8], int (&f)[8]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const bool in_ = 8 * c + q < nt;
      v[q] = in_ ? x[(size_t)(8 * c + q) * batch] : make_double2(0.0, 0.0);
      f[q] = in_ ? ec[8 * c + q] : 0;
    }
  };
  double2 v[8];  // a row of at most 64 tau is read once: one chunk per thread, kept
  int f[8];
  uint32_t h = 0;
  for (int c = ty; c < chunks; c += 8) {
    load(c, v, f);
#pragma unroll
    for (int q = 0; q < 8; ++q) h = max(h, max(hi_at(v[q].x, f[q]), hi_at(v[q].y, f[q])));
  }
  const int s = row_exp(h, sh, tx, ty);
  if (!live) return;
  if (ty == 0) ea[row] = s;
  unsigned char* tile = Ai + (size_t)(row >> 7) * chunks * XA_BYTES;
  for (int c = ty; c < chunks; c += 8) {
    if (chunks > 8) load(c, v, f);
    long long t[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] = to_fix(v[q].x, s - f[q]);
    put8<128>(tile + (size_t)c * XA_BYTES, row & 127, 0, t);
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] = to_fix(v[q].y, s - f[q]);
    put8<128>(tile + (size_t)c * XA_BYTES, row & 127, 1, t);
  }
}

// Backward tile t of transform z: 4 rows I x 32 columns J of a 32 x 32 block (bi <= bj)
struct BwdTile {
  int bi, bj, sub;
  __device__ BwdTile(int t, int nb) {
    sub = t & 7;
    int p = t >> 3;
    bi = 0;
    while (p >= nb - bi) {
      p -= nb - bi;
      ++bi;
    }
    bj = bi + p;
  }
  // Row r of the tile. A warp's 32 rows are 4 I x 8 J, so that both W_IJ and W_JI (and the outputs there)
  // come in runs of 64 bytes or more; 32 J of one I would touch 32 lines of W^T for 16 bytes each.
  __device__ bool element(int r, int m, int& I, int& J) const {  // false: beyond the matrix
    I = 32 * bi + 4 * sub + (r & 3);
    J = 32 * bj + 8 * (r >> 5) + ((r & 31) >> 2);
    return I < m && J < m;
  }
};

// g and h of the piece's tiles: images [tile][g, h][chunk]
__global__ void __launch_bounds__(256) k_bdig_bwd(const double2* __restrict__ W, const int* __restrict__ ec, int m, int nf,
                                                  int chunks, int64_t T0, int per_z, unsigned char* __restrict__ Ai,
                                                  int* __restrict__ ea) {
  __shared__ uint32_t sh[2][8][32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int tile = blockIdx.x >> 2, q4 = blockIdx.x & 3;
  const int64_t t = T0 + tile, z = t / per_z;
  const BwdTile B((int)(t - z * per_z), (m + 31) / 32);
  const int row = 32 * q4 + tx;
  int I, J;
  const int nv = B.element(row, m, I, J) ? nf : 0;
  const double2* w = W + (size_t)z * nf * m * m;
  const size_t mm = (size_t)m * m, o = (size_t)I * m + J, ot = (size_t)J * m + I;
  auto load = [&](int c, double2 (&g)[8], double2 (&d)[8], int (&f)[8]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int j = 8 * c + q;
      g[q] = j < nv ? w[j * mm + o] : make_double2(0.0, 0.0);
      d[q] = j < nv ? w[j * mm + ot] : make_double2(0.0, 0.0);
      f[q] = j < nv ? ec[j] : 0;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const double2 a = g[q], b = d[q];
      g[q] = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y + b.y));
      d[q] = make_double2(0.5 * (a.y - b.y), 0.5 * (b.x - a.x));  // (a - b) / 2i
    }
  };
  double2 g[8], d[8];  // a row of at most 64 frequencies is read once: one chunk per thread, kept
  int f[8];
  uint32_t hg = 0, h2 = 0;
  for (int c = ty; c < chunks; c += 8) {
    load(c, g, d, f);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      hg = max(hg, max(hi_at(g[q].x, f[q]), hi_at(g[q].y, f[q])));
      h2 = max(h2, max(hi_at(d[q].x, f[q]), hi_at(d[q].y, f[q])));
    }
  }
  const int sg = row_exp(hg, sh[0], tx, ty), s2 = row_exp(h2, sh[1], tx, ty);
  if (ty == 0) {
    ea[256 * tile + row] = sg;
    ea[256 * tile + 128 + row] = s2;
  }
  for (int c = ty; c < chunks; c += 8) {
    if (chunks > 8) load(c, g, d, f);
    unsigned char* ch = Ai + ((size_t)2 * tile * chunks + c) * XA_BYTES;
    long long t[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] = to_fix(g[q].x, sg - f[q]);
    put8<128>(ch, row, 0, t);
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] = to_fix(g[q].y, sg - f[q]);
    put8<128>(ch, row, 1, t);
    ch += (size_t)chunks * XA_BYTES;
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] = to_fix(d[q].x, s2 - f[q]);
    put8<128>(ch, row, 0, t);
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] = to_fix(d[q].y, s2 - f[q]);
    put8<128>(ch, row, 1, t);
  }
}

// ------------------------------------------------------------------ the products
struct BoseUnit {
  int m, n0, n1;
  template <class J>
  __device__ BoseUnit(const J& j, int u) : m(u), n0(0), n1(j.ntiles) {}
  template <class J>
  __device__ void range(const J& j, int, int& c0, int& c1) const {
    c0 = 0;
    c1 = j.chunks;
  }
};

struct OpBoseFwd {
  static constexpr int LV = 7;
  struct Job {
    const unsigned char *A, *B;
    const int *ea, *eb;
    int ntiles, chunks, rows, nf, sh;
    int64_t R0, batch;
    double2* out;
  };
  struct Unit : BoseUnit {
    __device__ Unit(const Job& J, int u) : BoseUnit(J, u) {}
    __device__ const unsigned char* A(const Job& J, int) const { return J.A + (size_t)m * J.chunks * XA_BYTES; }
    __device__ const unsigned char* B(const Job& J, int n) const { return J.B + (size_t)n * J.chunks * XB_BYTES; }
  };
  int part, ea = 0;
  double2* o = nullptr;  // the row's element of out, frequency 0
  __device__ OpBoseFwd(const Job& J, const Unit& U, int r, int p) : part(p) {
    const int row = 128 * U.m + r;
    if (row >= J.rows) return;
    ea = J.ea[row];
    const int64_t R = J.R0 + row, z = R / J.batch, b = R - z * J.batch;
    o = J.out + (size_t)z * J.nf * J.batch + b;
  }
  __device__ void tile(const Job& J, const Unit&, int n, const long long (&y)[16]) {
    if (!o) return;
    const int j0 = (XN * n + 16 * part) / 2;
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (j0 + q < J.nf) {
        const int e = ea + J.eb[2 * (j0 + q)] - 62 + J.sh;
        o[(size_t)(j0 + q) * J.batch] = make_double2(fix_to_double(y[2 * q], e), fix_to_double(y[2 * q + 1], e));
      }
  }
  __device__ void finish(const Job&, const Unit&, double (&)[3][128], bool) {}
};

struct OpBoseBwd {
  static constexpr int LV = 7;
  struct Job {
    const unsigned char *A, *B;
    const int *ea, *eb;
    int ntiles, chunks, m, nt, sh, per_z;  // ntiles: twice the N tiles (g, h of each)
    int64_t T0;
    double2* out;
  };
  struct Unit : BoseUnit {
    __device__ Unit(const Job& J, int u) : BoseUnit(J, u) {}
    __device__ const unsigned char* A(const Job& J, int n) const {
      return J.A + (size_t)(2 * m + (n & 1)) * J.chunks * XA_BYTES;
    }
    __device__ const unsigned char* B(const Job& J, int n) const { return J.B + (size_t)(n >> 1) * J.chunks * XB_BYTES; }
  };
  int part, row, I, J_;
  double* out;
  __device__ OpBoseBwd(const Job& J, const Unit& U, int r, int p) : part(p), row(256 * U.m + r) {
    const int64_t t = J.T0 + U.m, z = t / J.per_z;
    if (!BwdTile((int)(t - z * J.per_z), (J.m + 31) / 32).element(r, J.m, I, J_)) I = J_ + 1;
    out = reinterpret_cast<double*>(J.out + (size_t)z * J.nt * J.m * J.m);
  }
  // even n: the real parts, odd n: the imaginary parts of the same elements
  __device__ void tile(const Job& J, const Unit&, int n, const long long (&y)[16]) {
    if (I > J_) return;  // the other half of a diagonal block, or beyond the matrix
    const int i0 = XN * (n >> 1) + 16 * part, im = n & 1, ea = J.ea[row + 128 * im];
    const size_t o = 2 * ((size_t)I * J.m + J_) + im, ot = 2 * ((size_t)J_ * J.m + I) + im;
    double* p = out + 2 * (size_t)i0 * J.m * J.m;
#pragma unroll
    for (int e = 0; e < 16; ++e, p += 2 * (size_t)J.m * J.m) {
      if (i0 + e >= J.nt) break;
      const double v = fix_to_double(y[e], ea + J.eb[i0 + e] - 62 + J.sh);
      p[o] = v;
      if (I < J_) p[ot] = im ? -v : v;
    }
  }
  __device__ void finish(const Job&, const Unit&, double (&)[3][128], bool) {}
};

}  // namespace

// The digits of both maps, column scales and row exponents, made once with the context:
// [forward image][backward image][eb fwd][eb bwd][ec fwd][ec bwd]
struct BoseMap {
  int chunks, ntn;
  unsigned char* B;
  int *eb, *ec;
};
static BoseMap bose_map(const gw_ctx* c, bool fwd, size_t* bytes) {
  const int cf = (c->ntau + 7) / 8, cb = (c->nnu + 7) / 8, nf = (2 * c->nnu + XN - 1) / XN, nb = (c->ntau + XN - 1) / XN;
  const size_t bf = (size_t)nf * cf * XB_BYTES, bb = (size_t)nb * cb * XB_BYTES;
  if (bytes) *bytes = bf + bb + 4 * (size_t)(XN * (nf + nb) + c->ntau + c->nnu);
  unsigned char* p = (unsigned char*)c->d_bdig;
  int* e = (int*)(p + bf + bb);
  return fwd ? BoseMap{cf, nf, p, e, e + XN * (nf + nb)} : BoseMap{cb, nb, p + bf, e + XN * nf, e + XN * (nf + nb) + c->ntau};
}

gw_status bose_digits(gw_ctx* c) {
  size_t bytes = 0;
  bose_map(c, true, &bytes);
  if (cudaMalloc(&c->d_bdig, bytes) != cudaSuccess) {
    cudaGetLastError();
    return set_err(c, GW_ENOMEM, "transform digits");
  }
  gw_status st;
  for (int d = 0; d < 2; ++d) {
    const BoseMap m = bose_map(c, d == 0, nullptr);
    const int n = m.ntn * XN * m.chunks;
    k_bcol<<<1, 256, 0, c->stream>>>(d ? c->d_Bbwd : c->d_Bfwd, c->nnu, c->ntau, d, m.ec);
    if ((st = check_launch(c, "transform column scales")) != GW_OK) return st;
    if (d == 0)
      k_bdig_t<<<(n + 127) / 128, 128, 0, c->stream>>>((const double2*)c->d_Bfwd, m.ec, c->nnu, c->ntau, m.chunks,
                                                       m.ntn * XN, m.B, m.eb);
    else
      k_bdig_tb<<<(n + 127) / 128, 128, 0, c->stream>>>(c->d_Bbwd, m.ec, c->nnu, c->ntau, m.chunks, m.ntn * XN, m.B, m.eb);
    if ((st = check_launch(c, "transform digits")) != GW_OK) return st;
  }
  return GW_OK;
}

// count transforms, as gw_tau_to_freq_many stores them. GW_EUNSUPPORTED when the workspace cannot be had.
gw_status launch_bose_exact(gw_ctx* c, int dir, int count, int64_t batch, const double* in, double* out) {
  const bool fwd = dir == GW_TAU_TO_IW;
  const int nt = c->ntau, nf = c->nnu;
  const BoseMap T = bose_map(c, fwd, nullptr);
  const int chunks = T.chunks, ntn = T.ntn;
  const int64_t b32 = (batch + 31) / 32;
  const int per_z = fwd ? 0 : (int)(b32 * (b32 + 1) / 2) * 8;
  // M tiles (of 128 rows; backward: pairs of them) in all and per piece: whole waves within kPiece
  const int64_t tiles = fwd ? (batch * count + 127) / 128 : (int64_t)per_z * count;
  const size_t tile_bytes = (size_t)(fwd ? 1 : 2) * chunks * XA_BYTES;
  const int sms = num_sms(c);
  const int64_t waves = std::max<int64_t>(1, (int64_t)(kPiece / tile_bytes) / sms);
  const int per = (int)std::min<int64_t>(tiles, waves * sms);
  const size_t b_ea = align256(4 * 256 * (size_t)per);
  if (!x_workspace(c, XW_BOSE, b_ea + (size_t)per * tile_bytes)) return GW_EUNSUPPORTED;
  int* ea = (int*)c->x_ws[XW_BOSE];
  unsigned char* Ai = (unsigned char*)c->x_ws[XW_BOSE] + b_ea;
  gw_status st;
  for (int64_t t0 = 0; t0 < tiles; t0 += per) {
    const int tn = (int)std::min<int64_t>(per, tiles - t0);
    if (fwd) {
      const int rows = (int)std::min<int64_t>((int64_t)tn * 128, batch * count - t0 * 128);
      k_bdig_fwd<<<(rows + 31) / 32, 256, 0, c->stream>>>((const double2*)in, T.ec, batch, nt, chunks, t0 * 128, rows, Ai, ea);
      if ((st = check_launch(c, "bose digits")) != GW_OK) return st;
      OpBoseFwd::Job J{Ai, T.B, ea, T.eb, ntn, chunks, rows, nf, drop_bits(16 * chunks), t0 * 128, batch, (double2*)out};
      if ((st = run_gemm<OpBoseFwd>(c, J, tn, "bose gemm")) != GW_OK) return st;
    } else {
      k_bdig_bwd<<<4 * tn, 256, 0, c->stream>>>((const double2*)in, T.ec, (int)batch, nf, chunks, t0, per_z, Ai, ea);
      if ((st = check_launch(c, "bose digits")) != GW_OK) return st;
      OpBoseBwd::Job J{Ai, T.B, ea, T.eb, 2 * ntn, chunks, (int)batch, nt, drop_bits(16 * chunks), per_z, t0, (double2*)out};
      if ((st = run_gemm<OpBoseBwd>(c, J, tn, "bose gemm")) != GW_OK) return st;
    }
  }
  return GW_OK;
}

}  // namespace gwi
