// Fine Wilson-clover operator of Eq. (2): gauge import, clover term A_x
// and the stencil apply (one thread per site and vector).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "async_copy.cuh"
#include "kernels.cuh"
#include "wilson_ops.cuh"
#include "tune.cuh"

namespace gbmg {

namespace {

// gauge_int[mu][s] = gauge_ext[mu][s] * (t antiperiodic and mu = t and
// t(s) = Lt - 1 ? -1 : 1): the fermion boundary sign lives on the link
// that wraps, so hops need no special case.
// Links of Eq. (2) with the fermion boundary sign folded in.
template <typename R>
__global__ void k_gauge_import(cpx<R>* __restrict__ out, const cpx<double>* __restrict__ in,
                               Geom g, int antiperiodic) {
  size_t n = size_t(4) * g.vol * 9;
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n;
       i += size_t(gridDim.x) * blockDim.x) {
    size_t link = i / 9;
    int mu = int(link / g.vol);
    int s = int(link % g.vol);
    double sgn = 1.0;
    if (antiperiodic && mu == 3 && s / g.stride[3] == g.L[3] - 1) sgn = -1.0;
    out[i] = cpx<R>(sgn * in[i]);
  }
}

// First two rows of every (sign-folded) link in FP32, [mu][V][6] complex,
// and the largest deviation, over all links, of the rebuilt third row
// sgn * conj(row0 x row1) from the stored one (FP64, as float bits into
// *maxdev; non-negative floats order like their bit patterns).
// Two-row link form (gauge compression, Sec. 4).
__global__ void k_gauge_compress12(cpx<float>* __restrict__ out, unsigned* __restrict__ maxdev,
                                   const cpx<double>* __restrict__ in, Geom g, int antiperiodic) {
  const size_t n = size_t(4) * g.vol;
  float dev = 0.f;
  for (size_t link = blockIdx.x * size_t(blockDim.x) + threadIdx.x; link < n;
       link += size_t(gridDim.x) * blockDim.x) {
    const int mu = int(link / g.vol);
    const int s = int(link % g.vol);
    const double sgn = (antiperiodic && mu == 3 && s / g.stride[3] == g.L[3] - 1) ? -1.0 : 1.0;
    cpx<double> u[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) u[i] = sgn * in[link * 9 + i];
#pragma unroll
    for (int i = 0; i < 6; ++i) out[link * 6 + i] = cpx<float>(u[i]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int b = (a + 1) % 3, c = (a + 2) % 3;
      const cpx<double> r = sgn * conj(u[b] * u[3 + c] - u[c] * u[3 + b]);
      const cpx<double> d = r - u[6 + a];
      dev = fmaxf(dev, float(sqrt(d.re * d.re + d.im * d.im)));
    }
  }
  for (int o = 16; o > 0; o >>= 1) dev = fmaxf(dev, __shfl_xor_sync(0xffffffffu, dev, o));
  if ((threadIdx.x & 31) == 0) atomicMax(maxdev, __float_as_uint(dev));
}

// 8-real form of an SU(3) link (Sec. 4): U = [[a1 a2 a3][b1 b2 b3][c1 c2 c3]]
// is stored as a2, a3, b1 and the phases of a1 and c1.  Unit rows and
// columns give |a1|^2 = 1 - |a2|^2 - |a3|^2 =: n and |c1|^2 = n - |b1|^2;
// orthogonality of rows 0 and 1 and c1 = conj(a2 b3 - a3 b2) (row 2 =
// conj(row 0 x row 1), det U = 1) are two linear equations for b2, b3 with
// determinant -n:
//   b2 = -(conj(a3) conj(c1) + conj(a1) a2 b1) / n
//   b3 =  (conj(a2) conj(c1) - conj(a1) a3 b1) / n
// and then c2 = conj(a3 b1 - a1 b3), c3 = conj(a1 b2 - a2 b1).
__device__ __forceinline__ void rebuild8(const float w[8], cpx<float> u[9]) {
  const cpx<float> a2(w[0], w[1]), a3(w[2], w[3]), b1(w[4], w[5]);
  const float n = norm2(a2) + norm2(a3);
  const float ra1 = sqrtf(fmaxf(1.f - n, 0.f));
  const float rc1 = sqrtf(fmaxf(n - norm2(b1), 0.f));
  float sa, ca, sc, cc;
  sincosf(w[6], &sa, &ca);
  sincosf(w[7], &sc, &cc);
  const cpx<float> a1(ra1 * ca, ra1 * sa), c1(rc1 * cc, rc1 * sc);
  const float inv = 1.f / n;
  const cpx<float> ab = conj(a1) * b1;
  const cpx<float> cc1 = conj(c1);
  const cpx<float> b2 = -inv * (conj(a3) * cc1 + a2 * ab);
  const cpx<float> b3 = inv * (conj(a2) * cc1 - a3 * ab);
  u[0] = a1;
  u[1] = a2;
  u[2] = a3;
  u[3] = b1;
  u[4] = b2;
  u[5] = b3;
  u[6] = c1;
  u[7] = conj(a3 * b1 - a1 * b3);
  u[8] = conj(a1 * b2 - a2 * b1);
}

// FP64 links (no boundary sign) -> the 8-real form, with the rebuilt
// link's largest deviation (atomicMax on the float bits) and, per block,
// the sum of squared deviations (summed on the host in block order)
__global__ void __launch_bounds__(256) k_gauge_compress8(float* __restrict__ out,
                                                         unsigned* __restrict__ maxdev,
                                                         double* __restrict__ sq_part,
                                                         const cpx<double>* __restrict__ in,
                                                         Geom g) {
  const size_t n = size_t(4) * g.vol;
  float dev = 0.f;
  double sq = 0.0;
  for (size_t link = blockIdx.x * size_t(blockDim.x) + threadIdx.x; link < n;
       link += size_t(gridDim.x) * blockDim.x) {
    const cpx<double>* u = in + link * 9;
    float w[8] = {float(u[1].re), float(u[1].im), float(u[2].re), float(u[2].im),
                  float(u[3].re), float(u[3].im), float(atan2(u[0].im, u[0].re)),
                  float(atan2(u[6].im, u[6].re))};
#pragma unroll
    for (int i = 0; i < 8; ++i) out[link * 8 + i] = w[i];
    cpx<float> r[9];
    rebuild8(w, r);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const double dr = double(r[i].re) - u[i].re, di = double(r[i].im) - u[i].im;
      const double d2 = dr * dr + di * di;
      sq += d2;
      dev = fmaxf(dev, float(sqrt(d2)));
    }
  }
  __shared__ double sh[8];
  for (int o = 16; o > 0; o >>= 1) {
    dev = fmaxf(dev, __shfl_xor_sync(0xffffffffu, dev, o));
    sq += __shfl_xor_sync(0xffffffffu, sq, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(maxdev, __float_as_uint(dev));
    sh[threadIdx.x >> 5] = sq;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (blockDim.x >> 5); ++w) t += sh[w];
    sq_part[blockIdx.x] = t;
  }
}

struct M3 {
  cpx<double> a[9];
};

__device__ __forceinline__ M3 mload(const cpx<double>* __restrict__ g, int mu, int s, int vol) {
  M3 m;
  const cpx<double>* p = g + (size_t(mu) * vol + s) * 9;
#pragma unroll
  for (int i = 0; i < 9; ++i) m.a[i] = p[i];
  return m;
}
__device__ __forceinline__ M3 mmul(const M3& x, const M3& y) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cpx<double> t(0.0, 0.0);
#pragma unroll
      for (int k = 0; k < 3; ++k) cmac(t, x.a[i * 3 + k], y.a[k * 3 + j]);
      r.a[i * 3 + j] = t;
    }
  return r;
}
__device__ __forceinline__ M3 mdag(const M3& x) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) r.a[i * 3 + j] = conj(x.a[j * 3 + i]);
  return r;
}

__device__ __forceinline__ int shifted(const Geom& g, const int c[4], int mu, int dm, int nu,
                                       int dn) {
  int cc[4] = {c[0], c[1], c[2], c[3]};
  cc[mu] = (cc[mu] + dm + g.L[mu]) % g.L[mu];
  cc[nu] = (cc[nu] + dn + g.L[nu]) % g.L[nu];
  return cc[0] + g.stride[1] * cc[1] + g.stride[2] * cc[2] + g.stride[3] * cc[3];
}

// Fhat_{mu nu}(x) = (Q - Q^dag) / 8, Q the sum of the four plaquette
// leaves at x, all oriented (+mu, +nu, -mu, -nu).
__device__ M3 field_strength(const cpx<double>* __restrict__ U, const Geom& g, int s,
                             const int c[4], int mu, int nu) {
  const int V = g.vol;
  int x = s;
  int xpm = shifted(g, c, mu, 1, nu, 0), xpn = shifted(g, c, mu, 0, nu, 1);
  int xmm = shifted(g, c, mu, -1, nu, 0), xmn = shifted(g, c, mu, 0, nu, -1);
  int xmmpn = shifted(g, c, mu, -1, nu, 1), xmmmn = shifted(g, c, mu, -1, nu, -1);
  int xpmmn = shifted(g, c, mu, 1, nu, -1);
  M3 q = mmul(mmul(mload(U, mu, x, V), mload(U, nu, xpm, V)),
              mmul(mdag(mload(U, mu, xpn, V)), mdag(mload(U, nu, x, V))));
  M3 t = mmul(mmul(mload(U, nu, x, V), mdag(mload(U, mu, xmmpn, V))),
              mmul(mdag(mload(U, nu, xmm, V)), mload(U, mu, xmm, V)));
#pragma unroll
  for (int i = 0; i < 9; ++i) q.a[i] += t.a[i];
  t = mmul(mmul(mdag(mload(U, mu, xmm, V)), mdag(mload(U, nu, xmmmn, V))),
           mmul(mload(U, mu, xmmmn, V), mload(U, nu, xmn, V)));
#pragma unroll
  for (int i = 0; i < 9; ++i) q.a[i] += t.a[i];
  t = mmul(mmul(mdag(mload(U, nu, xmn, V)), mload(U, mu, xmn, V)),
           mmul(mload(U, nu, xpmmn, V), mdag(mload(U, mu, x, V))));
#pragma unroll
  for (int i = 0; i < 9; ++i) q.a[i] += t.a[i];
  M3 f;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) f.a[i * 3 + j] = 0.125 * (q.a[i * 3 + j] - conj(q.a[j * 3 + i]));
  return f;
}

// A_x = c_sw (i/4) sum_{mu != nu} sigma_{mu nu} (x) Fhat_{mu nu}
//     = c_sw (i/2) sum_{mu < nu} sigma_{mu nu} (x) Fhat_{mu nu}.
// In the chiral basis sigma_{mu nu} = diag(s_up, s_lo) with Pauli blocks
//   (01): s3, s3   (02): s2, s2   (03): -s1, s1
//   (12): s1, s1   (13): s2, -s2  (23): -s3, s3
// so per chirality A = c_sw (i/2) [s1 (x) G1 + s2 (x) G2 + s3 (x) G3].
// Clover term A_x of Eq. (2) (Sec. 3.2).
__global__ void k_clover(const cpx<double>* __restrict__ U, Geom g, double csw,
                         double* __restrict__ out64, float* __restrict__ out32,
                         float4* __restrict__ out32t) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.vol) return;
  int c[4];
  site_coords(g, s, c);
  M3 F01 = field_strength(U, g, s, c, 0, 1);
  M3 F02 = field_strength(U, g, s, c, 0, 2);
  M3 F03 = field_strength(U, g, s, c, 0, 3);
  M3 F12 = field_strength(U, g, s, c, 1, 2);
  M3 F13 = field_strength(U, g, s, c, 1, 3);
  M3 F23 = field_strength(U, g, s, c, 2, 3);
  const double h = 0.5 * csw;
#pragma unroll
  for (int chi = 0; chi < 2; ++chi) {
    double sg = chi == 0 ? -1.0 : 1.0;
    cpx<double> blk[6][6];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        int k = a * 3 + b;
        cpx<double> G1 = F12.a[k] + sg * F03.a[k];
        cpx<double> G2 = F02.a[k] - sg * F13.a[k];
        cpx<double> G3 = F01.a[k] + sg * F23.a[k];
        // (i/2) csw [[G3, G1 - i G2], [G1 + i G2, -G3]]
        blk[a][b] = h * times_i(G3);
        blk[a][3 + b] = h * (times_i(G1) + G2);
        blk[3 + a][b] = h * (times_i(G1) - G2);
        blk[3 + a][3 + b] = -(h * times_i(G3));
      }
    double* o64 = out64 + size_t(s) * 72 + chi * 36;
#pragma unroll
    for (int i = 0; i < 6; ++i) o64[i] = blk[i][i].re;
#pragma unroll
    for (int i = 1; i < 6; ++i)
#pragma unroll
      for (int j = 0; j < i; ++j) {
        int k = i * (i - 1) / 2 + j;
        o64[6 + 2 * k] = blk[i][j].re;
        o64[7 + 2 * k] = blk[i][j].im;
      }
    if (out32) {
      float* o32 = out32 + size_t(s) * 72 + chi * 36;
      for (int i = 0; i < 36; ++i) o32[i] = float(o64[i]);
      // transposed: word w of every site adjacent
      for (int w = 0; w < 9; ++w)
        out32t[size_t(chi * 9 + w) * g.vol + s] = make_float4(
            float(o64[4 * w]), float(o64[4 * w + 1]), float(o64[4 * w + 2]), float(o64[4 * w + 3]));
    }
  }
}

// LF = 18: links stored in full; LF = 12: the two-row form (16-byte loads,
// 48 B per FP32 link) with the third row rebuilt in registers, the rebuilt
// row carrying the boundary sign of the link (t-links leaving the last time
// slice); LF = 8 (FP32 only): the 8-real form (two 16-byte loads, 32 B per
// link) rebuilt by rebuild8, the boundary sign applied to the whole link.
// Several vectors (nvec > 1, stored vstride apart): CTAs are ordered
// vector-fastest, so the nvec CTAs of one site chunk run close together and
// the chunk's links and clover come from DRAM once and from L2 for the
// other vectors.
// A: the clover, FP32 as 18 words of 16 B by site ([word][site]: adjacent
// lanes read adjacent words; records of 288 B per lane cost eight times the
// L1 wavefronts and bound the kernel), FP64 as records.
// Eq. (2): the Wilson-clover matrix on one or several vectors.
template <typename R, int LF, int MINB>
__global__ void __launch_bounds__(128, MINB) k_wilson(cpx<R>* __restrict__ out, const cpx<R>* __restrict__ in,
                                                const cpx<R>* __restrict__ U, const R* __restrict__ A,
                                                Geom g, R diag, size_t vstride, int nvec,
                                                int antiperiodic) {
  const int vec = blockIdx.x % nvec;
  const int s = (blockIdx.x / nvec) * blockDim.x + threadIdx.x;
  if (s >= g.vol) return;
  in += vec * vstride;
  out += vec * vstride;
  int c[4];
  site_coords(g, s, c);
  cpx<R> psi[12], acc[12], u[9];
  // 16-byte vector loads of the 96 B (FP32) / 192 B (FP64) spinor records and
  // of the clover record; links (72 B / 144 B records) by complex number
  auto load_spinor = [&](int site) {
    const uint4* p = reinterpret_cast<const uint4*>(in + size_t(site) * 12);
    constexpr int W = sizeof(cpx<R>) * 12 / 16;
    uint4 w[W];
#pragma unroll
    for (int i = 0; i < W; ++i) w[i] = __ldg(p + i);
#pragma unroll
    for (int i = 0; i < 12; ++i) psi[i] = reinterpret_cast<const cpx<R>*>(w)[i];
  };
  auto load_link = [&](size_t idx, bool neg) {
    if constexpr (LF == 8) {
      const uint4* p = reinterpret_cast<const uint4*>(U) + idx * 2;
      const uint4 w0 = __ldg(p), w1 = __ldg(p + 1);
      const float w[8] = {__uint_as_float(w0.x), __uint_as_float(w0.y), __uint_as_float(w0.z),
                          __uint_as_float(w0.w), __uint_as_float(w1.x), __uint_as_float(w1.y),
                          __uint_as_float(w1.z), __uint_as_float(w1.w)};
      rebuild8(w, u);
      if (neg) {
#pragma unroll
        for (int i = 0; i < 9; ++i) u[i] = -u[i];
      }
    } else if constexpr (LF == 12) {
      const uint4* p = reinterpret_cast<const uint4*>(U + idx * 6);
      uint4 w[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) w[i] = __ldg(p + i);
#pragma unroll
      for (int i = 0; i < 6; ++i) u[i] = reinterpret_cast<const cpx<R>*>(w)[i];
      const R sg = neg ? R(-1) : R(1);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int b = (a + 1) % 3, c = (a + 2) % 3;
        u[6 + a] = sg * conj(u[b] * u[3 + c] - u[c] * u[3 + b]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 9; ++i) u[i] = U[idx * 9 + i];
    }
  };
  // boundary sign of the t-links that wrap (only the rebuilt row needs it)
  const bool tlast = antiperiodic && c[3] == g.L[3] - 1, tfirst = antiperiodic && c[3] == 0;
  load_spinor(s);
#pragma unroll
  for (int i = 0; i < 12; ++i) acc[i] = cpx<R>(R(0), R(0));
  {
    constexpr int W = sizeof(R) * 72 / 16;
    uint4 w[W];
    if constexpr (std::is_same<R, float>::value) {
      const uint4* p = reinterpret_cast<const uint4*>(A) + s;
#pragma unroll
      for (int i = 0; i < W; ++i) w[i] = __ldg(p + size_t(i) * g.vol);
    } else {
      const uint4* p = reinterpret_cast<const uint4*>(A + size_t(s) * 72);
#pragma unroll
      for (int i = 0; i < W; ++i) w[i] = __ldg(p + i);
    }
    clover_accum(reinterpret_cast<const R*>(w), diag, psi, acc);
  }
  const size_t V = g.vol;
#define GB_HOP(MU)                                       \
  {                                                      \
    int sf = neighbour(g, s, c, 1 + 2 * MU);             \
    load_spinor(sf);                                     \
    load_link(MU * V + s, MU == 3 && tlast);             \
    hop_accum<MU, true>(u, psi, acc);                    \
    int sb = neighbour(g, s, c, 2 + 2 * MU);             \
    load_spinor(sb);                                     \
    load_link(MU * V + sb, MU == 3 && tfirst);           \
    hop_accum<MU, false>(u, psi, acc);                   \
  }
  GB_HOP(0) GB_HOP(1) GB_HOP(2) GB_HOP(3)
#undef GB_HOP
#pragma unroll
  for (int i = 0; i < 12; ++i) out[size_t(s) * 12 + i] = acc[i];
}

// Batched form for the setup sweeps: one thread applies the operator at one
// site to NB vectors, so the site's links and clover are read once for NB
// vectors instead of once per vector.  Vectors are stored back to back
// (vector v at offset v * vstride); blockIdx.y picks a group of NB vectors.
// Eq. (2) on NB vectors per thread (setup sweeps, Sec. 3.4 step 1).
template <typename R, int NB>
__global__ void __launch_bounds__(128) k_wilson_mv(cpx<R>* __restrict__ out,
                                                   const cpx<R>* __restrict__ in,
                                                   const cpx<R>* __restrict__ U,
                                                   const R* __restrict__ A, Geom g, R diag,
                                                   size_t vstride) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.vol) return;
  in += size_t(blockIdx.y) * NB * vstride;
  out += size_t(blockIdx.y) * NB * vstride;
  int c[4];
  site_coords(g, s, c);
  cpx<R> acc[NB][12];
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int i = 0; i < 12; ++i) acc[b][i] = cpx<R>(R(0), R(0));
  constexpr int SW = sizeof(cpx<R>) * 12 / 16;  // 16-byte words of a spinor
  auto load_spinor = [&](int b, int site, cpx<R> psi[12]) {
    const uint4* p = reinterpret_cast<const uint4*>(in + b * vstride + size_t(site) * 12);
    uint4 w[SW];
#pragma unroll
    for (int i = 0; i < SW; ++i) w[i] = __ldg(p + i);
#pragma unroll
    for (int i = 0; i < 12; ++i) psi[i] = reinterpret_cast<const cpx<R>*>(w)[i];
  };
  // clover, one chirality block (36 reals) at a time
#pragma unroll
  for (int chi = 0; chi < 2; ++chi) {
    constexpr int CW = sizeof(R) * 36 / 16;
    uint4 w[CW];
    const uint4* p = reinterpret_cast<const uint4*>(A + size_t(s) * 72 + chi * 36);
#pragma unroll
    for (int i = 0; i < CW; ++i) w[i] = __ldg(p + i);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      cpx<R> psi[12];
      load_spinor(b, s, psi);
      clover_block_accum(reinterpret_cast<const R*>(w), diag, psi + chi * 6, acc[b] + chi * 6);
    }
  }
  const size_t V = g.vol;
  cpx<R> u[9];
  auto load_link = [&](size_t idx) {
#pragma unroll
    for (int i = 0; i < 9; ++i) u[i] = U[idx * 9 + i];
  };
#define GB_HOP_MV(MU)                                   \
  {                                                     \
    const int sf = neighbour(g, s, c, 1 + 2 * MU);      \
    load_link(MU * V + s);                              \
    _Pragma("unroll") for (int b = 0; b < NB; ++b) {    \
      cpx<R> psi[12];                                   \
      load_spinor(b, sf, psi);                          \
      hop_accum<MU, true>(u, psi, acc[b]);              \
    }                                                   \
    const int sb = neighbour(g, s, c, 2 + 2 * MU);      \
    load_link(MU * V + sb);                             \
    _Pragma("unroll") for (int b = 0; b < NB; ++b) {    \
      cpx<R> psi[12];                                   \
      load_spinor(b, sb, psi);                          \
      hop_accum<MU, false>(u, psi, acc[b]);             \
    }                                                   \
  }
  GB_HOP_MV(0) GB_HOP_MV(1) GB_HOP_MV(2) GB_HOP_MV(3)
#undef GB_HOP_MV
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    uint4* o = reinterpret_cast<uint4*>(out + b * vstride + size_t(s) * 12);
#pragma unroll
    for (int i = 0; i < SW; ++i) o[i] = reinterpret_cast<const uint4*>(acc[b])[i];
  }
}

// Batched form with the operator staged in shared memory: CTA b holds the
// eight hop links (two-row form when C12) and the clover of the 32 sites
// [32 b, 32 b + 32), stored transposed ([element][site]) so that the 32
// lanes of a warp (32 consecutive sites) read consecutive words.  Warp w
// then applies the operator to vectors w, w + 4, ...: per vector the same
// work and registers as the one-vector kernel, while links and clover come
// from HBM once for all nvec vectors.
// Eq. (2) with a tile of links and clover in shared memory.
template <bool C12>
__global__ void __launch_bounds__(128) k_wilson_tile(cpx<float>* __restrict__ out,
                                                     const cpx<float>* __restrict__ in,
                                                     const cpx<float>* __restrict__ U,
                                                     const float* __restrict__ A, Geom g,
                                                     float diag, size_t vstride, int nvec,
                                                     int antiperiodic) {
  constexpr int TS = 32;               // sites per CTA
  constexpr int LC = C12 ? 6 : 9;      // stored complex numbers per link
  __shared__ cpx<float> lk[8 * LC * TS];   // [hop][element][site]
  __shared__ float cl[72 * TS];             // [element][site]
  __shared__ int nbb[4 * TS];               // backward neighbour of each site, per mu
  const int tid = threadIdx.x;
  const int s0 = blockIdx.x * TS;
  const size_t V = g.vol;
  {
    const int sl = tid & (TS - 1), mu = tid >> 5;
    const int s = s0 + sl;
    if (s < g.vol) {
      int c[4];
      site_coords(g, s, c);
      nbb[mu * TS + sl] = neighbour(g, s, c, 2 + 2 * mu);
    }
  }
  __syncthreads();
  for (int i = tid; i < 8 * LC * TS; i += 128) {
    const int sl = i & (TS - 1), e = (i / TS) % LC, h = i / (TS * LC);
    const int s = s0 + sl;
    if (s < g.vol) {
      const int mu = h >> 1;
      const size_t link = size_t(mu) * V + ((h & 1) ? nbb[mu * TS + sl] : s);
      const float2 f = __ldg(reinterpret_cast<const float2*>(U + link * LC + e));
      lk[i] = cpx<float>(f.x, f.y);
    }
  }
  for (int i = tid; i < 72 * TS; i += 128) {
    const int sl = i & (TS - 1), k = i / TS;
    const int s = s0 + sl;
    if (s < g.vol) cl[i] = __ldg(A + size_t(s) * 72 + k);
  }
  __syncthreads();
  const int sl = tid & (TS - 1), w = tid >> 5;
  const int s = s0 + sl;
  if (s >= g.vol) return;
  int c[4];
  site_coords(g, s, c);
  int nbr[8];
#pragma unroll
  for (int d = 0; d < 8; ++d) nbr[d] = neighbour(g, s, c, 1 + d);
  const bool tlast = antiperiodic && c[3] == g.L[3] - 1, tfirst = antiperiodic && c[3] == 0;
  for (int v = w; v < nvec; v += 4) {
    const cpx<float>* x = in + size_t(v) * vstride;
    cpx<float> psi[12], acc[12], u[9];
    auto load_spinor = [&](int site) {
      const uint4* q = reinterpret_cast<const uint4*>(x + size_t(site) * 12);
      uint4 wv[6];
#pragma unroll
      for (int i = 0; i < 6; ++i) wv[i] = __ldg(q + i);
#pragma unroll
      for (int i = 0; i < 12; ++i) psi[i] = reinterpret_cast<const cpx<float>*>(wv)[i];
    };
    auto load_link = [&](int h, bool neg) {
#pragma unroll
      for (int e = 0; e < LC; ++e) u[e] = lk[(h * LC + e) * TS + sl];
      if constexpr (C12) {
        const float sg = neg ? -1.f : 1.f;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const int b = (r + 1) % 3, cc = (r + 2) % 3;
          u[6 + r] = sg * conj(u[b] * u[3 + cc] - u[cc] * u[3 + b]);
        }
      }
    };
    load_spinor(s);
#pragma unroll
    for (int i = 0; i < 12; ++i) acc[i] = cpx<float>(0.f, 0.f);
    clover_accum_strided(cl + sl, TS, diag, psi, acc);
#define GB_TILE_HOP(MU)                                  \
  {                                                      \
    load_spinor(nbr[2 * MU]);                            \
    load_link(2 * MU, MU == 3 && tlast);                 \
    hop_accum<MU, true>(u, psi, acc);                    \
    load_spinor(nbr[2 * MU + 1]);                        \
    load_link(2 * MU + 1, MU == 3 && tfirst);            \
    hop_accum<MU, false>(u, psi, acc);                   \
  }
    GB_TILE_HOP(0) GB_TILE_HOP(1) GB_TILE_HOP(2) GB_TILE_HOP(3)
#undef GB_TILE_HOP
    uint4* o = reinterpret_cast<uint4*>(out + size_t(v) * vstride + size_t(s) * 12);
#pragma unroll
    for (int i = 0; i < 6; ++i) o[i] = reinterpret_cast<const uint4*>(acc)[i];
  }
}


// Tiled form: one CTA per block of BX x BY x BZ x BT sites (one thread per
// site).  Before any arithmetic, tensor copies (TMA) bring into shared
// memory the block's spinors, the one-site-deep faces around it (eight
// boxes at wrapped coordinates, so every neighbour of the block is
// present), the block's two-row links in all four directions and the links
// on its four backward faces (the U_mu(x - mu) of the boundary sites); a
// neighbour spinor that nine sites share is read from L2 once per block
// instead of once per site, and no thread waits on a dependent gather.  The
// thread's clover stays in registers across the vectors; for several
// vectors the links stay in shared memory and only the spinor tile is
// copied again, into the other of two spinor buffers while the current
// vector is computed.  Smem layout (records of 96 B spinors / 48 B links,
// in the boxes' own order, x fastest): [interior][x-][x+][y-][y+][z-][z+]
// [t-][t+] spinors, then [link mu interior] x 4, [x-][y-][z-][t-] links,
// then (several vectors) the second spinor buffer.
//
// What bounds it: with thread-private 16-byte accesses to records of 96 B
// (spinors), 48 B (links) and 288 B (clover), the L1 data pipe, before HBM.
// Three choices cut its wavefronts:
//  * a record of 96 B starts at bank 0, 8, 16 or 24, so the eight lanes of
//    a 16-byte phase collide two by two; lanes of every second group of four
//    read the record's halves (chiralities) in the other order, 12 banks
//    on, and keep the two halves exchanged throughout: the projections of
//    directions 0..2 change sign for them (C_mu = -B_mu), those of direction
//    3 do not (C_3 = B_3), and their accumulators hold the other chirality
//    first (see hop_halves);
//  * the clover is read from a transposed store, [word][site], where the
//    16-byte words of consecutive sites are adjacent;
//  * x is merged into the innermost tensor dimension, so a copy moves rows
//    of BX records instead of single records.
// Extents that the block does not divide leave partial blocks: the faces
// sit at the valid extent, the rest of a box is zero-filled (or holds sites
// nobody reads) and the surplus threads repeat a valid site without storing.
// Tensor maps (innermost first): spinors (24 Lx floats, Ly, Lz, Lt, nvec),
// links (12 Lx floats, Ly, Lz, Lt, 4).  Index 0: the interior box, 1 + mu:
// the face box of direction mu (extent 1 in mu).
struct WilsonTileMaps {
  CUtensorMap sp[5];
  CUtensorMap lk[5];
};

template <int BX, int BY, int BZ, int BT>
struct WilsonBlock {
  static constexpr int NS = BX * BY * BZ * BT;
  __host__ __device__ static constexpr int B(int mu) {
    return mu == 0 ? BX : mu == 1 ? BY : mu == 2 ? BZ : BT;
  }
  __host__ __device__ static constexpr int F(int mu) { return NS / B(mu); }  // face records
  static constexpr int NSP = NS + 2 * (F(0) + F(1) + F(2) + F(3));  // spinor records
  static constexpr int NLK = 4 * NS + F(0) + F(1) + F(2) + F(3);      // link records
  // first record of spinor face (mu, side): side 0 at x_mu - 1, 1 at x_mu + B_mu
  __host__ __device__ static constexpr int face_sp(int mu, int side) {
    int o = NS;
    for (int nu = 0; nu < mu; ++nu) o += 2 * F(nu);
    return o + side * F(mu);
  }
  // first record of the backward link face of mu
  __host__ __device__ static constexpr int face_lk(int mu) {
    int o = 4 * NS;
    for (int nu = 0; nu < mu; ++nu) o += F(nu);
    return o;
  }
  // the same for a direction known at run time
  __device__ static __forceinline__ int face_sp_rt(int mu, int side) {
    const int f = mu == 0 ? F(0) : mu == 1 ? F(1) : mu == 2 ? F(2) : F(3);
    return (mu == 0   ? face_sp(0, 0)
            : mu == 1 ? face_sp(1, 0)
            : mu == 2 ? face_sp(2, 0)
                      : face_sp(3, 0)) +
           side * f;
  }
  __device__ static __forceinline__ int face_lk_rt(int mu) {
    return mu == 0 ? face_lk(0) : mu == 1 ? face_lk(1) : mu == 2 ? face_lk(2) : face_lk(3);
  }
};

// One vector: a grid of resident CTAs walks the blocks, so that launch,
// barrier set-up and the record offsets of a thread are paid once, not per
// block.  Several vectors: a CTA per block (they amortise the set-up, and
// static block lists measured 12 % slower).
// Measured, 8x2x2x2 block: one 32^3x64 vector 318 -> 265 us (672 B/site with
// two-row links: 5.3 TB/s), eight 24^3x48 vectors 491 -> 437 us.  L1
// wavefronts fell from 65-70 to 38-45 % of their peak; what is left is
// latency (issue slots 37-50 % busy with 6-10 warps per SM; two threads per
// site doubled the warps and gained nothing).
// MINB: resident CTAs per SM that the register budget allows; MULTI: several
// vectors per launch; DOT: also the inner products <out, in> and |out|^2 that
// an MR step needs, as partial sums [vector][2][part] (one part per warp of a
// CTA, and per block with several vectors; per-block sums in FP32, FP64 across
// blocks): the pass that reads both vectors again goes.  32^3x64, one vector:
// 70 us of reading for 15 us here; 24 vectors of 16^3x32: 101 us for
// 44 us.
template <int BX, int BY, int BZ, int BT, int MINB, bool MULTI, bool DOT>
__global__ void __launch_bounds__(BX * BY * BZ * BT, MINB)
    k_wilson_blk(cpx<float>* __restrict__ out, const float4* __restrict__ A, Geom g, float diag,
                 size_t vstride, int nvec, int antiperiodic, int nblocks,
                 const __grid_constant__ WilsonTileMaps maps, int* __restrict__ err,
                 double2* __restrict__ part, int stall) {
  using WB = WilsonBlock<BX, BY, BZ, BT>;
  constexpr int NS = WB::NS;
  extern __shared__ __align__(128) unsigned char wsm[];
  unsigned char* lk = wsm + size_t(WB::NSP) * 96;   // link records
  // spinor buffers, used in turn (every offset a multiple of 128 B)
  unsigned char* const sp0 = wsm;
  unsigned char* const sp1 = MULTI ? lk + size_t(WB::NLK) * 48 : wsm;
  __shared__ uint64_t bar[2];
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    fence_mbar_init();
  }
  __syncthreads();
  const int n0 = (g.L[0] + BX - 1) / BX, n1 = (g.L[1] + BY - 1) / BY,
            n2 = (g.L[2] + BZ - 1) / BZ;
  const bool even = g.L[0] % BX == 0 && g.L[1] % BY == 0 && g.L[2] % BZ == 0 && g.L[3] % BT == 0;
  // which half of a record this lane reads first, and the sign that the
  // exchange of halves brings to directions 0..2
  const int swap = (tid >> 2) & 1;
  const float sg = swap ? -1.f : 1.f;
  const int h0 = swap * 48, h1 = 48 - h0;
  // this thread's site in the block and the records of its neighbours and
  // backward links, for a block of valid extents be
  int l[4], st, nf[4], nb[4], lb[4];
  bool valid;
  auto place = [&](const int be[4]) {
    l[0] = tid % BX;
    l[1] = (tid / BX) % BY;
    l[2] = (tid / (BX * BY)) % BZ;
    l[3] = tid / (BX * BY * BZ);
    valid = true;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      valid = valid && l[mu] < be[mu];
      l[mu] = min(l[mu], be[mu] - 1);
    }
    const int lstride[4] = {1, BX, BX * BY, BX * BY * BZ};
    st = l[0] + BX * (l[1] + BY * (l[2] + BZ * l[3]));
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      // index of the site in the face boxes of mu (the other coordinates, in order)
      int f = 0, m = 1;
#pragma unroll
      for (int nu = 0; nu < 4; ++nu)
        if (nu != mu) {
          f += l[nu] * m;
          m *= WB::B(nu);
        }
      nf[mu] = l[mu] + 1 < be[mu] ? st + lstride[mu] : WB::face_sp(mu, 1) + f;
      nb[mu] = l[mu] > 0 ? st - lstride[mu] : WB::face_sp(mu, 0) + f;
      lb[mu] = l[mu] > 0 ? mu * NS + st - lstride[mu] : WB::face_lk(mu) + f;
    }
  };
  {
    const int be[4] = {BX, BY, BZ, BT};
    place(be);
  }
  // warp 0 issues the copies, one per lane: lane 0 the spinor interior, 1 +
  // 2 mu + side its faces, 9 + mu the link interiors, 13 + mu the backward
  // link faces
  const bool is_link = lane >= 9, is_face = is_link ? lane >= 13 : lane > 0;
  const int imu = !is_face ? 0 : is_link ? lane - 13 : (lane - 1) >> 1;  // face direction
  const int iside = is_link ? 0 : (lane - 1) & 1;
  const CUtensorMap* imap = (is_link ? maps.lk : maps.sp) + (is_face ? 1 + imu : 0);
  uint32_t ioff = 0;  // destination, bytes from the start of its buffer
  if (is_link) {
    ioff = 48u * uint32_t(is_face ? WB::face_lk_rt(imu) : (lane - 9) * NS);
  } else if (is_face) {
    ioff = 96u * uint32_t(WB::face_sp_rt(imu, iside));
  }
  int it = 0;  // tiles issued and consumed so far: tile `it` in buffer it & 1 (MULTI) or 0
  constexpr int NW = NS / 32;
  double2 spr = make_double2(0.0, 0.0);  // DOT: sums over this CTA's blocks
  double spp = 0.0;
  for (int blk = blockIdx.x; blk < nblocks; blk += gridDim.x) {
    // block origin and valid extents
    int o[4], be[4];
    {
      int b = blk;
      o[0] = (b % n0) * BX;
      b /= n0;
      o[1] = (b % n1) * BY;
      b /= n1;
      o[2] = (b % n2) * BZ;
      o[3] = (b / n2) * BT;
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) be[mu] = min(WB::B(mu), g.L[mu] - o[mu]);
    }
    int ic[4];
    if (tid < 32) {
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) {
        // a face sits at the wrapped coordinate next to the block
        const int lo = o[mu] == 0 ? g.L[mu] - 1 : o[mu] - 1;
        const int hi = o[mu] + be[mu] == g.L[mu] ? 0 : o[mu] + be[mu];
        ic[mu] = is_face && mu == imu ? (iside ? hi : lo) : o[mu];
      }
    }
    // the copies of vector v's spinor tile (and, for v = 0, of the links)
    // as tile k, completing on its buffer's barrier.  Every thread has passed
    // a block barrier since that buffer (and, for v = 0, the links) was read;
    // the fence orders those reads before the copies.
    auto issue = [&](int v, int k) {
      uint64_t* b = MULTI && (k & 1) ? &bar[1] : &bar[0];
      if (lane == 0) {
        fence_proxy_async_smem();
        // (stall, host-set fault injection: waits for bytes that never come)
        mbar_arrive_expect_tx(b, uint32_t(WB::NSP) * 96u +
                                     (v == 0 ? uint32_t(WB::NLK) * 48u : 0u) + (stall ? 16u : 0u));
      }
      __syncwarp();
      if (lane < (v == 0 ? 17 : 9))
        tma_load_5d((is_link ? lk : (k & 1) ? sp1 : sp0) + ioff, imap,
                    (is_link ? 12 : 24) * ic[0], ic[1], ic[2], ic[3],
                    is_link ? (is_face ? imu : lane - 9) : v, b);
    };
    if (tid < 32) issue(0, it);
    if (!even) place(be);
    const int site = (o[0] + l[0]) +
                     g.L[0] * ((o[1] + l[1]) + g.L[1] * ((o[2] + l[2]) + g.L[2] * (o[3] + l[3])));
    const bool tlast = antiperiodic && o[3] + l[3] == g.L[3] - 1;
    const bool tfirst = antiperiodic && o[3] + l[3] == 0;
    // the site's clover, loaded while the first copies are in flight: the
    // block of the first half's chirality, then the other
    float clv[72];
    {
      const float4* a = A + size_t(swap * 9) * g.vol + site;
      const float4* b = A + size_t((1 - swap) * 9) * g.vol + site;
#pragma unroll
      for (int i = 0; i < 9; ++i, a += g.vol, b += g.vol) {
        reinterpret_cast<uint4*>(clv)[i] = ld_early16(a);
        reinterpret_cast<uint4*>(clv)[9 + i] = ld_early16(b);
      }
    }
    for (int v = 0; v < (MULTI ? nvec : 1); ++v, ++it) {
      // the other buffer was last read before the barrier that ended tile it - 1
      if (MULTI && tid < 32 && v + 1 < nvec) issue(v + 1, it + 1);
      const unsigned char* sp = (it & 1) ? sp1 : sp0;
      uint64_t* wb = MULTI && (it & 1) ? &bar[1] : &bar[0];
      const uint32_t ph = uint32_t(MULTI ? it >> 1 : it) & 1u;
      if (!__all_sync(0xffffffffu, mbar_wait(wb, ph))) {
        // the copies did not land within the budget of some lane: its warp
        // records that and leaves as a whole (lanes that left alone would be
        // waited for at the next warp-wide step); the first warp gives the
        // copies in flight (this tile's and the next one's) a second bounded
        // wait.  The block barrier does not count warps that have left.
        if (lane == 0) atomicOr(err, 1);
        if (tid == 0) {
          mbar_wait(wb, ph);
          if (MULTI && v + 1 < nvec)
            mbar_wait((it & 1) ? &bar[0] : &bar[1], uint32_t((it + 1) >> 1) & 1u);
        }
        return;
      }
      cpx<float> ax[6], ay[6];
      // the operands of one hop: both halves of the neighbour and the link's
      // two rows, loaded one hop ahead of their use
      struct Hop {
        uint4 x[3], y[3], k[3];
      };
      auto load_spinor = [&](int rec, Hop& q) {
        const unsigned char* p = sp + size_t(rec) * 96;
#pragma unroll
        for (int i = 0; i < 3; ++i) q.x[i] = reinterpret_cast<const uint4*>(p + h0)[i];
#pragma unroll
        for (int i = 0; i < 3; ++i) q.y[i] = reinterpret_cast<const uint4*>(p + h1)[i];
      };
      auto load_hop = [&](int rec, int link, Hop& q) {
        load_spinor(rec, q);
        const uint4* p = reinterpret_cast<const uint4*>(lk + size_t(link) * 48);
#pragma unroll
        for (int i = 0; i < 3; ++i) q.k[i] = p[i];
      };
      auto hop = [&](auto mu, auto fwd, const Hop& q, bool neg) {
        cpx<float> u[9];
#pragma unroll
        for (int i = 0; i < 3; ++i) reinterpret_cast<uint4*>(u)[i] = q.k[i];
        const float sn = neg ? -1.f : 1.f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int b = (a + 1) % 3, cc = (a + 2) % 3;
          u[6 + a] = sn * conj(u[b] * u[3 + cc] - u[cc] * u[3 + b]);
        }
        hop_halves<decltype(mu)::value, decltype(fwd)::value>(
            u, reinterpret_cast<const cpx<float>*>(q.x),
            reinterpret_cast<const cpx<float>*>(q.y), ax, ay, sg);
      };
      Hop q[2];
      load_spinor(st, q[1]);
      if (MULTI) load_hop(nf[0], st, q[0]);
#pragma unroll
      for (int i = 0; i < 6; ++i) ax[i] = ay[i] = cpx<float>(0.f, 0.f);
      clover_block_accum(clv, diag, reinterpret_cast<const cpx<float>*>(q[1].x), ax);
      clover_block_accum(clv + 36, diag, reinterpret_cast<const cpx<float>*>(q[1].y), ay);
      // (one vector: only now, when the clover's registers are free)
      if (!MULTI) load_hop(nf[0], st, q[0]);
#define GB_BLK_HOP(MU)                                                                \
  load_hop(nb[MU], lb[MU], q[1]);                                                     \
  hop(std::integral_constant<int, MU>{}, std::true_type{}, q[0], MU == 3 && tlast);   \
  if (MU < 3) load_hop(nf[(MU + 1) & 3], (MU + 1) * NS + st, q[0]);                   \
  hop(std::integral_constant<int, MU>{}, std::false_type{}, q[1], MU == 3 && tfirst);
      GB_BLK_HOP(0) GB_BLK_HOP(1) GB_BLK_HOP(2) GB_BLK_HOP(3)
#undef GB_BLK_HOP
      if (valid) {
        unsigned char* op =
            reinterpret_cast<unsigned char*>(out + size_t(v) * vstride + size_t(site) * 12);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          reinterpret_cast<uint4*>(op + h0)[i] = reinterpret_cast<const uint4*>(ax)[i];
          reinterpret_cast<uint4*>(op + h1)[i] = reinterpret_cast<const uint4*>(ay)[i];
        }
      }
      if constexpr (DOT) {
        load_spinor(st, q[0]);
        cpx<float> pr(0.f, 0.f);
        float pp = 0.f;
        if (valid) {
#pragma unroll
          for (int i = 0; i < 6; ++i) {
            cmac_conj(pr, ax[i], reinterpret_cast<const cpx<float>*>(q[0].x)[i]);
            cmac_conj(pr, ay[i], reinterpret_cast<const cpx<float>*>(q[0].y)[i]);
            pp = fmaf(ax[i].re, ax[i].re, fmaf(ax[i].im, ax[i].im, pp));
            pp = fmaf(ay[i].re, ay[i].re, fmaf(ay[i].im, ay[i].im, pp));
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          pr.re += __shfl_xor_sync(0xffffffffu, pr.re, o);
          pr.im += __shfl_xor_sync(0xffffffffu, pr.im, o);
          pp += __shfl_xor_sync(0xffffffffu, pp, o);
        }
        if (MULTI) {
          if (lane == 0) {
            const size_t np = size_t(nblocks) * NW, at = size_t(blk) * NW + (tid >> 5);
            part[size_t(2 * v) * np + at] = make_double2(double(pr.re), double(pr.im));
            part[size_t(2 * v + 1) * np + at] = make_double2(double(pp), 0.0);
          }
        } else if (lane == 0) {
          spr.x += double(pr.re);
          spr.y += double(pr.im);
          spp += double(pp);
        }
      }
      // every thread is done with the tile before the copies of another one
      __syncthreads();
    }
  }
  if (DOT && !MULTI && lane == 0) {
    const size_t np = size_t(gridDim.x) * NW, at = size_t(blockIdx.x) * NW + (tid >> 5);
    part[at] = spr;
    part[np + at] = make_double2(spp, 0.0);
  }
}

// resident CTAs of the device for a kernel at a shared-memory size
template <typename K>
int resident_ctas(K kern, int threads, size_t smem) {
  int dev = 0, sms = 0, per = 0;
  GB_CHECK(cudaGetDevice(&dev));
  GB_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  GB_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem));
  return sms * (per > 0 ? per : 1);
}

// Host side of k_wilson_blk: the five tensor maps of the vectors (`in`, nvec of
// them stored back to back; those of the two-row links and the kernel's
// attributes are the plan's) and the launch.  On small lattices this host work
// is the call: ten maps, two attributes and the occupancy query on every call
// made one 6^4 vector 11.7 us (8.0 now; thread per site 8.5).  nparts (not
// null): with inner products; receives the parts per sum, left in the reduction
// buffer.
template <int BX, int BY, int BZ, int BT, int MINB, int MINM>
void launch_wilson_blk(mg_ctx* c, TilePlan& plan, int* nparts, cpx<float>* out,
                       const cpx<float>* in, const cpx<float>* U12, const float4* A,
                       const Geom& g, float diag, size_t vstride, int nvec, int ap, int* err,
                       cudaStream_t st, int stall) {
  using WB = WilsonBlock<BX, BY, BZ, BT>;
  const cuuint64_t X = g.L[0], Y = g.L[1], Z = g.L[2], T = g.L[3];
  // maps over records of `w` floats: 0 the block, 1 + mu its face in mu
  auto make_maps = [&](CUtensorMap m[5], const void* base, cuuint32_t w, cuuint64_t slices) {
    const cuuint64_t d[5] = {w * X, Y, Z, T, slices}, r = 4 * w;
    const cuuint64_t s[4] = {r * X, r * X * Y, r * X * Y * Z, r * X * Y * Z * T};
    for (int k = 0; k < 5; ++k) {
      cuuint32_t box[5] = {w * BX, BY, BZ, BT, 1};
      if (k > 0) box[k - 1] = k == 1 ? w : 1;
      m[k] = make_map_5d(base, d, s, box);
    }
  };
  std::call_once(plan.links_once, [&] { make_maps(plan.links, U12, 12, 4); });
  WilsonTileMaps m;
  make_maps(m.sp, in, 24, cuuint64_t(nvec));
  std::copy(plan.links, plan.links + 5, m.lk);
  // several vectors: shared memory allows few CTAs, so registers are not
  // held down for more
  auto k = nvec > 1 ? (nparts ? k_wilson_blk<BX, BY, BZ, BT, MINM, true, true>
                              : k_wilson_blk<BX, BY, BZ, BT, MINM, true, false>)
                    : (nparts ? k_wilson_blk<BX, BY, BZ, BT, MINB, false, true>
                              : k_wilson_blk<BX, BY, BZ, BT, MINB, false, false>);
  // several vectors: a second spinor buffer after the links
  const size_t smem =
      size_t(WB::NSP) * 96 * (nvec > 1 ? 2 : 1) + size_t(WB::NLK) * 48;
  const int which = (nvec > 1 ? 2 : 0) + (nparts ? 1 : 0);
  std::call_once(plan.kern_once[which], [&] {
    GB_CHECK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
    GB_CHECK(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                  cudaSharedmemCarveoutMaxShared));
    plan.ctas[which] = resident_ctas(k, WB::NS, smem);
  });
  const int blocks = ceil_div(g.L[0], BX) * ceil_div(g.L[1], BY) * ceil_div(g.L[2], BZ) *
                     ceil_div(g.L[3], BT);
  const int grid = nvec > 1 ? blocks : std::min(blocks, plan.ctas[which]);
  double2* part = nullptr;
  if (nparts) {
    *nparts = grid * (WB::NS / 32);
    part = reduction_parts(c, size_t(*nparts) * 2 * nvec);
  }
  k<<<grid, WB::NS, smem, st>>>(out, A, g, diag, vstride, nvec, ap, blocks, m, err, part, stall);
}

// the tiled form needs extents of at least a block and 16-byte aligned operands
bool wilson_blk_ok(const Geom& g, const int b[4], const void* in, const void* out, const void* U) {
  for (int mu = 0; mu < 4; ++mu)
    if (g.L[mu] < b[mu]) return false;
  return reinterpret_cast<uintptr_t>(in) % 16 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0 &&
         reinterpret_cast<uintptr_t>(U) % 16 == 0;
}
}  // namespace

void fine_operator_build(mg_ctx* c, const void* gauge_ext, cudaStream_t st) {
  Level& L = c->L[0];
  const size_t n = size_t(4) * L.g.vol * 9;
  L.gauge64.alloc(n * sizeof(cpx<double>));
  k_gauge_import<double><<<ceil_div(n, 256), 256, 0, st>>>(
      L.gauge64.as<cpx<double>>(), (const cpx<double>*)gauge_ext, L.g, c->p.t_antiperiodic);
  GB_LAUNCH_CHECK();
  L.clover64.alloc(size_t(L.g.vol) * 72 * sizeof(double));
  float* c32 = nullptr;
  if (L.prec == MG_F32) {
    L.gauge32.alloc(n * sizeof(cpx<float>));
    k_gauge_import<float><<<ceil_div(n, 256), 256, 0, st>>>(
        L.gauge32.as<cpx<float>>(), (const cpx<double>*)gauge_ext, L.g, c->p.t_antiperiodic);
    GB_LAUNCH_CHECK();
    L.clover32.alloc(size_t(L.g.vol) * 72 * sizeof(float));
    c32 = L.clover32.as<float>();
    L.clover32t.alloc(size_t(L.g.vol) * 72 * sizeof(float));
    // two-row link form, used only if every link rebuilds to FP32 precision
    L.gauge12.alloc(size_t(4) * L.g.vol * 6 * sizeof(cpx<float>));
    DevBuf dev;
    dev.alloc(sizeof(unsigned));
    GB_CHECK(cudaMemsetAsync(dev.p, 0, sizeof(unsigned), st));
    int blocks = ceil_div(size_t(4) * L.g.vol, 256);
    if (blocks > 152 * 32) blocks = 152 * 32;
    k_gauge_compress12<<<blocks, 256, 0, st>>>(L.gauge12.as<cpx<float>>(), dev.as<unsigned>(),
                                                (const cpx<double>*)gauge_ext, L.g,
                                                c->p.t_antiperiodic);
    GB_LAUNCH_CHECK();
    unsigned h = 0;
    GB_CHECK(cudaMemcpyAsync(&h, dev.p, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
    GB_CHECK(cudaStreamSynchronize(st));
    float maxdev;
    std::memcpy(&maxdev, &h, sizeof(float));
    L.gauge12_ok = maxdev < 1e-5f;
    c->launches++;
    // 8-real link form (from the FP64 field, boundary sign applied in the kernel)
    L.gauge8.alloc(size_t(4) * L.g.vol * 8 * sizeof(float));
    DevBuf part;
    part.alloc(size_t(blocks) * sizeof(double));
    GB_CHECK(cudaMemsetAsync(dev.p, 0, sizeof(unsigned), st));
    k_gauge_compress8<<<blocks, 256, 0, st>>>(L.gauge8.as<float>(), dev.as<unsigned>(),
                                               part.as<double>(), (const cpx<double>*)gauge_ext,
                                               L.g);
    GB_LAUNCH_CHECK();
    std::vector<double> hp(blocks);
    GB_CHECK(cudaMemcpyAsync(&h, dev.p, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
    GB_CHECK(cudaMemcpyAsync(hp.data(), part.p, size_t(blocks) * sizeof(double),
                             cudaMemcpyDeviceToHost, st));
    GB_CHECK(cudaStreamSynchronize(st));
    std::memcpy(&maxdev, &h, sizeof(float));
    double sq = 0.0;
    for (double v : hp) sq += v;
    L.gauge8_maxdev = maxdev;
    L.gauge8_rmsdev = std::sqrt(sq / (double(n) * 2.0));
    // the rebuild's error grows like 1 / (1 - |a1|^2) on the rare links
    // close to a diagonal matrix: the form is eligible when the deviation is
    // at FP32 rounding size on average and bounded everywhere
    L.gauge8_ok = L.gauge8_rmsdev < 1e-6 && maxdev < 1e-3f;
    c->launches++;
  }
  k_clover<<<ceil_div(L.g.vol, 128), 128, 0, st>>>(L.gauge64.as<cpx<double>>(), L.g, c->p.csw,
                                                    L.clover64.as<double>(), c32,
                                                    L.clover32t.as<float4>());
  GB_LAUNCH_CHECK();
  c->launches += L.prec == MG_F32 ? 3 : 2;
  L.diag = 4.0 + c->p.mass;
}

void wilson_apply(mg_ctx* c, Vec out, Vec in, int nvec, cudaStream_t st, int* nparts) {
  if (nparts) *nparts = 0;
  Level& L = c->L[0];
  GB_REQUIRE(out.prec == in.prec, MG_ERR_ARG, "wilson_apply: precision mismatch");
  GB_REQUIRE(out.p != in.p, MG_ERR_ARG, "wilson_apply: output aliases input");
  const size_t vs = size_t(L.g.vol) * 12;
  dim3 grid(ceil_div(L.g.vol, 128) * nvec);
  // algorithmic bytes per site: spinor in + out (2 x 24 reals) per vector,
  // four links (4 x 18 reals: each link serves two sites) and the clover
  // (72 reals) once for all vectors
  const double bytes =
      double(L.g.vol) * (48.0 * nvec + 144.0) * (out.prec == MG_F64 ? 8 : 4);
  ProfScope ps(c->prof, st, "wilson_clover", 0, bytes, double(nvec) * L.g.vol * 1824.0);
  if (out.prec == MG_F32) {
    // FP32: the autotuner picks one launch policy q:
    //   0 / 1   one vector per thread, stored / two-row links, default registers
    //   2 .. 5  the same with a register budget (minimum CTAs per SM 2, 2, 4, 6)
    //   6 / 7   2 / 4 vectors per thread (links and clover reused in registers)
    //   8 / 9   links (stored / two-row) and clover of 32 sites staged in
    //           shared memory, warps looping over the vectors (nvec >= 4)
    //   10 / 11 8-real links, default registers / at least 4 CTAs per SM
    //   12 .. 15 tiled: a 4x4x4x2 / 4x4x2x2 / 8x2x2x2 / 8x4x2x2 block with
    //           its halo staged in shared memory by tensor copies (two-row
    //           links)
    // Two-row and 8-real policies are candidates only when the field allows
    // them; tiled ones when every extent holds a block (extents it does not
    // divide leave partial blocks).
    GB_REQUIRE(L.gauge32.p, MG_ERR_STATE, "FP32 fine operator not built");
    const unsigned gx = ceil_div(L.g.vol, 128);
    const int ap = c->p.t_antiperiodic;
    const cpx<float>* U18 = L.gauge32.as<cpx<float>>();
    const cpx<float>* U12 = L.gauge12.as<cpx<float>>();
    const cpx<float>* U8 = L.gauge8.as<cpx<float>>();
    const float* A = L.clover32.as<float>();
    const float4* At = L.clover32t.as<float4>();
    const float* Ac = L.clover32t.as<float>();
    auto* o = (cpx<float>*)out.p;
    auto* i = (const cpx<float>*)in.p;
    const float dg = float(L.diag);
    const unsigned gt = ceil_div(L.g.vol, 32);
    int* err = c->status.as<int>() + 1;
    int* np = nullptr;  // (the autotuner times the plain launches)
    int stall = 0;      // (fault injection)
    auto launch = [&](int q) {
      switch (q) {
        case 1: k_wilson<float, 12, 0><<<grid, 128, 0, st>>>(o, i, U12, Ac, L.g, dg, vs, nvec, ap); break;
        case 2: k_wilson<float, 18, 2><<<grid, 128, 0, st>>>(o, i, U18, Ac, L.g, dg, vs, nvec, ap); break;
        case 3: k_wilson<float, 12, 2><<<grid, 128, 0, st>>>(o, i, U12, Ac, L.g, dg, vs, nvec, ap); break;
        case 4: k_wilson<float, 12, 4><<<grid, 128, 0, st>>>(o, i, U12, Ac, L.g, dg, vs, nvec, ap); break;
        case 5: k_wilson<float, 12, 6><<<grid, 128, 0, st>>>(o, i, U12, Ac, L.g, dg, vs, nvec, ap); break;
        case 6: k_wilson_mv<float, 2><<<dim3(gx, nvec / 2), 128, 0, st>>>(o, i, U18, A, L.g, dg, vs); break;
        case 7: k_wilson_mv<float, 4><<<dim3(gx, nvec / 4), 128, 0, st>>>(o, i, U18, A, L.g, dg, vs); break;
        case 8: k_wilson_tile<false><<<gt, 128, 0, st>>>(o, i, U18, A, L.g, dg, vs, nvec, ap); break;
        case 9: k_wilson_tile<true><<<gt, 128, 0, st>>>(o, i, U12, A, L.g, dg, vs, nvec, ap); break;
        case 10: k_wilson<float, 8, 0><<<grid, 128, 0, st>>>(o, i, U8, Ac, L.g, dg, vs, nvec, ap); break;
        case 11: k_wilson<float, 8, 4><<<grid, 128, 0, st>>>(o, i, U8, Ac, L.g, dg, vs, nvec, ap); break;
        case 12: launch_wilson_blk<4, 4, 4, 2, 3, 2>(c, L.tile[0], np, o, i, U12, At, L.g, dg, vs, nvec, ap, err, st, stall); break;
        case 13: launch_wilson_blk<4, 4, 2, 2, 6, 3>(c, L.tile[1], np, o, i, U12, At, L.g, dg, vs, nvec, ap, err, st, stall); break;
        case 14: launch_wilson_blk<8, 2, 2, 2, 6, 3>(c, L.tile[2], np, o, i, U12, At, L.g, dg, vs, nvec, ap, err, st, stall); break;
        case 15: launch_wilson_blk<8, 4, 2, 2, 3, 2>(c, L.tile[3], np, o, i, U12, At, L.g, dg, vs, nvec, ap, err, st, stall); break;
        default: k_wilson<float, 18, 0><<<grid, 128, 0, st>>>(o, i, U18, Ac, L.g, dg, vs, nvec, ap); break;
      }
    };
    std::vector<int> cands = {0, 2};
    if (L.gauge12_ok) cands.insert(cands.end(), {1, 3, 4, 5});
    if (L.gauge8_ok) cands.insert(cands.end(), {10, 11});
    if (L.gauge12_ok) {
      const int blk[4][4] = {{4, 4, 4, 2}, {4, 4, 2, 2}, {8, 2, 2, 2}, {8, 4, 2, 2}};
      for (int k = 0; k < 4; ++k)
        if (wilson_blk_ok(L.g, blk[k], i, o, U12)) cands.push_back(12 + k);
    }
    if (nvec % 2 == 0) cands.push_back(6);
    if (nvec % 4 == 0) cands.push_back(7);
    if (nvec >= 4) {
      cands.push_back(8);
      if (L.gauge12_ok) cands.push_back(9);
    }
    const std::string key = "wilson/v" + std::to_string(L.g.vol) + "/n" + std::to_string(nvec) +
                            "/c" + std::to_string(int(L.gauge12_ok));
    int q = Tuner::get().choose(key, cands, st, launch);
    if (nparts && (q < 12 || q > 15)) {
      // the inner products come with a tiled launch; after another one they are a
      // pass of their own, at least its launches and half of its reads longer
      // (16^3x8: the plain kernel won by 0.1 us, the MR step lost 5)
      const float pass_ms = 3e-3f + 96.f * float(nvec) * float(L.g.vol) / 6.8e9f;
      const int t = Tuner::get().within(key, 12, 15, pass_ms);
      if (std::find(cands.begin(), cands.end(), t) != cands.end()) q = t;
    }
    np = nparts;
    if (q >= 12 && q <= 15) stall = take_fault(c->inject_tile_stall);
    launch(q);
  } else {
    k_wilson<double, 18, 0><<<grid, 128, 0, st>>>(
        (cpx<double>*)out.p, (const cpx<double>*)in.p, L.gauge64.as<cpx<double>>(),
        L.clover64.as<double>(), L.g, L.diag, vs, nvec, c->p.t_antiperiodic);
  }
  GB_LAUNCH_CHECK();
  c->launches++;
}

}  // namespace gbmg
