// Galerkin product of the FP32 Wilson-clover level (Sec. 3.4 step 4) with the
// contractions P^dag T on the 5th-generation tensor cores at FP32 accuracy.
//
// For output block d of coarse site xc (see galerkin.cu):
//   out[(s,i),(s',j)] = sum_{x, a in chi s} conj(P(x)[a][i]) T(x)[a][(s',j)],
// T(x) = sum_e H_e(x) P(x + e).  The contractions are four fifths of the
// arithmetic (331,776 of 423,072 flop per fine site at Nv = 24, 4^4
// aggregates); on the FP32 pipe they bound the build (k_galerkin_chunk: 62 %
// issue, shared-memory reads as busy as the FMA pipe).  Here CUDA-core warps
// only form T; the contractions are real GEMMs
//   D_s[T rows][P rows] += sum_k A_s[T row][k] B_s[P row][k],   k = (site, a),
// T rows 2 c, 2 c + 1 = Re, Im of column c, P rows i, Nv + i = Re, Im of
// vector i: every product of the four a complex multiply needs, none twice.
//
// Accuracy: every FP32 operand v is split into three BF16 numbers, each the
// rounding of what the ones before it leave: 3 x 8 bits, so that their sum is v
// itself (BF16 has FP32's exponents: entries of any size, down to 2^-110).  Six
// products hold v w to 2^-26 of it: hi hi in one accumulator; hi mid, mid hi, hi
// lo, mid mid, lo hi, 2^-8 of it and less, in another.  (FP16 pairs held an
// operand to 2^-23, and numbers below 2^-13 to a fixed 2^-36: with vectors 1e-6
// of the others at the faces of their aggregate, face blocks were 0.1 to 0.3 of
// their norm off.)  The accumulators run over a unit of one chunk of eight sites
// (3 steps of K = 16) on the X blocks, of two on the face blocks, and are then
// added to FP32 registers: the tensor cores truncate when they accumulate, and on
// the X blocks, whose sums have one sign, that bias grows with the unit.
// Relative error of the links against 64 bits, 24 vectors (the FP32 pipe's own
// sums in brackets): Gaussian vectors 1.2e-7 on 2^4 [2.1e-7] and 1.3e-7 on 4^4
// [7.7e-7] aggregates; one site of each 2x4^3 aggregate large and the others 1e-3
// of it, 1.9e-7 [1.1e-6]; sites at the faces 1e-6 of the inner ones, worst face
// block 1.4e-7 [5.3e-7].  Units of two chunks on the X blocks too: 1.6e-7 on 4^4,
// 0.5 % faster; of one everywhere: 1.5 % slower.
//
// What bounds it now: the T warps, on the latency of the P and link gathers
// (issue 46 %, long-scoreboard stalls; the tensor pipe is 14 % busy).  24^3x48,
// Nv = 24, 4^4 aggregates, 281 GFLOP: 9.21 -> 5.43 ms (FP16 pairs 5.25: the third
// piece's conversions and stores), the call with its export 9.67 -> 5.89 ms.
// Two-row links with two hops loaded ahead were slower (spills).
// One resident CTA per SM walks its (xc, d) blocks, X blocks first.  Roles:
// 16 Nv T threads, one column of one of the chunk's 8 sites each (Nv = 24:
// 12 warps), writing the split operands into a ring of kRing stages; one
// thread issuing the 36 MMAs of a chunk; warps 0.. adding finished units from
// TMEM (two sets of accumulators in turn) and storing the block.  Every wait
// is bounded: the role whose time runs out sets the error word and the CTA's
// abort flag, which every waiting role reads, whole warps decide together
// (wait_or_abort_warp), the MMAs in flight are waited for (bounded), TMEM is
// freed and the CTA leaves.
#include <cuda_bf16.h>

#include <algorithm>

#include "kernels.cuh"
#include "tcgen05.cuh"
#include "wilson_ops.cuh"

namespace gbmg {

namespace {

constexpr int kCh = 8;         // fine sites per chunk: K = 48 per chirality
constexpr int kRing = 2;       // operand stages (a third does not fit)
constexpr int kMaxPer = 512;   // fine sites per aggregate (the site tables)
constexpr int kUnitX = 1, kUnitY = 2;  // chunks accumulated in TMEM, X and face blocks

template <int NV>
struct GM {
  static constexpr int N = 2 * NV;                 // P rows
  static constexpr int TT = 16 * NV;               // T threads
  static constexpr int NTW = TT / 32;              // T warps
  static constexpr int THREADS = 128 + TT;
  static constexpr int ND = (4 * NV + 31) / 32;    // warps that drain
  static constexpr uint32_t LBO = 128, SBO = 6 * 128 + 16;  // +16: fewer bank conflicts
  // (the MMA's T rows from 4 NV to 128 read on into the next operand; their
  // accumulator rows are never read)
  static constexpr uint32_t ASZ = uint32_t(NV / 2) * SBO, BSZ = uint32_t(N / 8) * SBO;
  static constexpr uint32_t STAGE = 6 * ASZ + 6 * BSZ;
  static constexpr uint32_t TMEM = N * 8 <= 256 ? 256 : 512;
  static constexpr size_t SMEM = size_t(kRing) * STAGE + kMaxPer * (8 + 16);
  static_assert(16 * SBO <= ASZ + BSZ * 6, "the last T operand's rows end inside the stage");
  static_assert(N * 8 <= 512 && TT % 32 == 0 && N % 16 == 0 && ND <= 3, "tile shape");
};

struct GalMap {
  Geom fine, coarse;
  int b[4];
  int per;
  // the last round of X blocks has `rem`, so `spare` CTAs go without; those take
  // the first `some` face blocks
  int rem, spare, some;
};

// two numbers as three BF16 pairs: w[0] + w[1] + w[2] is each of them exactly
__device__ __forceinline__ void split3(float a, float b, uint32_t (&w)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    w[k] = *reinterpret_cast<const uint32_t*>(&h);
    a -= __uint_as_float(w[k] << 16);
    b -= __uint_as_float(w[k] & 0xffff0000u);
  }
}

template <int E>
struct HopIdx {
  static constexpr int value = E;
};

// Column j of chirality SP of the diagonal block's T(x): the clover block and
// the hops that stay inside the aggregate (bit e - 1 of `leave` clear), the
// next hop's operands loaded while the current one is applied.  v0 receives
// P(x)'s six entries of the column.
template <int SP>
__device__ __forceinline__ void t_column_x(const cpx<float>* __restrict__ U,
                                           const float* __restrict__ A, float diag,
                                           const cpx<float>* __restrict__ Vp, const Geom& g,
                                           int nv, int x, int leave, int j, cpx<float> o[12],
                                           cpx<float> v0[6]) {
  auto load_v = [&](int y, cpx<float> v[6]) {
    const cpx<float>* src = Vp + (size_t(y) * 12 + 6 * SP) * nv + j;
#pragma unroll
    for (int a = 0; a < 6; ++a) v[a] = src[a * nv];
  };
  auto load_u = [&](int mu, int s, cpx<float> u[9]) {
    const cpx<float>* p = U + (size_t(mu) * g.vol + s) * 9;
#pragma unroll
    for (int k = 0; k < 9; ++k) u[k] = p[k];
  };
  // partner of hop e; the site itself when the hop leaves (its operands are
  // loaded but not used)
  auto partner = [&](int e) {
    const int st = g.stride[(e - 1) >> 1];
    return (leave >> (e - 1)) & 1 ? x : ((e & 1) ? x + st : x - st);
  };
#pragma unroll
  for (int a = 0; a < 12; ++a) o[a] = cpx<float>(0.f, 0.f);
  load_v(x, v0);
  cpx<float> v[6], u[9];
  load_v(partner(1), v);
  load_u(0, x, u);
  clover_block_accum(A + size_t(x) * 72 + 36 * SP, diag, v0, o + 6 * SP);
  auto step = [&](auto ic) {
    constexpr int E = decltype(ic)::value;
    constexpr int MU = (E - 1) >> 1;
    constexpr bool FWD = (E & 1) == 1;
    cpx<float> vn[6], un[9];
    if constexpr (E < 8) {
      const int y = partner(E + 1);
      load_v(y, vn);
      load_u(E >> 1, (E & 1) == 0 ? x : y, un);  // hop E + 1 is forward when E is even
    }
    if (!((leave >> (E - 1)) & 1)) {
      cpx<float> psi[12];
#pragma unroll
      for (int a = 0; a < 6; ++a) {
        psi[6 * SP + a] = v[a];
        psi[6 * (1 - SP) + a] = cpx<float>(0.f, 0.f);
      }
      hop_accum<MU, FWD>(u, psi, o);
    }
    if constexpr (E < 8) {
#pragma unroll
      for (int a = 0; a < 6; ++a) v[a] = vn[a];
#pragma unroll
      for (int k = 0; k < 9; ++k) u[k] = un[k];
    }
  };
  step(HopIdx<1>{});
  step(HopIdx<2>{});
  step(HopIdx<3>{});
  step(HopIdx<4>{});
  step(HopIdx<5>{});
  step(HopIdx<6>{});
  step(HopIdx<7>{});
  step(HopIdx<8>{});
}

// Column j of chirality SP of a face block's T(x): the hop d alone, to y.
template <int SP>
__device__ __forceinline__ void t_column_y(const cpx<float>* __restrict__ U,
                                           const cpx<float>* __restrict__ Vp, const Geom& g,
                                           int nv, int x, int y, int d, int j, cpx<float> o[12],
                                           cpx<float> v0[6]) {
  const int mu = (d - 1) >> 1;
  const bool fwd = (d & 1) == 1;
  cpx<float> v[6], u[9];
  const cpx<float>* s0 = Vp + (size_t(x) * 12 + 6 * SP) * nv + j;
  const cpx<float>* s1 = Vp + (size_t(y) * 12 + 6 * SP) * nv + j;
  const cpx<float>* p = U + (size_t(mu) * g.vol + (fwd ? x : y)) * 9;
#pragma unroll
  for (int a = 0; a < 6; ++a) v[a] = s1[a * nv];
#pragma unroll
  for (int k = 0; k < 9; ++k) u[k] = p[k];
#pragma unroll
  for (int a = 0; a < 6; ++a) v0[a] = s0[a * nv];
  cpx<float> psi[12];
#pragma unroll
  for (int a = 0; a < 6; ++a) {
    psi[6 * SP + a] = v[a];
    psi[6 * (1 - SP) + a] = cpx<float>(0.f, 0.f);
  }
#pragma unroll
  for (int a = 0; a < 12; ++a) o[a] = cpx<float>(0.f, 0.f);
  hop_accum_rt(mu, fwd, u, psi, o);
}

// Sec. 3.4 step 4: P^dag M P into the nine blocks of Eq. (3).
template <int NV, bool DEAL>
__global__ void __launch_bounds__(GM<NV>::THREADS, 1)
    k_galerkin_mma(const cpx<float>* __restrict__ U, const float* __restrict__ A, float diag,
                   const cpx<float>* __restrict__ Vp, GalMap m,
                   cpx<float>* __restrict__ out, int* __restrict__ err, int stall) {
  using G = GM<NV>;
  constexpr int N = G::N;
  extern __shared__ __align__(128) unsigned char sm[];
  // per aggregate-local site: offset from the aggregate's first site, leave
  // flags (bit e - 1: hop e leaves); then the sites of the eight faces
  int2* tab = reinterpret_cast<int2*>(sm + size_t(kRing) * G::STAGE);
  unsigned short* face = reinterpret_cast<unsigned short*>(tab + kMaxPer);
  __shared__ uint64_t full[kRing], empty[kRing], dfull[2], dempty[2], fin, stall_bar;
  __shared__ uint32_t tmem_sh;
  __shared__ volatile int abort_sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    tmem_alloc(&tmem_sh, G::TMEM);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int i = 0; i < kRing; ++i) {
      mbar_init(&full[i], G::NTW);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&dfull[i], 1);
      mbar_init(&dempty[i], G::ND);
    }
    mbar_init(&fin, 1);
    mbar_init(&stall_bar, 1);  // the injected stall's barrier; never arrived at
    fence_mbar_init();
    abort_sh = 0;
  }
  for (int ls = tid; ls < m.per; ls += G::THREADS) {
    int q = ls, off = 0, leave = 0, c[4];
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      c[mu] = q % m.b[mu];
      q /= m.b[mu];
      off += c[mu] * m.fine.stride[mu];
      leave |= (c[mu] == m.b[mu] - 1 ? 1 : 0) << (2 * mu);
      leave |= (c[mu] == 0 ? 1 : 0) << (2 * mu + 1);
    }
    tab[ls] = make_int2(off, leave);
    int base = 0;  // face lists in hop order, the other coordinates in order
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      int f = 0, mul = 1;
#pragma unroll
      for (int nu = 0; nu < 4; ++nu)
        if (nu != mu) {
          f += c[nu] * mul;
          mul *= m.b[nu];
        }
      if ((leave >> (2 * mu)) & 1) face[base + f] = (unsigned short)ls;
      if ((leave >> (2 * mu + 1)) & 1) face[base + mul + f] = (unsigned short)ls;
      base += 2 * mul;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_sh;
  const int cvol = m.coarse.vol, items = 9 * cvol;
  // block d of coarse site xc: items 0..cvol-1 are the X blocks, then the
  // eight face blocks of each site
  auto item_d = [&](int it) { return it < cvol ? 0 : 1 + ((it - cvol) & 7); };
  auto item_xc = [&](int it) { return it < cvol ? it : (it - cvol) >> 3; };
  // A role's walk over the CTA's blocks, dealt out round robin.  DEAL: X blocks
  // round robin; on the CTAs that got one X block less, their share of the first
  // m.some face blocks; then all others round robin.
  auto rest = [&] {
    const int turn = int(blockIdx.x) - m.rem;
    return cvol + m.some + (turn < 0 ? turn + int(gridDim.x) : turn);
  };
  auto faces = [&] {
    const int y = cvol + int(blockIdx.x) - m.rem;
    return y >= cvol && y < cvol + m.some ? y : rest();
  };
  auto first_item = [&] {
    return !DEAL || int(blockIdx.x) < cvol ? int(blockIdx.x) : faces();
  };
  auto next_item = [&](int it) {
    if (!DEAL || it >= cvol + m.some) return it + int(gridDim.x);
    if (it < cvol) return it + int(gridDim.x) < cvol ? it + int(gridDim.x) : faces();
    return it + m.spare < cvol + m.some ? it + m.spare : rest();
  };
  auto face_b = [&](int d) {
    const int mu = (d - 1) >> 1;
    return mu == 0 ? m.b[0] : mu == 1 ? m.b[1] : mu == 2 ? m.b[2] : m.b[3];
  };
  auto item_cnt = [&](int d) { return d == 0 ? m.per : m.per / face_b(d); };
  auto item_unit = [&](int d) { return d == 0 ? kUnitX : kUnitY; };  // chunks per unit

  if (warp >= 4) {
    // ---------------------------------------------------------- T threads
    const int t = tid - 128;
    // two sites side by side in a warp: their operand words fill each other's gaps,
    // 8-byte stores without bank conflicts (one column after the other: half of
    // the banks unused, 5.55 instead of 5.43 ms)
    const int sp = t / (kCh * NV), pair = (t / (2 * NV)) % (kCh / 2);
    const int sl = 2 * pair + (t & 1), j = (t % (2 * NV)) >> 1;
    const int col = sp * NV + j;
    // operand offsets of this thread's three k pairs.  The order of k is free as
    // long as both operands have the same: site sl's first two pairs are k = 4 sl
    // .. 4 sl + 3, one 8-byte word, its third k = 32 + 2 sl.
    const uint32_t ko8 = uint32_t((sl >> 1) * 128 + (sl & 1) * 8);
    const uint32_t ko4 = uint32_t((4 + (sl >> 2)) * 128 + (sl & 3) * 4);
    auto ro = [&](int row) { return uint32_t((row >> 3) * G::SBO + (row & 7) * 16); };
    const uint32_t ra = ro(2 * col), rai = ro(2 * col + 1), rb = ro(j), rbi = ro(NV + j);
    int q = 0;
    bool ok = true;
    for (int it = first_item(); it < items && ok; it = next_item(it)) {
      const int d = item_d(it), xc = item_xc(it), cnt = item_cnt(d);
      int cc[4];
      site_coords(m.coarse, xc, cc);
      int x0 = 0;
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) x0 += cc[mu] * m.b[mu] * m.fine.stride[mu];
      const int dmu = d > 0 ? (d - 1) >> 1 : 0;
      const bool dfwd = (d & 1) == 1;
      // the hop d from the face: one step, or the wrap at the lattice's edge
      int hop = 0, fbase = 0;
      if (d > 0) {
#pragma unroll
        for (int mu = 0; mu < 4; ++mu)
          if (mu == dmu) {
            const int st = m.fine.stride[mu], wrap = (m.fine.L[mu] - 1) * st;
            hop = dfwd ? (cc[mu] == m.coarse.L[mu] - 1 ? -wrap : st) : (cc[mu] == 0 ? wrap : -st);
            fbase += dfwd ? 0 : m.per / m.b[mu];
          } else if (mu < dmu) {
            fbase += 2 * (m.per / m.b[mu]);
          }
      }
      for (int k0 = 0; k0 < cnt; k0 += kCh, ++q) {
        const int sidx = k0 + sl;
        cpx<float> o[12], v0[6];
        if (sidx < cnt) {
          const int ls = d == 0 ? sidx : face[fbase + sidx];
          const int2 e = tab[ls];
          const int x = x0 + e.x;
          if (d == 0) {
            if (sp == 0)
              t_column_x<0>(U, A, diag, Vp, m.fine, NV, x, e.y, j, o, v0);
            else
              t_column_x<1>(U, A, diag, Vp, m.fine, NV, x, e.y, j, o, v0);
          } else {
            if (sp == 0)
              t_column_y<0>(U, Vp, m.fine, NV, x, x + hop, d, j, o, v0);
            else
              t_column_y<1>(U, Vp, m.fine, NV, x, x + hop, d, j, o, v0);
          }
        } else {  // past the last site: zeros in both operands
#pragma unroll
          for (int a = 0; a < 12; ++a) o[a] = cpx<float>(0.f, 0.f);
#pragma unroll
          for (int a = 0; a < 6; ++a) v0[a] = cpx<float>(0.f, 0.f);
        }
        const int sg = q % kRing;
        if (q >= kRing &&
            !wait_or_abort_warp(&empty[sg], uint32_t(q / kRing - 1) & 1u, &abort_sh, err)) {
          ok = false;
          break;
        }
        unsigned char* st = sm + size_t(sg) * G::STAGE;
        // rows r (real parts) and ri (imaginary parts) of an operand's three
        // pieces, sz bytes apart
        auto put = [&](unsigned char* base, uint32_t sz, uint32_t r, uint32_t ri,
                       const cpx<float>* v) {
#pragma unroll
          for (int im = 0; im < 2; ++im) {
            uint32_t w[3][3];  // [pair][piece]
#pragma unroll
            for (int p = 0; p < 3; ++p)
              split3(im ? v[2 * p].im : v[2 * p].re, im ? v[2 * p + 1].im : v[2 * p + 1].re, w[p]);
            unsigned char* row = base + (im ? ri : r);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              *reinterpret_cast<uint2*>(row + k * sz + ko8) = make_uint2(w[0][k], w[1][k]);
              *reinterpret_cast<uint32_t*>(row + k * sz + ko4) = w[2][k];
            }
          }
        };
        put(st, G::ASZ, ra, rai, o);
        put(st + 3 * G::ASZ, G::ASZ, ra, rai, o + 6);
        put(st + 6 * G::ASZ + 3 * sp * G::BSZ, G::BSZ, rb, rbi, v0);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&full[sg]);
      }
    }
  } else if (warp == 3) {
    // ---------------------------------------------------------- MMA issue
    if (lane == 0) {
      constexpr uint32_t idesc = mma_idesc(128, N, true);
      int q = 0, w = 0;
      // (fault injection, host-set: waits for what never comes)
      bool ok = !stall || wait_or_abort(&stall_bar, 0u, &abort_sh, err);
      for (int it = first_item(); it < items && ok; it = next_item(it)) {
        const int nch = (item_cnt(item_d(it)) + kCh - 1) / kCh, unit = item_unit(item_d(it));
        for (int c = 0; c < nch && ok; ++c, ++q) {
          const int set = w & 1;
          const bool first = c % unit == 0;
          if (first && w >= 2)
            ok = wait_or_abort(&dempty[set], uint32_t((w >> 1) - 1) & 1u, &abort_sh, err);
          const int sg = q % kRing;
          ok = ok && wait_or_abort(&full[sg], uint32_t(q / kRing) & 1u, &abort_sh, err);
          if (!ok) break;
          tc_fence_after();
          const uint32_t st = smem_u32(sm + size_t(sg) * G::STAGE);
          const uint32_t dmain = tmem + uint32_t(set) * 4 * N, dsmall = dmain + 2 * N;
#pragma unroll
          for (int chi = 0; chi < 2; ++chi)
#pragma unroll
            for (int ks = 0; ks < 3; ++ks) {
              const uint32_t a0 = st + (chi * 3) * G::ASZ + ks * 256;
              const uint32_t b0 = st + 6 * G::ASZ + (chi * 3) * G::BSZ + ks * 256;
              uint64_t a[3], b[3];
#pragma unroll
              for (int k = 0; k < 3; ++k) {
                a[k] = smem_desc(a0 + k * G::ASZ, G::LBO, G::SBO);
                b[k] = smem_desc(b0 + k * G::BSZ, G::LBO, G::SBO);
              }
              const uint32_t acc = (first && ks == 0) ? 0u : 1u;
              mma_f16(dsmall + chi * N, a[0], b[2], idesc, acc);
              mma_f16(dsmall + chi * N, a[1], b[1], idesc, 1u);
              mma_f16(dsmall + chi * N, a[2], b[0], idesc, 1u);
              mma_f16(dsmall + chi * N, a[0], b[1], idesc, 1u);
              mma_f16(dsmall + chi * N, a[1], b[0], idesc, 1u);
              mma_f16(dmain + chi * N, a[0], b[0], idesc, acc);
            }
          mma_commit(&empty[sg]);
          if (c % unit == unit - 1 || c == nch - 1) {
            mma_commit(&dfull[set]);
            ++w;
          }
        }
      }
      // every MMA issued has finished before TMEM and shared memory go
      mma_commit(&fin);
      mbar_wait(&fin, 0u);
    }
    __syncwarp();
  } else if (warp < G::ND) {
    // ---------------------------------------------------------- drain
    const uint32_t tl = tmem + (uint32_t(warp * 32) << 16);
    const int row = warp * 32 + lane;  // T row: column row / 2, re or im
    const bool odd = row & 1;
    int w = 0;
    bool ok = true;
    for (int it = first_item(); it < items && ok; it = next_item(it)) {
      const int d = item_d(it), xc = item_xc(it);
      const int unit = item_unit(d), nun = ((item_cnt(d) + kCh - 1) / kCh + unit - 1) / unit;
      float acc[2 * N];
#pragma unroll
      for (int i = 0; i < 2 * N; ++i) acc[i] = 0.f;
      for (int un = 0; un < nun; ++un, ++w) {
        const int set = w & 1;
        if (!wait_or_abort_warp(&dfull[set], uint32_t(w >> 1) & 1u, &abort_sh, err)) {
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int i = 0; i < 2 * N; i += 16) {
          float v[16];
          tmem_ld16(tl + uint32_t(set) * 4 * N + i, v);
#pragma unroll
          for (int k = 0; k < 16; ++k) acc[i + k] += v[k];
          tmem_ld16(tl + uint32_t(set) * 4 * N + 2 * N + i, v);
#pragma unroll
          for (int k = 0; k < 16; ++k) acc[i + k] += v[k];
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&dempty[set]);
      }
      if (!ok) break;
      // re = Tr.Pr + Ti.Pi (even lane), im = Ti.Pr - Tr.Pi (odd lane); then
      // the even lane stores output row i, the odd one row i + 1
      float* dst = reinterpret_cast<float*>(out + (size_t(xc) * 9 + d) * N * N +
                                            size_t(row >> 1) * N);
#pragma unroll
      for (int chi = 0; chi < 2; ++chi)
#pragma unroll
        for (int i = 0; i < NV; i += 2) {
          float r[2];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const float pr = acc[chi * N + i + k], pi = acc[chi * N + NV + i + k];
            const float other = __shfl_xor_sync(0xffffffffu, pi, 1);
            r[k] = odd ? pr - other : pr + other;
          }
          const float give = odd ? r[0] : r[1];
          const float got = __shfl_xor_sync(0xffffffffu, give, 1);
          const float2 z = odd ? make_float2(got, r[1]) : make_float2(r[0], got);
          if (row < 4 * NV)
            *reinterpret_cast<float2*>(dst + 2 * (chi * NV + i + (odd ? 1 : 0))) = z;
        }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, G::TMEM);
}

template <int NV>
void launch_galerkin_mma(mg_ctx* c, const Level& F, GalMap m, cpx<float>* out, int* err,
                         cudaStream_t st) {
  int dev = 0, sms = 0;
  GB_CHECK(cudaGetDevice(&dev));
  GB_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int items = 9 * m.coarse.vol, grid = items < sms ? items : sms;
  // An X block costs as much as 1.8 face blocks per chunk of sites (4^4 aggregates:
  // 133 us against 18 for 16 vectors, 150 against 22 for 24), so with few rounds of
  // large ones the CTAs that got one less are given face blocks for it: 189 coarse
  // sites, 16 vectors, 449 -> 373 us.  From about four rounds on, and on small
  // aggregates, the plain order is as even and 1 to 5 % faster.
  int xch = ceil_div(m.per, kCh), ych = 0;
  for (int mu = 0; mu < 4; ++mu) ych += 2 * ceil_div(m.per / m.b[mu], kCh);
  m.rem = m.coarse.vol % grid;
  m.spare = m.rem ? grid - m.rem : 0;
  m.some = std::min(8 * m.coarse.vol, m.spare * std::max(1, int(1.8 * 8 * xch / ych + 0.5)));
  auto k = m.per >= 64 && m.coarse.vol < 4 * grid ? k_galerkin_mma<NV, true>
                                                  : k_galerkin_mma<NV, false>;
  GB_CHECK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(GM<NV>::SMEM)));
  k<<<grid, GM<NV>::THREADS, GM<NV>::SMEM, st>>>(
      F.gauge32.as<cpx<float>>(), F.clover32.as<float>(), float(F.diag), F.Vp.as<cpx<float>>(), m,
      out, err, take_fault(c->inject_galerkin_stall));
  GB_LAUNCH_CHECK();
}

}  // namespace

bool galerkin_mma(mg_ctx* c, int level, cudaStream_t st) {
  const Level& F = c->L[level];
  const Level& C = c->L[level + 1];
  // FP32 Wilson-clover level with SU(3) links, 16 or 24 vectors
  if (level != 0 || F.vprec != MG_F32 || C.vprec != MG_F32 || !F.gauge12_ok) return false;
  if (F.nvec != 16 && F.nvec != 24) return false;
  GalMap m;
  m.fine = F.g;
  m.coarse = C.g;
  for (int i = 0; i < 4; ++i) m.b[i] = F.block[i];
  m.per = F.g.vol / C.g.vol;
  if (m.per > kMaxPer) return false;
  int* err = c->status.as<int>() + 1;
  if (F.nvec == 24)
    launch_galerkin_mma<24>(c, F, m, C.links.as<cpx<float>>(), err, st);
  else
    launch_galerkin_mma<16>(c, F, m, C.links.as<cpx<float>>(), err, st);
  return true;
}

}  // namespace gbmg
