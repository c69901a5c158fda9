// The FP64 form's volume M2L (Sec. 5.3 item 3) on the tensor cores, to FP64 accuracy: the lattice
// convolution of m2l_tc.cu (parity sub-images, shifts, windows, real 2p x 2p translation matrices)
// with the exact digit products of p2p_f64.cu.  On the FP64 units the 2.2e6 pairs of a 1024^2
// grid took 3623 us, half of it log, atan2, division and the powers of every pair's offset.
//
// Operands.  A cell's 2p real inputs (M~_k times 2^c_k, c_k = k / 2 + log2 k, which brings the
// scaled multipoles, |M~_k| <= 2^(-k/2) / k sum |w|, to one size) are cut into seven signed 9-bit digits
// below the cell's own exponent; the matrices, columns times 2^-c_k and each output row by a power of
// two that brings its largest entry over all offsets below 1, likewise.  K = 32 inputs of two
// digits fill one 128-byte row: four row images, and four row sets per B block.  A shift's products
// of one order sum at most seven terms of K <= 32 products below 2^16, below 2^24: exact.  The
// orders of a shift are joined in int64 and added up per target in a unit of the target's own
// (p2p_f64.cu), one rounding to FP64 at the end.
//
// A CTA takes 128 flattened targets and two of the four parity classes (N = 2 W, so that seven
// orders fit TMEM), and sweeps the shifts that hold an offset of either class.  Parts of the shifts
// write L~ images of their own, which a last kernel adds.
//
// Bound by the epilogue, as the near field (p2p_f64.cu): the tensor pipe is active 23% of the 268 us of a
// 1024^2 grid, DRAM 1%, and a scheduler's two epilogue warps wait for TMEM reads, conversions and each
// other's 64-bit chains.
#include <algorithm>
#include <array>
#include <cmath>
#include <complex>
#include <vector>

#include "handle.cuh"
#include "oz.cuh"
#include "tc.cuh"

namespace fmmpc {

namespace {

constexpr int OZM_WROWS = 144;  // window: 128 targets, shifts of -4 .. 4, alignment
constexpr int OZM_WPAIR = OZM_WROWS * 128;  // one digit pair's window
constexpr int OZM_WBYTES = 4 * OZM_WPAIR;
constexpr int OZM_NWIN = 2;
constexpr int OZM_TAIL = 384;   // zero rows after each sub-image
constexpr int OZM_MAXPART = 4;
constexpr int OZM_MAXSH = 255;
constexpr int OZM_THREADS = 352;  // window producer, MMA issuer, eight epilogue warps, B producer

template <int W>
struct OzmShape {
  static constexpr int N = 2 * W;
  static constexpr int BPAIR = N * 128;       // one digit pair of a shift's B block
  static constexpr int BBYTES = 4 * BPAIR;
  static constexpr int NB = W == 24 ? 3 : 2;  // B slots
  static constexpr int SMEM = OZM_NWIN * OZM_WBYTES + NB * BBYTES + 1024;
};

struct OzmArgs {
  const unsigned char *img;   // [nrhs][4 digit pairs][rows][128 B]
  const int2 *lexp;           // [nrhs][rows] exponent and L1 norm (see p2p_f64.cu)
  const unsigned char *bmat;  // [shift][4 digit pairs][2 W][128 B], the shifts of class pair 0, then of 1
  const int2 *tiles;          // (level, f0)
  const int4 *shifts;         // (source parity, dy, dx, flags) in that order; flags: 1 the first shift of a
                              // (source parity, dy) group, 2 << h: class h of the pair has an offset
  cpx<double> *L;             // [part][nrhs][ncell][p]
  int64_t rows, ncell, part_stride;
  int *err;
  int64_t lev_row0[24];
  int lev_P[24];
  int part_s[2][OZM_MAXPART + 1];  // shifts of each class pair's parts
  int rb[34];                 // exponent of each output row
  int p, n;
};

// power-of-two scale of coefficient k
__host__ __device__ __forceinline__ int ozm_col(int k) {
  int lg = 0;
  while ((2 << lg) <= k) ++lg;
  return k / 2 + lg;
}

// Digit rows of the multipoles: eight lanes per (rhs, cell at level >= 2); lane c forms inputs
// 8 (c % 4) .. + 7 and writes them as 16-byte chunk c (digit 2 pair + c / 4) of the cell's four rows.
__global__ void k_m2l_oz_pack(OzmArgs a, int nrhs, int64_t ncell_lo, int64_t ncell_hi, const cpx<double> *__restrict__ Mv,
                              unsigned char *__restrict__ img, int2 *__restrict__ lexp) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t per = (ncell_hi - ncell_lo) * 8;
  const bool in = t < (int64_t)nrhs * per;  // every lane takes part in the shuffles
  const int64_t rhs = in ? t / per : 0, rem = in ? t % per : 0;
  const int64_t gidx = ncell_lo + rem / 8;
  const int c = (int)(rem % 8);
  const double *M = reinterpret_cast<const double *>(Mv + (rhs * a.ncell + gidx) * a.p);
  double x[8];
  unsigned long long mx = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int v = 8 * (c & 3) + q;
    x[q] = v < 2 * a.p && in ? ldexp(M[v], ozm_col(v >> 1)) : 0.0;
    mx = max(mx, oz_bits(x[q]));
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const int em = oz_biased(mx);
  uint32_t pk[4][4];  // [pair][two digits a word]
  float l1 = 0.0f;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    int d[OZ_S];
    oz_digits(oz_fixed(x[q], em, l1), d);
#pragma unroll
    for (int pr = 0; pr < 4; ++pr) {
      const int dg = (c >> 2) ? (2 * pr + 1 < OZ_S ? d[2 * pr + 1 < OZ_S ? 2 * pr + 1 : 0] : 0) : d[2 * pr];
      const uint32_t hv = __half_as_ushort(__int2half_rn(dg));
      if (q & 1) pk[pr][q >> 1] |= hv << 16;
      else pk[pr][q >> 1] = hv;
    }
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) l1 += __shfl_xor_sync(0xffffffffu, l1, o);
  if (!in) return;
  int l = 2;
  while (level_offset(l + 1) <= gidx) ++l;
  int cx, cy;
  morton_decode((uint32_t)(gidx - level_offset(l)), cx, cy);
  const int P = a.lev_P[l], q = (cx & 1) + 2 * (cy & 1);
  const int64_t f = (int64_t)((cy >> 1) + 4) * P + (cx >> 1) + 4;
  const int64_t row = a.lev_row0[l] + (int64_t)q * ((int64_t)P * P + OZM_TAIL) + f;
  if (c == 0) lexp[rhs * a.rows + row] = oz_group(mx, em, l1);
#pragma unroll
  for (int pr = 0; pr < 4; ++pr)
    reinterpret_cast<uint4 *>(img + ((rhs * 4 + pr) * a.rows + row) * 128)[c ^ (int)(f & 7)] =
        make_uint4(pk[pr][0], pk[pr][1], pk[pr][2], pk[pr][3]);
}

template <int W>
__global__ void __launch_bounds__(OZM_THREADS, 1) k_m2l_oz(OzmArgs a) {
  using SH = OzmShape<W>;
  constexpr int N = SH::N, NB = SH::NB;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ uint64_t wfull[OZM_NWIN], wempty[OZM_NWIN], bfull[NB], bempty[NB], acc_full[2], acc_empty[2], done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  __shared__ int4 ssh[OZM_MAXSH];  // the part's shifts
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char *smem = smem_raw + ((1024u - (tc::smem_addr(smem_raw) & 1023u)) & 1023u);
  unsigned char *wbuf = smem, *bbuf = smem + OZM_NWIN * OZM_WBYTES;
  const int2 tile = a.tiles[blockIdx.x];
  const int l = tile.x, f0 = tile.y, cpair = blockIdx.y & 1, part = blockIdx.y >> 1, rhs = blockIdx.z;
  const int P = a.lev_P[l], s0 = a.part_s[cpair][part], ns = a.part_s[cpair][part + 1] - s0;
  for (int j = tid; j < ns; j += blockDim.x) {
    int4 v = a.shifts[s0 + j];
    if (j == 0) v.w |= 1;
    ssh[j] = v;
  }
  if (tid == 0) {
    for (int s = 0; s < OZM_NWIN; ++s) {
      tc::mbar_init(&wfull[s], 1);
      tc::mbar_init(&wempty[s], 1);
    }
    for (int s = 0; s < NB; ++s) {
      tc::mbar_init(&bfull[s], 1);
      tc::mbar_init(&bempty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&acc_full[b], 1);
      tc::mbar_init(&acc_empty[b], 8);
    }
    tc::mbar_init(&done, 1);
    tc::mbar_init_fence();
    abort_flag = 0;
  }
  if (warp == 0) tc::tmem_alloc(&tmem_base, 512);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_base;
  int w_issued = 0, b_issued = 0;
  const int64_t sub = (int64_t)P * P + OZM_TAIL;
  if (warp == 0) {
    if (lane == 0) {  // windows, one per (source parity, dy) group
      bool ok = true;
      for (int j = 0; j < ns && ok && !abort_flag; ++j) {
        const int4 g = ssh[j];
        if (!(g.w & 1)) continue;
        const int ws = w_issued % OZM_NWIN;
        if (w_issued >= OZM_NWIN && !tc::mbar_wait(&wempty[ws], ((w_issued / OZM_NWIN) - 1) & 1, &abort_flag)) {
          ok = false;
          break;
        }
        const int w0 = (f0 + g.y * P - 4) & ~7;
        tc::mbar_expect_tx(&wfull[ws], OZM_WBYTES);
        for (int pr = 0; pr < 4; ++pr)
          tc::bulk_g2s(wbuf + ws * OZM_WBYTES + pr * OZM_WPAIR,
                       a.img + (((int64_t)rhs * 4 + pr) * a.rows + a.lev_row0[l] + (int64_t)g.x * sub + w0) * 128,
                       OZM_WPAIR, &wfull[ws]);
        ++w_issued;
      }
      if (!ok) {
        abort_flag = 1;
        atomicOr(a.err, 1);
      }
    }
  } else if (warp == 10) {
    if (lane == 0) {  // B blocks, one per shift
      bool ok = true;
      for (int j = 0; j < ns && !abort_flag; ++j) {
        const int bs = j % NB;
        if (j >= NB && !tc::mbar_wait(&bempty[bs], ((j / NB) - 1) & 1, &abort_flag)) { ok = false; break; }
        tc::mbar_expect_tx(&bfull[bs], SH::BBYTES);
        tc::bulk_g2s(bbuf + bs * SH::BBYTES, a.bmat + (int64_t)(s0 + j) * SH::BBYTES, SH::BBYTES, &bfull[bs]);
        b_issued = j + 1;
      }
      if (!ok) {
        abort_flag = 1;
        atomicOr(a.err, 1);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24);
      const uint32_t wlo0 = tc::desc_lo(tc::smem_addr(wbuf)), blo0 = tc::desc_lo(tc::smem_addr(bbuf));
      bool ok = true;
      int wi = -1;
      for (int j = 0; j < ns && ok; ++j) {
        const int4 g = ssh[j];
        if (g.w & 1) {
          ++wi;
          if (!tc::mbar_wait(&wfull[wi % OZM_NWIN], (wi / OZM_NWIN) & 1, &abort_flag)) { ok = false; break; }
        }
        const int bs = j % NB;
        if (!tc::mbar_wait(&bfull[bs], (j / NB) & 1, &abort_flag)) { ok = false; break; }
        const int w0 = (f0 + g.y * P - 4) & ~7;
        // digit i: row image i / 2, columns 32 (i % 2) ..: +4 in 16-byte units
        const uint32_t al = wlo0 + (uint32_t)((wi % OZM_NWIN) * (OZM_WBYTES >> 4) + (f0 + g.y * P + g.z - w0) * 8);
        const uint32_t bl = blo0 + (uint32_t)(bs * (SH::BBYTES >> 4));
#pragma unroll
        for (int ph = 0; ph < 2; ++ph) {  // orders 6, 5, 4, then 3 .. 0
          if (j > 0 && !tc::mbar_wait(&acc_empty[ph], (j - 1) & 1, &abort_flag)) { ok = false; break; }
          tc::fence_after();
#pragma unroll
          for (int s = ph ? 3 : 6; s >= (ph ? 0 : 4); --s)
#pragma unroll
            for (int i = 0; i <= s; ++i)
#pragma unroll
              for (int k = 0; k < 2; ++k)
                tc::mma_f16(tmem + N * s, tc::desc_of(al + (i >> 1) * (OZM_WPAIR >> 4) + 4 * (i & 1) + 2 * k),
                            tc::desc_of(bl + ((s - i) >> 1) * (SH::BPAIR >> 4) + 4 * ((s - i) & 1) + 2 * k), idesc,
                            (i > 0 || k > 0) ? 1u : 0u);
          tc::commit(&acc_full[ph]);
        }
        tc::commit(&bempty[bs]);
        if (ok && (j + 1 == ns || (ssh[j + 1].w & 1))) tc::commit(&wempty[wi % OZM_NWIN]);
      }
      if (!ok) {
        abort_flag = 1;
        atomicOr(a.err, 1);
      }
      tc::commit(&done);
    }
  } else {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 (one target each) and the W columns of
    // class 2 cpair + h
    const int qd = warp & 3, h = (warp - 2) >> 2;
    const int f = f0 + 32 * qd + lane;
    const int2 *le = a.lexp + (int64_t)rhs * a.rows + a.lev_row0[l] + f;
    int emax = OZ_NONE;
    float l1 = 0.0f;
    for (int j = 0; j < ns; ++j) {
      const int4 g = ssh[j];
      if (!((g.w >> (1 + h)) & 1)) continue;  // not in this class's lists
      oz_bound(__ldg(le + (int64_t)g.x * sub + g.y * P + g.z), emax, l1);
    }
    const int lsb = oz_unit(l1);
    long long acc[W];
#pragma unroll
    for (int i = 0; i < W; ++i) acc[i] = 0;
    bool ok = true;
    const uint32_t tb = tmem + ((uint32_t)(32 * qd) << 16) + W * h;
    for (int j = 0; j < ns; ++j) {
      const int4 g = ssh[j];
      const bool mine = (g.w >> (1 + h)) & 1;  // else its sums are zero
      const int d = mine ? min(emax - __ldg(le + (int64_t)g.x * sub + g.y * P + g.z).x + OZ_LSB - lsb, 62) : 62;
      const long long half = d > 0 ? 1ll << (d - 1) : 0;
      int tl[W];
      if (!__all_sync(0xffffffffu, tc::mbar_wait(&acc_full[0], j & 1, &abort_flag))) { ok = false; break; }
      tc::fence_after();
#pragma unroll
      for (int c = 0; c < W / 8; ++c) {
        float v4[8], v5[8], v6[8];
        tc::tmem_ld8(tb + N * 6 + 8 * c, v6);
        tc::tmem_ld8(tb + N * 5 + 8 * c, v5);
        tc::tmem_ld8(tb + N * 4 + 8 * c, v4);
#pragma unroll
        for (int i = 0; i < 8; ++i) tl[8 * c + i] = oz_join_low(v4[i], v5[i], v6[i]);
      }
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&acc_empty[0]);
      if (!__all_sync(0xffffffffu, tc::mbar_wait(&acc_full[1], j & 1, &abort_flag))) { ok = false; break; }
      tc::fence_after();
#pragma unroll
      for (int c = 0; c < W / 8; ++c) {
        float v0[8], v1[8], v2[8], v3[8];
        tc::tmem_ld8(tb + 8 * c, v0);
        tc::tmem_ld8(tb + N + 8 * c, v1);
        tc::tmem_ld8(tb + 2 * N + 8 * c, v2);
        tc::tmem_ld8(tb + 3 * N + 8 * c, v3);
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[8 * c + i] += (oz_join(tl[8 * c + i], v0[i], v1[i], v2[i], v3[i]) + half) >> d;
      }
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&acc_empty[1]);
    }
    if (!ok) {
      abort_flag = 1;
      if (lane == 0) atomicOr(a.err, 2);
    }
    const int S = P - 8, ti = f % P - 4, tj = f / P - 4;
    if (ok && !abort_flag && ti >= 0 && ti < S && tj >= 0 && tj < S) {
      const int cls = 2 * cpair + h, x = 2 * ti + (cls & 1), y = 2 * tj + (cls >> 1);
      const int64_t gidx = level_offset(l) + morton_encode((uint32_t)x, (uint32_t)y);
      double *L = reinterpret_cast<double *>(a.L + (int64_t)part * a.part_stride + ((int64_t)rhs * a.ncell + gidx) * a.p);
      const double nan = __longlong_as_double(0x7ff8000000000000ll);
      auto val = [&](int u) {
        if (emax >= OZ_NAN) return nan;
        return emax > OZ_NONE ? ldexp((double)acc[u], emax + a.rb[u] - lsb) : 0.0;
      };
      const double lnrho = log((double)(a.n >> l));
      L[0] = fma(lnrho, val(W - 2), val(0));
      L[1] = fma(lnrho, val(W - 1), val(1));
#pragma unroll
      for (int u = 2; u < W - 2; ++u)
        if (u < 2 * a.p) L[u] = val(u);
    }
  }
  __syncwarp();
  const bool finished = __all_sync(0xffffffffu, tc::mbar_wait(&done, 0, nullptr));
  if (!finished && lane == 0) atomicOr(a.err, 4);
  tc::fence_before();
  __syncthreads();
  if (abort_flag && lane == 0) {  // copies still in flight land before the block exits
    if (warp == 0)
      for (int u = max(0, w_issued - OZM_NWIN); u < w_issued; ++u)
        tc::mbar_wait(&wfull[u % OZM_NWIN], (u / OZM_NWIN) & 1, nullptr);
    if (warp == 10)
      for (int u = max(0, b_issued - NB); u < b_issued; ++u) tc::mbar_wait(&bfull[u % NB], (u / NB) & 1, nullptr);
  }
  __syncthreads();
  if (warp == 0) {
    tc::fence_after();
    tc::tmem_dealloc(tmem, 512);
  }
}

// L~ of levels >= 2 from the parts' images; zero above (no M2L there).
__global__ void k_m2l_oz_sum(int64_t per_rhs, int64_t lo, int64_t total, int nparts, int64_t stride,
                             const double *__restrict__ Lp, double *__restrict__ L) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= total) return;
  double v = 0.0;
  if (t % per_rhs >= lo)
    for (int q = 0; q < nparts; ++q) v += Lp[q * stride + t];
  L[t] = v;
}

// The digits of every shift's B block: thread per (shift, row, 16 bytes of a digit's columns).  idx: the
// matrix of each shift's two classes (-1: none); mats [matrix][2 p + 2 outputs][2 p], scaled columns.
template <int W>
__global__ void k_ozm_table(OzmArgs a, int ns, const int2 *__restrict__ idx, const double *__restrict__ mats,
                            unsigned char *__restrict__ bmat) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)ns * 2 * W * 4) return;
  const int q = (int)(i / (2 * W * 4)), row = (int)(i >> 2) % (2 * W), vc = (int)i & 3;
  const int h = row / W, u = row % W, p2 = 2 * a.p, m = h ? idx[q].y : idx[q].x;
  const bool used = m >= 0 && (u < p2 || u >= W - 2);
  const double *x = mats + ((int64_t)(used ? m : 0) * (p2 + 2) + (u < p2 ? u : p2 + u - (W - 2))) * p2;
  uint32_t pk[8][4];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int v = 8 * vc + j;
    int d[OZ_S];
    oz_digits(used && v < p2 ? __double2ll_rn(ldexp(x[v], 62 - a.rb[u])) : 0, d);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const uint32_t hv = __half_as_ushort(__int2half_rn(e < OZ_S ? d[e < OZ_S ? e : 0] : 0));
      if (j & 1) pk[e][j >> 1] |= hv << 16;
      else pk[e][j >> 1] = hv;
    }
  }
#pragma unroll
  for (int e = 0; e < 8; ++e)  // digit e: row set e / 2, columns 32 (e % 2) ..
    reinterpret_cast<uint4 *>(bmat + ((int64_t)q * 4 + e / 2) * 2 * W * 128 + row * 128)[(vc + 4 * (e & 1)) ^ (row & 7)] =
        make_uint4(pk[e][0], pk[e][1], pk[e][2], pk[e][3]);
}

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace

void init_m2l_oz(fmmpc_handle &H, DevPool &tmp) {
  OzM2L &T = H.ozm;
  T.enabled = false;
  const Geo &g = H.g;
  // W - 2 >= 2p outputs, K = 32 >= 2p inputs
  if (H.prec != FMMPC_PREC_FP64 || g.L < 2 || 2 * g.p + 2 > 32) return;
  M2lShifts S;
  if (!m2l_shift_sets(H, tmp, S)) return;  // lists that are not one offset set per class: pair by pair
  const int L = g.L, p = g.p, ns = (int)S.dxs.size();
  for (int dx : S.dxs)
    if (dx < -4 || dx > 4) return;
  T.width = 2 * p + 2 <= 24 ? 24 : 32;
  const int W = T.width;
  int64_t rows = 0;
  std::vector<int2> tiles;
  for (int l = 2; l <= L; ++l) {
    const int s = 1 << (l - 1), P = s + 8;
    T.lev_P[l] = P;
    T.lev_row0[l] = rows;
    rows += 4 * ((int64_t)P * P + OZM_TAIL);
    const int fs = 4 * P + 4, fe = (s + 3) * P + s + 3;
    for (int f0 = fs; f0 <= fe; f0 += 128) tiles.push_back(make_int2(l, f0));
  }
  T.rows = rows;
  T.ntiles = (int)tiles.size();
  // a tile's two class pairs are two CTAs: where these do not fill the SMs twice, the shifts are split between
  // four of each (1024^2: 52 tiles, 104 CTAs a part); the choice depends on the geometry and the device's
  // SM count (152), not on the right-hand sides
  int dev = 0, nsm = 0;
  FMMPC_CUDA(cudaGetDevice(&dev));
  FMMPC_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const int ctas = 2 * T.ntiles;
  T.nparts = ctas >= 2 * nsm ? 1 : OZM_MAXPART;
  std::vector<int4> shifts;
  std::vector<int> shq;  // the shift (index of shift_ofs) of each entry
  int count[2] = {};
  for (int cp = 0; cp < 2; ++cp) {
    for (const int4 &gr : S.groups) {
      bool first = true;
      for (int k = 0; k < gr.w; ++k) {
        const auto &o = S.shift_ofs[gr.z + k];
        const int mask = (o[2 * cp] >= 0 ? 2 : 0) | (o[2 * cp + 1] >= 0 ? 4 : 0);
        if (!mask) continue;
        shifts.push_back(make_int4(gr.x, gr.y, S.dxs[gr.z + k], mask | (first ? 1 : 0)));
        shq.push_back(gr.z + k);
        first = false;
        ++count[cp];
      }
    }
    for (int q = 0; q <= T.nparts; ++q)
      T.part_s[cp][q] = (cp ? count[0] : 0) + (int)((int64_t)count[cp] * q / T.nparts);
    for (int q = 0; q < T.nparts; ++q)
      if (T.part_s[cp][q + 1] - T.part_s[cp][q] > OZM_MAXSH) return;
  }
  // real matrices of every offset, inputs scaled by 2^-c_k.  The powers of an offset in two doubles each
  // (106 bits), so that an entry is one multiply-add: in long double, which is software on this host,
  // they were a third of a 64^2 handle's set-up (with the digits, 10 of 27 ms).
  std::vector<double> fact(2 * p + 2, 1.0);
  for (int i = 1; i < (int)fact.size(); ++i) fact[i] = fact[i - 1] * i;
  struct Two {
    double hi, lo;
  };
  auto two = [](long double x) {
    const double hi = (double)x;
    return Two{hi, (double)(x - hi)};
  };
  typedef std::complex<long double> C;
  std::vector<Two> pre(2 * p), pim(2 * p);  // o^-j of the offset at hand
  double lre = 0.0, lim = 0.0;              // log o
  auto set_offset = [&](int oi) {
    const C o((long double)(oi % 15 - 7), (long double)(oi / 15 - 7)), inv = C(1) / o;
    C pw(1);
    for (int j = 0; j < 2 * p; ++j, pw = pw * inv) {
      pre[j] = two(pw.real());
      pim[j] = two(pw.imag());
    }
    lre = (double)(0.5L * std::log(std::norm(o)));
    lim = (double)std::atan2(o.imag(), o.real());
  };
  auto times = [](double f, const Two &x) {
    const double q = f * x.hi;
    return q + (std::fma(f, x.hi, -q) + f * x.lo);
  };
  auto over = [](const Two &x, double n) {
    const double q = x.hi / n;
    return q + (std::fma(-q, n, x.hi) + x.lo) / n;
  };
  // real and imaginary part of output coefficient n from input coefficient k
  auto coeff = [&](int n, int k, double &re, double &im) {
    if (n == 0 && k == 0) {
      re = lre, im = lim;
    } else if (k == 0) {
      const double s = (n % 2) ? 1.0 : -1.0;
      re = s * over(pre[n], n), im = s * over(pim[n], n);
    } else {
      const double f = n == 0 ? 1.0 : ((n % 2) ? -1.0 : 1.0) * (fact[n + k - 1] / (fact[n] * fact[k - 1]));
      re = times(f, pre[n + k]), im = times(f, pim[n + k]);
    }
  };
  const int p2 = 2 * p, nout = p2 + 2;  // outputs: 2p real parts, then the sums M~_0 (rows W - 2, W - 1)
  std::vector<int> mat_of(225, -1);
  std::vector<double> mats, rmax(W, 0.0);  // [matrix][nout][2p], scaled columns
  for (int q = 0; q < ns; ++q)
    for (int c = 0; c < 4; ++c) {
      const int oi = S.shift_ofs[q][c];
      if (oi < 0 || mat_of[oi] >= 0) continue;
      mat_of[oi] = (int)(mats.size() / ((size_t)nout * p2));
      mats.resize(mats.size() + (size_t)nout * p2, 0.0);
      double *m = mats.data() + (size_t)mat_of[oi] * nout * p2;
      set_offset(oi);
      for (int n = 0; n < p; ++n)
        for (int k = 0; k < p; ++k) {
          double re, im;
          coeff(n, k, re, im);
          const double sc = std::ldexp(1.0, -ozm_col(k));
          m[(2 * n) * p2 + 2 * k] = m[(2 * n + 1) * p2 + 2 * k + 1] = sc * re;
          m[(2 * n) * p2 + 2 * k + 1] = -(sc * im);
          m[(2 * n + 1) * p2 + 2 * k] = sc * im;
        }
      m[p2 * p2] = m[(p2 + 1) * p2 + 1] = 1.0;
      for (int u = 0; u < nout; ++u)
        for (int v = 0; v < p2; ++v) {
          double &r = rmax[u < p2 ? u : W - 2 + u - p2];
          r = std::max(r, std::fabs(m[u * p2 + v]));
        }
    }
  for (int u = 0; u < W; ++u) {
    int e = 0;
    if (rmax[u] > 0.0) std::frexp(rmax[u], &e);  // rmax < 2^e
    T.rb[u] = e;
  }
  std::vector<int2> idx(shifts.size());
  for (size_t q = 0; q < shifts.size(); ++q) {
    const auto &o = S.shift_ofs[shq[q]];
    const int c = q < (size_t)count[0] ? 0 : 2;
    idx[q] = make_int2(o[c] < 0 ? -1 : mat_of[o[c]], o[c + 1] < 0 ? -1 : mat_of[o[c + 1]]);
  }
  const size_t ibytes = (size_t)H.nrhs_max * 4 * rows * 128, nexp = (size_t)H.nrhs_max * rows;
  T.img = H.ozm_pool.get<unsigned char>(ibytes);
  FMMPC_CUDA(cudaMemsetAsync(T.img, 0, ibytes, H.stream));
  T.lexp = H.ozm_pool.get<int2>(nexp);
  k_oz_fill<<<nblk(nexp), 256, 0, H.stream>>>((int64_t)nexp, T.lexp);
  FMMPC_LAUNCH_CHECK();
  T.bmat = H.ozm_pool.get<unsigned char>(shifts.size() * 4 * 2 * W * 128);
  T.tiles = H.ozm_pool.get<int2>(tiles.size());
  T.shifts = H.ozm_pool.get<int4>(shifts.size());
  T.part_stride = (int64_t)H.nrhs_max * g.ncell * p;
  T.Lp = H.ozm_pool.get<double>((size_t)2 * T.nparts * T.part_stride);
  T.err = H.ozm_pool.get<int>(1);
  double *dmats = tmp.get<double>(mats.size());
  int2 *didx = tmp.get<int2>(idx.size());
  FMMPC_CUDA(cudaMemcpyAsync(dmats, mats.data(), sizeof(double) * mats.size(), cudaMemcpyHostToDevice, H.stream));
  FMMPC_CUDA(cudaMemcpyAsync(didx, idx.data(), sizeof(int2) * idx.size(), cudaMemcpyHostToDevice, H.stream));
  OzmArgs a{};
  a.p = p;
  for (int u = 0; u < W; ++u) a.rb[u] = T.rb[u];
  const int nsh = (int)shifts.size();
  if (W == 24) k_ozm_table<24><<<nblk((int64_t)nsh * 2 * W * 4), 256, 0, H.stream>>>(a, nsh, didx, dmats, T.bmat);
  else k_ozm_table<32><<<nblk((int64_t)nsh * 2 * W * 4), 256, 0, H.stream>>>(a, nsh, didx, dmats, T.bmat);
  FMMPC_LAUNCH_CHECK();
  FMMPC_CUDA(cudaMemcpyAsync(T.tiles, tiles.data(), sizeof(int2) * tiles.size(), cudaMemcpyHostToDevice, H.stream));
  FMMPC_CUDA(cudaMemcpyAsync(T.shifts, shifts.data(), sizeof(int4) * shifts.size(), cudaMemcpyHostToDevice, H.stream));
  FMMPC_CUDA(cudaMemsetAsync(T.err, 0, sizeof(int), H.stream));
  if (W == 24) raise_smem_limit(k_m2l_oz<24>);
  else raise_smem_limit(k_m2l_oz<32>);
  FMMPC_CUDA(cudaStreamSynchronize(H.stream));
  T.enabled = true;
}

// L~ of every volume cell from its M2L list (zero at levels 0 and 1).
int run_m2l_oz(fmmpc_handle &H, const void *Mv, void *Lv, int nrhs, cudaStream_t s) {
  const OzM2L &T = H.ozm;
  const Geo &g = H.g;
  OzmArgs a{};
  a.img = T.img;
  a.lexp = T.lexp;
  a.bmat = T.bmat;
  a.tiles = T.tiles;
  a.shifts = T.shifts;
  a.L = reinterpret_cast<cpx<double> *>(T.Lp);
  a.rows = T.rows;
  a.ncell = g.ncell;
  a.part_stride = T.part_stride;
  a.err = T.err;
  for (int l = 0; l < 24; ++l) {
    a.lev_row0[l] = T.lev_row0[l];
    a.lev_P[l] = T.lev_P[l];
  }
  for (int cp = 0; cp < 2; ++cp)
    for (int q = 0; q <= T.nparts; ++q) a.part_s[cp][q] = T.part_s[cp][q];
  for (int u = 0; u < T.width; ++u) a.rb[u] = T.rb[u];
  a.p = g.p;
  a.n = g.n;
  const int64_t lo = level_offset(2), hi = level_offset(g.L + 1);
  k_m2l_oz_pack<<<nblk((int64_t)nrhs * (hi - lo) * 8), 256, 0, s>>>(a, nrhs, lo, hi, (const cpx<double> *)Mv, T.img,
                                                                    T.lexp);
  const dim3 grid((unsigned)T.ntiles, (unsigned)(2 * T.nparts), (unsigned)nrhs);
  if (T.width == 24) k_m2l_oz<24><<<grid, OZM_THREADS, OzmShape<24>::SMEM, s>>>(a);
  else k_m2l_oz<32><<<grid, OZM_THREADS, OzmShape<32>::SMEM, s>>>(a);
  const int64_t per = g.ncell * g.p * 2, total = per * nrhs;
  k_m2l_oz_sum<<<nblk(total), 256, 0, s>>>(per, lo * g.p * 2, total, T.nparts, 2 * T.part_stride, T.Lp, (double *)Lv);
  FMMPC_LAUNCH_CHECK();
  return 3;
}

}  // namespace fmmpc
