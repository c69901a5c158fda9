// The FP64 form's lattice near field (P2P, Sec. 5.1 Eq. e:volume_integral restricted to
// neighbouring leaves) on the tensor cores, to FP64 accuracy.
//
// FP64 is scarce on this GPU (2 multiply-adds per clock and SM): the 2.4e9 pairs of a 1024^2 grid
// took 4768 us on the FP64 units.  Here each FP64 operand is cut into seven signed 9-bit digits
// (63 bits), the digits are multiplied as FP16 integers by tcgen05.mma, and the sums are
// integers that the FP32 accumulator holds exactly: the error-free splitting of Ozaki, Ogita,
// Oishi and Rump ("Error-free transformations of matrix multiplication", 2012), with fixed-point
// digits.
//   W = 2^E sum_i w_i 2^(-9i - 8) per source leaf (E the exponent of the leaf's largest weight),
//   B = 2^EB sum_j b_j 2^(-9j - 8) for the kernel table ln|d|, |w_i|, |b_j| <= 256.
// Order s collects the products of i + j = s; orders 0 .. 6 are kept (28 products), the dropped
// ones are below 2^-57 of the largest product.  A digit product is at most 2^16, so a K = 64 sum of
// up to four products stays within 2^24 and is exact (orders 0-3); orders 4-6 hold five to
// seven products, whose sums the accumulator could truncate by a unit of 2^-52 only where
// they pass 2^24, relative 2^-57.  Per offset the orders are joined into a 64-bit integer in units of
// 2^-56, shifted to a unit of the target leaf's own (the finest in which the sum of its sources'
// L1 norms fits 61 bits) and added up in int64, one rounding to FP64 per part at the end.  Against
// long-double sums of white-noise weights on a 64^2 grid (eight parts): relative L2 error 2.3e-16, the
// CUDA-core kernel's FP64 additions 1.2e-15.
//
// Layout.  The leaves' digit rows (64 digits, 128 bytes, 128-byte swizzle) are flattened over the
// padded leaf grid with pitch P = NL + 2R, one image per digit; a CTA takes 128 consecutive
// flattened targets (M = 128, padding targets computed and dropped, so any leaf grid fills the
// tiles), N = the 64 target nodes, K = the 64 source nodes, and sweeps the stencil offsets: per
// source row one strip per digit, per offset seven 8 KB table blocks.  TMEM holds orders 4-6 and 0-3
// apart, so the epilogue joins the first while the second are multiplied and the other way round.
//
// Bound by the epilogue: eight warps, two per scheduler, whose TMEM reads, conversions and 64-bit shifts
// and additions are chains of dependent instructions (52M warp instructions, 18% of the issue
// slots).  The MMAs, 28 x 4 of 48 cycles per offset (N = 64), are 96 of the 260 us at 1024^2; the tensor
// pipe is active 27% of the time, DRAM 1%.
#include <algorithm>
#include <cmath>
#include <vector>

#include "handle.cuh"
#include "oz.cuh"
#include "tc.cuh"

namespace fmmpc {

namespace {

constexpr int OZ_TILE = 128;       // flattened target leaves per CTA
constexpr int OZ_BLK = 8192;       // one digit of one offset's table: 64 x 64 FP16
constexpr int OZ_MAXB = 12;        // table block slots at most (7 in use, the rest ahead)
constexpr int OZ_MAXOFS = 64;      // offsets per part at most: an L1 bound of about 2^12, units of 2^-48 and finer
constexpr int OZ_MAXPART = 8;
constexpr int OZ_MAXROWS = 33;
constexpr int OZ_THREADS = 320;    // producer, MMA issuer, eight epilogue warps

struct OzArgs {
  const uint16_t *img;        // [nrhs][OZ_S][rows][64] digits, swizzled per row
  const int2 *lexp;           // [nrhs][rows] exponent E of each leaf's weights, their L1 norm / 2^E (FP32, rounded up)
  const unsigned char *bmat;  // [offset][slots 6, 5, 0, 1, 2, 3, 4][64][64] digits of the table
  double *out;                // [part][nrhs][n][n] near-field sums (unscaled)
  int64_t part_stride, rows;
  int *err;
  int n, NL, P, R, eb, nbs, sh, nsr, vec;
  int16_t row_oy[OZ_MAXROWS], row_ox0[OZ_MAXROWS], row_cnt[OZ_MAXROWS];
  int16_t part_r[OZ_MAXPART], part_q[OZ_MAXPART], part_n[OZ_MAXPART];
  int part_o[OZ_MAXPART];     // index of the part's first offset
};

// Digit rows of the weights w = h^2 r and the FP64 weight image.  Thread per (rhs, leaf, node row
// jr of the leaf), jr fastest: the eight lanes of a leaf find its largest |w| by shuffles, take every weight
// as a fixed-point number below it, and write their row's digits as the 16-byte chunk jr of the leaf's
// swizzled row in each digit's image.
__global__ void k_oz_strips(int n, int lgNL, int P, int R, int64_t rows, double h2, int nrhs,
                            const double *__restrict__ r, uint16_t *__restrict__ img, int2 *__restrict__ lexp,
                            double *__restrict__ wimg, int npad, int pad) {
  const int NL = 1 << lgNL;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = t < ((int64_t)nrhs << (2 * lgNL + 3));  // every lane takes part in the shuffles
  const int jr = (int)(t & 7), Xl = (int)((t >> 3) & (NL - 1)), Yl = (int)((t >> (3 + lgNL)) & (NL - 1));
  const int64_t rhs = t >> (3 + 2 * lgNL);
  const int j = 8 * Yl + jr, i0 = 8 * Xl;
  double w[8];
  unsigned long long mx = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    w[q] = in ? h2 * r[rhs * (int64_t)n * n + (int64_t)j * n + i0 + q] : 0.0;
    mx = max(mx, oz_bits(w[q]));
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const int em = oz_biased(mx);
  const int64_t f = (int64_t)(Yl + R) * P + Xl + R;
  uint32_t pk[OZ_S][4];
  float l1 = 0.0f;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    int d[OZ_S];
    oz_digits(oz_fixed(w[q], em, l1), d);
#pragma unroll
    for (int s = 0; s < OZ_S; ++s) {
      const uint32_t hv = __half_as_ushort(__int2half_rn(d[s]));  // exact
      if (q & 1) pk[s][q >> 1] |= hv << 16;
      else pk[s][q >> 1] = hv;
    }
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) l1 += __shfl_xor_sync(0xffffffffu, l1, o);
  if (!in) return;
  if (jr == 0) lexp[rhs * rows + f] = oz_group(mx, em, l1);
  const int pos = jr ^ (int)(f & 7);
#pragma unroll
  for (int s = 0; s < OZ_S; ++s)
    reinterpret_cast<uint4 *>(img + ((rhs * OZ_S + s) * rows + f) * 64)[pos] =
        make_uint4(pk[s][0], pk[s][1], pk[s][2], pk[s][3]);
  double2 *wr = reinterpret_cast<double2 *>(wimg + rhs * (int64_t)npad * npad + (int64_t)(j + pad) * npad + i0 + pad);
#pragma unroll
  for (int q = 0; q < 4; ++q) wr[q] = make_double2(w[2 * q], w[2 * q + 1]);
}

// digit held by position p of an offset's seven table blocks: 6 and 5 first, which are free again
// once orders 4-6 are multiplied
__host__ __device__ constexpr int oz_slice(int p) { return p < 2 ? 6 - p : p - 2; }
__host__ __device__ constexpr int oz_pos(int slice) { return slice >= 5 ? 6 - slice : slice + 2; }

__global__ void __launch_bounds__(OZ_THREADS, 1) k_p2p_oz(OzArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint64_t full_s, empty_s, full_b[OZ_MAXB], empty_b[OZ_MAXB], acc_full[2], acc_empty[2], done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char *strips = smem + ((1024u - (tc::smem_addr(smem) & 1023u)) & 1023u);  // [OZ_S][sh]
  unsigned char *bm = strips + OZ_S * a.sh;                                          // [nbs][OZ_BLK]
  const int part = blockIdx.y, rhs = blockIdx.z;
  const int f0 = a.R * a.P + a.R + blockIdx.x * OZ_TILE;
  const int rs = a.part_r[part], qs = a.part_q[part], ng = a.part_n[part], nbs = a.nbs;
  if (tid == 0) {
    tc::mbar_init(&full_s, 1);
    tc::mbar_init(&empty_s, 1);
    for (int b = 0; b < nbs; ++b) {
      tc::mbar_init(&full_b[b], 1);
      tc::mbar_init(&empty_b[b], 1);
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
  int issued_s = 0, issued_b = 0;
  // flattened row of the first target's source for row r, and the strip's 8-aligned start
  auto wrow = [&](int r) { return f0 + (int)a.row_oy[r] * a.P - a.R; };
  if (warp == 0) {
    if (lane == 0) {
      // producer: per offset its table blocks through a ring of nbs slots; per source row the
      // strips, once the row before is done (its first blocks are under way by then)
      bool ok = true;
      int r = rs, q = qs;
      for (int g = 0; g < ng && ok && !abort_flag; ++g) {
        const unsigned char *src = a.bmat + (int64_t)(a.part_o[part] + g) * (OZ_S * OZ_BLK);
        for (int p = 0; p < OZ_S && ok; ++p) {
          const int u = OZ_S * g + p, slot = u % nbs;
          if (u >= nbs && !tc::mbar_wait(&empty_b[slot], ((u / nbs) - 1) & 1, &abort_flag)) ok = false;
          else {
            tc::mbar_expect_tx(&full_b[slot], OZ_BLK);
            tc::bulk_g2s(bm + slot * OZ_BLK, src + p * OZ_BLK, OZ_BLK, &full_b[slot]);
            issued_b = u + 1;
          }
        }
        if (ok && (g == 0 || q == 0)) {
          if (issued_s && !tc::mbar_wait(&empty_s, (issued_s - 1) & 1, &abort_flag)) ok = false;
          else {
            tc::mbar_expect_tx(&full_s, OZ_S * a.nsr * 128);
            const uint16_t *src_s = a.img + ((int64_t)rhs * OZ_S * a.rows + (wrow(r) & ~7)) * 64;
            for (int s = 0; s < OZ_S; ++s)
              tc::bulk_g2s(strips + s * a.sh, src_s + (int64_t)s * a.rows * 64, a.nsr * 128, &full_s);
            ++issued_s;
          }
        }
        if (++q == a.row_cnt[r]) {
          q = 0;
          ++r;
        }
      }
      if (!ok) {
        abort_flag = 1;
        atomicOr(a.err, 1);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // MMA issuer: FP16 digits, FP32 accumulators of order s at columns 64 s
      const uint32_t idesc = (1u << 4) | ((64u >> 3) << 17) | ((128u >> 4) << 24);
      const uint32_t slo0 = tc::desc_lo(tc::smem_addr(strips)), blo0 = tc::desc_lo(tc::smem_addr(bm));
      const uint32_t sh16 = (uint32_t)(a.sh >> 4);
      bool ok = true;
      int r = rs, q = qs, nrow = 0;
      for (int g = 0; g < ng && ok; ++g) {
        if (g == 0 || q == 0) {
          if (!tc::mbar_wait(&full_s, nrow & 1, &abort_flag)) { ok = false; break; }
          ++nrow;
        }
        uint32_t bl[OZ_S];  // descriptor low word of each digit's block
#pragma unroll
        for (int p = 0; p < OZ_S; ++p) {
          const int u = OZ_S * g + p, slot = u % nbs;
          if (ok && !tc::mbar_wait(&full_b[slot], (u / nbs) & 1, &abort_flag)) ok = false;
          bl[oz_slice(p)] = blo0 + (uint32_t)(slot * (OZ_BLK >> 4));
        }
        if (!ok) break;
        const int w = wrow(r);
        const uint32_t al = slo0 + 8u * (uint32_t)(w - (w & ~7) + a.R + a.row_ox0[r] + q);
#pragma unroll
        for (int ph = 0; ph < 2; ++ph) {  // orders 6, 5, 4, then 3 .. 0
          if (g > 0 && !tc::mbar_wait(&acc_empty[ph], (g - 1) & 1, &abort_flag)) { ok = false; break; }
          tc::fence_after();
#pragma unroll
          for (int s = ph ? 3 : 6; s >= (ph ? 0 : 4); --s)
#pragma unroll
            for (int i = 0; i <= s; ++i)
#pragma unroll
              for (int k = 0; k < 4; ++k)
                tc::mma_f16(tmem + 64 * s, tc::desc_of(al + i * sh16 + 2 * k), tc::desc_of(bl[s - i] + 2 * k), idesc,
                            (i > 0 || k > 0) ? 1u : 0u);
#pragma unroll
          for (int p = ph ? 2 : 0; p < (ph ? OZ_S : 2); ++p) tc::commit(&empty_b[(OZ_S * g + p) % nbs]);
          tc::commit(&acc_full[ph]);
        }
        if (++q == a.row_cnt[r]) {
          tc::commit(&empty_s);
          q = 0;
          ++r;
        }
      }
      if (!ok) {
        abort_flag = 1;
        atomicOr(a.err, 1);
      }
      tc::commit(&done);
    }
  } else {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 (one target leaf each), nodes 32 hf .. + 31
    const int qd = warp & 3, hf = (warp - 2) >> 2;
    const int f = f0 + 32 * qd + lane;
    const int2 *le = a.lexp + (int64_t)rhs * a.rows + f;  // the rows reach past the last target's sources
    int emax = OZ_NONE;
    float l1 = 0.0f;  // bound of the sum in units of 2^(emax + EB)
    {
      int r = rs, q = qs;
      for (int g = 0; g < ng; ++g) {
        oz_bound(__ldg(le + (int)a.row_oy[r] * a.P + a.row_ox0[r] + q), emax, l1);
        if (++q == a.row_cnt[r]) q = 0, ++r;
      }
    }
    const int lsb = oz_unit(l1);
    long long acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0;
    bool ok = true;
    int r = rs, q = qs;
    const uint32_t tb = tmem + ((uint32_t)(32 * qd) << 16) + 32 * hf;
    for (int g = 0; g < ng; ++g) {
      const int d = min(emax - __ldg(le + (int)a.row_oy[r] * a.P + a.row_ox0[r] + q).x + OZ_LSB - lsb, 62);
      const long long half = d > 0 ? 1ll << (d - 1) : 0;
      if (++q == a.row_cnt[r]) q = 0, ++r;
      int tl[32];  // orders 4-6 in units of 2^-56
      if (!__all_sync(0xffffffffu, tc::mbar_wait(&acc_full[0], g & 1, &abort_flag))) {
        ok = false;
        break;
      }
      tc::fence_after();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float v4[16], v5[16], v6[16];
        tc::tmem_ld16(tb + 64 * 6 + 16 * c, v6);
        tc::tmem_ld16(tb + 64 * 5 + 16 * c, v5);
        tc::tmem_ld16(tb + 64 * 4 + 16 * c, v4);
#pragma unroll
        for (int i = 0; i < 16; ++i) tl[16 * c + i] = oz_join_low(v4[i], v5[i], v6[i]);
      }
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&acc_empty[0]);
      if (!__all_sync(0xffffffffu, tc::mbar_wait(&acc_full[1], g & 1, &abort_flag))) {
        ok = false;
        break;
      }
      tc::fence_after();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float v0[16], v1[16], v2[16], v3[16];
        tc::tmem_ld16(tb + 16 * c, v0);
        tc::tmem_ld16(tb + 64 + 16 * c, v1);
        tc::tmem_ld16(tb + 128 + 16 * c, v2);
        tc::tmem_ld16(tb + 192 + 16 * c, v3);
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[16 * c + i] += (oz_join(tl[16 * c + i], v0[i], v1[i], v2[i], v3[i]) + half) >> d;
      }
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&acc_empty[1]);
    }
    if (!ok) {
      abort_flag = 1;
      if (lane == 0) atomicOr(a.err, 2);
    }
    const int X = f % a.P - a.R, Y = f / a.P - a.R;
    if (ok && !abort_flag && X >= 0 && X < a.NL && Y >= 0 && Y < a.NL) {
      double *o = a.out + (int64_t)part * a.part_stride + (int64_t)rhs * a.n * a.n + (int64_t)(Y * 8 + 4 * hf) * a.n + X * 8;
      const int e = emax + a.eb - lsb;
#pragma unroll
      for (int i = 0; i < 32; i += 2) {
        double x = 0.0, y = 0.0;
        if (emax >= OZ_NAN) x = y = __longlong_as_double(0x7ff8000000000000ll);
        else if (emax > OZ_NONE) {
          x = ldexp((double)acc[i], e);
          y = ldexp((double)acc[i + 1], e);
        }
        double *oi = o + (int64_t)(i >> 3) * a.n + (i & 7);
        if (a.vec) {
          *reinterpret_cast<double2 *>(oi) = make_double2(x, y);
        } else {  // the caller's z, aligned for FP64 only
          oi[0] = x;
          oi[1] = y;
        }
      }
    }
  }
  __syncwarp();
  const bool finished = __all_sync(0xffffffffu, tc::mbar_wait(&done, 0, nullptr));
  if (!finished && lane == 0) atomicOr(a.err, 4);
  tc::fence_before();
  __syncthreads();
  if (abort_flag && warp == 0 && lane == 0) {  // copies still in flight land before the block exits
    if (issued_s) tc::mbar_wait(&full_s, (issued_s - 1) & 1, nullptr);
    for (int u = max(0, issued_b - nbs); u < issued_b; ++u) tc::mbar_wait(&full_b[u % nbs], (u / nbs) & 1, nullptr);
  }
  __syncthreads();
  if (warp == 0) {
    tc::fence_after();
    tc::tmem_dealloc(tmem, 512);
  }
}

// The digits of the kernel table's block of every stencil offset (rows of offsets as in OzArgs), from the
// CUDA-core kernel's table of ln|d|: thread per (offset, target node t, source node row).  On the host
// the logarithms and digits of 37 x 4096 pairs were half of a 64^2 handle's set-up (11 of 27 ms).
__global__ void k_oz_table(OzArgs a, int no, int nrows, int eb, const double *__restrict__ table, int Rn, int c0, int stride,
                           unsigned char *__restrict__ bmat) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)no * 512) return;
  const int o = (int)(i >> 9), t = (int)(i >> 3) & 63, kc = (int)i & 7;
  int r = 0, q = o;
  while (r + 1 < nrows && q >= a.row_cnt[r]) q -= a.row_cnt[r++];
  const int ox = a.row_ox0[r] + q, oy = a.row_oy[r], dy = (t >> 3) - kc - 8 * oy;
  const double *row = table + (int64_t)(dy < 0 ? -dy : dy) * stride + c0 + Rn;
  uint32_t pk[OZ_S][4];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    int d[OZ_S];
    oz_digits(__double2ll_rn(ldexp(row[(t & 7) - j - 8 * ox], 62 - eb)), d);
#pragma unroll
    for (int s = 0; s < OZ_S; ++s) {
      const uint32_t hv = __half_as_ushort(__int2half_rn(d[s]));
      if (j & 1) pk[s][j >> 1] |= hv << 16;
      else pk[s][j >> 1] = hv;
    }
  }
#pragma unroll
  for (int s = 0; s < OZ_S; ++s)
    reinterpret_cast<uint4 *>(bmat + ((int64_t)o * OZ_S + oz_pos(s)) * OZ_BLK + t * 128)[kc ^ (t & 7)] =
        make_uint4(pk[s][0], pk[s][1], pk[s][2], pk[s][3]);
}

__global__ void k_near_combine64(int64_t total, const double *__restrict__ a, int64_t stride, int nparts,
                                 double *__restrict__ out) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= total) return;
  double v = a[t];
  for (int p = 1; p < nparts; ++p) v += a[p * stride + t];
  out[t] = v * NEG_INV_2PI;
}

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// the stencil's rows of offsets
OzArgs rows_of(const OzP2P &T) {
  OzArgs a{};
  for (int r = 0; r < T.nrows; ++r) {
    a.row_oy[r] = (int16_t)T.row_oy[r];
    a.row_ox0[r] = (int16_t)T.row_ox0[r];
    a.row_cnt[r] = (int16_t)T.row_cnt[r];
  }
  return a;
}

}  // namespace

// 8x8 leaves, at least 8 leaves a row (smaller grids have no tile to fill), a stencil whose strips
// fit the shared memory beside eight table blocks and whose offsets fit the parts.
bool oz_p2p_eligible(const fmmpc_handle &H) {
  const Geo &g = H.g;
  return H.prec == FMMPC_PREC_FP64 && g.m == 8 && g.L >= 3 && 2 * g.R + 1 <= OZ_MAXROWS &&
         H.st.count <= OZ_MAXOFS * OZ_MAXPART;
}

void init_p2p_oz(fmmpc_handle &H) {
  OzP2P &T = H.ozp;
  T.enabled = false;
  if (!oz_p2p_eligible(H)) return;
  const Geo &g = H.g;
  const Stencil &st = H.st;
  const int NL = 1 << g.L, R = g.R, P = NL + 2 * R;
  int dev = 0, nsm = 0, maxsm = 0;
  FMMPC_CUDA(cudaGetDevice(&dev));
  FMMPC_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  FMMPC_CUDA(cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  T.nsr = OZ_TILE + 2 * R + 8;  // strip rows: targets, shifts, alignment
  T.sh = (T.nsr * 128 + 1023) & ~1023;
  T.nbs = std::min(OZ_MAXB, (maxsm - 2048 - 1024 - OZ_S * T.sh) / OZ_BLK);
  if (T.nbs < OZ_S + 1) return;
  T.smem = OZ_S * T.sh + T.nbs * OZ_BLK + 1024;
  T.P = P;
  T.rows = (int64_t)P * P + 256;  // strips and exponents of the last tile reach past the grid
  int no = 0;
  std::vector<std::pair<int, int>> ofs;
  for (int oy = -st.R; oy <= st.R; ++oy) {
    const int a0 = st.ox0[oy + st.R], a1 = st.ox1[oy + st.R];
    if (a0 > a1) continue;
    T.row_oy[T.nrows] = oy;
    T.row_ox0[T.nrows] = a0;
    T.row_cnt[T.nrows] = a1 - a0 + 1;
    for (int ox = a0; ox <= a1; ++ox) ofs.push_back({T.nrows, ox - a0});
    ++T.nrows;
  }
  no = (int)ofs.size();
  const int64_t span = (int64_t)(NL - 1) * P + NL;  // flattened targets, padding between rows included
  T.ntiles = (int)((span + OZ_TILE - 1) / OZ_TILE);
  // with few tiles the offsets are split between up to eight CTAs, whose sums the L2P pass adds (512^2: 35
  // tiles, four parts), as long as the parts' CTAs fit the SMs at once: the choice depends on the
  // geometry and the device's SM count (152), not on the right-hand sides
  T.nparts = (no + OZ_MAXOFS - 1) / OZ_MAXOFS;
  while (2 * T.nparts <= OZ_MAXPART && T.ntiles * 2 * T.nparts <= nsm && 4 * T.nparts <= no) T.nparts *= 2;
  for (int p = 0; p < T.nparts; ++p) {
    const int b = (int)((int64_t)no * p / T.nparts), e = (int)((int64_t)no * (p + 1) / T.nparts);
    T.part_o[p] = b;
    T.part_r[p] = ofs[b].first;
    T.part_q[p] = ofs[b].second;
    T.part_n[p] = e - b;
  }
  const size_t nimg = (size_t)H.nrhs_max * OZ_S * T.rows * 64;
  T.img = H.ozp_pool.get<uint16_t>(nimg);
  FMMPC_CUDA(cudaMemsetAsync(T.img, 0, sizeof(uint16_t) * nimg, H.stream));
  const size_t nexp = (size_t)H.nrhs_max * T.rows;
  T.lexp = H.ozp_pool.get<int2>(nexp);
  k_oz_fill<<<nblk(nexp), 256, 0, H.stream>>>((int64_t)nexp, T.lexp);  // padding leaves are empty
  FMMPC_LAUNCH_CHECK();
  const double cself = -0.5 * std::log(2.0) - 1.5 + 0.25 * PI;
  for (int variant = 0; variant < 2; ++variant) {  // without and with ln h
    auto value = [&](int dx, int dy) {  // as in the table
      const double v = (dx == 0 && dy == 0) ? cself : 0.5 * std::log((double)dx * dx + (double)dy * dy);
      return variant ? v + g.lnh : v;
    };
    double vmax = 0.0;
    const int dm = 8 * R + 7;
    for (auto d : {std::pair<int, int>{0, 0}, {1, 0}, {dm, dm}}) vmax = std::max(vmax, std::fabs(value(d.first, d.second)));
    int eb = 0;
    std::frexp(vmax, &eb);  // vmax < 2^eb
    unsigned char *dB = H.ozp_pool.get<unsigned char>((size_t)no * OZ_S * OZ_BLK);
    k_oz_table<<<nblk((int64_t)no * 512), 256, 0, H.stream>>>(
        rows_of(T), no, T.nrows, eb, (const double *)(variant ? H.fb.table_lnh : H.fb.table), H.fb.Rn, H.fb.table_c0,
        H.fb.table_stride, dB);
    FMMPC_LAUNCH_CHECK();
    T.bmat[variant] = dB;
    T.eb[variant] = eb;
  }
  T.part_stride = (int64_t)H.nrhs_max * g.n * g.n;
  if (T.nparts > 1) T.near = H.ozp_pool.get<double>((size_t)T.nparts * T.part_stride);
  T.err = H.ozp_pool.get<int>(1);
  FMMPC_CUDA(cudaMemsetAsync(T.err, 0, sizeof(int), H.stream));
  raise_smem_limit(k_p2p_oz);
  T.enabled = true;
}

// Digit rows and the FP64 weight image of the right-hand side r, in one pass.
int prep_p2p_oz(fmmpc_handle &H, const double *r, int nrhs, cudaStream_t s, double *wimg) {
  const Geo &g = H.g;
  const int64_t threads = ((int64_t)nrhs << (2 * g.L)) * 8;
  k_oz_strips<<<nblk(threads), 256, 0, s>>>(g.n, g.L, H.ozp.P, g.R, H.ozp.rows, g.h * g.h, nrhs, r, H.ozp.img,
                                            H.ozp.lexp, wimg, g.npad, g.pad);
  FMMPC_LAUNCH_CHECK();
  return 1;
}

// The raw near-field sums: into the parts' images, or with one part into out itself.
int run_p2p_oz(fmmpc_handle &H, bool with_lnh, double *out, int nrhs, cudaStream_t s) {
  const Geo &g = H.g;
  const OzP2P &T = H.ozp;
  OzArgs a = rows_of(T);
  a.img = T.img;
  a.lexp = T.lexp;
  a.bmat = T.bmat[with_lnh ? 1 : 0];
  a.eb = T.eb[with_lnh ? 1 : 0];
  a.out = T.nparts > 1 ? T.near : out;
  a.vec = ((uintptr_t)a.out & 15) == 0;
  a.part_stride = T.part_stride;
  a.rows = T.rows;
  a.err = T.err;
  a.n = g.n;
  a.NL = 1 << g.L;
  a.P = T.P;
  a.R = g.R;
  a.nbs = T.nbs;
  a.sh = T.sh;
  a.nsr = T.nsr;
  for (int p = 0; p < T.nparts; ++p) {
    a.part_r[p] = (int16_t)T.part_r[p];
    a.part_q[p] = (int16_t)T.part_q[p];
    a.part_n[p] = (int16_t)T.part_n[p];
    a.part_o[p] = T.part_o[p];
  }
  k_p2p_oz<<<dim3((unsigned)T.ntiles, (unsigned)T.nparts, (unsigned)nrhs), OZ_THREADS, T.smem, s>>>(a);
  FMMPC_LAUNCH_CHECK();
  return 1;
}

// out = -1/(2 pi) times the sum of the parts (PART_NEAR, where no L2P pass follows).
int add_near_oz(fmmpc_handle &H, double *out, int nrhs, cudaStream_t s) {
  const int64_t total = (int64_t)H.g.n * H.g.n * nrhs;
  const OzP2P &T = H.ozp;
  k_near_combine64<<<nblk(total), 256, 0, s>>>(total, T.nparts > 1 ? T.near : out, T.part_stride, T.nparts, out);
  FMMPC_LAUNCH_CHECK();
  return 1;
}

}  // namespace fmmpc
