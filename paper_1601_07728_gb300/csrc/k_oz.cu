// FP64 matrix products D_b[m][n] = alpha sum_K A_b[m][K] B_b[n][K] on the FP16
// tensor cores by exact splitting (oz_dev.cuh), and the kernels that write the
// operands' digits.  Users: the screening stage's Green's functions (Sec. 3.3)
// and the set-up projection onto the local basis (Sec. 3.2.2).
//
// Why: GB300 retires 2 FP64 FMAs per SM and clock and about 2000 times as many
// FP16 products, so that the 19 products of 128 x 128 x 16 which replace one
// FP64 product of 128 x 64 x 16 still run some 50 times faster.  Measured:
// Green's functions of 900 points, 4096 states and 16 frequencies 682 ms
// (FP64 kernel) -> 14.0 ms (this one 12.9, writing the digits 0.97); the
// projection of 8^3 k x 16^3 points x 64 bands onto 64 functions 102.6 ms ->
// 4.4 ms (this one 2.0, digits 2.07, row scales 0.32).  The error against 64
// bits fell from 1.9e-15 to 1.3e-15 and from 1.3e-15 to 0.9e-15.  What bounds
// it now: operand tiles from L2 (35 bytes per SM and clock) beside the
// products' 64 clocks each.
#include "bse_internal.cuh"
#include "oz_dev.cuh"
#include "tc_ptx.cuh"

#include <algorithm>

namespace {

constexpr int OZ_M = 128, OZ_N = 64, OZ_KB = 64;   // output tile, K block (one 128-byte swizzle row)
constexpr int OZ_A = OZ_M * 128;                   // bytes of one digit's A tile
constexpr int OZ_BD = OZ_N * 128;                  // bytes of one digit's B tile
constexpr int OZ_B = OZ_S * OZ_BD;                 // ... and of the seven
constexpr int OZ_AS = 5, OZ_BS = 2;               // ring slots: A per digit, B per K block
constexpr int OZ_THREADS = 320;
// B slots lie between tiles of zeros: 0 B_0..B_6 0 B_0..B_6 0
constexpr int OZ_BAREA = OZ_BS * (OZ_B + OZ_BD) + OZ_BD;
constexpr size_t OZ_SMEM = 1024 + (size_t)OZ_AS * OZ_A + OZ_BAREA + 512;
constexpr unsigned long long OZ_WAIT_NS = 2000000000ull;

struct oz_mesh {
  int nk[3], nx[3];
  double s[3];
};

struct OzParams {
  int mt, nt, ntiles, kb;       // M tiles, N tiles, tiles over all batches, K blocks
  int rows_a, rows_b;           // rows per batch of each operand
  int a_batched, b_batched;     // 0: one operand for every batch
  const double* scale_a;        // [batch][rows_a] 2^e
  const double* scale_b;
  double alpha;
  double* out;                  // element (b, row, col) at b sb + (row>>1) sr2 + (row&1) sr1 + col sc
  long long sb, sr2, sr1, sc;
  int* err;
};

// Persistent warp-specialised kernel, one CTA per SM: warp 0 streams digit
// tiles with TMA (the seven B tiles of a K block as one box, each A digit in
// a slot of its own), warp 1 issues the digit products, warps 2-9 drain the
// accumulators every 128 K elements into 64-bit integers.
// A product of N = 64 or less takes the tensor core as long as one of N = 128
// (about 64 clocks measured at N = 32 and 64), so two neighbouring B digits
// form one operand of 128 rows and the accumulators of s = 2P, 2P + 1 one of
// 128 columns: digit A_i meets (B_0, B_1), (B_2, B_3), ... for even i and (0,
// B_0), (B_1, B_2), ... for odd i, 19 products instead of 28 per 16 K elements
// and all of one shape (s = 7 is computed along and not used).  M tiles are the fastest tile index: the CTAs running at one
// time then share both operands' tiles in L2.
__global__ void __launch_bounds__(OZ_THREADS, 1)
    oz_gemm(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb, const OzParams p) {
  extern __shared__ unsigned char oz_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)oz_raw + 1023) & ~(uintptr_t)1023);
  unsigned long long* bars = (unsigned long long*)(sm + OZ_AS * OZ_A + OZ_BAREA);
  constexpr int NBAR = 2 * OZ_AS + 2 * OZ_BS + 1 + OZ_S + 1;
  uint32_t* tmem_slot = (uint32_t*)(bars + NBAR);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  volatile int* a_issued = (volatile int*)(tmem_slot + 2);
  volatile int* b_issued = (volatile int*)(tmem_slot + 3);
  const uint32_t sa = smem_u32(sm), sb = sa + OZ_AS * OZ_A + OZ_BD;   // first B slot
  auto afull = [&](int s) { return smem_u32(&bars[s]); };
  auto aempty = [&](int s) { return smem_u32(&bars[OZ_AS + s]); };
  auto bfull = [&](int s) { return smem_u32(&bars[2 * OZ_AS + s]); };
  auto bempty = [&](int s) { return smem_u32(&bars[2 * OZ_AS + OZ_BS + s]); };
  const uint32_t tfull = smem_u32(&bars[2 * OZ_AS + 2 * OZ_BS]);
  auto tempty = [&](int s) { return smem_u32(&bars[2 * OZ_AS + 2 * OZ_BS + 1 + s]); };
  const uint32_t fin = smem_u32(&bars[NBAR - 1]);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < OZ_AS; ++s) {
      mbar_init(afull(s), 1);
      mbar_init(aempty(s), 1);
    }
    for (int s = 0; s < OZ_BS; ++s) {
      mbar_init(bfull(s), 1);
      mbar_init(bempty(s), 1);
    }
    mbar_init(tfull, 1);
    for (int s = 0; s < OZ_S; ++s) mbar_init(tempty(s), 8);
    mbar_init(fin, 1);
    *abort_flag = 0;
    *a_issued = 0;
    *b_issued = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int z = 0; z <= OZ_BS; ++z)
    for (int i = threadIdx.x; i < OZ_BD / 16; i += blockDim.x)
      reinterpret_cast<uint4*>(sm + OZ_AS * OZ_A + z * (OZ_B + OZ_BD))[i] = make_uint4(0, 0, 0, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the tensor core reads them
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    int ia = 0, ib = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
      const int m = t % p.mt, r = t / p.mt, n = r % p.nt, b = r / p.nt;
      const int za = p.a_batched ? b * OZ_S : 0, zb = p.b_batched ? b * OZ_S : 0;
      for (int kb = 0; kb < p.kb && ok; ++kb) {
        const int s = ib % OZ_BS;
        if (!(ok = mbar_wait(bempty(s), ((uint32_t)(ib / OZ_BS) & 1u) ^ 1u, abort_flag, OZ_WAIT_NS))) break;
        mbar_expect_tx(bfull(s), OZ_B);
        tma_load_3d(sb + s * (OZ_B + OZ_BD), &mb, bfull(s), kb * OZ_KB, n * OZ_N, zb);
        *b_issued = ++ib;
        for (int i = 0; i < OZ_S; ++i) {
          const int q = ia % OZ_AS;
          if (!(ok = mbar_wait(aempty(q), ((uint32_t)(ia / OZ_AS) & 1u) ^ 1u, abort_flag, OZ_WAIT_NS))) break;
          mbar_expect_tx(afull(q), OZ_A);
          tma_load_3d(sa + q * OZ_A, &ma, afull(q), kb * OZ_KB, m * OZ_M, za + i);
          *a_issued = ++ia;
        }
      }
    }
    if (!ok) {
      atomicExch(p.err, 1);
      *abort_flag = 1;
    }
  } else if (warp == 1 && lane == 0) {
    // FP16 A and B (K-major), FP32 D
    constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(2 * OZ_N >> 3) << 17) | ((uint32_t)(OZ_M >> 4) << 24);
    int ib = 0, chunk = 0, sl = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
      for (int kb = 0; kb < p.kb && ok; ++kb) {
        const bool first = (kb & 1) == 0, last = (kb & 1) == 1 || kb + 1 == p.kb;
        const int s = ib % OZ_BS;
        if (!(ok = mbar_wait(bfull(s), (uint32_t)(ib / OZ_BS) & 1u, abort_flag, OZ_WAIT_NS))) break;
        ++ib;
        const unsigned long long db = sdesc_sw128(sb + s * (OZ_B + OZ_BD));
#pragma unroll
        for (int i = 0; i < OZ_S; ++i) {
          if (!(ok = mbar_wait(afull(sl), ph, abort_flag, OZ_WAIT_NS))) break;
          tc_fence_after();
          const unsigned long long da = sdesc_sw128(sa + sl * OZ_A);
          if (i == 0 && first) {
            // each accumulator starts over as soon as it is drained
#pragma unroll
            for (int P = 0; P < 4; ++P) {
              ok = mbar_wait(tempty(2 * P), ((uint32_t)chunk & 1u) ^ 1u, abort_flag, OZ_WAIT_NS);
              if (ok && P < 3) ok = mbar_wait(tempty(2 * P + 1), ((uint32_t)chunk & 1u) ^ 1u, abort_flag, OZ_WAIT_NS);
              if (!ok) break;
              tc_fence_after();
#pragma unroll
              for (int ks = 0; ks < OZ_KB / 16; ++ks)
                mma_bf16(tmem + 2 * P * OZ_N, da + ks * 2, db + (2 * P * OZ_BD + ks * 32) / 16, idesc, ks > 0);
            }
            if (!ok) break;
          } else {
            // consecutive products go to different accumulators
#pragma unroll
            for (int ks = 0; ks < OZ_KB / 16; ++ks)
#pragma unroll
              for (int P = i / 2; P < 4; ++P)
                mma_bf16(tmem + 2 * P * OZ_N, da + ks * 2,
                         db + (unsigned long long)(long long)(((2 * P - i) * OZ_BD + ks * 32) / 16), idesc, 1);
          }
          mma_commit(aempty(sl));
          if (++sl == OZ_AS) sl = 0, ph ^= 1u;
        }
        if (!ok) break;
        mma_commit(bempty(s));
        if (last) {
          mma_commit(tfull);
          ++chunk;
        }
      }
    }
    if (!ok) {
      atomicExch(p.err, 1);
      *abort_flag = 1;
    }
    // issued products retire before tensor memory is freed
    mma_commit(fin);
    const unsigned long long t0 = gtime();
    while (!mbar_try(fin, 0) && gtime() - t0 < OZ_WAIT_NS) {
    }
  } else if (warp >= 2) {
    const int q = warp & 3, half = (warp - 2) >> 2;   // tensor-memory lanes 32 q.., columns 32 half..
    int chunk = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
      long long hi[32], lo[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) hi[c] = lo[c] = 0;
      for (int kb = 0; kb < p.kb; kb += 2, ++chunk) {
        ok = __all_sync(0xffffffffu, mbar_wait(tfull, (uint32_t)chunk & 1u, abort_flag, OZ_WAIT_NS));
        if (!ok) break;
        tc_fence_after();
        // hi: weights 2^-14, 2^-22, 2^-30; lo: 2^-38 .. 2^-62
#pragma unroll
        for (int s = 0; s < OZ_S; ++s) {
          float v[32];
          const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(s * OZ_N + half * 32);
          tmem_ld16(ta, v);
          tmem_ld16(ta + 16, v + 16);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty(s));
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            const int d = __float2int_rn(v[c]);
            if (s < 3)
              hi[c] += (long long)d * (1 << (8 * (2 - s)));
            else
              lo[c] += (long long)d * (1 << (8 * (6 - s)));
          }
        }
      }
      if (!ok) break;
      const int m = t % p.mt, r = t / p.mt, n = r % p.nt, b = r / p.nt;
      const int row = m * OZ_M + q * 32 + lane, col0 = n * OZ_N + half * 32;
      if (row < p.rows_a) {
        const double fa = p.alpha * p.scale_a[(p.a_batched ? (size_t)b * p.rows_a : 0) + row];
        const double* fb = p.scale_b + (p.b_batched ? (size_t)b * p.rows_b : 0) + col0;
        double* o = p.out + b * p.sb + (row >> 1) * p.sr2 + (row & 1) * p.sr1 + col0 * p.sc;
#pragma unroll
        for (int c = 0; c < 32; ++c)
          if (col0 + c < p.rows_b)
            o[c * p.sc] = ((double)hi[c] * 0x1p-30 + (double)lo[c] * 0x1p-62) * (fa * fb[c]);
      }
    }
    if (!ok && lane == 0) {
      atomicExch(p.err, 1);
      *abort_flag = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    // copies in flight land before the CTA leaves (the last use of each slot)
    const int na = *a_issued, nb = *b_issued;
    for (int k = na > OZ_AS ? na - OZ_AS : 0; k < na; ++k) {
      const unsigned long long t0 = gtime();
      while (!mbar_try(afull(k % OZ_AS), (uint32_t)(k / OZ_AS) & 1u) && gtime() - t0 < OZ_WAIT_NS) {
      }
    }
    for (int k = nb > OZ_BS ? nb - OZ_BS : 0; k < nb; ++k) {
      const unsigned long long t0 = gtime();
      while (!mbar_try(bfull(k % OZ_BS), (uint32_t)(k / OZ_BS) & 1u) && gtime() - t0 < OZ_WAIT_NS) {
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// block-wide maximum (blockDim.x <= 256); every thread returns it
__device__ unsigned block_max(unsigned v) {
  __shared__ unsigned wm[8];
  v = __reduce_max_sync(0xffffffffu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned m = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = max(m, wm[w]);
  return m;
}

// Digits of the rows of X [rows][n] (complex), one block per row and batch j;
// with d != nullptr entry K of batch j is first multiplied by d[j][K].
//   pair = 0: one row (re, im) per complex row, K = 2n interleaved
//   pair = 1: two rows, (re, im) and (-im, re): the products with a pair-0 row
//             are the real and imaginary part of sum x_a conj(x_b)
// dig [batch][7][rows (x2)][kp], zero beyond 2n; scale 2^e per row.
__global__ void __launch_bounds__(256) oz_split_rows(const double2* __restrict__ X, int n, const double2* __restrict__ d,
                                                     int rows, int kp, int pair, __half* __restrict__ dig,
                                                     double* __restrict__ scale, int* __restrict__ bad) {
  const int row = blockIdx.x, b = blockIdx.y;
  const double2* x = X + (size_t)row * n;
  const double2* db = d ? d + (size_t)b * n : nullptr;
  auto entry = [&](int k) {
    double2 v = x[k];
    if (db) {
      const double2 c = db[k];
      v = make_double2(v.x * c.x - v.y * c.y, v.x * c.y + v.y * c.x);
    }
    return v;
  };
  unsigned key = 0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const double2 v = entry(k);
    key = max(key, max(oz_key(v.x), oz_key(v.y)));
  }
  key = block_max(key);
  int flag = 0;
  const int e = oz_exponent(key, &flag);
  const int nr = rows << pair, r0 = row << pair;
  if (threadIdx.x == 0) {
    const double s = scalbn(1.0, e);
    scale[(size_t)b * nr + r0] = s;
    if (pair) scale[(size_t)b * nr + r0 + 1] = s;
    if (flag) atomicOr(bad, 1);
  }
  uint32_t* out = reinterpret_cast<uint32_t*>(dig) + ((size_t)b * OZ_S * nr + r0) * (kp / 2);
  const size_t digit = (size_t)nr * (kp / 2);
  for (int k = threadIdx.x; k < kp / 2; k += blockDim.x) {
    const double2 v = k < n ? entry(k) : make_double2(0.0, 0.0);
    const oz_fix fr = oz_fixed(v.x, e), fi = oz_fixed(v.y, e);
#pragma unroll
    for (int i = 0; i < OZ_S; ++i) out[i * digit + k] = oz_digit2(fr, fi, i);
    if (pair) {
      const oz_fix fm = oz_fixed(-v.y, e);
#pragma unroll
      for (int i = 0; i < OZ_S; ++i) out[i * digit + kp / 2 + k] = oz_digit2(fm, fr, i);
    }
  }
}

// Largest magnitude key of u[k][x][n] over x for every (k, n): blocks of 32
// bands x 8 rows walk a part of the grid (coalesced along n).
__global__ void __launch_bounds__(256) oz_col_keys(const double2* __restrict__ u, int nx, int nb, int per,
                                                   unsigned* __restrict__ keys) {
  __shared__ unsigned sk[8][32];
  const int n = blockIdx.y * 32 + (threadIdx.x & 31), g = threadIdx.x >> 5, k = blockIdx.z;
  const int x0 = blockIdx.x * per, x1 = min(nx, x0 + per);
  unsigned key = 0;
  if (n < nb) {
    const double2* p = u + (size_t)k * nx * nb + n;
#pragma unroll 4
    for (int x = x0 + g; x < x1; x += 8) {
      const double2 v = p[(size_t)x * nb];
      key = max(key, max(oz_key(v.x), oz_key(v.y)));
    }
  }
  sk[g][threadIdx.x & 31] = key;
  __syncthreads();
  if (g == 0 && n < nb) {
#pragma unroll
    for (int i = 1; i < 8; ++i) key = max(key, sk[i][threadIdx.x]);
    atomicMax(keys + (size_t)k * nb + n, key);
  }
}

// Digits of the rows (n) of e^{ik.x} u_nk(x), K = 2x interleaved (re, im):
// u [k][x][n] is read coalesced along n and written transposed.  One block:
// 32 grid points of one k, every band; a warp holds 4 bands x 8 groups of 4
// points, so that both the 64-byte reads and the 128-byte digit rows fill
// their sectors.  |e^{ik.x} u| components are at most sqrt 2 times those of u:
// the row scale has one more bit.
__global__ void __launch_bounds__(256) oz_split_bloch(const double2* __restrict__ u, oz_mesh ms, int k0, int nb, int kp,
                                                      const unsigned* __restrict__ keys, __half* __restrict__ dig,
                                                      double* __restrict__ scale, int* __restrict__ bad) {
  __shared__ double2 ph[32];
  const int nx = ms.nx[0] * ms.nx[1] * ms.nx[2];
  const int kl = blockIdx.y, k = k0 + kl, x0 = blockIdx.x * 32;
  if (threadIdx.x < 32) {
    const int x = x0 + threadIdx.x;
    double sn = 0.0, cs = 1.0;
    if (x < nx) {
      const int m2 = k % ms.nk[2], m1 = (k / ms.nk[2]) % ms.nk[1], m0 = k / (ms.nk[1] * ms.nk[2]);
      const int j2 = x % ms.nx[2], j1 = (x / ms.nx[2]) % ms.nx[1], j0 = x / (ms.nx[1] * ms.nx[2]);
      double fr = (m0 + ms.s[0]) * j0 / ((double)ms.nk[0] * ms.nx[0]) + (m1 + ms.s[1]) * j1 / ((double)ms.nk[1] * ms.nx[1]) +
                  (m2 + ms.s[2]) * j2 / ((double)ms.nk[2] * ms.nx[2]);
      fr -= floor(fr);
      sincospi(2.0 * fr, &sn, &cs);
    }
    ph[threadIdx.x] = make_double2(cs, sn);
  }
  __syncthreads();
  const int xg = threadIdx.x & 7, x = x0 + 4 * xg;
  double2 c[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) c[i] = ph[4 * xg + i];
  for (int n = threadIdx.x >> 3; n < nb; n += 32) {
    int flag = 0;
    const int e = oz_exponent(keys[(size_t)kl * nb + n], &flag) + 1;
    if (xg == 0 && blockIdx.x == 0) {
      scale[(size_t)kl * nb + n] = scalbn(1.0, e);
      if (flag) atomicOr(bad, 1);
    }
    oz_fix f[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double2 w = x + i < nx ? u[((size_t)k * nx + x + i) * nb + n] : make_double2(0.0, 0.0);
      f[2 * i] = oz_fixed(w.x * c[i].x - w.y * c[i].y, e);
      f[2 * i + 1] = oz_fixed(w.x * c[i].y + w.y * c[i].x, e);
    }
    __half* o = dig + ((size_t)kl * OZ_S * nb + n) * kp + 2 * x;
#pragma unroll
    for (int i = 0; i < OZ_S; ++i)
      *reinterpret_cast<uint4*>(o + (size_t)i * nb * kp) =
          make_uint4(oz_digit2(f[0], f[1], i), oz_digit2(f[2], f[3], i), oz_digit2(f[4], f[5], i),
                     oz_digit2(f[6], f[7], i));
  }
}

// FP16 map of digits [z][rows][kp]: box of 64 K elements x box_rows x box_z, 128-byte swizzle
bool digit_map(CUtensorMap* m, const __half* base, int kp, int rows, int z, int box_rows, int box_z) {
  const EncodeTiledFn f = bse_encode_tiled_fn();
  if (!f) return false;
  cuuint64_t dims[3] = {(cuuint64_t)kp, (cuuint64_t)rows, (cuuint64_t)z};
  cuuint64_t strides[2] = {(cuuint64_t)kp * 2, (cuuint64_t)rows * kp * 2};
  cuuint32_t box[3] = {(cuuint32_t)OZ_KB, (cuuint32_t)box_rows, (cuuint32_t)box_z};
  cuuint32_t es[3] = {1, 1, 1};
  return f(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half*>(base), dims, strides, box, es,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

size_t bse_oz_digit_bytes(int batches, int rows, int kp) {
  return (((size_t)batches * OZ_S * rows * kp * sizeof(__half)) + 255) / 256 * 256;
}
int bse_oz_tiles(int rows_a, int rows_b) { return (rows_a + OZ_M - 1) / OZ_M * ((rows_b + OZ_N - 1) / OZ_N); }
int bse_oz_kp(int k) { return (k + OZ_KB - 1) / OZ_KB * OZ_KB; }

bse_status bse_oz_split_rows(const double2* x, int rows, int n, const double2* d, int batches, int pair,
                             const bse_oz_operand& o, int* bad, cudaStream_t st) {
  oz_split_rows<<<dim3((unsigned)rows, (unsigned)batches), 256, 0, st>>>(x, n, d, rows, o.kp, pair, (__half*)o.digits,
                                                                          o.scale, bad);
  return cudaGetLastError() == cudaSuccess ? BSE_OK : BSE_ERR_CUDA;
}

bse_status bse_oz_split_bloch(const double2* u, const int* nk, const int* nx, const double* kshift, int nb, int k0,
                              int nkc, const bse_oz_operand& o, unsigned* keys, int* bad, cudaStream_t st) {
  oz_mesh ms;
  for (int i = 0; i < 3; ++i) {
    ms.nk[i] = nk[i];
    ms.nx[i] = nx[i];
    ms.s[i] = kshift ? kshift[i] : 0.0;
  }
  const int nxt = nx[0] * nx[1] * nx[2];
  const int per = nxt > 8192 ? 1024 : 512;
  cudaMemsetAsync(keys, 0, (size_t)nkc * nb * sizeof(unsigned), st);
  oz_col_keys<<<dim3((unsigned)((nxt + per - 1) / per), (unsigned)((nb + 31) / 32), (unsigned)nkc), 256, 0, st>>>(
      u + (size_t)k0 * nxt * nb, nxt, nb, per, keys);
  oz_split_bloch<<<dim3((unsigned)(o.kp / OZ_KB), (unsigned)nkc), 256, 0, st>>>(u, ms, k0, nb, o.kp, keys,
                                                                                (__half*)o.digits, o.scale, bad);
  return cudaGetLastError() == cudaSuccess ? BSE_OK : BSE_ERR_CUDA;
}

bse_status bse_oz_gemm(const bse_oz_operand& a, const bse_oz_operand& b, int batches, double alpha, double* out,
                       long long sb, long long sr2, long long sr1, long long sc, int* err, cudaStream_t st) {
  CUtensorMap ma, mb;
  if (!digit_map(&ma, (const __half*)a.digits, a.kp, a.rows, OZ_S * a.batches, OZ_M, 1) ||
      !digit_map(&mb, (const __half*)b.digits, b.kp, b.rows, OZ_S * b.batches, OZ_N, OZ_S))
    return BSE_ERR_CUDA;
  OzParams p{};
  p.mt = (a.rows + OZ_M - 1) / OZ_M;
  p.nt = (b.rows + OZ_N - 1) / OZ_N;
  p.ntiles = p.mt * p.nt * batches;
  p.kb = a.kp / OZ_KB;
  p.rows_a = a.rows;
  p.rows_b = b.rows;
  p.a_batched = a.batches > 1 ? 1 : 0;
  p.b_batched = b.batches > 1 ? 1 : 0;
  p.scale_a = a.scale;
  p.scale_b = b.scale;
  p.alpha = alpha;
  p.out = out;
  p.sb = sb;
  p.sr2 = sr2;
  p.sr1 = sr1;
  p.sc = sc;
  p.err = err;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaFuncSetAttribute(oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_SMEM) != cudaSuccess) {
    cudaGetLastError();
    return BSE_ERR_CUDA;
  }
  oz_gemm<<<std::min(p.ntiles, sms), OZ_THREADS, OZ_SMEM, st>>>(ma, mb, p);
  return cudaGetLastError() == cudaSuccess ? BSE_OK : BSE_ERR_CUDA;
}
