// Band<->grid contractions of Algorithm 1 (Sec. 3.2.1) in the FP64 form on the
// FP16 tensor cores by exact splitting (oz_dev.cuh).  U = e^{ik.x} u_nk(x) stays
// FP64 in memory and is split on the way into shared memory, so a pass reads
// its 16 bytes per entry once:
//   band->grid  phi[k][c][x] = sum_n U[k][x][n] psi[c][k][n]: A rows x, K = (n; re, im)
//   grid->band  D[q][j] = sum_x U[k][x][q] phi[k][j][x]:      A rows q = (n; re, im), K = x
// for up to eight complex columns at a time (sixteen real ones).
//
// Digit products (i, j) with i + j <= 7 are formed (one diagonal more than the
// long sums of k_oz.cu need: at K = 2 N_b ~ 100 the FP64 sums that this
// replaces lose only two or three bits).  The digits of psi or phi are stacked
// between tiles of zeros, 0 0 0 0 0 0 B_0 .. B_6 0, sixteen rows each, and A
// digit i multiplies the eight tiles from B_-i on: its products land in the
// columns of s = i + j = 0..7 of one accumulator.  Seven products of 128 x 128 x
// 16 per 16 K elements, all of one shape (products of different N in turn take
// 118 clocks each instead of 48, and N = 128 takes 64 where N = 16 takes 39).
// An accumulator holds 128 K elements exactly and is then drained.
//
// The digits hold an entry to 2^-56 of its row's largest, so every sum comes with
// that of its magnitudes, and those for which this is not FP64 accuracy are
// formed on the FP64 pipe (oz_accept; columns with Inf or NaN and columns below
// 2^-960 wholly): band->grid's by ozh_repair, grid->band's in ozh_final.
//
// L2,3 workload (8^3 k, 16^3 grid, 64 bands, 6 columns): H psi 15.0 ms with the
// FP64 kernels -> 2.86 in calls that follow one another on several streams (2.84
// with the magnitude sums left out); 3.15 by itself, of it the k-transform 1.08,
// oz_contract 0.92 and 0.90, digits of psi and phi 0.12, ozh_final 0.07.  What
// bounds oz_contract: the integer instructions that make digits (ALU pipe 68 and
// 78 % of active cycles, tensor pipe 24 and 29 %, DRAM 32 and 37 %).
#include "bse_internal.cuh"
#include "oz_dev.cuh"
#include "tc_ptx.cuh"

#include <math.h>

#include <algorithm>
#include <new>

namespace {

constexpr int H_C = 8, H_J = 2 * H_C;                // complex and real columns of a pass
constexpr int H_M = 128, H_KB = 32;                  // A rows, K elements of a stage (64-byte swizzle rows)
constexpr int H_STAGES = 3;
constexpr int H_A = H_M * H_KB * 2;                  // bytes of one digit's A tile
constexpr int H_BD = H_J * H_KB * 2;                 // bytes of one digit's B tile
constexpr int H_B = OZ_S * H_BD;                     // ... and of the seven
constexpr int H_BSTRIDE = H_B + (OZ_S - 1) * H_BD;   // a stage's B and the zeros before it
constexpr int H_N = 8 * H_J;                         // accumulator columns, s = 0..7
constexpr int H_BAREA = H_STAGES * H_BSTRIDE + H_BD; // ... zeros after the last stage
constexpr int H_CONV = 16;                           // conversion warps
constexpr int H_MAG = 2;                             // warps of the magnitude sums
constexpr int H_THREADS = 32 * (2 + 4 + H_CONV + H_MAG);
constexpr size_t H_SMEM = 1024 + (size_t)H_STAGES * OZ_S * H_A + H_BAREA + 256;
constexpr int H_CHUNK = 128 / H_KB;                  // K blocks until an accumulator is drained
constexpr unsigned long long H_DRAIN_NS = 2000000000ull;

// K-major operand in rows of 64 bytes (64-byte swizzle, 8-row groups 512 bytes apart)
__device__ __forceinline__ unsigned long long sdesc_sw64(uint32_t saddr) {
  unsigned long long d = 0;
  d |= (unsigned long long)((saddr & 0x3FFFFu) >> 4);
  d |= (unsigned long long)1 << 16;
  d |= (unsigned long long)(512 >> 4) << 32;
  d |= (unsigned long long)1 << 46;
  d |= (unsigned long long)4 << 61;   // SWIZZLE_64B
  return d;
}

// (hi 2^32 + lo) 2^e: three FP64-pipe operations; the exponent is added to the
// bits where the result stays a normal number
__device__ __forceinline__ double h_value(long long hi, long long lo, int e) {
  const double v = fma((double)hi, 4294967296.0, (double)lo);
  const int h = __double2hiint(v), ex = ((h >> 20) & 0x7ff) + e;
  if (v == 0.0) return 0.0;
  if (ex < 1 || ex > 2046) return scalbn(v, e);
  return __hiloint2double(h + (e << 20), __double2loint(v));
}

__device__ __forceinline__ void ldmatrix4_abs(uint32_t a, uint32_t* r) {   // ... as magnitudes
  ldmatrix_x4(a, r);
#pragma unroll
  for (int i = 0; i < 4; ++i) r[i] &= 0x7fff7fffu;
}

// FP64 sums over i < n of u_i p_c,i for the H_C columns p_c = p + c cs (those
// from nc on repeat the first), by one warp: lane L returns part (L >> 1) & 1 of column L >> 2
__device__ double warp_columns(const double2* __restrict__ u, const double2* __restrict__ p, size_t cs, int nc,
                                            int n) {
  double v[2 * H_C];
#pragma unroll
  for (int j = 0; j < 2 * H_C; ++j) v[j] = 0.0;
  const int lane = threadIdx.x & 31;
  for (int i = lane; i < n; i += 32) {
    const double2 a = u[i];
#pragma unroll
    for (int c = 0; c < H_C; ++c) {
      const double2 b = p[(c < nc ? c : 0) * cs + i];
      v[2 * c] = fma(a.x, b.x, fma(-a.y, b.y, v[2 * c]));
      v[2 * c + 1] = fma(a.x, b.y, fma(a.y, b.x, v[2 * c + 1]));
    }
  }
  // sums by exchanged halves: lane L ends with number L >> 1
#pragma unroll
  for (int h = H_C; h >= 1; h >>= 1) {
    const bool up = (lane & (2 * h)) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double mine = up ? v[h + i] : v[i], other = up ? v[i] : v[h + i];
      v[i] = mine + __shfl_xor_sync(0xffffffffu, other, 2 * h);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}
// FP64 sum of conj(u_i) p_i over i < n, entries of u `us` apart, by one warp; every lane returns it
__device__ double2 warp_dot(const double2* __restrict__ u, long long us, const double2* __restrict__ p, int n) {
  double x = 0.0, y = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x & 31; i < n; i += 32) {
    const double2 a = u[i * us], b = p[i];
    x = fma(a.x, b.x, fma(a.y, b.y, x));
    y = fma(a.x, b.y, fma(-a.y, b.x, y));
  }
  for (int off = 16; off > 0; off >>= 1) {
    x += __shfl_xor_sync(0xffffffffu, x, off);
    y += __shfl_xor_sync(0xffffffffu, y, off);
  }
  return make_double2(x, y);
}

// A column of psi or phi: its norm in units of its scale and sqrt(2 n) of its n
// entries other than 0; norm < 0: not to be summed from digits (Inf, NaN, or too small for them)
struct __align__(8) HColumn {
  float norm, root;
};
// norm_a: norm of the row of U; m: sum of magnitudes
__device__ __forceinline__ bool column_accepts(HColumn c, float norm_a, float m) {
  return c.norm >= 0.f && (c.norm == 0.f || norm_a == 0.f || oz_accept(m, fminf(norm_a, c.root), c.norm));
}

struct HParams {
  const double2* u;       // [nk][nx][nb]
  const short* ea;        // exponent per A row: [nk][nx] (mode 0) or [nk][nb] (mode 1)
  const float* na;        // mode 0: norm per grid row in units of its scale
  const int* eb;          // exponent per column: [nk][H_C]
  const HColumn* cb;      // mode 0: columns [nk][H_C]
  unsigned char* refused; // mode 0: [nk][nx], a bit per column whose sum is to come from the FP64 pipe
  int* any;               // mode 0: set where there is one
  double2* out;           // mode 0: phi; mode 1: partial sums [split][nk][H_C][nb]
  float* sums;            // mode 1: sums of magnitudes, as out
  int nk, nx, nb, mt, nsplit, ntiles, kb, kb_per_split;
  int nc, c0, ncc;        // mode 0: columns of phi, first column, columns of this pass
  int* err;
  unsigned long long wait_ns;
};

// Persistent, one CTA per SM: warp 0 brings B with TMA, warp 1 issues the
// products, warps 2-5 drain tensor memory, warps 6-21 read U (the next stage's
// loads are in flight while one is split) and write its digits, warps 22 and 23
// sum the magnitudes and say which results they accept (oz_accept).
template <int MODE>
__global__ void __launch_bounds__(H_THREADS, 1) oz_contract(const __grid_constant__ CUtensorMap mb, const HParams p) {
  extern __shared__ unsigned char ozh_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)ozh_raw + 1023) & ~(uintptr_t)1023);
  unsigned long long* bars = (unsigned long long*)(sm + H_STAGES * OZ_S * H_A + H_BAREA);
  uint32_t* tmem_slot = (uint32_t*)(bars + 3 * H_STAGES + 5);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  volatile int* issued = (volatile int*)(tmem_slot + 2);
  const uint32_t sbase = smem_u32(sm);
  const uint32_t bbase = sbase + H_STAGES * OZ_S * H_A + (OZ_S - 1) * H_BD;   // B_0 of the first stage
  auto afull = [&](int s) { return smem_u32(&bars[s]); };
  auto bfull = [&](int s) { return smem_u32(&bars[H_STAGES + s]); };
  auto empty = [&](int s) { return smem_u32(&bars[2 * H_STAGES + s]); };
  auto tfull = [&](int a) { return smem_u32(&bars[3 * H_STAGES + a]); };
  auto tempty = [&](int a) { return smem_u32(&bars[3 * H_STAGES + 2 + a]); };
  const uint32_t fin = smem_u32(&bars[3 * H_STAGES + 4]);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < H_STAGES; ++s) {
      mbar_init(afull(s), H_CONV);
      mbar_init(bfull(s), 1);
      mbar_init(empty(s), 1 + H_MAG);   // read by the products and the magnitude sums
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull(a), 1);
      mbar_init(tempty(a), 4);
    }
    mbar_init(fin, 1);
    *abort_flag = 0;
    *issued = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < H_BAREA / 16; i += blockDim.x)
    reinterpret_cast<uint4*>(sm + H_STAGES * OZ_S * H_A)[i] = make_uint4(0, 0, 0, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), 2 * H_N);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // tile t: split fastest, then M tile, then k; its K blocks [b0, b1)
  auto tile = [&](int t, int& k, int& m, int& sp, int& b0, int& b1) {
    sp = t % p.nsplit;
    const int r = t / p.nsplit;
    m = r % p.mt;
    k = r / p.mt;
    b0 = sp * p.kb_per_split;
    b1 = b0 + p.kb_per_split < p.kb ? b0 + p.kb_per_split : p.kb;
  };

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
        int k, m, sp, b0, b1;
        tile(t, k, m, sp, b0, b1);
        for (int b = b0; b < b1; ++b, ++it) {
          const int s = it % H_STAGES;
          if (!(ok = mbar_wait(empty(s), ((uint32_t)(it / H_STAGES) & 1u) ^ 1u, abort_flag, p.wait_ns))) break;
          mbar_expect_tx(bfull(s), H_B);
          tma_load_3d(bbase + s * H_BSTRIDE, &mb, bfull(s), b * H_KB, 0, k * OZ_S);
          *issued = it + 1;
        }
      }
      if (!ok) {
        atomicExch(p.err, 1);
        *abort_flag = 1;
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int it = 0, chunk = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
        int k, m, sp, b0, b1;
        tile(t, k, m, sp, b0, b1);
        for (int b = b0; b < b1 && ok; ++b, ++it) {
          const int pos = (b - b0) % H_CHUNK, acc = chunk & 1;
          if (pos == 0) {
            if (!(ok = mbar_wait(tempty(acc), ((uint32_t)(chunk >> 1) & 1u) ^ 1u, abort_flag, p.wait_ns))) break;
            tc_fence_after();
          }
          const int s = it % H_STAGES;
          const uint32_t ph = (uint32_t)(it / H_STAGES) & 1u;
          if (!(ok = mbar_wait(bfull(s), ph, abort_flag, p.wait_ns) && mbar_wait(afull(s), ph, abort_flag, p.wait_ns))) break;
          tc_fence_after();
          // FP16 in, FP32 out, M = 128, N = 128
          constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(H_N >> 3) << 17) | ((uint32_t)(H_M >> 4) << 24);
          const unsigned long long da = sdesc_sw64(sbase + s * (OZ_S * H_A)), db = sdesc_sw64(bbase + s * H_BSTRIDE);
          const uint32_t d = tmem + acc * H_N;
#pragma unroll
          for (int ks = 0; ks < H_KB / 16; ++ks)
#pragma unroll
            for (int i = 0; i < OZ_S; ++i)
              mma_bf16(d, da + (i * H_A + ks * 32) / 16, db - (i * H_BD) / 16 + ks * 2, idesc, !(pos == 0 && ks == 0 && i == 0));
          mma_commit(empty(s));
          if (pos == H_CHUNK - 1 || b + 1 == b1) {
            mma_commit(tfull(acc));
            ++chunk;
          }
        }
      }
      if (!ok) {
        atomicExch(p.err, 1);
        *abort_flag = 1;
      }
      mma_commit(fin);   // issued products retire before tensor memory is freed
      const unsigned long long t0 = gtime();
      while (!mbar_try(fin, 0) && gtime() - t0 < H_DRAIN_NS) {
      }
    }
  } else if (warp < 6) {
    const int q = warp & 3, row = q * 32 + lane;
    const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16);
    int chunk = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
      int k, m, sp, b0, b1;
      tile(t, k, m, sp, b0, b1);
      long long hi[H_J], lo[H_J];   // units 2^-38 (s <= 3) and 2^-70 (s = 4..7)
#pragma unroll
      for (int c = 0; c < H_J; ++c) hi[c] = lo[c] = 0;
      for (int b = b0; b < b1; b += H_CHUNK, ++chunk) {
        const int acc = chunk & 1;
        ok = __all_sync(0xffffffffu, mbar_wait(tfull(acc), (uint32_t)(chunk >> 1) & 1u, abort_flag, p.wait_ns));
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          float v[H_J];
          tmem_ld16(ta + acc * H_N + s * H_J, v);
#pragma unroll
          for (int c = 0; c < H_J; ++c) {
            const int d = __float2int_rn(v[c]);
            if (s < 4)
              hi[c] += (long long)d * (1 << (8 * (3 - s)));
            else
              lo[c] += (long long)d * (1 << (8 * (7 - s)));
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty(acc));
      }
      if (!ok) break;
      const int* eb = p.eb + (size_t)k * H_C;
      if constexpr (MODE == 0) {
        const int x = m * H_M + row;
        if (x < p.nx) {
          const int ea = p.ea[(size_t)k * p.nx + x];
#pragma unroll
          for (int c = 0; c < H_C; ++c)
            if (c < p.ncc) {
              const int e = eb[c] + ea - 70;
              p.out[((size_t)k * p.nc + p.c0 + c) * p.nx + x] =
                  make_double2(h_value(hi[2 * c], lo[2 * c], e), h_value(hi[2 * c + 1], lo[2 * c + 1], e));
            }
        }
      } else {
        double v[H_J];
        const int n = (m * H_M + row) >> 1;
        const int ea = n < p.nb ? p.ea[(size_t)k * p.nb + n] : 0;
#pragma unroll
        for (int j = 0; j < H_J; ++j) {
          if ((j >> 1) >= p.ncc) continue;
          v[j] = h_value(hi[j], lo[j], ea + eb[j >> 1] - 70);
        }
        // psi'_{c,n} = (D[2n][2c] + D[2n+1][2c+1]) + i (D[2n][2c+1] - D[2n+1][2c])
        const size_t o = ((size_t)sp * p.nk + k) * H_C * p.nb + n;
#pragma unroll
        for (int c = 0; c < H_C; ++c) {
          if (c >= p.ncc) continue;
          const double w0 = __shfl_xor_sync(0xffffffffu, v[2 * c], 1), w1 = __shfl_xor_sync(0xffffffffu, v[2 * c + 1], 1);
          if ((lane & 1) == 0 && n < p.nb) p.out[o + (size_t)c * p.nb] = make_double2(v[2 * c] + w1, v[2 * c + 1] - w0);
        }
      }
    }
    if (!ok && lane == 0) {
      atomicExch(p.err, 1);
      *abort_flag = 1;
    }
  } else if (warp >= 6 + H_CONV) {
    // ---------------- sums of magnitudes ----------------
    // 64 rows x 16 columns each with a product of the older tensor-core form on
    // the leading digits' tiles, beside the stage's seven products of 128 x 128.
    // Done by the draining warps it held the stages up (band->grid 1.4 instead
    // of 0.98 ms); their comparison with the norms there alone cost 0.23 ms.
    const int w = warp - (6 + H_CONV), br = (lane & 7) + ((lane >> 4) << 3);
    const int row0 = w * 64 + (lane >> 2);   // first of this lane's rows, 8 apart; its columns lane & 3 and 4 on
    int it = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
      int k, m, sp, b0, b1;
      tile(t, k, m, sp, b0, b1);
      float c[4][2][4], na[8];
      HColumn cb[2];
      if constexpr (MODE == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int x = m * H_M + row0 + 8 * i;
          na[i] = x < p.nx ? p.na[(size_t)k * p.nx + x] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int col = (lane & 3) + 4 * i;
          cb[i] = col < p.ncc ? p.cb[(size_t)k * H_C + col] : HColumn{0.f, 0.f};
        }
      }
#pragma unroll
      for (int i = 0; i < 32; ++i) c[i >> 3][(i >> 2) & 1][i & 3] = 0.f;
      for (int b = b0; b < b1; ++b, ++it) {
        const int s = it % H_STAGES;
        const uint32_t ph = (uint32_t)(it / H_STAGES) & 1u;
        ok = __all_sync(0xffffffffu, mbar_wait(bfull(s), ph, abort_flag, p.wait_ns) &&
                                         mbar_wait(afull(s), ph, abort_flag, p.wait_ns));
        if (!ok) break;
        const uint32_t at = sbase + s * (OZ_S * H_A), bt = bbase + s * H_BSTRIDE;
#pragma unroll
        for (int ks = 0; ks < H_KB / 16; ++ks) {
          uint32_t bq[4];
          ldmatrix4_abs(bt + br * 64 + (((2 * ks + ((lane >> 3) & 1)) ^ ((br >> 1) & 3)) << 4), bq);
#pragma unroll
          for (int mt = 0; mt < 4; ++mt) {
            const int ar = w * 64 + mt * 16 + (lane & 15);
            uint32_t aq[4];
            ldmatrix4_abs(at + ar * 64 + (((2 * ks + (lane >> 4)) ^ ((ar >> 1) & 3)) << 4), aq);
            mma_16x8x16<false>(c[mt][0], aq, bq[0], bq[1]);
            mma_16x8x16<false>(c[mt][1], aq, bq[2], bq[3]);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty(s));
      }
      if (!ok) break;
      // both parts of a complex column together, in units of the two scales
      auto sum = [&](int i, int nt) { return (c[i >> 1][nt][2 * (i & 1)] + c[i >> 1][nt][2 * (i & 1) + 1]) * 0x1p-14f; };
      if constexpr (MODE == 0) {
        unsigned any = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int x = m * H_M + row0 + 8 * i;
          unsigned f = 0;
#pragma unroll
          for (int nt = 0; nt < 2; ++nt)
            if (!column_accepts(cb[nt], na[i], sum(i, nt))) f |= 1u << ((lane & 3) + 4 * nt);
          f |= __shfl_xor_sync(0xffffffffu, f, 1);
          f |= __shfl_xor_sync(0xffffffffu, f, 2);
          if (x < p.nx) {
            any |= f;
            if ((lane & 3) == 0) p.refused[(size_t)k * p.nx + x] = (unsigned char)f;
          }
        }
        if (any) *p.any = 1;
      } else {
        // rows 2n and 2n + 1 (lanes 4 apart) are the parts of band n
        const size_t o = ((size_t)sp * p.nk + k) * H_C * p.nb;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int n = (m * H_M + row0 + 8 * i) >> 1;
#pragma unroll
          for (int nt = 0; nt < 2; ++nt) {
            const int col = (lane & 3) + 4 * nt;
            float v = sum(i, nt);
            v += __shfl_xor_sync(0xffffffffu, v, 4);
            if ((lane & 4) == 0 && n < p.nb && col < p.ncc) p.sums[o + (size_t)col * p.nb + n] = v;
          }
        }
      }
    }
    if (!ok && lane == 0) {
      atomicExch(p.err, 1);
      *abort_flag = 1;
    }
  } else {
    // ---------------- U into digits ----------------
    // Four entries of U per thread and stage.  Mode 0: band r of the block in
    // rows q + 32 i (a warp reads two rows of 256 bytes and writes two rows of
    // 64 bytes per digit); mode 1: band r, points 8 q + 4 hf + i (the two
    // halves of a 16-byte chunk in neighbouring lanes).
    const int tid = threadIdx.x - 32 * 6;
    const int r = MODE == 0 ? tid & 15 : (tid >> 1) & 63, q = MODE == 0 ? tid >> 4 : tid >> 7, hf = tid & 1;
    int it = 0;
    bool ok = true;
    double2 w[4];
    // this thread's entries of block b of tile (k, m): base + b * step + i * pitch,
    // entry i present where i < left(b)
    const ptrdiff_t step = MODE == 0 ? H_KB / 2 : (ptrdiff_t)H_KB * p.nb, pitch = MODE == 0 ? (ptrdiff_t)32 * p.nb : p.nb;
    auto base = [&](int k, int m) {
      const int x = MODE == 0 ? m * H_M + q : 8 * q + 4 * hf, n = MODE == 0 ? r : m * (H_M / 2) + r;
      return p.u + ((size_t)k * p.nx + x) * p.nb + n;
    };
    auto left = [&](int m, int b) {
      if (MODE == 0) return b * (H_KB / 2) + r < p.nb ? (p.nx - m * H_M - q + 31) >> 5 : 0;
      return m * (H_M / 2) + r < p.nb ? p.nx - b * H_KB - 8 * q - 4 * hf : 0;
    };
    auto load = [&](const double2* a, int n) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        w[i] = make_double2(0.0, 0.0);
        if (i < n) w[i] = load_in_place(a + i * pitch);
      }
    };
    // lines of a block four ahead into L2, so that the register loads one block
    // ahead (32 KB per SM in flight) cover an L2 hit and not HBM's latency
    auto prefetch = [&](const double2* a, int n) {
      if (r & 7) return;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < n) asm volatile("prefetch.global.L2 [%0];" ::"l"(a + i * pitch));
    };
    int e[4], en[4];
    auto exponents = [&](int k, int m, int* o) {
#pragma unroll
      for (int i = 0; i < (MODE == 0 ? 4 : 1); ++i) {
        const int row = MODE == 0 ? m * H_M + q + 32 * i : m * (H_M / 2) + r, nr = MODE == 0 ? p.nx : p.nb;
        o[i] = row < nr ? p.ea[(size_t)k * nr + row] : 0;
      }
    };
    constexpr int AHEAD = 4;
    int t = blockIdx.x, k = 0, m = 0, sp = 0, b0 = 0, b1 = 0;
    int k2 = 0, m2 = 0, s2 = 0, c0 = 0, c1 = 0;
    const double2 *cur = nullptr, *nxt = nullptr;
#pragma unroll
    for (int i = 0; i < 4; ++i) e[i] = en[i] = 0;
    if (t < p.ntiles) {
      tile(t, k, m, sp, b0, b1);
      cur = base(k, m);
      load(cur + b0 * step, left(m, b0));
      exponents(k, m, e);
    }
    for (; t < p.ntiles && ok; t += gridDim.x) {
      const bool more = t + (int)gridDim.x < p.ntiles;
      if (more) {
        tile(t + gridDim.x, k2, m2, s2, c0, c1);
        nxt = base(k2, m2);
        exponents(k2, m2, en);
      }
      for (int b = b0; b < b1; ++b, ++it) {
        oz_fix f[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          f[2 * i] = oz_fixed(w[i].x, e[MODE == 0 ? i : 0]);
          f[2 * i + 1] = oz_fixed(w[i].y, e[MODE == 0 ? i : 0]);
        }
        // the next block's loads (of the next tile after the last one)
        if (b + 1 < b1)
          load(cur + (b + 1) * step, left(m, b + 1));
        else if (more)
          load(nxt + c0 * step, left(m2, c0));
        const int bn = c0 + b + AHEAD - b1;
        if (b + AHEAD < b1)
          prefetch(cur + (b + AHEAD) * step, left(m, b + AHEAD));
        else if (more && bn < c1)
          prefetch(nxt + bn * step, left(m2, bn));
        const int s = it % H_STAGES;
        if (!(ok = __all_sync(0xffffffffu, mbar_wait(empty(s), ((uint32_t)(it / H_STAGES) & 1u) ^ 1u, abort_flag, p.wait_ns))))
          break;
        // 64-byte rows, chunks of 16 bytes swizzled by the row
        unsigned char* st = sm + s * (OZ_S * H_A);
        if constexpr (MODE == 0) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int rr = q + 32 * i;
            uint32_t* o = reinterpret_cast<uint32_t*>(st + rr * 64 + (((r >> 2) ^ ((rr >> 1) & 3)) << 4) + (r & 3) * 4);
#pragma unroll
            for (int g = 0; g < OZ_S; ++g) o[g * (H_A / 4)] = oz_digit2(f[2 * i], f[2 * i + 1], g);
          }
        } else {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int rr = 2 * r + h;
            uint2* o = reinterpret_cast<uint2*>(st + rr * 64 + ((q ^ ((rr >> 1) & 3)) << 4) + hf * 8);
#pragma unroll
            for (int g = 0; g < OZ_S; ++g)
              o[g * (H_A / 8)] = make_uint2(oz_digit2(f[h], f[2 + h], g), oz_digit2(f[4 + h], f[6 + h], g));
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(afull(s));
      }
      m = m2, b0 = c0, b1 = c1, cur = nxt;
#pragma unroll
      for (int i = 0; i < 4; ++i) e[i] = en[i];
    }
    if (!ok && lane == 0) {
      atomicExch(p.err, 1);
      *abort_flag = 1;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    // copies of B in flight land before the CTA leaves (the last use of each slot)
    const int n = *issued;
    for (int j = n > H_STAGES ? n - H_STAGES : 0; j < n; ++j) {
      const unsigned long long t0 = gtime();
      while (!mbar_try(bfull(j % H_STAGES), (uint32_t)(j / H_STAGES) & 1u) && gtime() - t0 < H_DRAIN_NS) {
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 2 * H_N);
  }
}

__device__ __forceinline__ float warp_sum(float v) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// The sums of band->grid that oz_contract refuses, on the FP64 pipe: a warp looks
// at 32 grid rows and forms all columns of one at a time.  3 us where there are
// none; all 12.6 million of the L2,3 workload 9 ms (28 by the two warps of
// oz_contract that sum the magnitudes).
__global__ void __launch_bounds__(256) ozh_repair(const HParams p, const double2* __restrict__ psi) {
  if (!*p.any) return;
  const int lane = threadIdx.x & 31;
  const long long rows = (long long)p.nk * p.nx;
  for (long long r0 = 32ll * (blockIdx.x * 8 + (threadIdx.x >> 5)); r0 < rows; r0 += 32ll * 8 * gridDim.x) {
    const unsigned mine = r0 + lane < rows ? p.refused[r0 + lane] : 0;
    for (unsigned w = __ballot_sync(0xffffffffu, mine != 0); w; w &= w - 1) {
      const long long r = r0 + __ffs(w) - 1;
      const unsigned f = __shfl_sync(0xffffffffu, mine, __ffs(w) - 1);
      const int k = (int)(r / p.nx), x = (int)(r % p.nx), c = lane >> 2;
      const double v = warp_columns(p.u + r * p.nb, psi + (size_t)k * p.nb, (size_t)p.nk * p.nb, p.ncc, p.nb);
      if ((lane & 1) == 0 && (f >> c & 1))
        reinterpret_cast<double*>(p.out + ((size_t)k * p.nc + p.c0 + c) * p.nx + x)[(lane >> 1) & 1] = v;
    }
  }
}

// exponent and norm (in units of 2^exponent) of every grid row (k, x) over its bands: one warp per row
__global__ void __launch_bounds__(256) ozh_row_exponents(const double2* __restrict__ u, long long rows, int nb,
                                                         short* __restrict__ e, float* __restrict__ norm,
                                                         int* __restrict__ bad) {
  const int lane = threadIdx.x & 31;
  for (long long r = blockIdx.x * 8ll + (threadIdx.x >> 5); r < rows; r += gridDim.x * 8ll) {
    unsigned key = 0;
    for (int n = lane; n < nb; n += 32) {
      const double2 v = u[(size_t)r * nb + n];
      key = max(key, max(oz_key(v.x), oz_key(v.y)));
    }
    key = __reduce_max_sync(0xffffffffu, key);
    int flag = 0;
    const int er = oz_exponent(key, &flag);
    float s = 0.f;
    for (int n = lane; n < nb; n += 32) s += oz_unit_square(u[(size_t)r * nb + n], er);
    s = warp_sum(s);
    if (lane == 0) {
      e[r] = (short)er;
      norm[r] = sqrtf(s);
      if (flag) atomicOr(bad, 1);
    }
  }
}

// exponent and norm of every band (k, n) over the grid: blocks of 32 bands x 8 points
__global__ void __launch_bounds__(256) ozh_band_exponents(const double2* __restrict__ u, int nx, int nb,
                                                          short* __restrict__ e, float* __restrict__ norm,
                                                          int* __restrict__ bad) {
  __shared__ unsigned sk[8][32];
  __shared__ float ss[8][32];
  const int n = blockIdx.x * 32 + (threadIdx.x & 31), g = threadIdx.x >> 5, k = blockIdx.y;
  unsigned key = 0;
  if (n < nb)
    for (int x = g; x < nx; x += 8) {
      const double2 v = u[((size_t)k * nx + x) * nb + n];
      key = max(key, max(oz_key(v.x), oz_key(v.y)));
    }
  sk[g][threadIdx.x & 31] = key;
  __syncthreads();
  for (int i = 0; i < 8; ++i) key = max(key, sk[i][threadIdx.x & 31]);
  int flag = 0;
  const int en = oz_exponent(key, &flag);
  float s = 0.f;
  if (n < nb)
    for (int x = g; x < nx; x += 8) s += oz_unit_square(u[((size_t)k * nx + x) * nb + n], en);
  ss[g][threadIdx.x & 31] = s;
  __syncthreads();
  if (g == 0 && n < nb) {
    for (int i = 1; i < 8; ++i) s += ss[i][threadIdx.x];
    e[(size_t)k * nb + n] = (short)en;
    norm[(size_t)k * nb + n] = sqrtf(s);
    if (flag) atomicOr(bad, 1);
  }
}

// Exponent of a column from the key of its largest entry.  Digits cannot stand
// for columns with Inf or NaN, or whose largest entry is below 2^-960 (with 2^-e
// and its products out of range): exponent 0, the sums from the FP64 pipe.
__device__ __forceinline__ bool column_exponent(unsigned key, int* e) {
  *e = key ? (int)(key >> 20) - 1022 : 0;
  if (key < 0x7ff00000u && *e >= -960) return true;
  *e = 0;
  return false;
}
// thread 0 records the column of exponent e from every thread's sum of squares and count of entries
__device__ void record_column(bool fits, int e, float sq, int count, int* eb, HColumn* cb) {
  const float2 n = block_norm(sq, count);
  if (threadIdx.x != 0) return;
  *eb = e;
  *cb = HColumn{fits ? n.x : -1.f, n.y};
}
// Digits of psi for band->grid, one block per (k, column): rows 2c = (psi_r,
// -psi_i) and 2c + 1 = (psi_i, psi_r) along (n; re, im).  dig [k][7][H_J][kp]
__global__ void __launch_bounds__(64) ozh_psi_digits(const double2* __restrict__ psi, int nk, int nb, int kp,
                                                     __half* __restrict__ dig, int* __restrict__ eb,
                                                     HColumn* __restrict__ cb, int* __restrict__ any) {
  const int k = blockIdx.x, c = blockIdx.y;
  if (k == 0 && c == 0 && threadIdx.x == 0) *any = 0;   // refused sums of the pass that follows
  const double2* p = psi + ((size_t)c * nk + k) * nb;
  unsigned key = 0;
  for (int n = threadIdx.x; n < nb; n += blockDim.x) key = max(key, max(oz_key(p[n].x), oz_key(p[n].y)));
  int e;
  const bool fits = column_exponent(block_max(key), &e);
  float sq = 0.f;
  int count = 0;
  uint32_t* o = reinterpret_cast<uint32_t*>(dig) + ((size_t)k * OZ_S * H_J + 2 * c) * (kp / 2);
  for (int n = threadIdx.x; n < nb; n += blockDim.x) {
    const double2 v = p[n];
    sq += oz_unit_square(v, e);
    count += oz_nonzero(v);
    const oz_fix fr = oz_fixed(v.x, e), fi = oz_fixed(v.y, e), fm = oz_fixed(-v.y, e);
#pragma unroll
    for (int i = 0; i < OZ_S; ++i) {
      o[(size_t)i * H_J * (kp / 2) + n] = oz_digit2(fr, fm, i);
      o[(size_t)i * H_J * (kp / 2) + kp / 2 + n] = oz_digit2(fi, fr, i);
    }
  }
  record_column(fits, e, sq, count, eb + k * H_C + c, cb + k * H_C + c);
}

// Digits of phi[k][c][x] for grid->band, one block per (k, column): row 2c its
// real, 2c + 1 its imaginary part along x.  dig [k][7][H_J][kp]
__global__ void __launch_bounds__(256) ozh_phi_digits(const double2* __restrict__ phi, int nx, int nc, int c0, int kp,
                                                      __half* __restrict__ dig, int* __restrict__ eb,
                                                      HColumn* __restrict__ cb) {
  const int k = blockIdx.x, c = blockIdx.y;
  const double2* p = phi + ((size_t)k * nc + c0 + c) * nx;
  unsigned key = 0;
#pragma unroll 4
  for (int x = threadIdx.x; x < nx; x += blockDim.x) {
    const double2 v = p[x];
    key = max(key, max(oz_key(v.x), oz_key(v.y)));
  }
  int e;
  const bool fits = column_exponent(block_max(key), &e);
  float sq = 0.f;
  int count = 0;
  uint32_t* o = reinterpret_cast<uint32_t*>(dig) + ((size_t)k * OZ_S * H_J + 2 * c) * (kp / 2);
  for (int x = 2 * threadIdx.x; x < nx; x += 2 * blockDim.x) {
    const double2 v0 = p[x], v1 = x + 1 < nx ? p[x + 1] : make_double2(0.0, 0.0);
    sq += oz_unit_square(v0, e) + oz_unit_square(v1, e);
    count += oz_nonzero(v0) + oz_nonzero(v1);
    const oz_fix r0 = oz_fixed(v0.x, e), r1 = oz_fixed(v1.x, e), i0 = oz_fixed(v0.y, e), i1 = oz_fixed(v1.y, e);
#pragma unroll
    for (int i = 0; i < OZ_S; ++i) {
      o[(size_t)i * H_J * (kp / 2) + x / 2] = oz_digit2(r0, r1, i);
      o[(size_t)i * H_J * (kp / 2) + kp / 2 + x / 2] = oz_digit2(i0, i1, i);
    }
  }
  record_column(fits, e, sq, count, eb + k * H_C + c, cb + k * H_C + c);
}

// out[c][k][n] = sum_split part + E psi - sum_b chi psi_b + short-range out, FP64.
// Sums over the grid that the digits may not stand for are formed here again.
struct HFinal {
  const double2 *part, *psi;
  double2* out;
  const double* e_nk;
  const double2 *chi, *a_proj, *srcp, *u, *phi;
  const float *sums, *norm;   // sums of magnitudes (as part), norms of the bands [nk][nb]
  const HColumn* cb;          // columns of phi [nk][H_C]
  int nsplit, nk, nx, nb, na, np, c0, ncc, nc;
};
__global__ void __launch_bounds__(256) ozh_final(const HFinal p) {
  const size_t nkb = (size_t)p.nk * p.nb, total = nkb * p.ncc;
  const int lane = threadIdx.x & 31;
  for (size_t i0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x - lane; i0 < total; i0 += (size_t)gridDim.x * blockDim.x) {
    const bool in = i0 + lane < total;
    const size_t i = in ? i0 + lane : total - 1;
    const int cc = (int)(i / nkb), c = p.c0 + cc, v = c / p.na, a = c % p.na;
    const size_t kn = i % nkb;
    const int k = (int)(kn / p.nb), n = (int)(kn % p.nb);
    double2 lr = make_double2(0.0, 0.0), rest = make_double2(0.0, 0.0);
    float m = 0.f;
    for (int s = 0; s < p.nsplit; ++s) {
      const size_t o = (((size_t)s * p.nk + k) * H_C + cc) * p.nb + n;
      const double2 t = p.part[o];
      lr.x += t.x;
      lr.y += t.y;
      m += p.sums[o];
    }
    const bool good = column_accepts(p.cb[(size_t)k * H_C + cc], p.norm[kn], m);
    unsigned w = __ballot_sync(0xffffffffu, in && !good);
    if (__popc(w) >= 8) {   // many of a warp's bands: each lane its own, u read along the bands
      if (in && !good) {
        const double2 *u = p.u + (size_t)k * p.nx * p.nb + n, *f = p.phi + ((size_t)k * p.nc + c) * p.nx;
        lr = make_double2(0.0, 0.0);
#pragma unroll 8
        for (int x = 0; x < p.nx; ++x) {
          const double2 q = u[(size_t)x * p.nb], b = f[x];
          lr.x = fma(q.x, b.x, fma(q.y, b.y, lr.x));
          lr.y = fma(q.x, b.y, fma(-q.y, b.x, lr.y));
        }
      }
      w = 0;
      __syncwarp();
    }
    for (; w; w &= w - 1) {   // else one at a time, lanes along the grid
      const int r = __ffs(w) - 1;
      const int kr = __shfl_sync(0xffffffffu, k, r), nr = __shfl_sync(0xffffffffu, n, r), cr = __shfl_sync(0xffffffffu, c, r);
      const double2 t = warp_dot(p.u + (size_t)kr * p.nx * p.nb + nr, p.nb, p.phi + ((size_t)kr * p.nc + cr) * p.nx, p.nx);
      if (lane == r) lr = t;
    }
    if (!in) continue;
    for (int b = 0; b < p.na; ++b) {
      const double2 ch = p.chi[a * p.na + b], pb = p.psi[(size_t)(v * p.na + b) * nkb + kn];
      rest.x = fma(-ch.x, pb.x, fma(ch.y, pb.y, rest.x));
      rest.y = fma(-ch.x, pb.y, fma(-ch.y, pb.x, rest.y));
    }
    const double2* cp = p.srcp + (size_t)v * p.na * p.np + (size_t)a * p.np;
#pragma unroll 4
    for (int j = 0; j < p.np; ++j) {
      const double2 ap = p.a_proj[(size_t)j * nkb + kn], q = cp[j];
      rest.x = fma(ap.x, q.x, fma(ap.y, q.y, rest.x));
      rest.y = fma(ap.x, q.y, fma(-ap.y, q.x, rest.y));
    }
    const double2 ps = p.psi[(size_t)c * nkb + kn];
    const double e = p.e_nk[kn];
    p.out[(size_t)c * nkb + kn] = make_double2(lr.x + rest.x + e * ps.x, lr.y + rest.y + e * ps.y);
  }
}

// digits [nk * 7][H_J][kp] FP16: box of 32 K elements x 16 rows x 7 digits, 64-byte swizzle
bool stacked_map(CUtensorMap* m, const __half* base, int kp, int nk) {
  const EncodeTiledFn f = bse_encode_tiled_fn();
  if (!f) return false;
  cuuint64_t dims[3] = {(cuuint64_t)kp, (cuuint64_t)H_J, (cuuint64_t)nk * OZ_S};
  cuuint64_t strides[2] = {(cuuint64_t)kp * 2, (cuuint64_t)H_J * kp * 2};
  cuuint32_t box[3] = {(cuuint32_t)H_KB, (cuuint32_t)H_J, (cuuint32_t)OZ_S};
  cuuint32_t es[3] = {1, 1, 1};
  return f(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half*>(base), dims, strides, box, es,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct OzhState {
  short *ex = nullptr, *en = nullptr;           // exponents of U per grid row and per band
  int *epsi = nullptr, *ephi = nullptr;         // exponents of the columns, [nk][H_C]
  __half *dpsi = nullptr, *dphi = nullptr;      // digits, [nk][7][H_J][kp]
  unsigned char* refused = nullptr;             // [nk][nx], band->grid
  float *nx = nullptr, *nn = nullptr;           // norms of U's rows and bands in units of their scales
  HColumn *cpsi = nullptr, *cphi = nullptr;     // the columns, [nk][H_C]
  double2* part = nullptr;                      // [nsplit][nk][H_C][nb]
  float* sums = nullptr;                        // their sums of magnitudes
  int* err = nullptr;                           // {wait gave up, U out of range, sums refused}
  CUtensorMap mpsi, mphi;
  int kp = 0, kpx = 0, nsplit = 1, sms = 0;
};

void free_state(OzhState* z) {
  void* ptrs[] = {z->ex,   z->en,   z->epsi, z->ephi, z->dpsi, z->dphi, z->nx,
                  z->nn, z->cpsi, z->cphi, z->part, z->sums, z->refused, z->err};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete z;
}

// Which form a call of nc columns takes, from the two times (us) as measured
// over 1 to 512 k points, 216 to 13824 grid points, 8 to 150 bands and 1 to 18
// columns.  Split: per pass of eight columns 45 for its launches and 6.6e-6 per
// entry of U in whole tiles of each contraction.  FP64 pipe: one block's walk
// over the grid, and 1.4e-5 per entry and column.  (2^3 k, 8^3 points, 16
// bands: 24 us against 53 at one column, 83 against 64 at six; 4^3 k, 12^3, 12:
// 66 against 125 and 296 against 192; 8^3 k, 16^3, 64 at six: 12.6 ms against 1.8.)
bool split_is_faster(const bse_handle* h, int nc) {
  auto up = [](double v, double m) { return ceil(v / m) * m; };
  const double nk = h->nk, nx = h->nx, nb = h->nb;
  const double split = ceil(nc / 8.0) * (45.0 + 6.6e-6 * nk * (up(nx, H_M) * up(nb, 16) + up(nx, H_KB) * up(nb, H_M / 2)));
  const double fp64 = 8.0 + 0.015 * nx * nc + 1.4e-5 * nk * nx * nb * nc;
  return split < fp64;
}

template <int MODE>
cudaError_t launch(const CUtensorMap& map, const HParams& p, int sms, cudaStream_t st) {
  const cudaError_t e = cudaFuncSetAttribute(oz_contract<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)H_SMEM);
  if (e != cudaSuccess) return e;
  oz_contract<MODE><<<std::min(p.ntiles, sms), H_THREADS, H_SMEM, st>>>(map, p);
  return cudaGetLastError();
}

}  // namespace

// Tables and buffers of the tensor-core contractions of an FP64 handle; without
// them (small systems, U out of the scheme's range, no memory left for them)
// the handle keeps the FP64 kernels.  Called last in the set-up.
// The low part of a sum grows by at most 5.1 * 2^14 * 2^24 per K element: 2^22
// points, and 2^21 bands, stay below 2^63.
void bse_ozh_prepare(bse_handle* h) {
  if (h->nx > (1 << 22) || h->nb > (1 << 21)) return;
  if (!split_is_faster(h, h->na) && !split_is_faster(h, h->na * h->max_vec)) return;
  OzhState* z = new (std::nothrow) OzhState();
  if (!z) return;
  const std::string err = h->err;
  const size_t bytes0 = h->dev_bytes;
  cudaDeviceGetAttribute(&z->sms, cudaDevAttrMultiProcessorCount, h->dev);
  z->kp = (2 * h->nb + H_KB - 1) / H_KB * H_KB;
  z->kpx = (h->nx + H_KB - 1) / H_KB * H_KB;
  // grid->band: about two tiles per SM, at least eight K blocks each
  const int tiles = h->nk * ((2 * h->nb + H_M - 1) / H_M), kb = z->kpx / H_KB;
  z->nsplit = std::max(1, std::min({(2 * z->sms + tiles - 1) / tiles, kb / 8, 16}));
  const size_t nk = (size_t)h->nk;
  const size_t bpsi = nk * OZ_S * H_J * z->kp * sizeof(__half), bphi = nk * OZ_S * H_J * z->kpx * sizeof(__half);
  struct {
    void** p;
    size_t bytes;
  } want[] = {{(void**)&z->ex, nk * h->nx * sizeof(short)},
              {(void**)&z->en, nk * h->nb * sizeof(short)},
              {(void**)&z->epsi, nk * H_C * sizeof(int)},
              {(void**)&z->ephi, nk * H_C * sizeof(int)},
              {(void**)&z->dpsi, bpsi},
              {(void**)&z->dphi, bphi},
              {(void**)&z->refused, nk * h->nx},
              {(void**)&z->nx, nk * h->nx * sizeof(float)},
              {(void**)&z->nn, nk * h->nb * sizeof(float)},
              {(void**)&z->cpsi, nk * H_C * sizeof(HColumn)},
              {(void**)&z->cphi, nk * H_C * sizeof(HColumn)},
              {(void**)&z->part, (size_t)z->nsplit * nk * H_C * h->nb * sizeof(double2)},
              {(void**)&z->sums, (size_t)z->nsplit * nk * H_C * h->nb * sizeof(float)},
              {(void**)&z->err, 256}};
  bool ok = z->sms > 0;
  for (auto& w : want) ok = ok && bse_handle_malloc(h, w.p, w.bytes, "tensor-core form of the FP64 contractions") == BSE_OK;
  int bad = 1;
  if (ok) {
    cudaMemsetAsync(z->dpsi, 0, bpsi, h->stream);
    cudaMemsetAsync(z->dphi, 0, bphi, h->stream);
    cudaMemsetAsync(z->err, 0, 256, h->stream);
    const long long rows = (long long)h->nk * h->nx;
    ozh_row_exponents<<<(unsigned)std::min<long long>((rows + 7) / 8, 16 * z->sms), 256, 0, h->stream>>>(
        (const double2*)h->u, rows, h->nb, z->ex, z->nx, z->err + 1);
    ozh_band_exponents<<<dim3((unsigned)((h->nb + 31) / 32), (unsigned)h->nk), 256, 0, h->stream>>>(
        (const double2*)h->u, h->nx, h->nb, z->en, z->nn, z->err + 1);
    ok = cudaMemcpyAsync(&bad, z->err + 1, sizeof(int), cudaMemcpyDeviceToHost, h->stream) == cudaSuccess &&
         cudaStreamSynchronize(h->stream) == cudaSuccess && stacked_map(&z->mpsi, z->dpsi, z->kp, h->nk) &&
         stacked_map(&z->mphi, z->dphi, z->kpx, h->nk);
  }
  if (!ok || bad) {
    cudaGetLastError();
    free_state(z);
    h->dev_bytes = bytes0;
    h->err = err;
    return;
  }
  h->launches += 2;
  h->ozh = z;
}

bool bse_ozh_takes(const bse_handle* h, int nc) { return h->ozh && split_is_faster(h, nc); }

void bse_ozh_free(bse_handle* h) {
  if (h->ozh) free_state((OzhState*)h->ozh);
  h->ozh = nullptr;
}

bool bse_ozh_release(bse_handle* h) {
  if (!h->ozh || h->ozh_recorded) return false;
  int e = 0;
  cudaMemcpyAsync(&e, ((OzhState*)h->ozh)->err, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
  if (cudaStreamSynchronize(h->stream) != cudaSuccess) return false;
  h->gave_up = h->gave_up || e;
  bse_drop_graph(h);   // its kernels use the tables
  bse_ozh_free(h);
  return true;
}

// phi[k][c][x] = sum_n U psi for every column
bse_status bse_ozh_band_to_grid(bse_handle* h, const double2* psi, int nc) {
  OzhState* z = (OzhState*)h->ozh;
  HParams p{};
  p.u = (const double2*)h->u;
  p.ea = z->ex;
  p.na = z->nx;
  p.eb = z->epsi;
  p.cb = z->cpsi;
  p.refused = z->refused;
  p.any = z->err + 2;
  p.out = (double2*)h->phi;
  p.nk = h->nk, p.nx = h->nx, p.nb = h->nb;
  p.mt = (h->nx + H_M - 1) / H_M;
  p.nsplit = 1;
  p.ntiles = h->nk * p.mt;
  p.kb = p.kb_per_split = z->kp / H_KB;
  p.nc = nc;
  p.err = z->err;
  p.wait_ns = h->tc_wait_ns;
  cudaError_t e = cudaSuccess;
  for (int c0 = 0; c0 < nc && e == cudaSuccess; c0 += H_C) {
    p.c0 = c0;
    p.ncc = std::min(H_C, nc - c0);
    const double2* pc = psi + (size_t)c0 * h->nk * h->nb;
    BSE_PROF(h, BSE_K_PREP,
             ozh_psi_digits<<<dim3((unsigned)h->nk, (unsigned)p.ncc), 64, 0, h->stream>>>(
                 pc, h->nk, h->nb, z->kp, z->dpsi, z->epsi, z->cpsi, p.any));
    BSE_PROF(h, BSE_K_BAND_TO_GRID, e = launch<0>(z->mpsi, p, z->sms, h->stream));
    BSE_PROF(h, BSE_K_BAND_TO_GRID, ozh_repair<<<(unsigned)(8 * z->sms), 256, 0, h->stream>>>(p, pc));
  }
  return bse_cuda_check(h, e == cudaSuccess ? cudaGetLastError() : e, "band->grid (split FP64)");
}

// out = grid->band of phi + diagonal, spin-orbit and short-range terms
bse_status bse_ozh_grid_to_band(bse_handle* h, const double2* psi, double2* hpsi, int nc) {
  OzhState* z = (OzhState*)h->ozh;
  HParams p{};
  p.u = (const double2*)h->u;
  p.ea = z->en;
  p.eb = z->ephi;
  p.out = z->part;
  p.sums = z->sums;
  p.nk = h->nk, p.nx = h->nx, p.nb = h->nb;
  p.mt = (2 * h->nb + H_M - 1) / H_M;
  p.kb = z->kpx / H_KB;
  p.kb_per_split = (p.kb + z->nsplit - 1) / z->nsplit;
  p.nsplit = (p.kb + p.kb_per_split - 1) / p.kb_per_split;
  p.ntiles = h->nk * p.mt * p.nsplit;
  p.err = z->err;
  p.wait_ns = h->tc_wait_ns;
  HFinal f = {z->part, psi, hpsi, h->e_nk, h->chi, h->a_proj, h->sr_cp, (const double2*)h->u, (const double2*)h->phi,
                      z->sums, z->nn, z->cphi, p.nsplit, h->nk, h->nx, h->nb, h->na, h->np, 0, 0, nc};
  cudaError_t e = cudaSuccess;
  const size_t nkb = (size_t)h->nk * h->nb;
  for (int c0 = 0; c0 < nc && e == cudaSuccess; c0 += H_C) {
    p.ncc = std::min(H_C, nc - c0);
    BSE_PROF(h, BSE_K_PREP,
             ozh_phi_digits<<<dim3((unsigned)h->nk, (unsigned)p.ncc), 256, 0, h->stream>>>(
                 (const double2*)h->phi, h->nx, nc, c0, z->kpx, z->dphi, z->ephi, z->cphi));
    BSE_PROF(h, BSE_K_GRID_TO_BAND, e = launch<1>(z->mphi, p, z->sms, h->stream));
    if (h->np > 0 && c0 == 0) cudaStreamWaitEvent(h->stream, h->ev_join, 0);   // short-range c' ready
    f.c0 = c0;
    f.ncc = p.ncc;
    BSE_PROF(h, BSE_K_GRID_TO_BAND,
             ozh_final<<<(unsigned)std::min<size_t>((nkb * p.ncc + 255) / 256, (size_t)32 * z->sms), 256, 0, h->stream>>>(f));
  }
  return bse_cuda_check(h, e == cudaSuccess ? cudaGetLastError() : e, "grid->band (split FP64)");
}

// the device word that a wait which gave up sets
int* bse_ozh_word(const bse_handle* h) { return ((OzhState*)h->ozh)->err; }
