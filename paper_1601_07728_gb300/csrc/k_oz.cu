// FP64 matrix products D_b[m][n] = alpha sum_K A_b[m][K] B_b[n][K] on the FP16
// tensor cores by exact splitting (oz_dev.cuh), and the kernels that write the
// operands' digits.  Users: the screening stage's Green's functions (Sec. 3.3)
// and the set-up projection onto the local basis (Sec. 3.2.2).
//
// Why: GB300 retires 2 FP64 FMAs per SM and clock and about 2000 times as many
// FP16 products, so that the 19 products of 128 x 128 x 16 which replace one
// FP64 product of 128 x 64 x 16 still run some 50 times faster.  Measured:
// Green's functions of 900 points, 4096 states and 16 frequencies 682 ms
// (FP64 kernel) -> 13.6 ms (this one 12.2, writing the digits 0.97, magnitudes 0.29); the
// projection of 8^3 k x 16^3 points x 64 bands onto 64 functions 102.6 ms ->
// 5.4 ms with the Bloch functions' digits in memory -> 3.2 ms with the digits
// made on the way into shared memory (oz_project 2.55, scales and magnitudes
// 0.38).  The error against 64 bits fell from 1.9e-15 to 1.4e-15 and from 1.4e-15
// to 0.7e-15.  What bounds oz_gemm now: operand tiles from L2 (35 bytes per SM and
// clock) beside the products' 64 clocks each.
//
// The digits hold an entry to 2^-56 of its row's largest.  Where that is not
// FP64's accuracy (oz_accept) the elements are formed again on the FP64 pipe, and
// all of them if these are more than one in 32.
#include "bse_internal.cuh"
#include "oz_dev.cuh"
#include "tc_ptx.cuh"

#include <stdlib.h>

#include <algorithm>

namespace {

constexpr int OZ_M = 128, OZ_N = 64, OZ_KB = 64;   // output tile, K block (one 128-byte swizzle row)
constexpr int OZ_A = OZ_M * 128;                   // bytes of one digit's A tile
constexpr int OZ_BD = OZ_N * 128;                  // bytes of one digit's B tile
constexpr int OZ_B = OZ_S * OZ_BD;                 // ... and of the seven
constexpr int OZ_AS = 5, OZ_BS = 2;               // ring slots: A per digit, B per K block
constexpr int OZ_D = 8;                            // accumulators, s = 0..7
constexpr int OZ_SF = 8;                           // digits of the local functions in the projection
constexpr int OZ_THREADS = 320;
// B slots lie between tiles of zeros: 0 B_0..B_6 0 B_0..B_6 0
constexpr int OZ_BAREA = OZ_BS * (OZ_B + OZ_BD) + OZ_BD;
constexpr size_t OZ_SMEM = 1024 + (size_t)OZ_AS * OZ_A + OZ_BAREA + 512;
constexpr unsigned long long OZ_WAIT_NS = 2000000000ull;   // limit of a wait, and of the drain after an abort

// limit of the pipeline waits of one call: OZ_WAIT_NS, or BSE_SPLIT_WAIT_NS of the environment (see bse.h)
unsigned long long wait_limit() {
  const char* v = getenv("BSE_SPLIT_WAIT_NS");
  if (!v) return OZ_WAIT_NS;
  char* end = nullptr;
  const unsigned long long n = strtoull(v, &end, 10);
  return end == v || *end != '\0' || n < 1000 || n > OZ_WAIT_NS ? OZ_WAIT_NS : n;
}

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
  unsigned long long wait_ns;
};

// bounded wait, inlined: at a call the draining warps' sums would go through memory
__device__ __forceinline__ bool oz_wait(uint32_t a, uint32_t parity, volatile int* abort_flag, unsigned long long limit_ns) {
  if (mbar_try(a, parity)) return true;
  const unsigned long long t0 = gtime();
  while (!mbar_try(a, parity))
    if (*abort_flag || gtime() - t0 > limit_ns) return false;
  return true;
}

// Chunks of 128 K elements.  The accumulators s = 4, 5 hold one chunk's sums
// (at most 6 * 128 * 2^14 < 2^24), s = 2, 3 two and s = 0, 1 four (4 * 256 and
// 2 * 512 times 2^14): c counts the chunks of a tile, `last` its last one.
// s = 6, 7 are kept for 32 (7 * 4096 * 2^14 < 2^31 still converts to an integer).
// Past 2^24 an addition of 16 K elements is rounded, by up to 2^-23 of the sum so
// far.  Digits of random signs stay below (2^20 after 4096 elements).  If all of
// K elements' digits were at their largest with one sign, the 56 * 32 additions
// until a drain, at half of 7 * 4096 * 2^14 on average, would add up to K 2^-58
// in units of the two scales: at most K 2^-55 sum |a| |b| for an accepted sum (a
// tenth and more), a quarter of what K roundings of an FP64 sum may add.
// Draining costs as much as converting u (float to integer runs at 16 per SM and
// clock): all seven of s < 7 after every chunk 12.9 ms for the Green's functions
// below, s >= 4 after every chunk 12.4 (with s = 7 13.0), as it is 12.2; oz_project
// 2.6, 2.4 (2.7) and 2.55.
// Issuing the products of s < 4 first while the others drain holds four A slots
// of five and was slower (14.5 ms).
__device__ __forceinline__ bool drains(int s, int c, bool last) {
  return last || (s >= 6 ? (c & 31) == 31 : s >= 4 || (s >= 2 ? (c & 1) == 1 : (c & 3) == 3));
}

// state of the issuing thread: A ring slot and phase, restarts of the accumulators s = 0, 1 / 2, 3 / 4, 5 / 6, 7
struct oz_issue {
  int sl = 0, r0 = 0, r1 = 0, r2 = 0, r3 = 0;
  uint32_t ph = 0;
};

// Digit products of one K block against the B tiles at descriptor db, the A
// digits from the ring.  First block of a chunk (c: its number in the tile): the
// accumulators that were drained start over, each as soon as that is done.
// A product of N = 64 or less takes the tensor core as long as one of N = 128
// (about 64 clocks measured at N = 32 and 64), so two neighbouring B digits
// form one operand of 128 rows and the accumulators of s = 2P, 2P + 1 one of
// 128 columns: digit A_i meets (B_0, B_1), (B_2, B_3), ... for even i and (0,
// B_0), (B_1, B_2), ... for odd i: 19 products per 16 K elements for seven A
// digits (34 pairs of digits), 20 for eight, and all of one shape.
template <int SA>   // A digits
__device__ __forceinline__ bool issue_block(uint32_t tmem, uint32_t sa, unsigned long long db, bool first, int c,
                                            oz_issue& z, uint32_t afull, uint32_t aempty, uint32_t tempty,
                                            volatile int* abort_flag, unsigned long long limit_ns) {
  // FP16 A and B (K-major), FP32 D
  constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(2 * OZ_N >> 3) << 17) | ((uint32_t)(OZ_M >> 4) << 24);
  auto products = [&](int i, int p0, int p1, uint32_t keep) {   // bit P of keep: add to accumulator P
    const unsigned long long da = sdesc_sw128(sa + z.sl * OZ_A);
#pragma unroll
    for (int ks = 0; ks < OZ_KB / 16; ++ks)
#pragma unroll
      for (int P = p0; P < p1; ++P)
        mma_bf16(tmem + 2 * P * OZ_N, da + ks * 2,
                 db + (unsigned long long)(long long)(((2 * P - i) * OZ_BD + ks * 32) / 16), idesc,
                 ks > 0 ? 1u : (keep >> P) & 1u);
  };
  auto drained = [&](int s, int n) { return oz_wait(tempty + 8 * s, ((uint32_t)n & 1u) ^ 1u, abort_flag, limit_ns); };
#pragma unroll
  for (int i = 0; i < SA; ++i) {
    if (!oz_wait(afull + 8 * z.sl, z.ph, abort_flag, limit_ns)) return false;
    tc_fence_after();
    if (i == 0 && first) {
      const bool n0 = (c & 3) == 0, n1 = (c & 1) == 0, n3 = (c & 31) == 0;
      if (n0 && !(drained(0, z.r0) && drained(1, z.r0))) return false;
      tc_fence_after();
      products(0, 0, 1, n0 ? 0u : 1u);
      if (n1 && !(drained(2, z.r1) && drained(3, z.r1))) return false;
      tc_fence_after();
      products(0, 1, 2, n1 ? 0u : 2u);
      if (!(drained(4, z.r2) && drained(5, z.r2))) return false;
      tc_fence_after();
      products(0, 2, 3, 0u);
      if (n3 && !(drained(6, z.r3) && drained(7, z.r3))) return false;
      tc_fence_after();
      products(0, 3, 4, n3 ? 0u : 8u);
      z.r0 += n0, z.r1 += n1, z.r2 += 1, z.r3 += n3;
    } else {
      products(i, i / 2, 4, 15u);   // consecutive products go to different accumulators
    }
    mma_commit(aempty + 8 * z.sl);
    if (++z.sl == OZ_AS) z.sl = 0, z.ph ^= 1u;
  }
  return true;
}

// hi 2^32 + lo += d 2^sh
__device__ __forceinline__ void add96(long long& hi, uint32_t& lo, int d, int sh) {
  const uint32_t l = (uint32_t)d << sh;
  const int m = sh ? d >> (32 - sh) : d >> 31, t = d >> 31;
  asm("{\n .reg .u32 a, b;\n mov.b64 {a, b}, %0;\n add.cc.u32 %1, %1, %2;\n addc.cc.u32 a, a, %3;\n"
      " addc.u32 b, b, %4;\n mov.b64 %0, {a, b};\n}\n"
      : "+l"(hi), "+r"(lo)
      : "r"(l), "r"(m), "r"(t));
}

// Accumulators of 32 TMEM lanes x C columns at ta into sums hi 2^-38 + lo 2^-70
// (lo unsigned; s < 4 have the weights 2^-14 .. 2^-38, the rest 2^-46 ..
// 2^-70).  Each is given back as soon as it is read.  |hi| <= 2^48 per 512 K
// elements: K <= 2^21.
template <int C>
__device__ __forceinline__ void drain_chunk(uint32_t ta, int c, bool last, uint32_t tempty, int lane, long long* hi,
                                            uint32_t* lo) {
#pragma unroll
  for (int s = 0; s < OZ_D; ++s) {
    if (!drains(s, c, last)) continue;
#pragma unroll
    for (int h = 0; h < C / 16; ++h) {
      float v[16];
      tmem_ld16(ta + s * OZ_N + 16 * h, v);
      if (h == C / 16 - 1) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty + 8 * s);
      }
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int d = __float2int_rn(v[k]), j = 16 * h + k;
        if (s < 4) {
          hi[j] += (long long)d * (1 << (8 * (3 - s)));
        } else {
          // 96-bit addition; as 64-bit arithmetic lo would take a pair of registers
          add96(hi[j], lo[j], d, 8 * (7 - s));
        }
      }
    }
  }
}
__device__ __forceinline__ double oz_value(long long hi, long long lo) {
  return (double)hi * 0x1p-38 + (double)lo * 0x1p-70;
}

// Persistent warp-specialised kernel, one CTA per SM: warp 0 streams digit
// tiles with TMA (the seven B tiles of a K block as one box, each A digit in
// a slot of its own), warp 1 issues the digit products, warps 2-9 drain the
// accumulators every 128 K elements into 64-bit integers.  M tiles are the
// fastest tile index: the CTAs running at one time then share both operands'
// tiles in L2.
__global__ void __launch_bounds__(OZ_THREADS, 1)
    oz_gemm(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb, const OzParams p) {
  extern __shared__ unsigned char oz_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)oz_raw + 1023) & ~(uintptr_t)1023);
  unsigned long long* bars = (unsigned long long*)(sm + OZ_AS * OZ_A + OZ_BAREA);
  constexpr int NBAR = 2 * OZ_AS + 2 * OZ_BS + 1 + OZ_D + 1;
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
    for (int s = 0; s < OZ_D; ++s) mbar_init(tempty(s), 8);
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
        if (!(ok = oz_wait(bempty(s), ((uint32_t)(ib / OZ_BS) & 1u) ^ 1u, abort_flag, p.wait_ns))) break;
        mbar_expect_tx(bfull(s), OZ_B);
        tma_load_3d(sb + s * (OZ_B + OZ_BD), &mb, bfull(s), kb * OZ_KB, n * OZ_N, zb);
        *b_issued = ++ib;
        for (int i = 0; i < OZ_S; ++i) {
          const int q = ia % OZ_AS;
          if (!(ok = oz_wait(aempty(q), ((uint32_t)(ia / OZ_AS) & 1u) ^ 1u, abort_flag, p.wait_ns))) break;
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
    int ib = 0;
    oz_issue z;
    bool ok = true;
    for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
      for (int kb = 0; kb < p.kb && ok; ++kb) {
        const bool first = (kb & 1) == 0, last = (kb & 1) == 1 || kb + 1 == p.kb;
        const int s = ib % OZ_BS;
        if (!(ok = oz_wait(bfull(s), (uint32_t)(ib / OZ_BS) & 1u, abort_flag, p.wait_ns))) break;
        ++ib;
        const unsigned long long db = sdesc_sw128(sb + s * (OZ_B + OZ_BD));
        if (!(ok = issue_block<OZ_S>(tmem, sa, db, first, kb >> 1, z, afull(0), aempty(0), tempty(0), abort_flag, p.wait_ns))) break;
        mma_commit(bempty(s));
        if (last) mma_commit(tfull);
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
      long long hi[32];
      uint32_t lo[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) hi[c] = 0, lo[c] = 0;
      for (int kb = 0; kb < p.kb; kb += 2, ++chunk) {
        ok = __all_sync(0xffffffffu, oz_wait(tfull, (uint32_t)chunk & 1u, abort_flag, p.wait_ns));
        if (!ok) break;
        tc_fence_after();
        drain_chunk<32>(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 32), kb >> 1, kb + 2 >= p.kb, tempty(0), lane,
                    hi, lo);
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
            o[c * p.sc] = oz_value(hi[c], lo[c]) * (fa * fb[c]);
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

// Digits of the rows of X [rows][n] (complex), one block per row and batch j;
// with d != nullptr entry K of batch j is first multiplied by d[j][K].
//   pair = 0: one row (re, im) per complex row, K = 2n interleaved
//   pair = 1: two rows, (re, im) and (-im, re): the products with a pair-0 row
//             are the real and imaginary part of sum x_a conj(x_b)
// dig [batch][7][rows (x2)][kp], zero beyond 2n; scale 2^e per row; norm [batch][rows]
// of the complex rows in units of that, with 2^1/2 of their number of entries.
__global__ void __launch_bounds__(256) oz_split_rows(const double2* __restrict__ X, int n, const double2* __restrict__ d,
                                                     int rows, int kp, int pair, __half* __restrict__ dig,
                                                     double* __restrict__ scale, float2* __restrict__ norm,
                                                     int* __restrict__ bad) {
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
  float sq = 0.f;
  int count = 0;
  for (int k = threadIdx.x; k < kp / 2; k += blockDim.x) {
    const double2 v = k < n ? entry(k) : make_double2(0.0, 0.0);
    sq += oz_unit_square(v, e);
    count += oz_nonzero(v);
    const oz_fix fr = oz_fixed(v.x, e), fi = oz_fixed(v.y, e);
#pragma unroll
    for (int i = 0; i < OZ_S; ++i) out[i * digit + k] = oz_digit2(fr, fi, i);
    if (pair) {
      const oz_fix fm = oz_fixed(-v.y, e);
#pragma unroll
      for (int i = 0; i < OZ_S; ++i) out[i * digit + kp / 2 + k] = oz_digit2(fm, fr, i);
    }
  }
  const float2 v = block_norm(sq, count);
  if (threadIdx.x == 0) norm[(size_t)b * rows + row] = v;
}

// two registers of interleaved (re, im) to one of two |re| + |im|
__device__ __forceinline__ uint32_t abs_sum(uint32_t x, uint32_t y) {
  const uint32_t re = __byte_perm(x, y, 0x5410) & 0x7fff7fffu, im = __byte_perm(x, y, 0x7632) & 0x7fff7fffu;
  const __half2 s = __hadd2(*reinterpret_cast<const __half2*>(&re), *reinterpret_cast<const __half2*>(&im));
  return *reinterpret_cast<const uint32_t*>(&s);
}

// Lists the elements (batch, r, r') of the product of rows A (pair = 0, batched)
// and B (pair = 1, of the same vectors, so that the magnitudes' sum is the same
// with r and r' exchanged: tiles on and below the diagonal only) whose magnitudes
// do not cover the digits' error: sum |a| |b| from the leading digits on the
// older tensor-core form (mma.sync m16n8k16 on |re| + |im|, K in any order as
// long as both sides have it).  Tiles of 128 x 128, K blocks of 64 in three
// buffers, a warp 64 x 32.  Part of the K blocks is enough for most: the first
// launch takes every `step`-th, and only where that refuses more than the list
// holds does a second one take them all (`after`: its count).  900 rows, 8192 K
// elements, 16 batches: 0.29 ms with every fourth.
constexpr int RF_T = 128, RF_S = 3, RF_BYTES = 2 * RF_T * 128;   // buffers, bytes of one: 128 rows of each operand
struct OzRefused {
  const __half *a, *b;              // digits [batch][7][nr][kp], [7][2 nr][kp]
  const double *sa, *sb;            // scales [batch][nr], [2 nr]
  const float2 *na, *nb;            // [batch][nr], [nr]
  int nr, kp, mt;                   // rows, padded K, tiles per side
  unsigned long long* list;
  unsigned cap;
  unsigned* count;
  int step;
  const unsigned* after;
  int* bad;
};
__global__ void __launch_bounds__(256, 2) oz_gemm_refused(const OzRefused p) {
  extern __shared__ __align__(128) unsigned char rf_sm[];
  if (p.after && *p.after <= p.cap) return;
  int m = (int)((sqrtf(8.f * blockIdx.x + 1.f) - 1.f) * 0.5f);   // row of the triangle
  while ((m + 1) * (m + 2) / 2 <= (int)blockIdx.x) ++m;
  while (m * (m + 1) / 2 > (int)blockIdx.x) --m;
  const int q = blockIdx.x - m * (m + 1) / 2, bt = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wm = (warp & 1) * 64, wn = (warp >> 1) * 32;
  const __half* a = p.a + (size_t)bt * OZ_S * p.nr * p.kp;
  // 16-byte chunks: row of A or B, chunk of the K block, swizzled by the row
  const int nkb = (p.kp / OZ_KB + p.step - 1) / p.step;
  auto load = [&](int i0) {
    const uint32_t base = smem_u32(rf_sm) + i0 % RF_S * RF_BYTES;
#pragma unroll
    for (int i = 0; i < 2 * RF_T * 8 / 256 && i0 < nkb; ++i) {
      const int e = threadIdx.x + 256 * i, r = e >> 3, c = e & 7;
      const __half* src = r < RF_T ? a + (size_t)min(m * RF_T + r, p.nr - 1) * p.kp
                                   : p.b + (size_t)2 * min(q * RF_T + r - RF_T, p.nr - 1) * p.kp;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(base + r * 128 + ((c ^ (r & 7)) << 4)),
                   "l"(src + (size_t)i0 * p.step * OZ_KB + c * 8)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");   // empty past the end: the waits count groups
  };
  float c[4][4][4];
#pragma unroll
  for (int i = 0; i < 64; ++i) c[i >> 4][(i >> 2) & 3][i & 3] = 0.f;
  load(0);
  load(1);
  for (int kb = 0; kb < nkb; ++kb) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();   // block kb is there, and every warp is done with kb - 1, whose buffer the next load takes
    load(kb + 2);
    const uint32_t base = smem_u32(rf_sm) + kb % RF_S * RF_BYTES;
    auto ldm = [&](int row, int chunk, uint32_t* r) { ldmatrix_x4(base + row * 128 + ((chunk ^ (row & 7)) << 4), r); };
#pragma unroll
    for (int h = 0; h < 2; ++h) {   // 32 K elements, 16 complex ones
      uint32_t b[4][2];
#pragma unroll
      for (int nt = 0; nt < 4; nt += 2) {
        const int row = RF_T + wn + nt * 8 + (lane & 7) + ((lane >> 4) << 3), ch = 4 * h + ((lane >> 3) & 1);
        uint32_t x[4], y[4];
        ldm(row, ch, x);
        ldm(row, ch + 2, y);
        b[nt][0] = abs_sum(x[0], x[1]), b[nt][1] = abs_sum(y[0], y[1]);
        b[nt + 1][0] = abs_sum(x[2], x[3]), b[nt + 1][1] = abs_sum(y[2], y[3]);
      }
#pragma unroll
      for (int mt = 0; mt < 4; ++mt) {
        const int row = wm + mt * 16 + (lane & 15), ch = 4 * h + (lane >> 4);
        uint32_t x[4], y[4];
        ldm(row, ch, x);
        ldm(row, ch + 2, y);
        const uint32_t v[4] = {abs_sum(x[0], x[2]), abs_sum(x[1], x[3]), abs_sum(y[0], y[2]), abs_sum(y[1], y[3])};
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) mma_16x8x16<false>(c[mt][nt], v, b[nt][0], b[nt][1]);
      }
    }
  }
  const double* sa = p.sa + (size_t)bt * p.nr;
  const float2* na = p.na + (size_t)bt * p.nr;
  // s: the sum in units of the scales of A's row r and B's row c
  auto refused = [&](int r, int c2, float s) {
    const float2 x = na[r], y = p.nb[c2];
    return x.x != 0.f && y.x != 0.f && !oz_accept(s, fminf(x.x, y.y), fminf(y.x, x.y));
  };
  auto put = [&](int r, int c2) {
    const unsigned at = atomicAdd(p.count, 1u);
    if (at < p.cap)
      p.list[at] = ((unsigned long long)bt << 32) | ((unsigned long long)r << 16) | (unsigned long long)c2;
    else if (p.step == 1)
      *p.bad = 1;
  };
#pragma unroll
  for (int mt = 0; mt < 4; ++mt)
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = m * RF_T + wm + mt * 16 + (lane >> 2) + 8 * (i >> 1);
        const int c2 = q * RF_T + wn + nt * 8 + 2 * (lane & 3) + (i & 1);
        if (r >= p.nr || c2 >= p.nr) continue;
        const float s = c[mt][nt][i] * 0x1p-14f;
        if (refused(r, c2, s)) put(r, c2);
        if (m != q) {   // the element across the diagonal: in other units, powers of two (FP64 divisions took 0.1 ms a launch)
          auto ex = [](double v) { return __double2hiint(v) >> 20; };
          const int u = ex(sa[r]) - ex(sa[c2]) + ex(p.sb[2 * c2]) - ex(p.sb[2 * r]);
          if (refused(c2, r, s * __uint_as_float((uint32_t)(min(max(u, -126), 127) + 127) << 23))) put(c2, r);
        }
      }
}

// Digits of the local functions' rows f [np][n], eight each (a function that
// falls off keeps FP64's digits to 2^-10 of its largest value, and what it loses
// below is 2^-64 of that): rows (Re f, Im f) and (-Im f, Re f) as in
// oz_split_rows with pair = 1, dig [8][2 np][kp]; with them its magnitudes max(|Re|,
// |Im|) as BF16 in units of the row's scale, mag [np][kp / 2], the row's norm in
// these units and 2^1/2 of its number of entries.  One block per function.
__global__ void __launch_bounds__(256) oz_split_functions(const double2* __restrict__ f, int n, int np, int kp,
                                                          __half* __restrict__ dig, unsigned short* __restrict__ mag,
                                                          double* __restrict__ scale, float2* __restrict__ norm,
                                                          int* __restrict__ bad) {
  const int row = blockIdx.x;
  const double2* x = f + (size_t)row * n;
  unsigned key = 0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) key = max(key, max(oz_key(x[k].x), oz_key(x[k].y)));
  key = block_max(key);
  int flag = 0;
  const int e = oz_exponent(key, &flag);
  uint32_t* out = reinterpret_cast<uint32_t*>(dig) + (size_t)2 * row * (kp / 2);
  const size_t digit = (size_t)2 * np * (kp / 2);
  float sq = 0.f;
  int count = 0;
  for (int k = threadIdx.x; k < kp / 2; k += blockDim.x) {
    const double2 v = k < n ? x[k] : make_double2(0.0, 0.0);
    int dr[OZ_SF], di[OZ_SF], dm[OZ_SF];
    oz_digits8(v.x, e, dr);
    oz_digits8(v.y, e, di);
    oz_digits8(-v.y, e, dm);
#pragma unroll
    for (int i = 0; i < OZ_SF; ++i) {
      const __half2 a = __floats2half2_rn((float)dr[i], (float)di[i]), b = __floats2half2_rn((float)dm[i], (float)dr[i]);
      out[i * digit + k] = *reinterpret_cast<const uint32_t*>(&a);
      out[i * digit + kp / 2 + k] = *reinterpret_cast<const uint32_t*>(&b);
    }
    const float ur = oz_unit(v.x, e), ui = oz_unit(v.y, e);
    mag[(size_t)row * (kp / 2) + k] = (unsigned short)(__float_as_uint(fmaxf(ur, ui)) >> 16);
    sq += ur * ur + ui * ui;
    count += oz_nonzero(v);
  }
  const float2 nr = block_norm(sq, count);
  if (threadIdx.x != 0) return;
  const double s = scalbn(1.0, e);
  scale[2 * row] = scale[2 * row + 1] = s;
  norm[row] = nr;
  if (flag) atomicOr(bad, 1);
}

// exponent that the magnitudes of column n are taken relative to: its first entry's
__device__ __forceinline__ int first_exponent(double2 v) {
  const unsigned key = max(oz_key(v.x), oz_key(v.y));
  return key ? (int)(key >> 20) - 1022 : 0;
}

// One reading of u[k][x][n] for the row scales and for what oz_accept asks:
//   keys[k][n]          largest magnitude key over x
//   cover[part][k][p][n] sum over the part's grid points of |f_p(x)| |u_kn(x)|, of the
//                       larger component's BF16 each, rounded down, in units of
//                       f's scale and 2^first_exponent
// Blocks of 64 bands x `per` grid points; a warp takes 8 bands, whose values it
// loads as they stand in the product's registers, and 64 functions at a time
// from shared memory (mma.sync m16n8k16).  Bound by HBM: 2.1 GB in 0.36 ms (the
// keys alone 0.29).
constexpr int CV_P = 64, CV_X = 256, CV_LD = CV_X + 8;
__global__ void __launch_bounds__(256) oz_cover(const double2* __restrict__ u, int nx, int nb, int per,
                                                const unsigned short* __restrict__ mag, int np, int xp,
                                                unsigned* __restrict__ keys, float* __restrict__ cover) {
  __shared__ __align__(16) unsigned short fs[CV_P * CV_LD];
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, k = blockIdx.z;
  const int n0 = blockIdx.y * 64 + (threadIdx.x >> 5) * 8, n = n0 + g;
  const int xa = blockIdx.x * per, xb = min(nx, xa + per);
  const bool in = n < nb;
  const double2* p = u + (size_t)k * nx * nb + (in ? n : 0);
  const int shift = (first_exponent(p[0]) + (1023 - 127)) << 7;   // of the exponent, above BF16's 7 bits
  unsigned key = 0;
  auto bf16 = [&](double2 v) {
    const int m = max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff);
    return (uint32_t)min(max((m >> 13) - shift, 0), 0x7f7f);
  };
  double2 w[8];   // the next 32 points: of each 16, this lane's four
  auto load = [&](int x0) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int x = x0 + 2 * t + (i & 1) + 8 * (i >> 1);
      w[i] = make_double2(0.0, 0.0);
      if (in && x < xb) w[i] = load_in_place(p + (size_t)x * nb);
    }
  };
  for (int p0 = 0; p0 < np; p0 += CV_P) {
    load(xa);
    float c[CV_P / 16][4];
#pragma unroll
    for (int i = 0; i < CV_P / 4; ++i) c[i >> 2][i & 3] = 0.f;
    for (int x0 = xa; x0 < xb; x0 += CV_X) {
      __syncthreads();
#pragma unroll
      for (int i = threadIdx.x; i < CV_P * (CV_X / 8); i += 256) {
        const int r = i / (CV_X / 8), x = i % (CV_X / 8) * 8;
        *reinterpret_cast<uint4*>(&fs[r * CV_LD + x]) =
            p0 + r < np && x0 + x < xp ? *reinterpret_cast<const uint4*>(&mag[(size_t)(p0 + r) * xp + x0 + x])
                                       : make_uint4(0, 0, 0, 0);
      }
      __syncthreads();
      for (int xs = 0; xs < CV_X && x0 + xs < xb; xs += 32) {
        double2 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = w[i];
        if (x0 + xs + 32 < xb) load(x0 + xs + 32);   // across the barriers above too
        if (p0 == 0)
#pragma unroll
          for (int i = 0; i < 8; ++i) key = max(key, max(oz_key(v[i].x), oz_key(v[i].y)));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t b0 = bf16(v[4 * h]) | bf16(v[4 * h + 1]) << 16, b1 = bf16(v[4 * h + 2]) | bf16(v[4 * h + 3]) << 16;
#pragma unroll
          for (int mt = 0; mt < CV_P / 16; ++mt) {
            uint32_t a[4];
            ldmatrix_x4(smem_u32(&fs[(mt * 16 + (lane & 15)) * CV_LD + xs + 16 * h + (lane >> 4) * 8]), a);
            mma_16x8x16<true>(c[mt], a, b0, b1);
          }
        }
      }
    }
    float* o = cover + ((size_t)blockIdx.x * gridDim.z + k) * np * nb;
#pragma unroll
    for (int mt = 0; mt < CV_P / 16; ++mt)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int q = p0 + mt * 16 + g + 8 * (i >> 1), m = n0 + 2 * t + (i & 1);
        if (q < np && m < nb) o[(size_t)q * nb + m] = c[mt][i];
      }
  }
  key = max(key, __shfl_xor_sync(0xffffffffu, key, 1));
  key = max(key, __shfl_xor_sync(0xffffffffu, key, 2));
  if (t == 0 && in) atomicMax(keys + (size_t)k * nb + n, key);
}

// Lists the elements [k][p][n] of a pass whose magnitudes do not cover the
// digits' error.  u's rounding counts with f's norm; f's own is 2^-8 of u's.
struct OzRepair {
  const double2 *u, *f, *phase;   // u, phase: the pass's first k point
  const float* cover;
  const unsigned* keys;
  const int* expo;
  const float2* norm;   // of f's rows {norm, root}
  int parts, nk, nx, xp, nb, np, nkt, k0;
  double alpha;
  double2* out;
  unsigned* list;    // [cap]
  unsigned cap;
  unsigned* count;
};
__global__ void __launch_bounds__(256) oz_refused(const OzRepair p, int* __restrict__ bad) {
  const size_t total = (size_t)p.nk * p.np * p.nb, i = blockIdx.x * (size_t)256 + threadIdx.x;
  bool refused = false;
  if (i < total) {
    const int n = (int)(i % p.nb), q = (int)(i / p.nb % p.np), k = (int)(i / p.nb / p.np);
    const float2 f = p.norm[q];
    if (f.x > 0.f && p.keys[(size_t)k * p.nb + n]) {
      float s = 0.f;
      for (int j = 0; j < p.parts; ++j) s += p.cover[j * total + i];
      s = ldexpf(s, first_exponent(p.u[(size_t)k * p.nx * p.nb + n]) - p.expo[(size_t)k * p.nb + n]);
      refused = !(isfinite(s) && oz_accept(s, f.x, f.y * 0x1p-8f));
    }
  }
  const unsigned w = __ballot_sync(0xffffffffu, refused), lane = threadIdx.x & 31;
  if (!w) return;
  unsigned at = 0;
  if (lane == 0) {
    at = atomicAdd(p.count, __popc(w));
    if (at + __popc(w) > p.cap) *bad = 1;
  }
  at = __shfl_sync(0xffffffffu, at, 0) + __popc(w & ((1u << lane) - 1u));
  if (refused && at < p.cap) p.list[at] = (unsigned)i;
}

// ... and forms them on the FP64 pipe, one warp each
__global__ void __launch_bounds__(256) oz_repair(const OzRepair p) {
  const unsigned m = min(*p.count, p.cap), lane = threadIdx.x & 31;
  for (unsigned w = blockIdx.x * 8 + (threadIdx.x >> 5); w < m; w += gridDim.x * 8) {
    const unsigned i = p.list[w];
    const int n = (int)(i % p.nb), q = (int)(i / p.nb % p.np), k = (int)(i / p.nb / p.np);
    const double2 *f = p.f + (size_t)q * p.nx, *ph = p.phase + (size_t)k * p.xp, *u = p.u + (size_t)k * p.nx * p.nb + n;
    double2 s = make_double2(0.0, 0.0);
    for (int x = lane; x < p.nx; x += 32) {
      const double2 a = f[x];
      if (a.x == 0.0 && a.y == 0.0) continue;
      const double2 b = u[(size_t)x * p.nb], e = ph[x];
      const double br = b.x * e.x - b.y * e.y, bi = b.x * e.y + b.y * e.x;
      s.x = fma(a.x, br, fma(a.y, bi, s.x));
      s.y = fma(a.x, bi, fma(-a.y, br, s.y));
    }
    for (int off = 16; off > 0; off >>= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
    }
    if (lane == 0) p.out[((size_t)q * p.nkt + p.k0 + k) * p.nb + n] = make_double2(p.alpha * s.x, p.alpha * s.y);
  }
}

// e^{ik.x} per dimension: tab_d[m][j] = e^{2 pi i (m + s_d) j / (nk_d nx_d)}, the
// three tables one after the other
__global__ void __launch_bounds__(256) oz_tables(oz_mesh ms, double2* __restrict__ tab) {
  long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  double2* t = tab;
  for (int d = 0; d < 3; ++d) {
    const long long n = (long long)ms.nk[d] * ms.nx[d];
    if (i < n) {
      double fr = ((int)(i / ms.nx[d]) + ms.s[d]) * (double)(i % ms.nx[d]) / ((double)ms.nk[d] * ms.nx[d]), sn, cs;
      fr -= floor(fr);
      sincospi(2.0 * fr, &sn, &cs);
      t[i] = make_double2(cs, sn);
      return;
    }
    i -= n;
    t += n;
  }
}

// phases [k][xp] of the k points from k0, xp grid points (zero beyond nx)
__global__ void __launch_bounds__(256) oz_phases(oz_mesh ms, const double2* __restrict__ tab, int k0, int xp,
                                                 double2* __restrict__ phase) {
  const int x = blockIdx.x * 256 + threadIdx.x, k = k0 + blockIdx.y;
  if (x >= xp) return;
  double2 r = make_double2(0.0, 0.0);
  if (x < ms.nx[0] * ms.nx[1] * ms.nx[2]) {
    const int m2 = k % ms.nk[2], m1 = (k / ms.nk[2]) % ms.nk[1], m0 = k / (ms.nk[1] * ms.nk[2]);
    const int j2 = x % ms.nx[2], j1 = (x / ms.nx[2]) % ms.nx[1], j0 = x / (ms.nx[1] * ms.nx[2]);
    const double2* t1 = tab + (size_t)ms.nk[0] * ms.nx[0];
    const double2* t2 = t1 + (size_t)ms.nk[1] * ms.nx[1];
    const double2 a = tab[(size_t)m0 * ms.nx[0] + j0], b = t1[(size_t)m1 * ms.nx[1] + j1],
                  c = t2[(size_t)m2 * ms.nx[2] + j2];
    const double2 ab = make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
    r = make_double2(ab.x * c.x - ab.y * c.y, ab.x * c.y + ab.y * c.x);
  }
  phase[(size_t)blockIdx.y * xp + x] = r;
}

// row scales 2^e of the rotated Bloch functions: |e^{ik.x} u| components are at
// most sqrt 2 times those of u, one more bit
__global__ void __launch_bounds__(256) oz_bloch_scales(const unsigned* __restrict__ keys, int n, int* __restrict__ expo,
                                                       double* __restrict__ scale, int* __restrict__ bad) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  int flag = 0;
  const int e = oz_exponent(keys[i], &flag) + 1;
  expo[i] = e;
  scale[i] = scalbn(1.0, e);
  if (flag) atomicOr(bad, 1);
}

constexpr int OZ_W = 16;                               // worker warps of oz_project
constexpr int OZ_PT = 64 + 32 * OZ_W;                  // its threads
constexpr int OZ_PH = 4;                               // phase slots
constexpr size_t OZ_PSMEM = OZ_SMEM + OZ_PH * OZ_KB / 2 * sizeof(double2);

struct OzProject {
  const double2* u;       // the pass's first k point: [k][x][n]
  const double2* phase;   // [k][32 kb]
  const int* expo;        // [k][nb]
  const double* scale;    // [k][nb]
  const double* scale_a;
  int nx, nb, np2, nkt, k0;
  int mt, nt, ntiles, kb, cpt;   // M tiles, N tiles, all tiles, K blocks and chunks of a tile
  double alpha;
  double* out;            // [np][nkt][nb] complex
  long long* part_hi;     // [CTA][2][128][64] sums of the tiles that CTAs share
  uint32_t* part_lo;
  int* err;
  unsigned long long wait_ns;
};

// first chunk of CTA c: all tiles' chunks in one line, cut into equal parts
__host__ __device__ inline long long oz_start(long long c, long long chunks, int grid) { return c * chunks / grid; }

__device__ __forceinline__ void oz_store(const OzProject& p, int t, int row, int col, long long hi, long long lo) {
  const int m = t % p.mt, r = t / p.mt, n = r % p.nt, k = r / p.nt;
  const int gr = m * OZ_M + row, gc = n * OZ_N + col;
  if (gr < p.np2 && gc < p.nb)
    p.out[2 * (((size_t)(gr >> 1) * p.nkt + p.k0 + k) * p.nb + gc) + (gr & 1)] =
        oz_value(hi, lo) * (p.alpha * p.scale_a[gr] * p.scale[(size_t)k * p.nb + gc]);
}

// Projections a = alpha F (e^{ik.x} u)^T: the product kernel above with the Bloch
// functions turned into digits on the way into shared memory instead of
// written to memory in 14 bytes per 8 and read back.  Warp 0 streams the
// projectors' digits and the phases of a K block (32 grid points), warp 1
// issues, warps 2-17 both convert (thread: band tid / 8, four grid points: 64-
// byte reads, and 16-byte stores that fill all banks) and drain (32 rows x 16
// columns each).  A chunk is drained after the first block of the next one is
// converted, so that the tensor core has that block while they drain.  The
// phases' products (4 FP64 operations per complex entry: 4096 clocks a block at
// two per SM and clock) run beside the digit products' 5120 clocks; a block
// takes about 11,300, in which the 16 warps' FP64, integer and load phases
// overlap only in part (FP64 pipe 39 %, tensor pipe 47 %).  With conversion and
// draining on warps of their own (eight each) it was 12,300.
// The CTAs take equal shares of all tiles' chunks; sums of a tile that two or more share
// go to part_hi and part_lo, exact as they are, and oz_join adds them.
__global__ void __launch_bounds__(OZ_PT, 1) oz_project(const __grid_constant__ CUtensorMap ma, const OzProject p) {
  extern __shared__ unsigned char oz_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)oz_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* const bs = sm + OZ_AS * OZ_A + OZ_BD;   // first B slot
  double2* phs = (double2*)(sm + OZ_AS * OZ_A + OZ_BAREA);
  unsigned long long* bars = (unsigned long long*)(phs + OZ_PH * (OZ_KB / 2));
  constexpr int NBAR = 2 * OZ_AS + 2 * OZ_BS + 2 * OZ_PH + 1 + OZ_D + 1;
  uint32_t* tmem_slot = (uint32_t*)(bars + NBAR);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  volatile int* a_issued = (volatile int*)(tmem_slot + 2);
  volatile int* p_issued = (volatile int*)(tmem_slot + 3);
  const uint32_t sa = smem_u32(sm), sb = sa + OZ_AS * OZ_A + OZ_BD, sp = smem_u32(phs), b0 = smem_u32(bars);
  auto afull = [&](int s) { return b0 + 8 * s; };
  auto aempty = [&](int s) { return b0 + 8 * (OZ_AS + s); };
  auto bfull = [&](int s) { return b0 + 8 * (2 * OZ_AS + s); };
  auto bempty = [&](int s) { return b0 + 8 * (2 * OZ_AS + OZ_BS + s); };
  auto pfull = [&](int s) { return b0 + 8 * (2 * OZ_AS + 2 * OZ_BS + s); };
  auto pempty = [&](int s) { return b0 + 8 * (2 * OZ_AS + 2 * OZ_BS + OZ_PH + s); };
  const uint32_t tfull = b0 + 8 * (2 * OZ_AS + 2 * OZ_BS + 2 * OZ_PH), tempty = tfull + 8, fin = b0 + 8 * (NBAR - 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < OZ_AS; ++s) {
      mbar_init(afull(s), 1);
      mbar_init(aempty(s), 1);
    }
    for (int s = 0; s < OZ_BS; ++s) {
      mbar_init(bfull(s), OZ_W);
      mbar_init(bempty(s), 1);
    }
    for (int s = 0; s < OZ_PH; ++s) {
      mbar_init(pfull(s), 1);
      mbar_init(pempty(s), OZ_W);
    }
    mbar_init(tfull, 1);
    for (int s = 0; s < OZ_D; ++s) mbar_init(tempty + 8 * s, OZ_W);
    mbar_init(fin, 1);
    *abort_flag = 0;
    *a_issued = 0;
    *p_issued = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int z = 0; z <= OZ_BS; ++z)   // the tiles of zeros
    for (int i = threadIdx.x; i < OZ_BD / 16; i += blockDim.x)
      reinterpret_cast<uint4*>(sm + OZ_AS * OZ_A + z * (OZ_B + OZ_BD))[i] = make_uint4(0, 0, 0, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // this CTA's blocks: from block bq of tile tq, `total` of them
  const long long chunks = (long long)p.ntiles * p.cpt;
  const long long q0 = oz_start(blockIdx.x, chunks, gridDim.x), q1 = oz_start(blockIdx.x + 1, chunks, gridDim.x);
  const int tq = (int)(q0 / p.cpt), bq = 2 * (int)(q0 % p.cpt), te = (int)((q1 - 1) / p.cpt);
  const int be = min(2 * (int)((q1 - 1) % p.cpt) + 2, p.kb);
  const int total = (te - tq) * p.kb + be - bq;

  if (warp == 0 && lane == 0) {
    int ia = 0, ip = 0, t = tq, b = bq, tp = tq, bp = bq;
    bool ok = true;
    auto phases = [&]() {
      const int s = ip % OZ_PH;
      if (!oz_wait(pempty(s), ((uint32_t)(ip / OZ_PH) & 1u) ^ 1u, abort_flag, p.wait_ns)) return false;
      mbar_expect_tx(pfull(s), OZ_KB / 2 * sizeof(double2));
      bulk_load(sp + s * (OZ_KB / 2) * (int)sizeof(double2),
                p.phase + ((size_t)(tp / p.mt / p.nt) * p.kb + bp) * (OZ_KB / 2), OZ_KB / 2 * sizeof(double2), pfull(s));
      *p_issued = ++ip;
      if (++bp == p.kb) bp = 0, ++tp;
      return true;
    };
    for (int i = 0; i < total && ok; ++i) {
      while (ok && ip < total && ip < i + OZ_PH - 1) ok = phases();
      const int m = t % p.mt;
      for (int j = 0; j < OZ_SF && ok; ++j) {
        const int q = ia % OZ_AS;
        if (!(ok = oz_wait(aempty(q), ((uint32_t)(ia / OZ_AS) & 1u) ^ 1u, abort_flag, p.wait_ns))) break;
        mbar_expect_tx(afull(q), OZ_A);
        tma_load_3d(sa + q * OZ_A, &ma, afull(q), b * OZ_KB, m * OZ_M, j);
        *a_issued = ++ia;
      }
      if (++b == p.kb) b = 0, ++t;
    }
    if (!ok) {
      atomicExch(p.err, 1);
      *abort_flag = 1;
    }
  } else if (warp == 1 && lane == 0) {
    int c = 0, b = bq;   // chunk of the tile, as this CTA counts
    oz_issue z;
    bool ok = true;
    for (int i = 0; i < total; ++i) {
      const int s = i % OZ_BS;
      if (!(ok = oz_wait(bfull(s), (uint32_t)(i / OZ_BS) & 1u, abort_flag, p.wait_ns))) break;
      const unsigned long long db = sdesc_sw128(sb + s * (OZ_B + OZ_BD));
      if (!(ok = issue_block<OZ_SF>(tmem, sa, db, (b & 1) == 0, c, z, afull(0), aempty(0), tempty, abort_flag, p.wait_ns))) break;
      mma_commit(bempty(s));
      if ((b & 1) == 1 || b + 1 == p.kb) {
        mma_commit(tfull);
        ++c;
      }
      if (++b == p.kb) b = 0, c = 0;
    }
    if (!ok) {
      atomicExch(p.err, 1);
      *abort_flag = 1;
    }
    mma_commit(fin);   // issued products retire before tensor memory is freed
    const unsigned long long t0 = gtime();
    while (!mbar_try(fin, 0) && gtime() - t0 < OZ_WAIT_NS) {
    }
  } else if (warp >= 2) {
    const int tid = threadIdx.x - 64, nl = tid >> 3, xg = tid & 7;
    const int row = (warp & 3) * 32 + lane, col0 = ((warp - 2) >> 2) * 16;
    const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)col0;
    const uint32_t dst = smem_u32(bs) + nl * 128 + ((xg ^ (nl & 7)) << 4);
    long long hi[16];
    uint32_t lo[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) hi[c] = 0, lo[c] = 0;
    int chunk = 0, cc = 0;   // drained so far, of them in this tile
    // the accumulators of the oldest chunk not yet drained, which ends with block b of tile t
    auto drain = [&](int t, int b, bool last) {
      if (!__all_sync(0xffffffffu, oz_wait(tfull, (uint32_t)chunk & 1u, abort_flag, p.wait_ns))) return false;
      ++chunk;
      tc_fence_after();
      const bool end = b + 1 == p.kb || last;
      drain_chunk<16>(ta, cc, end, tempty, lane, hi, lo);
      ++cc;
      if (!end) return true;
      cc = 0;
      const size_t o = ((size_t)(2 * blockIdx.x + (t > tq ? 1 : 0)) * OZ_M + row) * OZ_N + col0;
      const bool whole = b + 1 == p.kb && (t > tq || bq == 0);
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        if (whole) {
          oz_store(p, t, row, col0 + c, hi[c], lo[c]);
        } else {
          p.part_hi[o + c] = hi[c];
          p.part_lo[o + c] = lo[c];
        }
        hi[c] = 0, lo[c] = 0;
      }
      return true;
    };
    double2 w[4];
    const double2* base = nullptr;   // this thread's first entry of the tile, nullptr: a column beyond the last
    int e = 0, en = 0;
    auto tile = [&](int t) {
      const int r = t / p.mt, n = (r % p.nt) * OZ_N + nl, k = r / p.nt;
      const bool in = t <= te && n < p.nb;
      base = in ? p.u + ((size_t)k * p.nx + 4 * xg) * p.nb + n : nullptr;
      en = in ? p.expo[(size_t)k * p.nb + n] : 0;
    };
    auto load = [&](int b) {
      const int left = base ? p.nx - b * (OZ_KB / 2) - 4 * xg : 0;
      const double2* a = base + (size_t)b * (OZ_KB / 2) * p.nb;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        w[i] = make_double2(0.0, 0.0);
        if (i < left) w[i] = load_in_place(a + (size_t)i * p.nb);
      }
      // lines of a block four ahead into L2: the loads then cover an L2 hit, not HBM's latency
      if ((nl & 7) == 0 && b + 4 < p.kb) {
        a += (size_t)4 * (OZ_KB / 2) * p.nb;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i < left - 4 * (OZ_KB / 2)) asm volatile("prefetch.global.L2 [%0];" ::"l"(a + (size_t)i * p.nb));
      }
    };
    tile(tq);
    load(bq);
    int t = tq, b = bq, t1 = tq, b1 = bq;
    bool ok = true;
    for (int i = 0; i < total; ++i) {
      if (b == 0 || i == 0) e = en;
      const int s = i % OZ_BS, q = i % OZ_PH;
      ok = __all_sync(0xffffffffu, oz_wait(pfull(q), (uint32_t)(i / OZ_PH) & 1u, abort_flag, p.wait_ns) &&
                                       oz_wait(bempty(s), ((uint32_t)(i / OZ_BS) & 1u) ^ 1u, abort_flag, p.wait_ns));
      if (!ok) break;
      oz_fix f[8];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double2 c = phs[q * (OZ_KB / 2) + 4 * xg + j];
        f[2 * j] = oz_fixed(w[j].x * c.x - w[j].y * c.y, e);
        f[2 * j + 1] = oz_fixed(w[j].x * c.y + w[j].y * c.x, e);
      }
#pragma unroll
      for (int j = 0; j < OZ_S; ++j)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + s * (OZ_B + OZ_BD) + j * OZ_BD),
                     "r"(oz_digit2(f[0], f[1], j)), "r"(oz_digit2(f[2], f[3], j)), "r"(oz_digit2(f[4], f[5], j)),
                     "r"(oz_digit2(f[6], f[7], j))
                     : "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bfull(s));
        mbar_arrive(pempty(q));
      }
      const int tc = t, bc = b;
      if (++b == p.kb) b = 0, tile(++t);
      if (i + 1 < total) load(b);
      if (i > 0 && (bc & 1) == 0 && !(ok = drain(t1, b1, false))) break;
      t1 = tc, b1 = bc;
    }
    if (ok) ok = drain(t1, b1, true);
    if (!ok && lane == 0) {
      atomicExch(p.err, 1);
      *abort_flag = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    // copies in flight land before the CTA leaves (the last use of each slot)
    const int na = *a_issued, np = *p_issued;
    for (int k = na > OZ_AS ? na - OZ_AS : 0; k < na; ++k) {
      const unsigned long long t0 = gtime();
      while (!mbar_try(afull(k % OZ_AS), (uint32_t)(k / OZ_AS) & 1u) && gtime() - t0 < OZ_WAIT_NS) {
      }
    }
    for (int k = np > OZ_PH ? np - OZ_PH : 0; k < np; ++k) {
      const unsigned long long t0 = gtime();
      while (!mbar_try(pfull(k % OZ_PH), (uint32_t)(k / OZ_PH) & 1u) && gtime() - t0 < OZ_WAIT_NS) {
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// tiles shared by several CTAs of oz_project (grid of them): the sum of their
// partial sums, one block per tile and 16 rows
__global__ void __launch_bounds__(256) oz_join(const OzProject p, int grid) {
  const int t = blockIdx.x;
  const long long chunks = (long long)p.ntiles * p.cpt, qa = (long long)t * p.cpt, qb = qa + p.cpt - 1;
  auto owner = [&](long long q) {
    long long c = q * grid / chunks;
    while (oz_start(c + 1, chunks, grid) <= q) ++c;
    return (int)c;
  };
  const int ca = owner(qa), cb = owner(qb);
  if (ca == cb) return;
  for (int i = threadIdx.x; i < 16 * OZ_N; i += 256) {
    const int row = blockIdx.y * 16 + i / OZ_N, col = i % OZ_N;
    long long hi = 0, lo = 0;
    for (int c = ca; c <= cb; ++c) {
      const int slot = 2 * c + (oz_start(c, chunks, grid) / p.cpt < t ? 1 : 0);
      const size_t o = ((size_t)slot * OZ_M + row) * OZ_N + col;
      hi += p.part_hi[o];
      lo += p.part_lo[o];
    }
    oz_store(p, t, row, col, hi, lo);
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
int bse_oz_kp(int k) { return (k + OZ_KB - 1) / OZ_KB * OZ_KB; }

bse_status bse_oz_split_rows(const double2* x, int rows, int n, const double2* d, int batches, int pair,
                             const bse_oz_operand& o, int* bad, cudaStream_t st) {
  oz_split_rows<<<dim3((unsigned)rows, (unsigned)batches), 256, 0, st>>>(x, n, d, rows, o.kp, pair, (__half*)o.digits,
                                                                          o.scale, o.norm, bad);
  return cudaGetLastError() == cudaSuccess ? BSE_OK : BSE_ERR_CUDA;
}

// The scratch holds the projectors' digits, the phases and magnitude sums of as
// many k points per pass as fit 256 MB, and the shared tiles' sums: 128 MB for
// 8^3 k x 16^3 points.
bse_status bse_oz_project(const double2* u, const int* nk, const int* nx, int nb, const double* kshift,
                          const double2* f, int np, double dv, double2* a, cudaStream_t st, bool* done) {
  *done = false;
  oz_mesh ms;
  for (int i = 0; i < 3; ++i) {
    ms.nk[i] = nk[i];
    ms.nx[i] = nx[i];
    ms.s[i] = kshift ? kshift[i] : 0.0;
  }
  const int nkt = nk[0] * nk[1] * nk[2], nxt = nx[0] * nx[1] * nx[2], kp = bse_oz_kp(2 * nxt);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaFuncSetAttribute(oz_project, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_PSMEM) != cudaSuccess) {
    cudaGetLastError();
    return BSE_OK;
  }
  // parts of the grid in oz_cover: of 1024 points, and enough to fill the SMs
  const int nbt = (nb + 63) / 64, want = std::max((nxt + 1023) / 1024, (4 * sms + nkt * nbt - 1) / (nkt * nbt));
  const int xpart = (nxt + CV_X * std::min(want, 64) - 1) / (CV_X * std::min(want, 64)) * CV_X;
  const int parts = (nxt + xpart - 1) / xpart;
  const size_t per = (size_t)kp / 2 * sizeof(double2), outs = (size_t)np * nb, pcov = (size_t)parts * outs * sizeof(float);
  const int nkc = (int)std::min<size_t>({(size_t)nkt, std::max<size_t>(((size_t)256 << 20) / (per + pcov), 1), (size_t)32768,
                                         std::max<size_t>(((size_t)1 << 31) / outs, 1)});
  auto pad = [](size_t n) { return (n + 255) / 256 * 256; };
  long long ntab = 0;
  for (int i = 0; i < 3; ++i) ntab += (long long)nk[i] * nx[i];
  const size_t sd = bse_oz_digit_bytes(1, 2 * np, kp) / OZ_S * OZ_SF, sf = pad((size_t)2 * np * sizeof(double)), sph = pad(nkc * per);
  const size_t stab = pad((size_t)ntab * sizeof(double2)), skey = pad((size_t)nkc * nb * sizeof(unsigned));
  const size_t ssc = pad((size_t)nkc * nb * sizeof(double)), npart = (size_t)2 * sms * OZ_M * OZ_N;
  const size_t smag = pad((size_t)np * (kp / 2) * sizeof(short)), snrm = pad((size_t)np * sizeof(float2));
  const size_t scov = pad(nkc * pcov), cap = nkc * outs / 32 + 1024, slist = pad(cap * sizeof(unsigned));
  bse_scratch sc(st);
  if (!sc.get(sd + sf + sph + stab + 2 * skey + ssc + npart * 12 + smag + snrm + scov + slist + 256)) return BSE_OK;
  char* q = (char*)sc.p;
  bse_oz_operand A;
  A.digits = q, q += sd;
  A.scale = (double*)q, q += sf;
  A.rows = 2 * np, A.kp = kp;
  OzProject p{};
  double2* phase = (double2*)q;
  q += sph;
  double2* tab = (double2*)q;
  q += stab;
  unsigned* keys = (unsigned*)q;
  q += skey;
  int* expo = (int*)q;
  q += skey;
  double* scale = (double*)q;
  q += ssc;
  p.part_hi = (long long*)q, q += npart * 8;
  p.part_lo = (uint32_t*)q, q += npart * 4;
  unsigned short* mag = (unsigned short*)q;
  q += smag;
  float2* norm = (float2*)q;
  q += snrm;
  float* cover = (float*)q;
  q += scov;
  unsigned* list = (unsigned*)q;
  q += slist;
  int* word = (int*)q;   // {wait gave up, out of range or too many elements refused, elements refused}
  p.phase = phase;
  p.expo = expo;
  p.scale = scale;
  p.scale_a = A.scale;
  p.nx = nxt;
  p.nb = nb;
  p.np2 = 2 * np;
  p.nkt = nkt;
  p.mt = (2 * np + OZ_M - 1) / OZ_M;
  p.nt = (nb + OZ_N - 1) / OZ_N;
  p.kb = kp / OZ_KB;
  p.cpt = (p.kb + 1) / 2;
  p.alpha = dv;
  p.out = (double*)a;
  p.err = word;
  p.wait_ns = wait_limit();
  CUtensorMap ma;
  if (!digit_map(&ma, (const __half*)A.digits, kp, A.rows, OZ_SF, OZ_M, 1)) return BSE_OK;
  cudaMemsetAsync(word, 0, 2 * sizeof(int), st);
  // rows (Re f, Im f) and (-Im f, Re f): real and imaginary part of conj(f) times a column
  oz_split_functions<<<(unsigned)np, 256, 0, st>>>(f, nxt, np, kp, (__half*)A.digits, mag, A.scale, norm, word + 1);
  bse_status s = BSE_OK;
  OzRepair rp{};
  rp.f = f, rp.phase = phase, rp.cover = cover, rp.keys = keys, rp.expo = expo, rp.norm = norm;
  rp.parts = parts, rp.nx = nxt, rp.xp = kp / 2, rp.nb = nb, rp.np = np, rp.nkt = nkt;
  rp.alpha = dv;
  rp.out = a;
  rp.list = list;
  rp.cap = (unsigned)cap;
  rp.count = (unsigned*)word + 2;
  oz_tables<<<(unsigned)((ntab + 255) / 256), 256, 0, st>>>(ms, tab);
  for (int k = 0; k < nkt && s == BSE_OK; k += nkc) {
    const int n = std::min(nkc, nkt - k);
    p.u = u + (size_t)k * nxt * nb;
    p.k0 = k;
    p.ntiles = p.mt * p.nt * n;
    cudaMemsetAsync(keys, 0, (size_t)n * nb * sizeof(unsigned), st);
    cudaMemsetAsync(rp.count, 0, sizeof(unsigned), st);
    oz_cover<<<dim3((unsigned)parts, (unsigned)nbt, (unsigned)n), 256, 0, st>>>(p.u, nxt, nb, xpart, mag, np, kp / 2, keys,
                                                                                cover);
    oz_bloch_scales<<<(unsigned)(((long long)n * nb + 255) / 256), 256, 0, st>>>(keys, n * nb, expo, scale, word + 1);
    oz_phases<<<dim3((unsigned)((kp / 2 + 255) / 256), (unsigned)n), 256, 0, st>>>(ms, tab, k, kp / 2, phase);
    const int grid = (int)std::min<long long>(sms, (long long)p.ntiles * p.cpt);
    oz_project<<<grid, OZ_PT, OZ_PSMEM, st>>>(ma, p);
    oz_join<<<dim3((unsigned)p.ntiles, OZ_M / 16), 256, 0, st>>>(p, grid);
    rp.u = p.u;
    rp.nk = n;
    rp.k0 = k;
    oz_refused<<<(unsigned)((n * outs + 255) / 256), 256, 0, st>>>(rp, word + 1);
    oz_repair<<<(unsigned)(4 * sms), 256, 0, st>>>(rp);
    if (cudaGetLastError() != cudaSuccess) s = BSE_ERR_CUDA;
  }
  int hw[2] = {0, 0};
  if (s == BSE_OK && (cudaMemcpyAsync(hw, word, sizeof(hw), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                      cudaStreamSynchronize(st) != cudaSuccess))
    s = BSE_ERR_CUDA;
  if (s != BSE_OK) return s;
  *done = hw[0] == 0 && hw[1] == 0;
  return BSE_OK;
}

bse_status bse_oz_gemm(const bse_oz_operand& a, const bse_oz_operand& b, int batches, double alpha, double* out,
                       long long sb, long long sr2, long long sr1, long long sc, int* err, cudaStream_t st) {
  CUtensorMap ma, mb;
  if (!digit_map(&ma, (const __half*)a.digits, a.kp, a.rows, OZ_S * a.batches, OZ_M, 1) ||
      !digit_map(&mb, (const __half*)b.digits, b.kp, b.rows, OZ_S * b.batches, OZ_N, OZ_S))
    return BSE_ERR_UNSUPPORTED;
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
  p.wait_ns = wait_limit();
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaFuncSetAttribute(oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_SMEM) != cudaSuccess) {
    cudaGetLastError();
    return BSE_ERR_UNSUPPORTED;
  }
  oz_gemm<<<std::min(p.ntiles, sms), OZ_THREADS, OZ_SMEM, st>>>(ma, mb, p);
  return cudaGetLastError() == cudaSuccess ? BSE_OK : BSE_ERR_CUDA;
}

bse_status bse_oz_refused(const bse_oz_operand& a, const bse_oz_operand& b, int batches, unsigned long long* list,
                          unsigned cap, unsigned* count, int* bad, cudaStream_t st) {
  OzRefused p{};
  p.a = (const __half*)a.digits, p.b = (const __half*)b.digits;
  p.sa = a.scale, p.sb = b.scale;
  p.na = a.norm, p.nb = b.norm;
  p.nr = a.rows;
  p.kp = a.kp;
  p.mt = (a.rows + RF_T - 1) / RF_T;
  p.list = list;
  p.cap = cap;
  p.bad = bad;
  if (cudaFuncSetAttribute(oz_gemm_refused, cudaFuncAttributeMaxDynamicSharedMemorySize, RF_S * RF_BYTES) != cudaSuccess) {
    cudaGetLastError();
    return BSE_ERR_UNSUPPORTED;
  }
  // every fourth K block from 64 of them on (a random sum's magnitudes are then
  // still some 20 times the limit)
  cudaMemsetAsync(count, 0, 2 * sizeof(unsigned), st);
  for (int all = 0; all < 2; ++all) {
    p.step = all || a.kp < 64 * OZ_KB ? 1 : 4;
    p.count = count + all;
    p.after = all ? count : nullptr;
    oz_gemm_refused<<<dim3((unsigned)(p.mt * (p.mt + 1) / 2), (unsigned)batches), 256, RF_S * RF_BYTES, st>>>(p);
    if (p.step == 1) break;
  }
  return cudaGetLastError() == cudaSuccess ? BSE_OK : BSE_ERR_CUDA;
}
