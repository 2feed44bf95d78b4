// Grouped FP64 GEMM on the tensor cores by exact digit products.
//
// Same work lists and results as gemm_fp64_kernel (lrt_kernels.cu): an output tile sums,
// over its segments, scale_q op(A_q) op(B_q), the segments concatenated along one K axis and
// taken 32 positions (a chunk) at a time.  GB300 issues 2 FP64 FMA per clock and SM but 1024
// FP16 FMA with FP32 accumulation through mma.sync, so each chunk is multiplied in integers:
//
//  - every K position is first given the exponent it has over one operand (its largest element
//    among the tile's rows of A, or columns of B, there): that power of two moves to the other
//    operand, so that a chunk may join operators of any size and operands that are graded in
//    opposite directions along K.  The vectors of a call lie along the other operand, whose rows
//    then do not see each other;
//  - every row of A and column of B of the chunk is scaled by a power of two (its largest
//    exponent) and cut into 7 balanced digits of 9 bits, g_d in [-256, 256]: 63 bits, so an
//    element within 2^9 of its row's largest keeps all of its 53;
//  - digit products A_i B_j with i + j = d <= 6 are summed over the chunk in FP32 (28
//    mma.sync per 16 x 8 x 16): at most 7 * 32 * 2^16 < 2^24, so every sum is exact;
//  - the 7 sums are joined in a 64-bit integer, rounded once to FP64 and added to the tile's
//    FP64 accumulator with the row's and column's power of two: one FP64 instruction per
//    element and chunk instead of 32.
//
// (The splitting is the error-free transformation of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix multiplication",
// Numer. Algorithms 59, 2012, with a fixed digit grid per chunk.)  What a chunk loses is
// relative to its row's largest times its column's largest element (after the exponents above):
// the dropped products (6 pairs of i + j = 7) are below 2^-53.4 of that, cut operands and the
// join's rounding add up to 2^-52.4, and with digits of random sign it is about 2^-59.  That is
// less than the 32 roundings of an FMA chain where the products of the row and column are of
// one size, and more where all of them are far below the two largest elements: sums of small
// products are not as accurate by themselves as an FMA chain's.  Elements whose row or column
// holds an infinity, a NaN, subnormals alone or lies outside 2^-423 .. 2^477 are multiplied in
// plain FP64 from the staged operands.
//
// Measured on the k = 24, M = 500, 6-vector sigma (23.7 G multiply-adds): 44.0 ms by FP64 FMAs,
// 16.3 ms here (15.2 with the exponents taken out of the K positions of phase 2 alone: one more
// pass over the staged operand and one more barrier per chunk); error against 64-bit exact values
// 3.7e-16 (8.3e-16 by FMAs) at k = 8, 3.5e-15 (7.3e-15) on the PPP chain.  The kernel is bound by
// issued instructions (48% of the issue slots; tensor pipe 20%, FP64 pipe 24%): cutting the
// operands (a third of them) and staging cost more than the products.  Hence tiles of 128 staged
// rows for up to 16 16 x 16 units and 16 warps per SM, 2 CTAs of 8 warps at 128 registers (96 rows
// for 8 units, 3 CTAs of 4 warps: 16.9 ms where this split took 15.2); and one row or column scale
// per 32 positions, so a chunk needs no look at the rest of K.  Operands cut ahead into digit
// matrices and fetched by bulk copies were not faster (19.3 ms then: pools of 14 bytes per
// element, chunks that end with every segment, fewer warps).
#include "lrt_kernels.h"
#include "lrt_fp64_tile.h"

#include <atomic>

namespace lrt {

static_assert(GEMM_KC == 32, "the lane mappings below");
constexpr int MMA_ND = 7;                 // digits
constexpr int MMA_WARPS = 8;              // warps of a CTA tile
constexpr int MMA_EMIN = 600, MMA_EMAX = 1500;   // exponent fields the integer path takes
constexpr int MMA_E0 = 1023;
constexpr int MMA_NOBAL = -4096;                  // exponent of a K position where that operand is zero
constexpr int MMA_NONE = -1100;                   // largest exponents of rows up to here: no product but zeros
constexpr int MMA_WILD = (int)0x80000000;        // exponent word of a row the integer path does not take

struct MmaSmem {
  double raw[MMA_ROWS][GEMM_KC];          // chunk operands: A rows, then B columns; 16-byte groups XOR row
  uint32_t dig[MMA_ND][MMA_ROWS][GEMM_KC / 2];   // digits as FP16 pairs, 16-byte groups XOR row / 2
  alignas(16) int ex[MMA_ROWS];           // (E - 539) << 20 of each row (read in pairs)
  double sc[GEMM_KC];                     // segment scale of each K position
  SegS sd[GEMM_SEGB];
  int kst[GEMM_SEGB + 1];
  alignas(16) int bal[GEMM_KC];           // exponents taken out of the K positions
  alignas(8) int2 vl[MMA_ROWS];           // vector block and index inside it of each row
  int wild[2];                            // chunk (by parity) holds a row outside the integer path
  uint32_t neg;                           // K positions of negative scale
  int mode;                               // scales of the chunk: 0 all 1, 1 all +-1, 2 general
};

__device__ __forceinline__ void cp_async8z(void* dst, const void* src, int bytes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm2(uint32_t (&r)[2], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t s) { return __byte_perm(a, b, s); }
// (x & mask) | 0x64006400 as FP16 pairs is 1024 + field; times the signs minus 1280 times the
// signs leaves +-(field - 256)
__device__ __forceinline__ uint32_t digit_pair(uint32_t x, uint32_t mask, uint32_t sign, uint32_t off) {
  uint32_t r;
  const uint32_t h = (x & mask) | 0x64006400u;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(h), "r"(sign), "r"(off));
  return r;
}

// magnitude (its leading bit at bit 61 - sh) biased by 256 in every digit
__device__ __forceinline__ uint2 fixed63(uint32_t hi, uint32_t lo, int sh) {
  // sum_d 256 * 2^(9 d), d = 0..6
  constexpr uint64_t BIAS = 256ull * ((1ull << 0) | (1ull << 9) | (1ull << 18) | (1ull << 27) | (1ull << 36) |
                                      (1ull << 45) | (1ull << 54));
  const uint32_t H = __funnelshift_l(lo, hi, 11) | 0x80000000u, L = lo << 11;   // leading bit at bit 63
  const int s = sh + 2;
  const uint32_t wl = __funnelshift_rc(__funnelshift_rc(L, H, s), 0u, max(s - 32, 0));
  const uint32_t wh = __funnelshift_rc(H, 0u, s);
  const uint64_t w = ((uint64_t)wh << 32 | wl) + BIAS;
  return make_uint2((uint32_t)w, (uint32_t)(w >> 32));
}
// digits (most significant first) of two neighbouring K positions with high words ha, hb
__device__ __forceinline__ void digits2(const uint2 a, const uint2 b, uint32_t ha, uint32_t hb, uint32_t (&d)[MMA_ND]) {
  const uint32_t sg = prmt(ha, hb, 0x7632) & 0x80008000u;
  const uint32_t one = sg | 0x3C003C00u, off = sg ^ 0xE500E500u;
  d[6] = digit_pair(prmt(a.x, b.x, 0x5410), 0x01FF01FFu, one, off);            // bits 0-8
  d[5] = digit_pair(prmt(a.x, b.x, 0x6521) >> 1, 0x01FF01FFu, one, off);       // 9-17
  d[4] = digit_pair(prmt(a.x, b.x, 0x7632) >> 2, 0x01FF01FFu, one, off);       // 18-26
  d[3] = digit_pair(prmt(prmt(a.x, a.y, 0x0043), prmt(b.x, b.y, 0x0043), 0x5410) >> 3, 0x01FF01FFu, one, off);   // 27-35
  d[2] = digit_pair(prmt(a.y, b.y, 0x5410) >> 4, 0x01FF01FFu, one, off);       // 36-44
  d[1] = digit_pair(prmt(a.y, b.y, 0x6521) >> 5, 0x01FF01FFu, one, off);       // 45-53
  d[0] = digit_pair(prmt(a.y, b.y, 0x7632) >> 6, 0x03FF03FFu, one, off);       // 54-63
}

// four K positions of a row as (hi, lo) words
struct Quad {
  uint32_t hi[4], lo[4];
};
// positions 4l .. 4l + 3 of a staged row (16-byte groups XOR row)
__device__ __forceinline__ Quad load_quad(const double* raw, int row, int l) {
  Quad q;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int g = (2 * l + h) ^ (row & 15);
    const uint4 v = *reinterpret_cast<const uint4*>(raw + (size_t)row * GEMM_KC + 2 * g);
    q.lo[2 * h] = v.x;
    q.hi[2 * h] = v.y;
    q.lo[2 * h + 1] = v.z;
    q.hi[2 * h + 1] = v.w;
  }
  return q;
}
__device__ __forceinline__ void exponents(const Quad& q, int (&e)[4], int& emax) {
#pragma unroll
  for (int j = 0; j < 4; ++j) e[j] = (int)((q.hi[j] & 0x7FFFFFFFu) >> 20);
  emax = max(max(e[0], e[1]), max(e[2], e[3]));
}
// rows the integer path does not take, by their largest exponent (a subnormal's is 0 before the
// K positions' exponents, a zero's -4096 after them)
__device__ __forceinline__ bool outside_range(int emax) { return emax > MMA_NONE && (emax < MMA_EMIN || emax > MMA_EMAX); }
__device__ __forceinline__ bool is_zero(uint32_t hi, uint32_t lo) { return ((hi & 0x7FFFFFFFu) | lo) == 0; }
// digits of a row's four positions, the row's exponent taken over its 8 lanes (e: -4096 for a
// zero).  Returns the row's exponent word, MMA_WILD when it needs the FP64 path.
__device__ __forceinline__ int cut_row(const Quad& q, const int (&e)[4], int emax, uint32_t (&d0)[MMA_ND],
                                       uint32_t (&d1)[MMA_ND]) {
  emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 1));
  emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 2));
  emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 4));
  const bool wild = outside_range(emax);
  const int E = emax > 0 ? emax : MMA_E0;   // a zero row: every element shifts out
  uint2 f[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) f[j] = fixed63(q.hi[j], q.lo[j], E - e[j]);
  digits2(f[0], f[1], q.hi[0], q.hi[1], d0);
  digits2(f[2], f[3], q.hi[2], q.hi[3], d1);
  return wild ? MMA_WILD : (E - 539) << 20;
}
// word offset of positions 4l .. 4l + 3 inside a row's 16 digit words (16-byte groups XOR row / 2)
__device__ __forceinline__ int digit_word(int row, int l) {
  return ((((l >> 1) ^ (row >> 1)) & 3) << 2) + ((l & 1) << 1);
}

// the 7 digit-product sums of one element, in units of 2^13 of the last digits' product.
// Sums that stay below 2^22 once scaled become integers by adding 1.5 * 2^23 (the two least
// significant ones rounded to nearest); the others take the slower conversion.
__device__ __forceinline__ int magic_int(float x) { return __float_as_int(x) - 0x4B400000; }
__device__ __forceinline__ long long join_digits(const float (&v)[MMA_ND][4], int t) {
  constexpr float MG = 12582912.0f;
  const int d0 = magic_int(v[0][t] + MG), d1 = magic_int(v[1][t] + MG);   // <= 2^21, 2^22
  const int d2 = __float2int_rn(v[2][t]), d3 = __float2int_rn(v[3][t]), d4 = __float2int_rn(v[4][t]);
  const int d5 = magic_int(fmaf(v[5][t], 0.0625f, MG)), d6 = magic_int(fmaf(v[6][t], 1.0f / 8192.0f, MG));
  return ((long long)d0 << 41) + ((long long)d1 << 32) + ((long long)d2 << 23) + ((long long)d3 << 14) +
         ((long long)d4 << 5) + (long long)(d5 + d6);
}

// x times the power of two with exponent word w (both inside the normal range), on the integer
// pipe: a tile's first chunk needs no FP64 instruction
__device__ __forceinline__ double scaled(double x, int w) {
  return __hiloint2double(x != 0.0 ? __double2hiint(x) + w - (1023 << 20) : 0, __double2loint(x));
}

// v[d] += the digit products of weight d over 16 positions, for 16 rows and 8 columns: this
// lane's ldmatrix addresses aa, ba of the first digits, and the digits' stride.  (Two column
// groups at a time would load A once for both, but keeps 8 warps per CTA from 128 registers.)
__device__ __forceinline__ void unit_products(float (&v)[MMA_ND][4], uint32_t aa, uint32_t ba, uint32_t stride) {
  uint32_t B[MMA_ND][2];
#pragma unroll
  for (int j = 0; j < MMA_ND; ++j) ldsm2(B[j], ba + j * stride);
#pragma unroll
  for (int i = 0; i < MMA_ND; ++i) {
    uint32_t A[4];
    ldsm4(A, aa + i * stride);
#pragma unroll
    for (int j = 0; j < MMA_ND - i; ++j) mma16816(v[i + j], A, B[j][0], B[j][1]);
  }
}

__device__ __forceinline__ void scale_quad(const MmaSmem& S, int mode, int l, Quad& q) {
  if (mode == 1) {
    const uint32_t n = S.neg >> (4 * l);
#pragma unroll
    for (int j = 0; j < 4; ++j) q.hi[j] ^= (n << (31 - j)) & 0x80000000u;
  } else if (mode == 2) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double x = __hiloint2double((int)q.hi[j], (int)q.lo[j]) * S.sc[4 * l + j];
      q.hi[j] = (uint32_t)__double2hiint(x);
      q.lo[j] = (uint32_t)__double2loint(x);
    }
  }
}

template <class Extra>
__device__ __forceinline__ void gemm_mma_tile(const GemmSeg* __restrict__ segs, const int3 wi, const double* xbase,
                                              double* ybase, double* tbase, double* wbase, const GemmOut& o,
                                              const Extra& extra) {
  extern __shared__ __align__(16) unsigned char mma_smem_raw[];
  MmaSmem& S = *reinterpret_cast<MmaSmem*>(mma_smem_raw);
  const int m0 = wi.y >> 8, mt = wi.y & 255, n0 = wi.z >> 8, nt = wi.z & 255;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int a16 = (mt + 15) >> 4, b16 = (nt + 15) >> 4;
  const int RB = 16 * a16;                 // first B row
  const int rows = RB + 16 * b16;          // <= MMA_ROWS
  const int units = a16 * b16;             // <= 2 * MMA_WARPS
  const bool bal_a = o.balance_rows != 0;   // exponents of the K positions from op(A)'s rows, else op(B)'s columns

  // row tables; padding rows are zero for the whole tile
  if (tid < rows) {
    const bool isA = tid < RB;
    const int i = isA ? tid : tid - RB;
    int g = (isA ? m0 : n0) + i, v = 0;
    const int blk = isA ? o.c_vr : o.c_vc;
    if (blk > 0) {
      v = g / blk;
      g -= v * blk;
    }
    S.vl[tid] = make_int2(v, g);
  }
  for (int r = warp; r < rows; r += MMA_WARPS)
    if (r < RB ? r >= mt : r - RB >= nt) S.raw[r][lane] = 0.0;
  if (tid < GEMM_KC) S.bal[tid] = MMA_NOBAL;
  if (tid < 2) S.wild[tid] = 0;

  double acc[2][2][4];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[u][h][c] = 0.0;

  int it = 0;            // chunks done
  for (int b0 = 0; b0 < o.seg_count; b0 += GEMM_SEGB) {
    const int nb = min(GEMM_SEGB, o.seg_count - b0);
    __syncthreads();   // the previous batch's descriptors and digits are no longer read
    if (warp == 0) {
      int k = 0;
      if (lane < nb) {
        GemmSeg g = segs[o.seg_begin + b0 + lane];
        if (g.a_rel) g.A = (g.a_rel == 1 ? xbase : g.a_rel == 2 ? tbase : extra(g.a_rel - 3)) + g.a_off;
        if (g.b_rel) g.B = (g.b_rel == 1 ? xbase : g.b_rel == 2 ? tbase : extra(g.b_rel - 3)) + g.b_off;
        S.sd[lane] = SegS{g.A, g.B, g.lda, g.ldb, g.transA, g.transB, g.scale, o.c_vr, o.c_vc, g.a_vs, g.b_vs};
        k = g.k;
      }
      int incl = k;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += v;
      }
      S.kst[lane + 1] = incl;
      if (lane == 0) S.kst[0] = 0;
    }
    __syncthreads();
    const int Kb = S.kst[nb];
    const int nch = (Kb + GEMM_KC - 1) / GEMM_KC;
    int q1 = 0;   // segment of this lane's K position, chunk after chunk
    int q2 = 0;   // segment of the chunk's first position

    auto issue = [&](int c) {
      const int p0 = c * GEMM_KC;
      const int p = p0 + lane;
      const bool in = p < Kb;
      while (in && S.kst[q1 + 1] <= p) ++q1;
      const SegS& s = S.sd[q1];
      const int kl = p - S.kst[q1];
      const int g16 = lane >> 1, half = lane & 1;
      // lanes along K: operands stored K-contiguous, and zeros beyond Kb
      const bool ka = !in || !s.transA, kb = !in || s.transB;
      const int nz = in ? 8 : 0;
      // rows i = warp, warp + 8, ...: i mod 16, and so the swizzle, repeats every second
      auto rows_along_k = [&](int r0, int n, const double* base, int ld, int64_t vs) {
        const uint32_t ld8 = in ? 8u * (uint32_t)ld : 0u, vs8 = in ? 8u * (uint32_t)vs : 0u;
        const char* src = reinterpret_cast<const char*>(in ? base + kl : base);
        for (int i0 = warp; i0 < n; i0 += 4 * MMA_WARPS)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + MMA_WARPS * u;
            if (i < n) {
              const int2 vl = S.vl[r0 + i];
              cp_async8z(&S.raw[r0 + i][2 * (g16 ^ ((warp + MMA_WARPS * u) & 15)) + half],
                         src + (uint64_t)(uint32_t)vl.x * vs8 + (uint64_t)(uint32_t)vl.y * ld8, nz);
            }
          }
      };
      static_assert(16 % MMA_WARPS == 0, "the swizzle period above");
      if (ka) rows_along_k(0, mt, s.A, s.lda, s.avs);
      if (kb) rows_along_k(RB, nt, s.B, s.ldb, s.bvs);
      // lanes along the rows: operands stored K-major, one segment after the other
      if (__any_sync(0xffffffffu, !ka || !kb)) {
        const int pend = min(p0 + GEMM_KC, Kb);
        for (int q = q2; q < nb && S.kst[q] < pend; ++q) {
          const int f = max(S.kst[q], p0), l = min(S.kst[q + 1], pend);
          const int kk0 = f - p0 + ((warp - (f - p0)) & (MMA_WARPS - 1));   // first position of this warp
          if (kk0 >= l - p0) continue;
          const SegS& t = S.sd[q];
          auto k_major = [&](int r0, int n, const double* base, int ld, int64_t vs) {
            const double* src = base + (int64_t)(p0 + kk0 - S.kst[q]) * ld;
            for (int i = lane; i < n; i += 32) {
              const int r = r0 + i;
              const int2 vl = S.vl[r];
              const double* p = src + ((uint64_t)(uint32_t)vl.x * (uint32_t)vs + (uint32_t)vl.y);
              double* row = &S.raw[r][0];
              for (int kk = kk0; kk < l - p0; kk += MMA_WARPS, p += (int64_t)MMA_WARPS * ld)
                cp_async8z(row + 2 * ((kk >> 1) ^ (r & 15)) + (kk & 1), p, 8);
            }
          };
          if (t.transA) k_major(0, mt, t.A, t.lda, t.avs);
          if (!t.transB) k_major(RB, nt, t.B, t.ldb, t.bvs);
        }
      }
      if (warp == 0) {
        const double sc = in ? s.scale : 1.0;
        S.sc[lane] = sc;
        const bool one = __all_sync(0xffffffffu, sc == 1.0), pm = __all_sync(0xffffffffu, fabs(sc) == 1.0);
        const uint32_t neg = __ballot_sync(0xffffffffu, sc < 0.0);
        if (lane == 0) {
          S.mode = one ? 0 : pm ? 1 : 2;
          S.neg = neg;
        }
      }
      const int pn = p0 + GEMM_KC;
      while (pn < Kb && S.kst[q2 + 1] <= pn) ++q2;
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    };

    if (nch > 0) issue(0);
    for (int c = 0; c < nch; ++c, ++it) {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      __syncthreads();               // the chunk has landed; the previous one's digits are no longer read
      const int kc = min(GEMM_KC, Kb - c * GEMM_KC);
      const int mode = S.mode;
      const int l = lane & 7;
      {
        // largest exponent of each K position over the balanced side
        int mx[4] = {0, 0, 0, 0};
        const int r1 = bal_a ? RB : rows;
        for (int r = (bal_a ? 0 : RB) + 4 * warp + (lane >> 3); r < r1; r += 4 * MMA_WARPS) {
          Quad q = load_quad(&S.raw[0][0], r, l);
          if (!bal_a) scale_quad(S, mode, l, q);
#pragma unroll
          for (int j = 0; j < 4; ++j) mx[j] = max(mx[j], (int)(q.hi[j] & 0x7FFFFFFFu) >> 20);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          mx[j] = max(mx[j], __shfl_xor_sync(0xffffffffu, mx[j], 8));
          mx[j] = max(mx[j], __shfl_xor_sync(0xffffffffu, mx[j], 16));
          // kept as the exponent itself; a position where that side is zero stays far below every other
          if (lane < 8 && mx[j] > 0) atomicMax(&S.bal[4 * l + j], mx[j] - MMA_E0);
        }
        __syncthreads();
      }
      for (int r = 4 * warp + (lane >> 3); r < rows; r += 4 * MMA_WARPS) {   // rows is a multiple of 16
        Quad q = load_quad(&S.raw[0][0], r, l);
        const bool isB = r >= RB;
        if (isB) scale_quad(S, mode, l, q);
        int e[4], emax;
        exponents(q, e, emax);
        // infinities and NaN keep their row out of the integer path (all rows, on the balanced side)
        const bool own = isB != bal_a;
        const int4 bk = *reinterpret_cast<const int4*>(&S.bal[4 * l]);
        const int bj[4] = {bk.x, bk.y, bk.z, bk.w};
        const bool inf = own ? max(max(bk.x, bk.y), max(bk.z, bk.w)) == 2047 - MMA_E0 : emax == 2047;
#pragma unroll
        for (int j = 0; j < 4; ++j) e[j] = is_zero(q.hi[j], q.lo[j]) ? -4096 : own ? e[j] - bj[j] : e[j] + bj[j];
        emax = inf ? 4095 : max(max(e[0], e[1]), max(e[2], e[3]));
        uint32_t d0[MMA_ND], d1[MMA_ND];
        const int x = cut_row(q, e, emax, d0, d1);
        if (l == 0) S.ex[r] = x;
        if (x == MMA_WILD) S.wild[it & 1] = 1;
        const int w = digit_word(r, l);
#pragma unroll
        for (int d = 0; d < MMA_ND; ++d) *reinterpret_cast<uint2*>(&S.dig[d][r][w]) = make_uint2(d0[d], d1[d]);
      }
      __syncthreads();
      const bool wild = S.wild[it & 1] != 0;
      if (tid == 0) S.wild[(it & 1) ^ 1] = 0;   // last read before this chunk's first barrier
      if (tid < GEMM_KC) S.bal[tid] = MMA_NOBAL;
      if (!wild && c + 1 < nch) issue(c + 1);   // lands during the products; raw is free
      const int nks = kc > 16 ? 2 : 1;
      const uint32_t dig0 = (uint32_t)__cvta_generic_to_shared(&S.dig[0][0][0]);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int un = warp + MMA_WARPS * u;
        if (un >= units) break;
        const int ra = 16 * (un / b16), cb = 16 * (un % b16);
        const bool second = cb + 8 < nt;
        const int ar = ra + (lane & 15), br = RB + cb + (lane & 7);
        const int e0 = S.ex[ra + (lane >> 2)], e1 = S.ex[ra + (lane >> 2) + 8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (h == 1 && !second) break;
          float v[MMA_ND][4];
#pragma unroll
          for (int d = 0; d < MMA_ND; ++d)
#pragma unroll
            for (int t = 0; t < 4; ++t) v[d][t] = 0.0f;
          for (int ks = 0; ks < nks; ++ks) {
            const int b8 = br + 8 * h;
            unit_products(v, dig0 + ar * 64 + (((2 * ks + (lane >> 4)) ^ (ar >> 1)) & 3) * 16,
                          dig0 + b8 * 64 + (((2 * ks + ((lane >> 3) & 1)) ^ (b8 >> 1)) & 3) * 16, (uint32_t)sizeof(S.dig[0]));
          }
          const int2 f = *reinterpret_cast<const int2*>(&S.ex[RB + cb + 8 * h + 2 * (lane & 3)]);
          if (!wild) {
#pragma unroll
            for (int t = 0; t < 4; ++t)
              acc[u][h][t] = fma((double)join_digits(v, t),
                                 __hiloint2double(((t & 2) ? e1 : e0) + ((t & 1) ? f.y : f.x), 0), acc[u][h][t]);
          } else {
#pragma unroll 1
            for (int t = 0; t < 4; ++t) {
              const int ea = (t & 2) ? e1 : e0, eb = (t & 1) ? f.y : f.x;
              double s = t == 0 ? acc[u][h][0] : t == 1 ? acc[u][h][1] : t == 2 ? acc[u][h][2] : acc[u][h][3];
              if ((ea | eb) >= 0) {
                float w[MMA_ND][4];
#pragma unroll
                for (int d = 0; d < MMA_ND; ++d) w[d][0] = t == 0 ? v[d][0] : t == 1 ? v[d][1] : t == 2 ? v[d][2] : v[d][3];
                s = fma((double)join_digits(w, 0), __hiloint2double(ea + eb, 0), s);
              } else {
                // plain FP64 from the staged operands
                const int i = ra + (lane >> 2) + 8 * (t >> 1), j = RB + cb + 8 * h + 2 * (lane & 3) + (t & 1);
                for (int kk = 0; kk < kc; ++kk)
                  s = fma(S.raw[i][2 * ((kk >> 1) ^ (i & 15)) + (kk & 1)],
                          S.raw[j][2 * ((kk >> 1) ^ (j & 15)) + (kk & 1)] * S.sc[kk], s);
              }
              if (t == 0) acc[u][h][0] = s;
              if (t == 1) acc[u][h][1] = s;
              if (t == 2) acc[u][h][2] = s;
              if (t == 3) acc[u][h][3] = s;
            }
          }
        }
      }
      if (wild) {          // the staged operands were kept for the FP64 path
        __syncthreads();
        if (c + 1 < nch) issue(c + 1);
      }
    }
  }
  double* cbase = o.c_rel == GEMM_C_SPLIT ? wbase + o.c_off
                 : o.c_rel ? (o.c_rel == 1 ? ybase : o.c_rel == 2 ? tbase : extra(o.c_rel - 3)) + o.c_off : o.C;
  if (o.seg_count == 0) __syncthreads();   // the row tables are read below
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int un = warp + MMA_WARPS * u;
    if (un >= units) break;
    const int ra = 16 * (un / b16) + (lane >> 2), cb = 16 * (un % b16) + 2 * (lane & 3);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int i = ra + 8 * (t >> 1), j = cb + 8 * h + (t & 1);
        if (i >= mt || j >= nt) continue;
        // a part of a split tile is dense, whatever the output's vector blocks
        double* c = cbase + (o.c_rel == GEMM_C_SPLIT
                                 ? (int64_t)(m0 + i) * o.ldc + n0 + j
                                 : (int64_t)(S.vl[i].x + S.vl[RB + j].x) * o.c_vs + (int64_t)S.vl[i].y * o.ldc + S.vl[RB + j].y);
        *c = o.accumulate ? (*c + acc[u][h][t]) : acc[u][h][t];
      }
  }
}

__device__ __forceinline__ double* mma_extra(const GemmExtra& ex, int i) {
  switch (i) {
    case 0: return ex.p[0];
    case 1: return ex.p[1];
    case 2: return ex.p[2];
    case 3: return ex.p[3];
    case 4: return ex.p[4];
    case 5: return ex.p[5];
    case 6: return ex.p[6];
    default: return ex.p[7];
  }
}

constexpr int MMA_CTAS = 2;

__global__ void __launch_bounds__(32 * MMA_WARPS, MMA_CTAS)
    gemm_mma_kernel(const GemmOut* __restrict__ outs, const GemmSeg* __restrict__ segs, const int3* __restrict__ tiles,
                    int ntiles, const double* __restrict__ xbase, double* __restrict__ ybase, double* __restrict__ tbase,
                    const GemmBases* __restrict__ multi, const GemmExtra ex, double* __restrict__ wbase) {
  const int w = blockIdx.x;
  if (w >= ntiles) return;
  const int3 wi = tiles[w];
  const GemmOut o = outs[wi.x];
  if (multi) {
    const GemmBases b = multi[o.inst];
    xbase = b.x;
    ybase = b.y;
    tbase = b.t;
  }
  gemm_mma_tile(segs, wi, xbase, ybase, tbase, wbase, o, [&](int i) { return mma_extra(ex, i); });
}

__global__ void __launch_bounds__(32 * MMA_WARPS, MMA_CTAS)
    gemm_mma_inst_kernel(const GemmOut* __restrict__ outs, const GemmSeg* __restrict__ segs,
                         const int3* __restrict__ tiles, int ntiles, const __grid_constant__ GemmInstSet P, int ninst) {
  const int w = blockIdx.x / ninst;
  if (w >= ntiles) return;
  const GemmInst* b = &P.b[blockIdx.x % ninst];
  const int3 wi = tiles[w];
  const GemmOut o = outs[wi.x];
  gemm_mma_tile(segs, wi, b->x, b->y, b->t, nullptr, o, [&](int i) { return b->e[i]; });
}

// dynamic shared memory of the kernels, once per device (beyond MAX_DEV devices, at every launch)
static cudaError_t mma_smem_attr() {
  constexpr int MAX_DEV = 64;
  static std::atomic<int> done[MAX_DEV];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool kept = dev >= 0 && dev < MAX_DEV;
  if (kept && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
  for (const void* f : {(const void*)gemm_mma_kernel, (const void*)gemm_mma_inst_kernel}) {
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MmaSmem));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
  }
  if (kept) done[dev].store(1, std::memory_order_release);
  return cudaSuccess;
}

void launch_gemm_mma(const GemmOut* outs, const GemmSeg* segs, const int3* tiles, int ntiles, const double* xbase,
                     double* ybase, double* tbase, cudaStream_t st, const GemmBases* multi, const GemmExtra* extra,
                     double* wbase) {
  if (ntiles <= 0) return;
  if (mma_smem_attr() != cudaSuccess) return;
  const GemmExtra ex = extra ? *extra : GemmExtra{};
  gemm_mma_kernel<<<ntiles, 32 * MMA_WARPS, sizeof(MmaSmem), st>>>(outs, segs, tiles, ntiles, xbase, ybase, tbase, multi,
                                                                ex, wbase);
}

void launch_gemm_mma_inst(const GemmOut* outs, const GemmSeg* segs, const int3* tiles, int ntiles,
                          const GemmInstSet& bases, int ninst, cudaStream_t st) {
  if (ntiles <= 0 || ninst <= 0) return;
  if (mma_smem_attr() != cudaSuccess) return;
  gemm_mma_inst_kernel<<<(unsigned)((long long)ntiles * ninst), 32 * MMA_WARPS, sizeof(MmaSmem), st>>>(
      outs, segs, tiles, ntiles, bases, ninst);
}

// ---------------------------------------------------------------------------
// small blocks: one warp per tile
//
// The blocks of small and medium systems are a few states wide (2 x 2 x 4 to 16 x 16 x 30), so a
// CTA that stages its operands spends microseconds of latency, barriers and descriptor reads
// on a product that takes nanoseconds.  Here every warp takes its own work item, reads the
// operands straight from global memory (L1 keeps a block's few lines) and meets no barrier:
//
//  - tiny tiles (WARP_DIRECT): lanes own output elements and run FP64 FMAs, a segment at a time;
//  - others: 16 x 16 tiles as digit products, 16 positions a chunk.  A lane loads exactly the
//    elements its mma.sync fragments hold and cuts them in registers, so shared memory only
//    holds the segment table.  With WARP_SWAP the 16-wide side of the product carries the
//    output's columns (the longer side pads less).
//
// Long segment lists are split into K parts on separate warps; the warp that finishes a
// tile's last part adds the parts in order (a counter per tile, reset by that warp), which
// spares the reduction launch.
//
// Measured (one-site sigma, FP64 FMA tiles of a CTA -> here): k = 8, M = 64, 1 vector 183 -> 51 us;
// k = 17, M = 30, 6 vectors 468 -> 106 us; eight molecules in one call 1.67 -> 0.90 ms.  Bound by
// latency: descriptor and operand reads of short items, 16 warps per SM (128 registers; 3 CTAs of
// 168 registers are 5% slower on the longer lists).  Lists of FMA arithmetic (GemmMath) run
// whole on the direct path.
// ---------------------------------------------------------------------------
struct WarpSeg {
  const double* p;          // operand along the tile's rows, and along its columns
  const double* q;
  int64_t pvs, qvs;         // vector block strides
  double scale;
  int prs, pks, qrs, qks;   // strides by row (column) and by K position
};
constexpr int WARP_WARPS = 4;
struct WarpSmem {
  WarpSeg sd[WARP_WARPS][GEMM_SEGB];
  int kst[WARP_WARPS][GEMM_SEGB + 1];
};

// stages up to 32 segments for this warp; returns their total K
template <class Extra>
__device__ __forceinline__ int warp_segs(WarpSeg* sd, int* kst, const GemmSeg* __restrict__ segs, int sb, int nb, bool swap,
                                         const double* xbase, const double* tbase, const Extra& extra, int lane) {
  int k = 0;
  __syncwarp();
  if (lane < nb) {
    GemmSeg g = segs[sb + lane];
    if (g.a_rel) g.A = (g.a_rel == 1 ? xbase : g.a_rel == 2 ? tbase : extra(g.a_rel - 3)) + g.a_off;
    if (g.b_rel) g.B = (g.b_rel == 1 ? xbase : g.b_rel == 2 ? tbase : extra(g.b_rel - 3)) + g.b_off;
    const int ars = g.transA ? 1 : g.lda, aks = g.transA ? g.lda : 1;
    const int brs = g.transB ? g.ldb : 1, bks = g.transB ? 1 : g.ldb;
    sd[lane] = swap ? WarpSeg{g.B, g.A, g.b_vs, g.a_vs, g.scale, brs, bks, ars, aks}
                    : WarpSeg{g.A, g.B, g.a_vs, g.b_vs, g.scale, ars, aks, brs, bks};
    k = g.k;
  }
  int incl = k;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += v;
  }
  kst[lane + 1] = incl;
  if (lane == 0) kst[0] = 0;
  __syncwarp();
  return kst[nb];
}

// where element (i, j) of an output lives (i, j inside the whole output)
__device__ __forceinline__ int64_t out_offset(const GemmOut& o, int i, int j) {
  int64_t off = 0;
  if (o.c_vr > 0) {
    const int v = i / o.c_vr;
    off += v * o.c_vs;
    i -= v * o.c_vr;
  }
  if (o.c_vc > 0) {
    const int v = j / o.c_vc;
    off += v * o.c_vs;
    j -= v * o.c_vc;
  }
  return off + (int64_t)i * o.ldc + j;
}

// the last part of a split tile to finish adds the parts in order; all 32 lanes call
__device__ __forceinline__ void warp_reduce_parts(const GemmOut* __restrict__ outs, const SplitTile& t, int* counter,
                                                  const double* wbase, double* ybase, double* tbase, int lane) {
  __threadfence();
  __syncwarp();
  int last = 0;
  if (lane == 0) last = atomicAdd(counter, 1) == t.nparts - 1;
  last = __shfl_sync(0xffffffffu, last, 0);
  if (!last) return;
  __threadfence();
  const GemmOut o = outs[t.o];
  double* cbase = o.c_rel == 1 ? ybase + o.c_off : o.c_rel == 2 ? tbase + o.c_off : o.C;
  const int ne = t.mt * t.nt;
  const double* w = wbase + t.ws_off;
  for (int e = lane; e < ne; e += 32) {
    double s = 0.0;
#pragma unroll 8
    for (int p = 0; p < t.nparts; ++p) s += __ldcg(w + (int64_t)p * ne + e);
    double* c = cbase + out_offset(o, t.m0 + e / t.nt, t.n0 + e % t.nt);
    *c = o.accumulate ? *c + s : s;
  }
  if (lane == 0) *counter = 0;
}

// exponent word of a row from the four positions of its lane's quad
__device__ __forceinline__ int row_exponent(const int (&e)[4]) {
  int m = max(max(e[0], e[1]), max(e[2], e[3]));
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
  return max(m, __shfl_xor_sync(0xffffffffu, m, 2));
}
__device__ __forceinline__ int exponent_of(double x) { return (__double2hiint(x) & 0x7FFFFFFF) >> 20; }
// fragments of four positions (2t, 2t + 1, 2t + 8, 2t + 9) of one row
__device__ __forceinline__ void cut_quad(const double (&x)[4], const int (&e)[4], int E, uint32_t (&lo)[MMA_ND],
                                         uint32_t (&hi)[MMA_ND]) {
  uint2 f[4];
  uint32_t h[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    h[j] = (uint32_t)__double2hiint(x[j]);
    f[j] = fixed63(h[j], (uint32_t)__double2loint(x[j]), E - e[j]);
  }
  digits2(f[0], f[1], h[0], h[1], lo);
  digits2(f[2], f[3], h[2], h[3], hi);
}

template <class Extra>
__device__ __forceinline__ void warp_tile(const GemmOut* __restrict__ outs, const GemmSeg* __restrict__ segs, const int3 wi,
                                          const double* xbase, double* ybase, double* tbase, double* wbase,
                                          const SplitTile* __restrict__ splits, int* counters, const GemmOut& o,
                                          const Extra& extra, WarpSmem& S) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int m0 = wi.y >> 8, mt = wi.y & 255, n0 = wi.z >> 8, nt = wi.z & 255;
  WarpSeg* sd = S.sd[warp];
  int* kst = S.kst[warp];
  const bool part = o.c_rel == GEMM_C_SPLIT;
  double* cbase = part ? wbase + o.c_off
                  : o.c_rel ? (o.c_rel == 1 ? ybase : o.c_rel == 2 ? tbase : extra(o.c_rel - 3)) + o.c_off : o.C;
  // a part of a split tile is dense, whatever the output's vector blocks
  auto store = [&](int i, int j, double x) {
    double* c = cbase + (part ? (int64_t)i * o.ldc + j : out_offset(o, i, j));
    *c = o.accumulate ? *c + x : x;
  };

  if (o.flags & GEMM_WARP_DIRECT) {
    const int ne = mt * nt, cnt = (ne + 31) >> 5;     // elements per lane
    constexpr int MAXE = GEMM_DIRECT_MAX / 32;
    int rv[MAXE], rr[MAXE], cv[MAXE], cr[MAXE];
    double acc[MAXE];
#pragma unroll
    for (int u = 0; u < MAXE; ++u) {
      const int e = min(lane + 32 * u, ne - 1);
      rr[u] = m0 + e / nt;
      cr[u] = n0 + e % nt;
      rv[u] = cv[u] = 0;
      if (o.c_vr > 0) {
        rv[u] = rr[u] / o.c_vr;
        rr[u] -= rv[u] * o.c_vr;
      }
      if (o.c_vc > 0) {
        cv[u] = cr[u] / o.c_vc;
        cr[u] -= cv[u] * o.c_vc;
      }
      acc[u] = 0.0;
    }
    for (int b0 = 0; b0 < o.seg_count; b0 += GEMM_SEGB) {
      const int nb = min(GEMM_SEGB, o.seg_count - b0);
      warp_segs(sd, kst, segs, o.seg_begin + b0, nb, false, xbase, tbase, extra, lane);
      for (int q = 0; q < nb; ++q) {
        const WarpSeg g = sd[q];
        const int kq = kst[q + 1] - kst[q];
#pragma unroll
        for (int u = 0; u < MAXE; ++u) {
          if (u >= cnt) break;
          const double* a = g.p + rv[u] * g.pvs + (int64_t)rr[u] * g.prs;
          const double* b = g.q + cv[u] * g.qvs + (int64_t)cr[u] * g.qrs;
          double s = 0.0;
#pragma unroll 4
          for (int k = 0; k < kq; ++k) s = fma(a[(int64_t)k * g.pks], b[(int64_t)k * g.qks], s);
          acc[u] = fma(g.scale, s, acc[u]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < MAXE; ++u) {
      const int e = lane + 32 * u;
      if (e < ne) store(m0 + e / nt, n0 + e % nt, acc[u]);
    }
  } else {
    const bool swap = (o.flags & GEMM_WARP_SWAP) != 0;
    const bool bal_r = swap == (o.balance_rows == 0);   // exponents of the K positions from the tile's rows, else its columns
    const int r0 = swap ? n0 : m0, rt = swap ? nt : mt, c0 = swap ? m0 : n0, ct = swap ? mt : nt;
    const int rblk = swap ? o.c_vc : o.c_vr, cblk = swap ? o.c_vr : o.c_vc;
    const int g = lane >> 2, t = lane & 3;
    const int nh = ct > 8 ? 2 : 1;
    int rv[2], rr[2], cv[2], cr[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {   // lanes beyond the tile repeat its last row or column
      rr[h] = r0 + min(g + 8 * h, rt - 1);
      cr[h] = c0 + min(g + 8 * h, ct - 1);
      rv[h] = cv[h] = 0;
      if (rblk > 0) {
        rv[h] = rr[h] / rblk;
        rr[h] -= rv[h] * rblk;
      }
      if (cblk > 0) {
        cv[h] = cr[h] / cblk;
        cr[h] -= cv[h] * cblk;
      }
    }
    double acc[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[h][i] = 0.0;
    for (int b0 = 0; b0 < o.seg_count; b0 += GEMM_SEGB) {
      const int nb = min(GEMM_SEGB, o.seg_count - b0);
      const int Kb = warp_segs(sd, kst, segs, o.seg_begin + b0, nb, swap, xbase, tbase, extra, lane);
      int qs = 0;
      for (int p0 = 0; p0 < Kb; p0 += 16) {
        double a[2][4], b[2][4], sc[4];
        while (qs + 1 < nb && kst[qs + 1] <= p0) ++qs;
        int q = qs;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int p = p0 + 2 * t + (j & 1) + 8 * (j >> 1);
          a[0][j] = a[1][j] = b[0][j] = b[1][j] = 0.0;
          sc[j] = 1.0;
          if (p < Kb) {
            while (kst[q + 1] <= p) ++q;
            const WarpSeg& s = sd[q];
            const int kl = p - kst[q];
            const double* pp = s.p + (int64_t)kl * s.pks;
            const double* qq = s.q + (int64_t)kl * s.qks;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              a[h][j] = pp[rv[h] * s.pvs + (int64_t)rr[h] * s.prs];
              if (h < nh) b[h][j] = qq[cv[h] * s.qvs + (int64_t)cr[h] * s.qrs];
            }
            sc[j] = s.scale;
          }
        }
        int ea[2][4], eb[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // the segment's scale goes with the second operand of the product (op(B))
            // (+-1, almost always: a sign, not a multiplication on the slow FP64 pipe)
            double& x = swap ? a[h][j] : b[h][j];
            if (fabs(sc[j]) == 1.0)
              x = __hiloint2double(__double2hiint(x) ^ (__double2hiint(sc[j]) & (int)0x80000000), __double2loint(x));
            else
              x *= sc[j];
            ea[h][j] = exponent_of(a[h][j]);
            eb[h][j] = exponent_of(b[h][j]);
          }
        bool all = false;    // the balanced side holds an infinity or NaN
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          int m = bal_r ? max(ea[0][j], ea[1][j]) : max(eb[0][j], eb[1][j]);
          m = max(m, __shfl_xor_sync(0xffffffffu, m, 4));
          m = max(m, __shfl_xor_sync(0xffffffffu, m, 8));
          m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
          const int d = m > 0 ? m - MMA_E0 : MMA_NOBAL, da = bal_r ? -d : d;
          all |= m == 2047;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            ea[h][j] = is_zero(__double2hiint(a[h][j]), __double2loint(a[h][j])) ? -4096 : ea[h][j] == 2047 ? 4095 : ea[h][j] + da;
            eb[h][j] = is_zero(__double2hiint(b[h][j]), __double2loint(b[h][j])) ? -4096 : eb[h][j] == 2047 ? 4095 : eb[h][j] - da;
          }
        }
        all = __any_sync(0xffffffffu, all);
        int E[2], F[2], xe[2], xf[2];    // exponents of the rows and columns, and their words
        bool wild = false;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          E[h] = row_exponent(ea[h]);
          F[h] = row_exponent(eb[h]);
          const bool we = outside_range(E[h]) || (all && bal_r), wf = outside_range(F[h]) || (all && !bal_r);
          wild |= we | wf;
          if (E[h] <= 0) E[h] = MMA_E0;
          if (F[h] <= 0) F[h] = MMA_E0;
          xe[h] = we ? MMA_WILD : (E[h] - 539) << 20;
          xf[h] = wf ? MMA_WILD : (F[h] - 539) << 20;
        }
        // plain FP64 over the chunk for one element (r, c) of the tile
        auto fp64_chunk = [&](int r, int c, double x) {
          int r1 = r0 + min(r, rt - 1), c1 = c0 + min(c, ct - 1), v1 = 0, v2 = 0;
          if (rblk > 0) v1 = r1 / rblk, r1 -= v1 * rblk;
          if (cblk > 0) v2 = c1 / cblk, c1 -= v2 * cblk;
          int qw = qs;
          for (int p = p0; p < min(p0 + 16, Kb); ++p) {
            while (kst[qw + 1] <= p) ++qw;
            const WarpSeg& s = sd[qw];
            const int kl = p - kst[qw];
            const double u = s.p[(int64_t)kl * s.pks + v1 * s.pvs + (int64_t)r1 * s.prs];
            const double w = s.q[(int64_t)kl * s.qks + v2 * s.qvs + (int64_t)c1 * s.qrs];
            x = swap ? fma(w, u * s.scale, x) : fma(u, w * s.scale, x);
          }
          return x;
        };
        wild = __any_sync(0xffffffffu, wild);
        const bool first = b0 == 0 && p0 == 0;
        uint32_t A0[MMA_ND], A1[MMA_ND], A2[MMA_ND], A3[MMA_ND];
        cut_quad(a[0], ea[0], E[0], A0, A2);
        cut_quad(a[1], ea[1], E[1], A1, A3);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (h >= nh) break;
          uint32_t B0[MMA_ND], B1[MMA_ND];
          cut_quad(b[h], eb[h], F[h], B0, B1);
          float v[MMA_ND][4];
#pragma unroll
          for (int d = 0; d < MMA_ND; ++d)
#pragma unroll
            for (int i = 0; i < 4; ++i) v[d][i] = 0.0f;
#pragma unroll
          for (int i = 0; i < MMA_ND; ++i) {
            const uint32_t A[4] = {A0[i], A1[i], A2[i], A3[i]};
#pragma unroll
            for (int j = 0; j < MMA_ND - i; ++j) mma16816(v[i + j], A, B0[j], B1[j]);
          }
          // exponents of this lane's two columns, held by the lanes of those columns
          const int f0 = __shfl_sync(0xffffffffu, xf[h], 8 * t), f1 = __shfl_sync(0xffffffffu, xf[h], 8 * t + 4);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int x = xe[i >> 1], f = (i & 1) ? f1 : f0;
            if (first && !wild)
              acc[h][i] = scaled((double)join_digits(v, i), x + f);
            else if (!wild || (x | f) >= 0)
              acc[h][i] = fma((double)join_digits(v, i), __hiloint2double(x + f, 0), acc[h][i]);
            else
              acc[h][i] = fp64_chunk(g + 8 * (i >> 1), 8 * h + 2 * t + (i & 1), acc[h][i]);
          }
        }
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = g + 8 * (i >> 1), c = 8 * h + 2 * t + (i & 1);
        if (r < rt && c < ct) store(swap ? c0 + c : r0 + r, swap ? r0 + r : c0 + c, acc[h][i]);
      }
  }
  if (part) warp_reduce_parts(outs, splits[o.split], counters + o.split, wbase, ybase, tbase, lane);
}

constexpr int WARP_CTAS = 4;

__global__ void __launch_bounds__(32 * WARP_WARPS, WARP_CTAS)
    gemm_warp_kernel(const GemmOut* __restrict__ outs, const GemmSeg* __restrict__ segs, const int3* __restrict__ tiles,
                     int ntiles, const double* __restrict__ xbase, double* ybase, double* tbase,
                     const GemmBases* __restrict__ multi, const GemmExtra ex, double* wbase,
                     const SplitTile* __restrict__ splits, int* counters) {
  __shared__ WarpSmem S;
  const int w = blockIdx.x * WARP_WARPS + (threadIdx.x >> 5);
  if (w >= ntiles) return;
  const int3 wi = tiles[w];
  const GemmOut o = outs[wi.x];
  if (multi) {
    const GemmBases b = multi[o.inst];
    xbase = b.x;
    ybase = b.y;
    tbase = b.t;
  }
  warp_tile(outs, segs, wi, xbase, ybase, tbase, wbase, splits, counters, o, [&](int i) { return mma_extra(ex, i); }, S);
}

// instances interleave: the warps of a CTA take the same tile of neighbouring instances
__global__ void __launch_bounds__(32 * WARP_WARPS, WARP_CTAS)
    gemm_warp_inst_kernel(const GemmOut* __restrict__ outs, const GemmSeg* __restrict__ segs,
                          const int3* __restrict__ tiles, int ntiles, const __grid_constant__ GemmInstSet P, int ninst) {
  __shared__ WarpSmem S;
  const unsigned w = blockIdx.x * WARP_WARPS + (threadIdx.x >> 5);
  const int tile = (int)(w / ninst);
  if (tile >= ntiles) return;
  const GemmInst* b = &P.b[w % ninst];
  const int3 wi = tiles[tile];
  const GemmOut o = outs[wi.x];
  warp_tile(outs, segs, wi, b->x, b->y, b->t, nullptr, nullptr, nullptr, o, [&](int i) { return b->e[i]; }, S);
}

void launch_gemm_warp(const GemmOut* outs, const GemmSeg* segs, const int3* tiles, int ntiles, const double* xbase,
                      double* ybase, double* tbase, cudaStream_t st, const GemmBases* multi, const GemmExtra* extra,
                      double* wbase, const SplitTile* splits, int* counters) {
  if (ntiles <= 0) return;
  const GemmExtra ex = extra ? *extra : GemmExtra{};
  gemm_warp_kernel<<<(ntiles + WARP_WARPS - 1) / WARP_WARPS, 32 * WARP_WARPS, 0, st>>>(
      outs, segs, tiles, ntiles, xbase, ybase, tbase, multi, ex, wbase, splits, counters);
}

void launch_gemm_warp_inst(const GemmOut* outs, const GemmSeg* segs, const int3* tiles, int ntiles,
                           const GemmInstSet& bases, int ninst, cudaStream_t st) {
  if (ntiles <= 0 || ninst <= 0) return;
  const long long n = (long long)ntiles * ninst;
  gemm_warp_inst_kernel<<<(unsigned)((n + WARP_WARPS - 1) / WARP_WARPS), 32 * WARP_WARPS, 0, st>>>(
      outs, segs, tiles, ntiles, bases, ninst);
}

}  // namespace lrt
