// FP64 kernels of the sigma / renormalization path.
//
//  gather:    scaled, optionally transposed block copies summed into destination
//             sub-blocks (building enlarged-block operators, the "x h_i" of
//             Eq. lopr1st); 32x32 tiles, source descriptors staged in shared memory.
//  gemm_fp64: grouped GEMM whose output tiles each loop over a list of
//             (A, B, scale) products (K-concatenation), so all contributions to
//             one output block are summed in registers without atomics.
//  diag:      outer products of operator diagonals (preconditioner of Eq. error).
#include "lrt_kernels.h"
#include "lrt_fp64_tile.h"

#include <algorithm>
#include <atomic>

namespace lrt {

// ---------------------------------------------------------------------------
// gather
// ---------------------------------------------------------------------------
// The sources of a task (a dozen on average for an enlarged operator set, most of them
// blocks of a few tens of rows) are staged as descriptors in shared memory, and their
// loads are unrolled so that several are in flight: a tile costs a few memory round trips
// instead of two per source.  Transposed sources are read straight from global memory;
// the CTA's reads of one source block stay in L1.
// A work item is a chunk of GATHER_CHUNK consecutive elements of the task's row-major
// destination (thread t owns elements t, t + 256, ...): blocks only a few columns wide
// still fill every lane, where square 32 x 32 tiles left most of them idle.  Each
// element sums its sources in the order they are listed.
constexpr int GATHER_SRC_STAGE = 64;
constexpr int GATHER_PER_THREAD = GATHER_CHUNK / 256;

__device__ __forceinline__ void gather_item(const GatherTask* __restrict__ tasks, const GatherSrc* __restrict__ srcs,
                                            const int3 wi, double* dbase, const double* sbase1,
                                            const double* sbase2, GatherSrc* sd) {
  GatherTask t = tasks[wi.x];
  if (dbase) t.dst = dbase + t.dst_off;
  const int tid = threadIdx.x;
  const int64_t n = (int64_t)t.rows * t.cols;
  const int64_t e0 = (int64_t)wi.y * GATHER_CHUNK + tid;
  int rr[GATHER_PER_THREAD], cc[GATHER_PER_THREAD];
  double acc[GATHER_PER_THREAD];
#pragma unroll
  for (int i = 0; i < GATHER_PER_THREAD; ++i) {
    const int64_t e = e0 + 256 * i;
    rr[i] = e < n ? (int)(e / t.cols) : -1;
    cc[i] = e < n ? (int)(e - (int64_t)rr[i] * t.cols) : 0;
    acc[i] = 0.0;
  }
  for (int s0 = 0; s0 < t.src_count; s0 += GATHER_SRC_STAGE) {
    const int ns = min(GATHER_SRC_STAGE, t.src_count - s0);
    __syncthreads();   // the previous descriptors are no longer read
    if (tid < ns) {
      GatherSrc g = srcs[t.src_begin + s0 + tid];
      if (g.rel) g.src = (g.rel == 1 ? sbase1 : sbase2) + g.src_off;
      sd[tid] = g;
    }
    __syncthreads();
#pragma unroll 4
    for (int s = 0; s < ns; ++s) {
      const double* src = sd[s].src;
      const int64_t ld = sd[s].ld;
      const double sc = sd[s].scale;
      const bool tr = sd[s].trans != 0;
#pragma unroll
      for (int i = 0; i < GATHER_PER_THREAD; ++i)
        if (rr[i] >= 0) acc[i] += sc * (tr ? src[(int64_t)cc[i] * ld + rr[i]] : src[(int64_t)rr[i] * ld + cc[i]]);
    }
  }
#pragma unroll
  for (int i = 0; i < GATHER_PER_THREAD; ++i)
    if (rr[i] >= 0) t.dst[(int64_t)rr[i] * t.ld_dst + cc[i]] += acc[i];
}

__global__ void __launch_bounds__(256) gather_kernel(const GatherTask* __restrict__ tasks,
                                                     const GatherSrc* __restrict__ srcs,
                                                     const int3* __restrict__ tiles, int ntiles,
                                                     double* __restrict__ dbase,
                                                     const double* __restrict__ sbase1,
                                                     const double* __restrict__ sbase2) {
  __shared__ GatherSrc sd[GATHER_SRC_STAGE];
  if ((int)blockIdx.x >= ntiles) return;
  gather_item(tasks, srcs, tiles[blockIdx.x], dbase, sbase1, sbase2, sd);
}

__global__ void __launch_bounds__(256) gather_inst_kernel(const GatherTask* __restrict__ tasks,
                                                          const GatherSrc* __restrict__ srcs,
                                                          const int3* __restrict__ tiles, int ntiles,
                                                          const __grid_constant__ GatherInstSet P, int ninst) {
  __shared__ GatherSrc sd[GATHER_SRC_STAGE];
  const int w = blockIdx.x / ninst;
  if (w >= ntiles) return;
  const GatherBases* b = &P.b[blockIdx.x % ninst];
  gather_item(tasks, srcs, tiles[w], b->d, b->s1, b->s2, sd);
}

void launch_gather(const GatherTask* tasks, const GatherSrc* srcs, const int3* tiles, int ntiles,
                   cudaStream_t st, double* dbase, const double* sbase1, const double* sbase2) {
  if (ntiles <= 0) return;
  gather_kernel<<<ntiles, 256, 0, st>>>(tasks, srcs, tiles, ntiles, dbase, sbase1, sbase2);
}

void launch_gather_inst(const GatherTask* tasks, const GatherSrc* srcs, const int3* tiles, int ntiles,
                        const GatherInstSet& bases, int ninst, cudaStream_t st) {
  // the caller checks 1 <= ninst <= 64 and ntiles * ninst < 2^31
  if (ntiles <= 0 || ninst <= 0) return;
  gather_inst_kernel<<<(unsigned)((long long)ntiles * ninst), 256, 0, st>>>(tasks, srcs, tiles, ntiles, bases, ninst);
}

// ---------------------------------------------------------------------------
// enlargement
//
// A sub-block of an enlarged operator sums up to a few hundred scaled source blocks (the
// complementary operators of a cut combine every pair operator).  A host list of those sources
// has millions of entries, one per sector, and took 50 ms to write and upload for a 1.5 ms
// gather; the references that generate it do not depend on the sector.  So a warp takes up to
// ENL_CHUNK elements of a sub-block, its lanes look up 32 references at a time (does the
// reference have a block between these sectors, where, with which sign), and all lanes then
// sum the blocks found, in reference order.  Sub-blocks of 16 elements and fewer spread the
// references over the idle lanes.  One two-site sweep position at k = 12, M = 128: 92.7 -> 17.2 ms
// (host list, upload and gather before; the rest is the sigma plan), TDA on PPP M = 128 240 ->
// 153 ms.  Bound by the FP64 pipe (one FMA per source element) when the
// blocks are large, by the reference reads when they are small.
// ---------------------------------------------------------------------------
constexpr int ENL_WARPS = 8;
struct EnlSrc {
  const double* p;
  int rs, cs;          // strides of the block's rows and columns
  double scale;
};
struct EnlSmem {
  EnlSrc s[ENL_WARPS][32];
};

__device__ __forceinline__ void enlarge_item(const EnlTables& t, const int3 wi, double* __restrict__ d,
                                             const double* __restrict__ x, const double* __restrict__ xrev, EnlSrc* S) {
  const int lane = threadIdx.x & 31;
  const int o = wi.x, fk = wi.y >> 4, n1 = (wi.y >> 2) & 3, n0 = wi.y & 3;
  const int fb = t.ebra[o * t.nse + fk];
  const int ke = t.fsub[4 * fk + n0], be = t.fsub[4 * fb + n1];
  const int rows = t.xdim[be], cols = t.xdim[ke], n = rows * cols;
  const int odd1 = (n1 == 1) | (n1 == 2), odd0 = (n0 == 1) | (n0 == 2);
  // the sign that comes with an odd operator of X (site on the left) or with the site's own
  const bool neg_odd = t.right && odd0, neg_all = !t.right && (odd1 ^ odd0) && t.xpar[ke];
  // lanes: element wi.z + lane + 32 i, or (n <= 16) element lane mod n, every groups-th source
  const int groups = n <= 16 ? 32 / n : 1;
  const int e0 = groups > 1 ? lane % n : wi.z + lane, grp = groups > 1 ? lane / n : 0;
  int rr[4], cc[4];
  double acc[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int e = min(e0 + 32 * i, n - 1);
    rr[i] = e / cols;
    cc[i] = e - rr[i] * cols;
    acc[i] = 0.0;
  }
  const int left = n - wi.z, cnt = groups > 1 ? 1 : min(4, (left + 31) >> 5);
  const int r1 = t.rbeg[o + 1];
  for (int r0 = t.rbeg[o]; r0 < r1; r0 += 32) {
    bool ok = false;
    EnlSrc src{};
    if (r0 + lane < r1) {
      const EnlRef r = t.refs[r0 + lane];
      const EnlSite& g = t.sites[r.site];
      if ((g.mask >> (4 * n1 + n0)) & 1) {
        const int j = r.op >> 1, tr = r.op & 1;
        const int s = tr ? be : ke;
        const EnlBlock b = t.blk[j * t.ns + s];
        const bool rev = tr && xrev;
        if (b.bra == (tr ? ke : be) && (b.nz & (rev ? 2 : 1))) {
          ok = true;
          const int ld = t.xdim[s];
          const bool neg = neg_all || (neg_odd && t.opar[j]);
          src.p = (rev ? xrev : x) + b.off;
          src.rs = tr ? 1 : ld;
          src.cs = tr ? ld : 1;
          src.scale = (neg ? -r.c : r.c) * g.e[4 * n1 + n0];
        }
      }
    }
    const uint32_t m = __ballot_sync(0xffffffffu, ok);
    __syncwarp();                 // the previous sources are no longer read
    if (ok) S[__popc(m & ((1u << lane) - 1))] = src;
    __syncwarp();
    const int ns = __popc(m);
    if (cnt == 1) {
#pragma unroll 4
      for (int s = grp; s < ns; s += groups)
        acc[0] = fma(S[s].scale, S[s].p[(int64_t)rr[0] * S[s].rs + (int64_t)cc[0] * S[s].cs], acc[0]);
    } else {
#pragma unroll 2
      for (int s = 0; s < ns; ++s) {
        const EnlSrc g = S[s];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i < cnt) acc[i] = fma(g.scale, g.p[(int64_t)rr[i] * g.rs + (int64_t)cc[i] * g.cs], acc[i]);
      }
    }
  }
  const int ldd = t.fdim[fk];
  double* dst = d + t.eoff[o * t.nse + fk] + (int64_t)t.foff[4 * fb + n1] * ldd + t.foff[4 * fk + n0];
  if (groups > 1) {
    double s = 0.0;               // the groups' sums, in order
    for (int g = 0; g < groups; ++g) s += __shfl_sync(0xffffffffu, acc[0], g * n + e0);
    if (lane < n) dst[(int64_t)rr[0] * ldd + cc[0]] = s;
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (i < cnt && lane + 32 * i < left) dst[(int64_t)rr[i] * ldd + cc[i]] = acc[i];
}

__global__ void __launch_bounds__(32 * ENL_WARPS) enlarge_kernel(const EnlTables t, const int3* __restrict__ items,
                                                                  int nitems, double* __restrict__ d,
                                                                  const double* __restrict__ x,
                                                                  const double* __restrict__ xrev) {
  __shared__ EnlSmem S;
  const int warp = threadIdx.x >> 5, w = blockIdx.x * ENL_WARPS + warp;
  if (w >= nitems) return;
  enlarge_item(t, items[w], d, x, xrev, S.s[warp]);
}

__global__ void __launch_bounds__(32 * ENL_WARPS) enlarge_inst_kernel(const EnlTables t, const int3* __restrict__ items,
                                                                       int nitems, const __grid_constant__ GatherInstSet P,
                                                                       int ninst) {
  __shared__ EnlSmem S;
  const int warp = threadIdx.x >> 5;
  const unsigned w = blockIdx.x * ENL_WARPS + warp;
  const int it = (int)(w / ninst);
  if (it >= nitems) return;
  const GatherBases* b = &P.b[w % ninst];
  enlarge_item(t, items[it], b->d, b->s1, b->s2, S.s[warp]);
}

void launch_enlarge(const EnlTables& t, const int3* items, int nitems, double* d, const double* x, const double* xrev,
                    cudaStream_t st) {
  if (nitems <= 0) return;
  enlarge_kernel<<<(nitems + ENL_WARPS - 1) / ENL_WARPS, 32 * ENL_WARPS, 0, st>>>(t, items, nitems, d, x, xrev);
}

void launch_enlarge_inst(const EnlTables& t, const int3* items, int nitems, const GatherInstSet& bases, int ninst,
                         cudaStream_t st) {
  // the caller checks 1 <= ninst <= 64 and nitems * ninst < 2^31
  if (nitems <= 0 || ninst <= 0) return;
  const long long n = (long long)nitems * ninst;
  enlarge_inst_kernel<<<(unsigned)((n + ENL_WARPS - 1) / ENL_WARPS), 32 * ENL_WARPS, 0, st>>>(t, items, nitems, bases,
                                                                                            ninst);
}

// ---------------------------------------------------------------------------
// grouped FP64 GEMM with K-concatenated segments
//
// GB300 issues about 2 FP64 FMA per clock per SM, so the kernel is bound by the
// number of DFMA warp instructions once its operands arrive in time.  Padding is
// the enemy: each lane owns individual output elements of a <= GEMM_TM x GEMM_TN
// tile (flattened, so only the last warp of a tile is partly idle).  The segments
// of a tile (often a dozen or more, each contracting only ~8 indices) are packed
// along one K axis and staged GEMM_KC positions at a time with cp.async into a
// double buffer, so a chunk's copies are all in flight at once and overlap the
// previous chunk's FMAs (the staging plan is in lrt_fp64_tile.h).
// ---------------------------------------------------------------------------
constexpr int GEMM_MAXE = GEMM_TM * GEMM_TN / GEMM_THREADS;   // outputs per thread
constexpr int GEMM_CTAS = 4;                                   // resident CTAs per SM (registers, shared memory)
static_assert(GEMM_TM == GEMM_TILE_M && GEMM_TN == GEMM_TILE_N, "tile shape of the staging plan");

struct GemmSmem {
  double As[2][GEMM_TM][GEMM_KC + 1];
  double Bs[2][GEMM_KC][GEMM_TN + 1];
  double sc[2][GEMM_KC];          // scale of the segment holding each K position of a chunk
  SegS sd[GEMM_SEGB];
  int kst[GEMM_SEGB + 1];
  int unit[2];                    // every scale of the chunk is 1
};

__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// extra base i of a launch (a switch, so the parameter block is not copied to local memory)
__device__ __forceinline__ double* extra_base(const GemmExtra& ex, int i) {
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

// acc[j] += sum_kk As[row_j][kk] Bs[kk][col_j] over a staged chunk, for the first N outputs
template <int N>
__device__ __forceinline__ void fma_chunk(double (&acc)[GEMM_MAXE], const uint32_t (&rc)[GEMM_MAXE],
                                          const double* __restrict__ As, const double* __restrict__ Bs, int kc) {
  for (int kk = 0; kk < kc; ++kk) {
#pragma unroll
    for (int j = 0; j < N; ++j)
      acc[j] = fma(As[(rc[j] >> 16) * (GEMM_KC + 1) + kk], Bs[kk * (GEMM_TN + 1) + (rc[j] & 0xFFFFu)], acc[j]);
  }
}

// the FMA loop is dispatched by a switch (one indirect branch) over these output counts;
// a chain of compares measured ~10% slower on the small tiles of phase 1
static_assert(GEMM_MAXE == 16, "the switch below lists the output counts 1..16");

// one tile of the grouped GEMM; extra(i) resolves extra base i of the tile's instance
template <class Extra>
__device__ __forceinline__ void gemm_fp64_tile(const GemmOut* __restrict__ outs, const GemmSeg* __restrict__ segs,
                                               const int3 wi, const double* xbase, double* ybase, double* tbase,
                                               double* wbase, const GemmOut& o, const Extra& extra) {
  extern __shared__ __align__(16) unsigned char gemm_smem_raw[];
  GemmSmem& S = *reinterpret_cast<GemmSmem*>(gemm_smem_raw);
  const int m0 = wi.y >> 8, mt = wi.y & 255, n0 = wi.z >> 8, nt = wi.z & 255;
  const int ne = mt * nt;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t rc[GEMM_MAXE];        // (row << 16) | col of each owned output element
  double acc[GEMM_MAXE];
#pragma unroll
  for (int j = 0; j < GEMM_MAXE; ++j) {
    const int e = tid + GEMM_THREADS * j;
    rc[j] = e < ne ? ((uint32_t)(e / nt) << 16) | (uint32_t)(e % nt) : 0u;
    acc[j] = 0.0;
  }
  const int cnt = ne > tid ? (ne - tid + GEMM_THREADS - 1) / GEMM_THREADS : 0;
  // outputs of lane 0, the most of any lane of the warp; the other lanes' extra slots
  // accumulate (0, 0)-element products that are never stored
  const int cntw = ne > 32 * warp ? (ne - 32 * warp + GEMM_THREADS - 1) / GEMM_THREADS : 0;

  for (int b0 = 0; b0 < o.seg_count; b0 += GEMM_SEGB) {
    const int nb = min(GEMM_SEGB, o.seg_count - b0);
    __syncthreads();   // the previous batch's descriptors and buffers are no longer read
    if (warp == 0) {
      int k = 0;
      if (lane < nb) {
        GemmSeg g = segs[o.seg_begin + b0 + lane];
        if (g.a_rel) g.A = (g.a_rel == 1 ? xbase : g.a_rel == 2 ? tbase : extra(g.a_rel - 3)) + g.a_off;
        if (g.b_rel) g.B = (g.b_rel == 1 ? xbase : g.b_rel == 2 ? tbase : extra(g.b_rel - 3)) + g.b_off;
        S.sd[lane] = SegS{g.A, g.B, g.lda, g.ldb, g.transA, g.transB, g.scale, o.c_vr, o.c_vc, g.a_vs, g.b_vs};
        k = g.k;
      }
      int incl = k;   // inclusive prefix of k over the lanes
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

    auto issue = [&](int c, int buf) {
      const int p0 = c * GEMM_KC;
      stage_chunk(tid, S.sd, S.kst, Kb, p0, m0, mt, n0, nt, [&](int which, int r, int col, const double* src) {
        if (which == 0) cp_async8(&S.As[buf][r][col], src);
        else cp_async8(&S.Bs[buf][r][col], src);
      });
      if (warp == 0) {
        const int p = p0 + lane;
        const double s = p < Kb ? S.sd[seg_at(S.kst, p, 0)].scale : 1.0;
        S.sc[buf][lane] = s;
        const bool u = __all_sync(0xffffffffu, s == 1.0);
        if (lane == 0) S.unit[buf] = u ? 1 : 0;
      }
      cp_async_commit();
    };

    if (nch > 0) issue(0, 0);
    for (int c = 0; c < nch; ++c) {
      const int buf = c & 1;
      if (c + 1 < nch) {
        issue(c + 1, buf ^ 1);   // buffer buf ^ 1 was last read before the previous iteration's barrier
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();           // chunk c has landed for every thread
      const int kc = min(GEMM_KC, Kb - c * GEMM_KC);
      if (!S.unit[buf]) {        // scale row kk of B by its segment's scale
        if (lane < nt)
          for (int kk = warp; kk < kc; kk += GEMM_WARPS) S.Bs[buf][kk][lane] *= S.sc[buf][kk];
        __syncthreads();
      }
      const double* As = &S.As[buf][0][0];
      const double* Bs = &S.Bs[buf][0][0];
      switch (cntw) {            // warp-uniform trip count: no predicated-off DFMA occupies the pipe
#define LRT_FMA_CASE(N) \
  case N: fma_chunk<N>(acc, rc, As, Bs, kc); break;
        LRT_FMA_CASE(1) LRT_FMA_CASE(2) LRT_FMA_CASE(3) LRT_FMA_CASE(4) LRT_FMA_CASE(5) LRT_FMA_CASE(6)
        LRT_FMA_CASE(7) LRT_FMA_CASE(8) LRT_FMA_CASE(9) LRT_FMA_CASE(10) LRT_FMA_CASE(11) LRT_FMA_CASE(12)
        LRT_FMA_CASE(13) LRT_FMA_CASE(14) LRT_FMA_CASE(15) LRT_FMA_CASE(16)
#undef LRT_FMA_CASE
        default: break;
      }
      __syncthreads();           // buffer buf is free for chunk c + 2
    }
  }
  double* cbase = o.c_rel == GEMM_C_SPLIT ? wbase + o.c_off
                 : o.c_rel ? (o.c_rel == 1 ? ybase : o.c_rel == 2 ? tbase : extra(o.c_rel - 3)) + o.c_off : o.C;
#pragma unroll
  for (int j = 0; j < GEMM_MAXE; ++j) {
    if (j >= cnt) break;
    int r = m0 + (int)(rc[j] >> 16), col = n0 + (int)(rc[j] & 0xFFFFu);
    double* c = cbase;
    if (o.c_rel == GEMM_C_SPLIT) {
      // a part of a split tile is dense, whatever the output's vector blocks
    } else if (o.c_vr > 0) {     // row blocks of the vectors
      const int v = r / o.c_vr;
      c += (int64_t)v * o.c_vs;
      r -= v * o.c_vr;
    } else if (o.c_vc > 0) {     // column blocks of the vectors
      const int v = col / o.c_vc;
      c += (int64_t)v * o.c_vs;
      col -= v * o.c_vc;
    }
    c += (int64_t)r * o.ldc + col;
    *c = o.accumulate ? (*c + acc[j]) : acc[j];
  }
}

// Per-device state: a process may drive several GPUs (one context per device), and a
// function attribute set with cudaFuncSetAttribute applies to the current device only.
constexpr int MAX_DEVICES = 64;

int gemm_fp64_slots() {
  static std::atomic<int> slots[MAX_DEVICES];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return GEMM_CTAS;
  int n = slots[dev].load(std::memory_order_acquire);
  if (!n) {
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    n = std::max(1, nsm) * GEMM_CTAS;
    slots[dev].store(n, std::memory_order_release);
  }
  return n;
}

// Opt the FP64 GEMM into its dynamic shared memory on the current device, once per device.
// On failure the attribute stays unset, the error is the runtime's last error, and the
// caller's launch check reports it.
__global__ void __launch_bounds__(GEMM_THREADS, GEMM_CTAS) gemm_fp64_kernel(const GemmOut* __restrict__ outs,
                                                                    const GemmSeg* __restrict__ segs,
                                                                    const int3* __restrict__ tiles, int ntiles,
                                                                    const double* __restrict__ xbase,
                                                                    double* __restrict__ ybase,
                                                                    double* __restrict__ tbase,
                                                                    const GemmBases* __restrict__ multi,
                                                                    const GemmExtra ex, double* __restrict__ wbase) {
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
  gemm_fp64_tile(outs, segs, wi, xbase, ybase, tbase, wbase, o, [&](int i) { return extra_base(ex, i); });
}

__global__ void __launch_bounds__(GEMM_THREADS, GEMM_CTAS) gemm_fp64_inst_kernel(const GemmOut* __restrict__ outs,
                                                                         const GemmSeg* __restrict__ segs,
                                                                         const int3* __restrict__ tiles,
                                                                         int ntiles,
                                                                         const __grid_constant__ GemmInstSet P,
                                                                         int ninst) {
  const int w = blockIdx.x / ninst;
  if (w >= ntiles) return;
  const GemmInst* b = &P.b[blockIdx.x % ninst];
  const int3 wi = tiles[w];
  const GemmOut o = outs[wi.x];
  gemm_fp64_tile(outs, segs, wi, b->x, b->y, b->t, nullptr, o, [&](int i) { return b->e[i]; });
}

static cudaError_t gemm_fp64_smem_attr() {
  static std::atomic<int> done[MAX_DEVICES];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  if (done[dev].load(std::memory_order_acquire)) return cudaSuccess;
  for (const void* f : {(const void*)gemm_fp64_kernel, (const void*)gemm_fp64_inst_kernel}) {
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GemmSmem));
    if (e != cudaSuccess) return e;
    // all of the unified L1 as shared memory, so GEMM_CTAS CTAs fit on an SM
    e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
  }
  done[dev].store(1, std::memory_order_release);   // concurrent first calls set the same values
  return cudaSuccess;
}

void launch_gemm_fp64(const GemmOut* outs, const GemmSeg* segs, const int3* tiles, int ntiles,
                      const double* xbase, double* ybase, double* tbase, cudaStream_t st, const GemmExtra* extra,
                      double* wbase) {
  if (ntiles <= 0) return;
  if (gemm_fp64_smem_attr() != cudaSuccess) return;
  const GemmExtra ex = extra ? *extra : GemmExtra{};
  gemm_fp64_kernel<<<ntiles, GEMM_THREADS, sizeof(GemmSmem), st>>>(outs, segs, tiles, ntiles, xbase, ybase, tbase,
                                                                  nullptr, ex, wbase);
}

// 256 elements of a split tile per CTA: each sums its parts in part order (deterministic), eight
// loads in flight, then lands where the tile's output puts it, vector blocking included, as in
// the GEMM epilogue.  (One CTA for a whole tile of 100 parts: 385 us on the k = 24, M = 500
// workload, most SMs idle at the end.)
__global__ void __launch_bounds__(256) split_reduce_kernel(const GemmOut* __restrict__ outs,
                                                           const SplitTile* __restrict__ tiles,
                                                           const double* __restrict__ wbase,
                                                           double* __restrict__ ybase, double* __restrict__ tbase,
                                                           const GemmBases* __restrict__ multi) {
  const SplitTile t = tiles[blockIdx.x];
  const int ne = t.mt * t.nt;
  const int e = blockIdx.y * blockDim.x + threadIdx.x;
  if (e >= ne) return;
  const GemmOut o = outs[t.o];
  if (multi) {
    ybase = multi[o.inst].y;
    tbase = multi[o.inst].t;
  }
  double* cbase = o.c_rel == 1 ? ybase + o.c_off : o.c_rel == 2 ? tbase + o.c_off : o.C;
  const double* w = wbase + t.ws_off + e;
  double s = 0.0;
#pragma unroll 8
  for (int p = 0; p < t.nparts; ++p) s += w[(int64_t)p * ne];
  int r = t.m0 + e / t.nt, col = t.n0 + e % t.nt;
  double* c = cbase;
  if (o.c_vr > 0) {
    const int v = r / o.c_vr;
    c += (int64_t)v * o.c_vs;
    r -= v * o.c_vr;
  } else if (o.c_vc > 0) {
    const int v = col / o.c_vc;
    c += (int64_t)v * o.c_vs;
    col -= v * o.c_vc;
  }
  c += (int64_t)r * o.ldc + col;
  *c = o.accumulate ? (*c + s) : s;
}

void launch_split_reduce(const GemmOut* outs, const SplitTile* tiles, int ntiles, const double* wbase, double* ybase,
                         double* tbase, cudaStream_t st, const GemmBases* multi) {
  if (ntiles <= 0) return;
  constexpr int most = GEMM_TM * GEMM_TN > 16 * 256 ? GEMM_TM * GEMM_TN : 16 * 256;   // elements of a tile (either kernel)
  split_reduce_kernel<<<dim3(ntiles, (most + 255) / 256), 256, 0, st>>>(outs, tiles, wbase, ybase, tbase, multi);
}

void launch_gemm_fp64_inst(const GemmOut* outs, const GemmSeg* segs, const int3* tiles, int ntiles,
                           const GemmInstSet& bases, int ninst, cudaStream_t st) {
  // the caller checks 1 <= ninst <= GEMM_MAX_INST and ntiles * ninst < 2^31
  if (ntiles <= 0 || ninst <= 0) return;
  if (gemm_fp64_smem_attr() != cudaSuccess) return;
  gemm_fp64_inst_kernel<<<(unsigned)((long long)ntiles * ninst), GEMM_THREADS, sizeof(GemmSmem), st>>>(
      outs, segs, tiles, ntiles, bases, ninst);
}

void launch_gemm_fp64_multi(const GemmOut* outs, const GemmSeg* segs, const int3* tiles, int ntiles,
                            const GemmBases* bases, double* wbase, cudaStream_t st) {
  if (ntiles <= 0) return;
  if (gemm_fp64_smem_attr() != cudaSuccess) return;
  gemm_fp64_kernel<<<ntiles, GEMM_THREADS, sizeof(GemmSmem), st>>>(outs, segs, tiles, ntiles, nullptr, nullptr,
                                                                  nullptr, bases, GemmExtra{}, wbase);
}

// ---------------------------------------------------------------------------
// diagonal of H_eff
// ---------------------------------------------------------------------------
// One CTA per output block; term diagonals are staged through shared memory in
// chunks so each element reads them from there instead of from global memory.
constexpr int DIAG_CHUNK = 16;
constexpr int DIAG_MAXD = 128;     // rows and columns of a block staged per chunk (32 KB of shared memory)

__global__ void __launch_bounds__(256) diag_kernel(const DiagOut* __restrict__ outs,
                                                   const DiagTerm* __restrict__ terms,
                                                   double* __restrict__ dbase) {
  __shared__ double xs[DIAG_CHUNK][DIAG_MAXD];   // scale_t * x_t, so one DFMA per term and element
  __shared__ double ys[DIAG_CHUNK][DIAG_MAXD];
  const DiagOut o = outs[blockIdx.x];
  for (int r0 = 0; r0 < o.rows; r0 += DIAG_MAXD)
    for (int c0 = 0; c0 < o.cols; c0 += DIAG_MAXD) {
      const int rt = min(DIAG_MAXD, o.rows - r0), ct = min(DIAG_MAXD, o.cols - c0);
      const int n = rt * ct;
      // each thread keeps up to 8 partial sums in registers, more are revisited below
      for (int base = 0; base < n; base += 8 * blockDim.x) {
        double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int t0 = 0; t0 < o.term_count; t0 += DIAG_CHUNK) {
          const int tc = min(DIAG_CHUNK, o.term_count - t0);
          __syncthreads();
          for (int e = threadIdx.x; e < tc * (rt + ct); e += blockDim.x) {
            const int t = e / (rt + ct), u = e % (rt + ct);
            const DiagTerm d = terms[o.term_begin + t0 + t];
            if (u < rt) xs[t][u] = d.x ? d.scale * d.x[(int64_t)(r0 + u) * d.xs] : d.scale;
            else ys[t][u - rt] = d.y ? d.y[(int64_t)(c0 + u - rt) * d.ys] : 1.0;
          }
          __syncthreads();
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int e = base + threadIdx.x + j * blockDim.x;
            if (e < n) {
              const int i = e / ct, jj = e % ct;
              double a = acc[j];
              for (int t = 0; t < tc; ++t) a = fma(xs[t][i], ys[t][jj], a);
              acc[j] = a;
            }
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int e = base + threadIdx.x + j * blockDim.x;
          if (e < n) dbase[o.d_off + (int64_t)(r0 + e / ct) * o.cols + (c0 + e % ct)] = acc[j];
        }
      }
    }
}

void launch_diag(const DiagOut* outs, const DiagTerm* terms, int nouts, double* dbase,
                 cudaStream_t st) {
  if (nouts <= 0) return;
  diag_kernel<<<nouts, 256, 0, st>>>(outs, terms, dbase);
}

}  // namespace lrt

// ---------------------------------------------------------------------------
// Davidson vector operations
// ---------------------------------------------------------------------------
namespace lrt {

__global__ void __launch_bounds__(256) dots_kernel(const double* __restrict__ V, int64_t ld, int m,
                                                   const double* __restrict__ w, int64_t n,
                                                   double* __restrict__ out) {
  __shared__ double red[256];
  const int j = blockIdx.x;
  if (j >= m) return;
  double acc = 0.0;
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) acc = fma(V[j * ld + e], w[e], acc);
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[j] = red[0];
}

void launch_dots(const double* V, int64_t ld, int m, const double* w, int64_t n, double* out, cudaStream_t st) {
  if (m <= 0) return;
  dots_kernel<<<m, 256, 0, st>>>(V, ld, m, w, n, out);
}

// out[a * nb + b] = A[a] . B[b] for vectors given by pointer arrays (one block per pair)
__global__ void __launch_bounds__(256) pair_dots_kernel(const double* const* __restrict__ A,
                                                        const double* const* __restrict__ B, int nb, int64_t n,
                                                        double* __restrict__ out) {
  __shared__ double red[256];
  const int a = blockIdx.x / nb, b = blockIdx.x % nb;
  const double* x = A[a];
  const double* y = B[b];
  double acc = 0.0;
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) acc = fma(x[e], y[e], acc);
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = red[0];
}

void launch_pair_dots(const double* const* A, const double* const* B, int na, int nb, int64_t n, double* out,
                      cudaStream_t st) {
  if (na <= 0 || nb <= 0) return;
  pair_dots_kernel<<<na * nb, 256, 0, st>>>(A, B, nb, n, out);
}

__global__ void __launch_bounds__(256) lincomb_kernel(const double* __restrict__ V, int64_t ld, int m,
                                                      const double* __restrict__ coef, double sign, int64_t n,
                                                      double* __restrict__ out, double beta) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double acc = beta == 0.0 ? 0.0 : beta * out[e];
    for (int j = 0; j < m; ++j) acc = fma(sign * coef[j], V[j * ld + e], acc);
    out[e] = acc;
  }
}

void launch_lincomb(const double* V, int64_t ld, int m, const double* coef, int64_t n, double* out, double beta,
                    cudaStream_t st, double sign) {
  if (n <= 0) return;
  const int grid = (int)std::min<int64_t>((n + 255) / 256, 152 * 8);
  lincomb_kernel<<<grid, 256, 0, st>>>(V, ld, m, coef, sign, n, out, beta);
}

// Davidson: a direction's norm, Ritz pair and next direction stay on the device, so that an
// iteration waits for the host once (to test convergence) and not six times: 373 -> 278 ms for a
// ground-state sweep pair at k = 8, M = 64, whose vectors of a few thousand elements take
// microseconds and a round trip 20.  A direction of norm below DAV_MIN_NORM ends the iteration:
// the last Ritz vector is kept.
__device__ __forceinline__ double dav_norm(double t2) { return sqrt(t2 > 0.0 ? t2 : 0.0); }

// v = t / |t|
__global__ void __launch_bounds__(256) dav_unit_kernel(const double* __restrict__ t, const double* __restrict__ t2,
                                                       int64_t n, double* __restrict__ v) {
  const double nt = dav_norm(*t2), f = nt < DAV_MIN_NORM ? 0.0 : 1.0 / nt;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    v[e] = f == 0.0 ? 0.0 : f * t[e];
}

void launch_dav_unit(const double* t, const double* t2, int64_t n, double* v, cudaStream_t st) {
  if (n <= 0) return;
  const int grid = (int)std::min<int64_t>((n + 255) / 256, 152 * 8);
  dav_unit_kernel<<<grid, 256, 0, st>>>(t, t2, n, v);
}

// u = V z, au = AV z, r = au - theta u, t = -r / (d - theta) for the lowest pair (theta, z) of the
// m-dimensional subspace
__global__ void __launch_bounds__(256) dav_ritz_kernel(const double* __restrict__ V, const double* __restrict__ AV,
                                                       int64_t ld, int m, const double* __restrict__ Z,
                                                       const double* __restrict__ w, const double* __restrict__ t2,
                                                       const double* __restrict__ d, int64_t n, double* __restrict__ u,
                                                       double* __restrict__ au, double* __restrict__ r,
                                                       double* __restrict__ t) {
  if (dav_norm(*t2) < DAV_MIN_NORM) return;
  const double theta = *w;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double x = 0.0, ax = 0.0;
    for (int j = 0; j < m; ++j) {
      const double z = Z[(int64_t)j * m];
      x = fma(z, V[j * ld + e], x);
      ax = fma(z, AV[j * ld + e], ax);
    }
    const double res = fma(-theta, x, ax);
    double den = d[e] - theta;
    if (fabs(den) < 1e-4) den = den < 0.0 ? -1e-4 : 1e-4;
    u[e] = x;
    au[e] = ax;
    r[e] = res;
    t[e] = -res / den;
  }
}

void launch_dav_ritz(const double* V, const double* AV, int64_t ld, int m, const double* Z, const double* w,
                     const double* t2, const double* d, int64_t n, double* u, double* au, double* r, double* t,
                     cudaStream_t st) {
  if (n <= 0) return;
  const int grid = (int)std::min<int64_t>((n + 255) / 256, 152 * 8);
  dav_ritz_kernel<<<grid, 256, 0, st>>>(V, AV, ld, m, Z, w, t2, d, n, u, au, r, t);
}

// ---------------------------------------------------------------------------
// batched vector operations of the TDA sweeps
// ---------------------------------------------------------------------------
static int vec_grid(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 4)); }

__global__ void __launch_bounds__(256) rank1_batch_kernel(const double* __restrict__ w, int64_t ldw,
                                                          const double* __restrict__ coef, double alpha, int nv,
                                                          double* __restrict__ V, int64_t ld, int64_t n) {
  const int v = blockIdx.y;
  const double c = coef ? alpha * coef[v] : alpha;
  if (c == 0.0) return;
  double* x = V + (int64_t)v * ld;
  const double* y = w + (int64_t)v * ldw;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    x[e] = fma(c, y[e], x[e]);
}

void launch_rank1_batch(const double* w, int64_t ldw, const double* coef, double alpha, int nv, double* V,
                        int64_t ld, int64_t n, cudaStream_t st) {
  if (nv <= 0 || n <= 0) return;
  rank1_batch_kernel<<<dim3(vec_grid(n), nv), 256, 0, st>>>(w, ldw, coef, alpha, nv, V, ld, n);
}

// Products with diagonal matrices (Schmidt values, their inverses): one multiplication per
// element, rounded once, however far the values span.  (As D x D products they cost D / 2 times
// the operations of this bandwidth-bound pass.)
__global__ void __launch_bounds__(256) diag_scale_kernel(const double* __restrict__ A, int64_t lda,
                                                         const double* __restrict__ w, const int* __restrict__ state,
                                                         int64_t n, double* __restrict__ out, int64_t ldo, bool acc) {
  const double* a = A + (int64_t)blockIdx.y * lda;
  double* o = out + (int64_t)blockIdx.y * ldo;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const double x = __dmul_rn(a[e], w[state[e]]);
    o[e] = acc ? __dadd_rn(o[e], x) : x;
  }
}

void launch_diag_scale(const double* A, int64_t lda, const double* w, const int* state, int nv, int64_t n, double* out,
                       int64_t ldo, bool acc, cudaStream_t st) {
  if (nv <= 0 || n <= 0) return;
  diag_scale_kernel<<<dim3(vec_grid(n), nv), 256, 0, st>>>(A, lda, w, state, n, out, ldo, acc);
}

// one thread per element and up to ROT_MU outputs at a time: every old vector is read once
// per group of ROT_MU new vectors
constexpr int ROT_MU = 16;
__global__ void __launch_bounds__(256) rotate_kernel(const double* __restrict__ Vold, int64_t ld_old, int lold,
                                                     const double* __restrict__ a, int m, int mu0, int mcnt,
                                                     double* __restrict__ Vnew, int64_t ld_new, int64_t n) {
  __shared__ double sa[JACOBI_MAXN * ROT_MU];
  for (int t = threadIdx.x; t < lold * mcnt; t += blockDim.x) sa[t] = a[(t / mcnt) * m + mu0 + t % mcnt];
  __syncthreads();
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double acc[ROT_MU];
#pragma unroll
    for (int q = 0; q < ROT_MU; ++q) acc[q] = 0.0;
    for (int j = 0; j < lold; ++j) {
      const double x = Vold[(int64_t)j * ld_old + e];
#pragma unroll
      for (int q = 0; q < ROT_MU; ++q)
        if (q < mcnt) acc[q] = fma(sa[j * mcnt + q], x, acc[q]);
    }
#pragma unroll
    for (int q = 0; q < ROT_MU; ++q)
      if (q < mcnt) Vnew[(int64_t)(mu0 + q) * ld_new + e] = acc[q];
  }
}

void launch_rotate(const double* Vold, int64_t ld_old, int lold, const double* a, int m, double* Vnew,
                   int64_t ld_new, int64_t n, cudaStream_t st) {
  if (m <= 0 || n <= 0) return;
  if (lold <= 0) {
    for (int mu = 0; mu < m; ++mu) cudaMemsetAsync(Vnew + (int64_t)mu * ld_new, 0, (size_t)n * sizeof(double), st);
    return;
  }
  for (int mu0 = 0; mu0 < m; mu0 += ROT_MU)
    rotate_kernel<<<vec_grid(n), 256, 0, st>>>(Vold, ld_old, lold, a, m, mu0, std::min(ROT_MU, m - mu0), Vnew,
                                               ld_new, n);
}

__global__ void __launch_bounds__(256) precond_batch_kernel(const double* __restrict__ R, int64_t ldr,
                                                            const double* __restrict__ d,
                                                            const double* __restrict__ theta, int64_t n,
                                                            double* __restrict__ Z, int64_t ldz, double sign) {
  const int v = blockIdx.y;
  const double th = theta[v];
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double den = d[e] - th;
    if (fabs(den) < 1e-4) den = den < 0.0 ? -1e-4 : 1e-4;
    Z[(int64_t)v * ldz + e] = -sign * R[(int64_t)v * ldr + e] / den;
  }
}

__global__ void __launch_bounds__(256) precond_abs_kernel(const double* __restrict__ R, const double* __restrict__ d,
                                                          double shift, int64_t n, double* __restrict__ Z) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    Z[e] = R[e] / fmax(fabs(d[e] - shift), 1e-4);
}

void launch_precond_abs(const double* R, const double* d, double shift, int64_t n, double* Z, cudaStream_t st) {
  if (n <= 0) return;
  precond_abs_kernel<<<vec_grid(n), 256, 0, st>>>(R, d, shift, n, Z);
}

void launch_precond_batch(const double* R, int64_t ldr, const double* d, const double* theta, int nv, int64_t n,
                          double* Z, int64_t ldz, double sign, cudaStream_t st) {
  if (nv <= 0 || n <= 0) return;
  precond_batch_kernel<<<dim3(vec_grid(n), nv), 256, 0, st>>>(R, ldr, d, theta, n, Z, ldz, sign);
}

// first pass: CTA (pair p, chunk c) sums its share of the elements of pair p
__device__ __forceinline__ double block_sum256(double v, double* red) {
  red[threadIdx.x] = v;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  return red[0];
}

__global__ void __launch_bounds__(256) vdots_part_kernel(const double* __restrict__ A, int64_t lda,
                                                         const double* __restrict__ B, int64_t ldb, int nb,
                                                         int64_t n, int pairs_mode, double* __restrict__ work) {
  __shared__ double red[256];
  const int p = blockIdx.y, c = blockIdx.x;
  const int a = pairs_mode ? p / nb : p;
  const int b = pairs_mode ? p % nb : p;
  const double* x = A + (int64_t)a * lda;
  const double* y = B + (int64_t)b * ldb;
  const int64_t per = (n + DOT_CHUNKS - 1) / DOT_CHUNKS;
  const int64_t e0 = (int64_t)c * per, e1 = min(n, e0 + per);
  double acc = 0.0;
  for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) acc = fma(x[e], y[e], acc);
  const double s = block_sum256(acc, red);
  if (threadIdx.x == 0) work[(int64_t)p * DOT_CHUNKS + c] = s;
}

__global__ void vdots_sum_kernel(const double* __restrict__ work, int np, double* __restrict__ out, int accumulate) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= np) return;
  double s = 0.0;
  for (int c = 0; c < DOT_CHUNKS; ++c) s += work[(int64_t)p * DOT_CHUNKS + c];
  out[p] = accumulate ? out[p] + s : s;
}

void launch_vdots(const double* A, int64_t lda, const double* B, int64_t ldb, int nv, int64_t n, double* out,
                  bool accumulate, double* work, cudaStream_t st) {
  if (nv <= 0) return;
  vdots_part_kernel<<<dim3(DOT_CHUNKS, nv), 256, 0, st>>>(A, lda, B, ldb, 1, n, 0, work);
  vdots_sum_kernel<<<(nv + 127) / 128, 128, 0, st>>>(work, nv, out, accumulate ? 1 : 0);
}

void launch_pair_dots_strided(const double* A, int64_t lda, int na, const double* B, int64_t ldb, int nb, int64_t n,
                              double* out, double* work, cudaStream_t st) {
  if (na <= 0 || nb <= 0) return;
  vdots_part_kernel<<<dim3(DOT_CHUNKS, na * nb), 256, 0, st>>>(A, lda, B, ldb, nb, n, 1, work);
  vdots_sum_kernel<<<(na * nb + 127) / 128, 128, 0, st>>>(work, na * nb, out, 0);
}

__global__ void gather_sum_kernel(const double* __restrict__ src, const int* __restrict__ beg,
                                  const int* __restrict__ idx, const double* __restrict__ coef, int nout,
                                  double* __restrict__ out) {
  const int d = blockIdx.x * blockDim.x + threadIdx.x;
  if (d >= nout) return;
  double s = 0.0;
  for (int j = beg[d]; j < beg[d + 1]; ++j) s = fma(coef[j], src[idx[j]], s);
  out[d] += s;
}

void launch_gather_sum(const double* src, const int* beg, const int* idx, const double* coef, int nout, double* out,
                       cudaStream_t st) {
  if (nout <= 0) return;
  gather_sum_kernel<<<(nout + 127) / 128, 128, 0, st>>>(src, beg, idx, coef, nout, out);
}

__global__ void reduced_acc_kernel(const double* __restrict__ D1, const double* __restrict__ D2,
                                   const double* __restrict__ D3, int l, double* __restrict__ Hr,
                                   double* __restrict__ Sr) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= l * l) return;
  const int a = t / l, b = t % l;
  Hr[t] += D1[t] + D2[t] + D2[b * l + a];
  Sr[t] += D3[t];
}

void launch_reduced_acc(const double* D1, const double* D2, const double* D3, int l, double* Hr, double* Sr,
                        cudaStream_t st) {
  if (l <= 0) return;
  reduced_acc_kernel<<<(l * l + 127) / 128, 128, 0, st>>>(D1, D2, D3, l, Hr, Sr);
}

// Jacobi eigenvalue iteration for a small symmetric matrix held in shared memory (n <=
// JACOBI_MAXN = 48), n / 2 disjoint rotations at a time (round-robin ordering, Brent and Luk,
// SIAM J. Sci. Stat. Comput. 6, 1985): a step's rotations are computed by one thread each, then
// every thread applies two of them to 2 x 2 blocks of A, one to pairs of Z.  Sweeps stop when the
// off-diagonal norm is below 1e-15 of the Frobenius norm, or after a fixed number.  One
// rotation at a time, the chain of n (n - 1) / 2 rotations a sweep took 1.48 ms at n <= 24 (60%
// of a ground-state run).  What is left is a serial chain of steps: the rotation (square root,
// quotient, reciprocal square root), two barriers and the FP64 pipe of one SM.  Hence only the
// blocks on and above the diagonal, no work for rotations that are the identity, a thread's
// blocks found once and a step's pairs once by the thread that rotates them (n = 12 / 24: 233 /
// 631 -> 178 / 472 us, the residual of a pair and the orthogonality 2 to 3 times smaller).
// The tangent in FP32, its element's rest kept, was 10% faster there but half as fast on matrices
// of rank one: not kept.
constexpr int JACOBI_THREADS = 256;
constexpr int JACOBI_NP = JACOBI_MAXN / 2;
constexpr int JACOBI_ITEMS = (JACOBI_NP * (JACOBI_NP + 1) / 2 + JACOBI_MAXN * JACOBI_NP + JACOBI_THREADS - 1) / JACOBI_THREADS;
__global__ void __launch_bounds__(JACOBI_THREADS) jacobi_kernel(double* __restrict__ Ag, int ld, int n,
                                                                const double* __restrict__ col, double* __restrict__ w,
                                                                double* __restrict__ Zg) {
  __shared__ double A[JACOBI_MAXN][JACOBI_MAXN + 1];
  __shared__ double Z[JACOBI_MAXN][JACOBI_MAXN + 1];
  __shared__ double2 rot[JACOBI_NP];              // cosine and sine of a step's pairs
  __shared__ int2 pair[JACOBI_NP];                // their indices, the smaller first
  __shared__ double red[2][JACOBI_THREADS / 32];
  __shared__ int order[JACOBI_MAXN];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ne = (n + 1) & ~1, np = ne / 2;       // an odd n gets a row that pairs with nobody
  for (int e = tid; e < n * n; e += JACOBI_THREADS) {
    const int i = e / n, j = e % n;
    if (col && max(i, j) == n - 1) {              // the new row and column
      A[i][j] = Ag[i * ld + j] = col[min(i, j)];
    } else {
      A[i][j] = 0.5 * (Ag[i * ld + j] + Ag[j * ld + i]);
    }
    Z[i][j] = (i == j) ? 1.0 : 0.0;
  }
  // this thread's items, u | v << 8: rows of pair u times columns of pair v >= u of A, then
  // (1 << 16 set) row u of Z times pair v; -1 none
  int item[JACOBI_ITEMS];
  const int na = np * (np + 1) / 2;
#pragma unroll
  for (int h = 0; h < JACOBI_ITEMS; ++h) {
    const int e = tid + h * JACOBI_THREADS;
    item[h] = -1;
    if (e < na) {                                 // row u of the triangle starts at u np - u (u - 1) / 2
      int u = 0, f = e;
      while (f >= np - u) f -= np - u++;
      item[h] = u | (u + f) << 8;
    } else if (e < na + n * np) {
      item[h] = (e - na) / np | (e - na) % np << 8 | 1 << 16;
    }
  }
  // pair k of step r: player ne - 1 (k = 0) or (r + k) mod (ne - 1), against (r - k) mod (ne - 1)
  const int m = ne - 1;
  int pa = tid == 0 ? m : tid, pb = tid == 0 ? 0 : m - tid;
  __syncthreads();
  for (int sweep = 0; sweep < 60; ++sweep) {
    double off = 0.0, fro = 0.0;
    for (int e = tid; e < n * n; e += JACOBI_THREADS) {
      const int i = e / n, j = e % n;
      const double x = A[i][j] * A[i][j];
      fro += x;
      if (i != j) off += x;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, d);
      fro += __shfl_xor_sync(0xffffffffu, fro, d);
    }
    if (lane == 0) {
      red[0][warp] = off;
      red[1][warp] = fro;
    }
    __syncthreads();
    off = fro = 0.0;
    for (int k = 0; k < JACOBI_THREADS / 32; ++k) {
      off += red[0][k];
      fro += red[1][k];
    }
    // (a matrix with NaN or infinities ends after its 60 sweeps)
    if (off <= 1e-30 * fro) break;
    for (int r = 0; r < m; ++r) {                 // m steps bring every pair back to its start
      bool turns = false;
      if (tid < np) {
        const int p = min(pa, pb), q = max(pa, pb);
        double c = 1.0, s = 0.0;
        if (q < n) {
          const double apq = A[p][q];
          // elements that together stay below a tenth of the stopping norm are left alone
          if (apq * apq * (double)(n * n) > 1e-31 * fro) {
            // t = sgn(d / b) |b| / (|d| + sqrt(d^2 + b^2)), both scaled by a power of two to
            // keep the squares in range
            double d = A[q][q] - A[p][p], b = 2.0 * apq;
            const bool neg = d != 0.0 && (d < 0.0) != (b < 0.0);
            const int ex = min(max(__double2hiint(fmax(fabs(d), fabs(b))) >> 20, 1), 2045);
            const double f = __hiloint2double((2046 - ex) << 20, 0);
            d = fabs(d) * f;
            b = fabs(b) * f;
            const double t = b / (d + sqrt(d * d + b * b));
            c = rsqrt(1.0 + t * t);
            s = neg ? -t * c : t * c;
          }
        }
        rot[tid] = make_double2(c, s);
        pair[tid] = make_int2(p, q);
        turns = s != 0.0;
        if (tid > 0) pa = pa + 1 == m ? 0 : pa + 1;
        pb = pb + 1 == m ? 0 : pb + 1;
      }
      if (!__syncthreads_or(turns)) continue;
      // A <- J^T A J by 2 x 2 blocks (rows of pair u, columns of pair v >= u, mirrored), Z <- Z J
#pragma unroll
      for (int h = 0; h < JACOBI_ITEMS; ++h) {
        if (item[h] < 0) break;
        const int u = item[h] & 255, v = item[h] >> 8 & 255;
        const double c = rot[v].x, s = rot[v].y;
        const int p = pair[v].x, q = pair[v].y;
        if (item[h] < 1 << 16) {
          const double cu = rot[u].x, su = rot[u].y;
          if (s == 0.0 && su == 0.0) continue;
          const int i = pair[u].x, j = pair[u].y;
          // rows or columns of the bye player (index n) do not exist
          const bool hi = j < n, hq = q < n;
          const double a00 = A[i][p], a01 = hq ? A[i][q] : 0.0, a10 = hi ? A[j][p] : 0.0, a11 = hi && hq ? A[j][q] : 0.0;
          const double b00 = c * a00 - s * a01, b01 = s * a00 + c * a01;
          const double b10 = c * a10 - s * a11, b11 = s * a10 + c * a11;
          const double d00 = cu * b00 - su * b10, d11 = su * b01 + cu * b11;
          const double d01 = u == v ? 0.0 : cu * b01 - su * b11, d10 = u == v ? 0.0 : su * b00 + cu * b10;
          A[i][p] = A[p][i] = d00;
          if (hq) A[i][q] = A[q][i] = d01;
          if (hi) A[j][p] = A[p][j] = d10;
          if (hi && hq) A[j][q] = A[q][j] = d11;
        } else if (s != 0.0) {
          const double zp = Z[u][p], zq = Z[u][q];
          Z[u][p] = c * zp - s * zq;
          Z[u][q] = s * zp + c * zq;
        }
      }
      __syncthreads();
    }
  }
  // rank of every eigenvalue (ties by index)
  const double x = tid < n ? A[tid][tid] : 0.0;
  const bool nan = __syncthreads_or(x != x);      // then they keep their places
  if (tid < n) {
    int rank = tid;
    if (!nan) {
      rank = 0;
      for (int j = 0; j < n; ++j) rank += A[j][j] < x || (A[j][j] == x && j < tid);
    }
    order[rank] = tid;
  }
  __syncthreads();
  for (int e = tid; e < n * n; e += JACOBI_THREADS) {
    const int i = e / n, j = e % n;
    Zg[i * n + j] = Z[i][order[j]];
  }
  for (int i = tid; i < n; i += JACOBI_THREADS) w[i] = A[order[i]][order[i]];
}

void launch_jacobi_eigh(double* A, int n, double* w, double* Z, cudaStream_t st, const double* col, int ld) {
  if (n <= 0) return;
  jacobi_kernel<<<1, JACOBI_THREADS, 0, st>>>(A, ld > 0 ? ld : n, n, col, w, Z);
}

}  // namespace lrt
