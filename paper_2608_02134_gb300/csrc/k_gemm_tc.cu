// General C = diag(r) (A B^T) diag(c) on the tcgen05 tensor cores (bf16 operands,
// fp32 accumulation in tensor memory, fp32 output): the dense contractions of
// the long-prefix path.
//
//   * the fixed rank-r Rademacher projection of the boundary states, y_i = R h_i
//     (A = visual hidden rows, B = R, no scaling);
//   * the bounded appearance bank's cosines x~_{c(m)} . x~_i over the projected
//     unit states (A, B = the states split into bf16 hi/lo terms, laid out so
//     one product over 3r columns sums hi.hi + hi.lo + lo.hi);
//   * the support cosines of the assignment, cos(h_{S_k}, h_i), as K x N rows
//     (A = the selected rows gathered, B = the visual hidden rows, scaled by
//     the reciprocal norms of both).
//   * the cosine Gram of the boundary states for large or batched problems
//     (symmetric mode: A = B = the visual rows, scaled by their reciprocal
//     norms; only tiles on or above the diagonal are computed).
// (Appendix "Appearance and spatial clients", last paragraph; the cost notes
// after Algorithm 1: the bounded bank and the chunked N x K assignment product;
// Eq. (cond-aux-clients), (cond-assignment) for the cosines.)
//
// Persistent: one CTA per SM takes every gridDim.x-th 128 x BN output tile (BN = 128
// or 256, launch_gemm_tc).  Warp 0 / lane 0 streams 64-wide K slices of the A and B row blocks with
// TMA (128-byte swizzle) through an mbarrier ring of four stages; warp 1 / lane 0
// issues tcgen05.mma (M = 128, N = BN, K = 16) into one of two accumulators in
// tensor memory (BN columns each); warps 4 to 11 drain the other one: warp w reads
// lane quarter w % 4 and half of the columns in 32-column chunks, and stores each
// chunk through a 32 x 32 shared-memory transpose, so every store instruction writes
// whole 128-byte row segments (four of them where the rows lie on 16 bytes), scaled by
// row and column.  So a tile's products run while the last one is stored,
// with all four stages' loads in flight behind them.  Before, two CTAs of two
// stages shared an SM, and one's products waited for their own two loads whenever
// the other was storing: tensor pipe active 49% on a full SM, 4,096 x 15,876 x
// 3,584 344 us, now 313; the Gram of 4,096 states 58, now 57, of
// 32 x 1,296 272, now 215; 4,096 x 15,876 x 384, bound by its stores, 101, now 72.
//
// Ragged edges: TMA fills K columns past the operands' extents with zeros.  The
// last row block of an operand with at least one full tile of rows is shifted
// inward (start M - 128, likewise Nn - BN) so every box lies inside the image's own
// rows -- the hidden states' visual rows are followed by text rows whose count only
// the device knows -- and stores only the rows and columns the previous tile does
// not own; a smaller operand reads zeros past its declared rows.  Symmetric
// mode (M == Nn, A and B the same rows): the tiles are those that hold an entry
// with j >= i; a tile stores its own entries and, from registers (coalesced over
// the lanes), the mirror C[j][i] of each entry j > i whose own tile is not computed
// -- every entry is written exactly once, so the result does not depend on the order
// of the stores.  Every mbarrier wait is bounded (about two seconds after its tile
// began); on timeout the kernel records GMC_STATUS_TIMEOUT, drains its copies and
// products and frees its tensor memory.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "tc.cuh"

namespace gmc {

namespace {
constexpr int GM = 128, GK = 64, GST = 4;  // tile rows, K slice, ring stages
constexpr int G_EPI = 8;                   // epilogue warps, after four others
constexpr int G_THREADS = 32 * (4 + G_EPI);
constexpr int GA_BYTES = GM * GK * 2;      // 16 KiB per stage
constexpr long long G_WAIT = 4000000000LL;

struct GemmCtl {
  uint64_t full[GST];
  uint64_t empty[GST];
  uint64_t tfull[2];   // an accumulator holds its tile
  uint64_t tempty[2];  // and has been read
  uint64_t done;       // every product issued has ended
  uint32_t tmem;
  volatile int abort;
};

// Symmetric mode: tile (I, J) (rows 128 I.., columns BN J..) is computed when it
// holds an entry with j >= i.
template <int BN> __host__ __device__ __forceinline__ bool sym_tile(int I, int J) {
  return BN * J + BN - 1 >= GM * I;
}
template <int BN> __host__ __device__ __forceinline__ int sym_first_col(int I) {
  const int x = GM * I - (BN - 1);
  return x <= 0 ? 0 : (x + BN - 1) / BN;
}

template <int BN> constexpr size_t gemm_smem() {
  return 1024 + (size_t)GST * (GA_BYTES + BN * GK * 2) + G_EPI * 32 * 32 * sizeof(float) +
         sizeof(GemmCtl);
}

// Output tile t of the grid's list.
struct GemmTile {
  int b, m0, n0;   // image, first row and column it owns
  int ml, nl;      // first row and column it loads: shifted inward at the ragged end
  int arow, brow;  // the operands' first rows of the image
};
// false: the image has no text (its offsets are invalid), nothing to compute
template <int BN>
__device__ __forceinline__ bool gemm_tile(const GemmArgs& g, int t, int per_image, GemmTile* o) {
  const int b = t / per_image;
  t -= b * per_image;
  int tI, tJ;
  const int nJ = ceil_div(g.Nn, BN);
  if (g.sym) {  // the computed tiles, row block by row block
    tI = 0;
    while (t >= nJ - sym_first_col<BN>(tI)) {
      t -= nJ - sym_first_col<BN>(tI);
      ++tI;
    }
    tJ = sym_first_col<BN>(tI) + t;
  } else if (g.m_fast) {
    // consecutive CTAs share a B tile (the larger operand is B and stays in L2 while
    // the A tiles stream past it), else an A tile
    const int nI = ceil_div(g.M, GM);
    tJ = t / nI;
    tI = t - tJ * nI;
  } else {
    tI = t / nJ;
    tJ = t - tI * nJ;
  }
  o->b = b;
  o->m0 = tI * GM;
  o->n0 = tJ * BN;
  o->ml = g.M >= GM ? min(o->m0, g.M - GM) : o->m0;
  o->nl = g.Nn >= BN ? min(o->n0, g.Nn - BN) : o->n0;
  o->arow = (int)((long long)b * g.a_img);
  o->brow = (int)((long long)b * g.b_img);
  if (g.a_text || g.b_text) {
    const TextGeom tg = text_geom(g.toff, b, g.B, g.Tmax, g.status);
    if (tg.T == 0) return false;
    if (g.a_text) o->arow += tg.off;
    if (g.b_text) o->brow += tg.off;
  }
  return true;
}
}  // namespace

template <int BN>
__global__ void __launch_bounds__(G_THREADS, 1)
    k_gemm_tc(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap,
              GemmArgs g, int per_image) {
  grid_dep_wait();
  constexpr int B_BYTES = BN * GK * 2;
  extern __shared__ uint8_t sm_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(sm_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* tilesA = base;
  uint8_t* tilesB = base + GST * GA_BYTES;
  float* stage = reinterpret_cast<float*>(base + GST * (GA_BYTES + B_BYTES));  // [G_EPI][32][32]
  GemmCtl* ctl = reinterpret_cast<GemmCtl*>(stage + G_EPI * 32 * 32);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nk = ceil_div(g.Kd, GK);
  const int ntiles = per_image * g.B;

  if (threadIdx.x == 0) {
    for (int s = 0; s < GST; ++s) {
      tc::mbar_init(&ctl->full[s], 1);
      tc::mbar_init(&ctl->empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(&ctl->tfull[s], 1);
      tc::mbar_init(&ctl->tempty[s], G_EPI);
    }
    tc::mbar_init(&ctl->done, 1);
    ctl->abort = 0;
    tc::fence_mbar_init();
    tc::prefetch_tmap(&amap);
    tc::prefetch_tmap(&bmap);
  }
  if (warp == 0) {
    tc::tmem_alloc(&ctl->tmem, 2 * BN);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = ctl->tmem;
  int issued = 0;  // K slices asked for, over all tiles (warp 0 / lane 0)

  if (warp == 0) {
    if (lane == 0) {
      for (int t = blockIdx.x; t < ntiles && !ctl->abort; t += gridDim.x) {
        GemmTile o;
        if (!gemm_tile<BN>(g, t, per_image, &o)) continue;
        const long long deadline = clock64() + G_WAIT;
        for (int kb = 0; kb < nk; ++kb) {
          const int s = issued % GST;
          if (issued >= GST &&
              !tc::mbar_wait(&ctl->empty[s], ((uint32_t)(issued / GST) & 1u) ^ 1u, deadline))
            ctl->abort = 1;
          if (ctl->abort) break;
          tc::mbar_arrive_expect_tx(&ctl->full[s], GA_BYTES + B_BYTES);
          tc::tma_load_2d(tilesA + s * GA_BYTES, &amap, kb * GK, o.arow + o.ml, &ctl->full[s]);
          tc::tma_load_2d(tilesB + s * B_BYTES, &bmap, kb * GK, o.brow + o.nl, &ctl->full[s]);
          ++issued;
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = tc::idesc_bf16_f32(GM, BN);
      int it = 0, n = 0;  // slices and tiles so far
      for (int t = blockIdx.x; t < ntiles && !ctl->abort; t += gridDim.x) {
        GemmTile o;
        if (!gemm_tile<BN>(g, t, per_image, &o)) continue;
        const long long deadline = clock64() + G_WAIT;
        const int buf = n & 1;
        if (n >= 2 && !tc::mbar_wait(&ctl->tempty[buf], ((uint32_t)(n >> 1) & 1u) ^ 1u, deadline)) {
          ctl->abort = 1;
          break;
        }
        tc::fence_after_sync();
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int s = it % GST;
          if (!tc::mbar_wait(&ctl->full[s], (uint32_t)(it / GST) & 1u, deadline)) {
            ctl->abort = 1;
            break;
          }
          tc::fence_after_sync();
          const uint64_t ad = tc::desc_sw128_kmajor(tilesA + s * GA_BYTES);
          const uint64_t bd = tc::desc_sw128_kmajor(tilesB + s * B_BYTES);
#pragma unroll
          for (int kk = 0; kk < GK / 16; ++kk)
            tc::mma_bf16(tmem + buf * BN, ad + 2 * kk, bd + 2 * kk, idesc, (kb | kk) != 0);
          tc::mma_commit(&ctl->empty[s]);
        }
        if (ctl->abort) break;
        tc::mma_commit(&ctl->tfull[buf]);
        ++n;
      }
      // every arrival of the products has landed before the block ends, also on abort
      tc::mma_commit(&ctl->done);
      if (!tc::mbar_wait(&ctl->done, 0, clock64() + G_WAIT)) ctl->abort = 1;
    }
    __syncwarp();
  } else if (warp >= 4) {
    const int quarter = warp & 3, half = (warp - 4) >> 2;
    float* st = stage + (warp - 4) * (32 * 32);
    // rows of C on 16 bytes, for tiles that start on a multiple of four columns
    const bool quads = (g.ldc & 3) == 0 && (g.c_img & 3) == 0 &&
                       (reinterpret_cast<uintptr_t>(g.C) & 15) == 0;
    int n = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
      GemmTile o;
      if (!gemm_tile<BN>(g, t, per_image, &o)) continue;
      const int buf = n & 1;
      const bool here = tc::mbar_wait(&ctl->tfull[buf], (uint32_t)(n >> 1) & 1u, clock64() + G_WAIT);
      if (!__all_sync(FULL, here)) {
        if (lane == 0) ctl->abort = 1;
        break;
      }
      ++n;
      tc::fence_after_sync();
      const int row = quarter * 32 + lane;  // this thread's TMEM lane = tile row
      const int i = o.ml + row;
      float r = 1.f;  // scales of the tile's rows and columns (1 where none is given)
      if (g.rscale && i < g.M) r = g.rscale[(size_t)o.b * g.M + i];
      const uint32_t trow = tmem + buf * BN + ((uint32_t)(quarter * 32) << 16);
      float* Cimg = g.C + (size_t)o.b * g.c_img;
      const bool full = o.m0 == o.ml && o.n0 == o.nl && o.ml + GM <= g.M && o.nl + BN <= g.Nn;
#pragma unroll 1
      for (int c = 0; c < BN / 64; ++c) {
        const int cl = half * (BN / 2) + c * 32;  // first column of the chunk, within the tile
        const int i0 = o.ml + quarter * 32, j0 = o.nl + cl;  // the chunk's first entry
        float v[32];
        tc::tmem_ld32(trow + (uint32_t)cl, v);
        if (c == BN / 64 - 1) {  // the accumulator is read: the next products may have it
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&ctl->tempty[buf]);
        }
        // the transpose: 16-byte unit u of row l in unit u ^ (l & 7)
        float4* st4 = reinterpret_cast<float4*>(st);
#pragma unroll
        for (int u = 0; u < 8; ++u)
          st4[lane * 8 + (u ^ (lane & 7))] =
              make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
        const int col = j0 + lane;
        float cs = 1.f;
        if (g.cscale && col < g.Nn) cs = g.cscale[(size_t)o.b * g.Nn + col];
        if (g.sym) {  // mirrors of owned entries j > i whose own tile is not computed
          // a tile that owns all it loads: one answer for 32 x 32 entries off the diagonal
          // (128 and 256 are multiples of 32, and so are i0 and j0)
          const bool all = full && j0 > i0 + 31;
          const bool any = !all || !sym_tile<BN>(j0 / GM, i0 / BN);
          const bool own_i = i >= o.m0 && i < g.M;
          float* mir = Cimg + (size_t)j0 * g.ldc + i;
          if (any) {
#pragma unroll  // fully: v stays in registers
            for (int q = 0; q < 32; ++q) {
              const int j = j0 + q;
              const float x = v[q] * (r * __shfl_sync(FULL, cs, q));
              if (all || (own_i && j >= o.n0 && j < g.Nn && j > i && !sym_tile<BN>(j / GM, i / BN)))
                mir[(size_t)q * g.ldc] = x;
            }
          }
        }
        __syncwarp();
        if (full && quads) {  // four columns a lane, four rows a store
          const int u = lane & 7, r0 = lane >> 3;
          float4 c4;
          c4.x = __shfl_sync(FULL, cs, 4 * u);
          c4.y = __shfl_sync(FULL, cs, 4 * u + 1);
          c4.z = __shfl_sync(FULL, cs, 4 * u + 2);
          c4.w = __shfl_sync(FULL, cs, 4 * u + 3);
          float* out = Cimg + (size_t)(i0 + r0) * g.ldc + j0 + 4 * u;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int rr = 4 * k + r0;
            const float rk = __shfl_sync(FULL, r, rr);
            float4 x = st4[rr * 8 + (u ^ (rr & 7))];
            x.x *= rk * c4.x;
            x.y *= rk * c4.y;
            x.z *= rk * c4.z;
            x.w *= rk * c4.w;
            *reinterpret_cast<float4*>(out) = x;
            out += 4 * (size_t)g.ldc;
          }
        } else {
          const bool col_ok = col >= o.n0 && col < g.Nn;  // owned by this tile
#pragma unroll 4
          for (int rr = 0; rr < 32; ++rr) {
            const int m = i0 + rr;
            const float rk = __shfl_sync(FULL, r, rr);
            const float x = st[rr * 32 + (((lane >> 2) ^ (rr & 7)) << 2) + (lane & 3)];
            if (m >= o.m0 && m < g.M && col_ok) Cimg[(size_t)m * g.ldc + col] = x * (rk * cs);
          }
        }
        __syncwarp();
      }
    }
  }
  __syncthreads();
  const bool ok = !ctl->abort;
  if (!ok && threadIdx.x == 0) {
    set_status(g.status, GMC_STATUS_TIMEOUT);
    // drain the copies still in flight
    const long long d2 = clock64() + G_WAIT;
    for (int q = (issued > GST ? issued - GST : 0); q < issued; ++q)
      if (!tc::mbar_wait(&ctl->full[q % GST], (uint32_t)(q / GST) & 1u, d2)) break;
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 2 * BN);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {
int gemm_sms() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      sms = 152;
    }
  }
  return sms;
}

// Tiles of an image in symmetric mode.
template <int BN> int sym_tiles(int N) {
  int nt = 0;
  for (int I = 0; I < ceil_div(N, GM); ++I) nt += ceil_div(N, BN) - sym_first_col<BN>(I);
  return nt;
}
}  // namespace

template <int BN>
static cudaError_t launch_gemm_bn(const GemmArgs& g, const void* A, long long a_rows, int lda,
                                  const void* Bm, long long b_rows, int ldb, cudaStream_t st) {
  CUtensorMap am, bm;
  cudaError_t e = make_tmap_bf16(&am, A, (uint64_t)g.Kd, (uint64_t)a_rows, (uint64_t)lda, GM);
  if (e != cudaSuccess) return e;
  if ((e = make_tmap_bf16(&bm, Bm, (uint64_t)g.Kd, (uint64_t)b_rows, (uint64_t)ldb, BN)) !=
      cudaSuccess)
    return e;
  const int per_image = g.sym ? sym_tiles<BN>(g.M) : ceil_div(g.Nn, BN) * ceil_div(g.M, GM);
  const int sms = gemm_sms();
  const long long tiles = (long long)per_image * g.B;
  if (tiles > 0x7fffffffLL - sms) return cudaErrorInvalidValue;
  constexpr size_t smem = gemm_smem<BN>();
  if ((e = set_smem_limit((const void*)k_gemm_tc<BN>, smem)) != cudaSuccess) return e;
  launch_k(k_gemm_tc<BN>, (int)std::min<long long>(tiles, sms), G_THREADS, smem, st, 1, am, bm, g,
           per_image);
  return cudaGetLastError();
}

int gemm_sym_ctas(int N, int B) { return sym_tiles<256>(N) * B; }

cudaError_t launch_gemm_tc(const GemmArgs& g, const void* A, long long a_rows, int lda,
                           const void* Bm, long long b_rows, int ldb, cudaStream_t st) {
  if (g.M < 1 || g.Nn < 1 || g.Kd < 1 || g.B < 1) return cudaErrorInvalidValue;
  if (g.sym && (g.M != g.Nn || g.Nn <= 128 || g.m_fast)) return cudaErrorInvalidValue;
  // an operand addressed from the hidden states (a_text / b_text) must hold a
  // full box of rows, so the shifted last box stays inside the image's visual
  // rows (the buffer may end right after the last image's text rows)
  if ((g.a_text && g.M < GM) || (g.b_text && g.Nn < (g.Nn <= 128 ? 128 : 256)))
    return cudaErrorInvalidValue;
  bool narrow = g.Nn <= 128;
  if (g.sym) {
    // 128 x 128 tiles where they take no more turns of the SMs than 128 x 256 ones (each
    // turn is then shorter): a call of gmc_cosine, 4 images of N = 1,296 67 us, 57 so; 20 of
    // 576 88 and 75; 80 of 256 (D = 256) 36 and 26.  With one turn more the wide tiles
    // win (5 of 1,296: 69 and 76; 32: 276 and 327).
    const int sms = gemm_sms();
    const long long wide = (long long)sym_tiles<256>(g.M) * g.B;
    const long long half = (long long)sym_tiles<128>(g.M) * g.B;
    narrow = (half + sms - 1) / sms <= (wide + sms - 1) / sms;
  }
  if (narrow) return launch_gemm_bn<128>(g, A, a_rows, lda, Bm, b_rows, ldb, st);
  return launch_gemm_bn<256>(g, A, a_rows, lda, Bm, b_rows, ldb, st);
}

}  // namespace gmc
