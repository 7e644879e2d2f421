// The first (dense) round of the batched responsibility solver (Eq. (4)) over
// the whole GPU.  With S empty, b_m = 0 and the gains are the column sums of
// Cbar (computed while the clients were built).  Three kernels:
//   k_r0_pool   one block per image: the pool of the largest gains;
//   k_r0_rho    warp per client row: responsibilities over the pool, summed
//               into the scores in 64-bit fixed point (global atomics);
//   k_r0_filter warp per client row: the batch (top scores), the coverage
//               b_m = max over the batch, and the row's survivors
//               {i : Cbar_mi > b_m} compacted in place; the next round's gains
//               are summed in fixed point (global atomics).
// The next sparse_gpu_rounds() rounds run the same three steps over the survivor
// lists left in place by the previous round (row m: values Cbar[m][0..cnt_m),
// tokens scol[m][0..cnt_m), ascending):
//   k_rg_pool   the pool of the current gains among the unselected tokens;
//   k_rg_rho    warp per row: the row's pool entries are found through a
//               token -> pool slot table; pool tokens without a survivor in
//               the row have R = 0 and still count in its softmax denominator;
//   k_rg_filter warp per row: batch, coverage over the batch's entries, the
//               survivors compacted in place, the next gains.
// While many survivors remain, a whole-GPU round is cheaper than a round of
// the cluster kernel (16 SMs).  Every reduction is an integer sum, so the
// result does not depend on the order blocks run in.  The cluster kernel
// (k_select) continues from the first round not done here; info[b] carries the
// pool size, the tokens selected so far and the rounds done.
#include "common.cuh"
#include "kernels.cuh"
#include "select_common.cuh"

namespace gmc {

namespace {
// Threads of a sparse round's pool block: a turn takes four tokens a thread.  1,024
// above N = 2,048 (a second turn costs more than the wider barriers).
constexpr int POOL_THREADS = 1024;
int pool_threads(int N) { return N > 2048 ? POOL_THREADS : POOL_THREADS / 2; }

// The responsibility and filter kernels have ROWS warps a block (a template
// parameter: 16 for one image, 8 for a batch) and take `rpw` consecutive rows per
// warp.  Every block pays for tables of N tokens, and the filters end with a global
// addition per touched token, so a batch takes more rows per block; the next row
// is loaded while one is worked on.  At most eight: with 32 the images of a ragged
// batch that have the most rows ran alone at the end.
int rows_per_warp(int B, int M, int rows) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      sms = 152;
    }
  }
  const long long rpw = (long long)B * M / ((long long)rows * 4 * sms);
  return rpw < 1 ? 1 : (rpw > 8 ? 8 : (int)rpw);
}

// The first 64 entries of a row's survivor list, loaded ahead of their use by the
// kernels with several rows per warp (a batch).  With one row per warp there is
// nothing to load ahead of, and the registers cost a block per SM (document page:
// the eight responsibility launches 71 us without, 91 us with them).
template <bool AHEAD>
struct RowHead {
  static constexpr int U = AHEAD ? 2 : 0;
  int j[2];
  float v[2];
  __device__ __forceinline__ void load(const float* vals, const uint16_t* cols, int n, int lane) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = 32 * u + lane;
      j[u] = e < n ? (int)cols[e] : -1;
      v[u] = e < n ? vals[e] : 0.f;
    }
  }
};
}  // namespace

__global__ void __launch_bounds__(512) k_r0_pool(const long long* __restrict__ u0, int B, int N,
                                                   int P, const int32_t* toff, int Tmax, int I,
                                                   int32_t* pool0, int32_t* info, long long* s0,
                                                   long long* u1, long long* fv, uint32_t* status,
                                                   TraceView tv) {
  grid_dep_wait();
  extern __shared__ __align__(16) char sm_r0p[];
  const int b = blockIdx.x;
  // the accumulators of the next two kernels start at zero; nothing selected yet
  for (int k = threadIdx.x; k < P; k += blockDim.x) s0[(size_t)b * P + k] = 0;
  for (int j = threadIdx.x; j < N; j += blockDim.x) u1[(size_t)b * N + j] = 0;
  if (threadIdx.x < 4) fv[(size_t)b * 4 + threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    info[b * INFO_W + 1] = 0;
    info[b * INFO_W + 2] = 0;
    info[b * INFO_W + 3] = 0;
    info[b * INFO_W + 4] = 0;
    info[b * INFO_W + 5] = -1;  // boundary bucket of the last pool: none yet
  }
  if (toff && text_geom(toff, b, B, Tmax, nullptr).T == 0) {
    if (threadIdx.x == 0) info[b * INFO_W] = 0;
    return;
  }
  sel::PoolScratch w{};  // gains in shared memory: no boundary staging
  char* p = sm_r0p;
  long long* ug = reinterpret_cast<long long*>(p);  p += sizeof(long long) * (size_t)N;
  w.hist = reinterpret_cast<int*>(p);       p += sizeof(int) * sel::HBINS;
  w.bnd = reinterpret_cast<int*>(p);        p += sizeof(int) * N;
  w.wsum = reinterpret_cast<int*>(p);       p += sizeof(int) * 32;
  w.scal = reinterpret_cast<int*>(p);       p += sizeof(int) * 8;
  w.coarse = reinterpret_cast<int*>(p);     p += sizeof(int) * sel::CBINS;
  int* pool = reinterpret_cast<int*>(p);    p += sizeof(int) * P;
  w.key = reinterpret_cast<short*>(p);     p += sizeof(short) * (size_t)N;
  w.pk = reinterpret_cast<unsigned char*>(p); p += (size_t)N;
  unsigned char* selz = reinterpret_cast<unsigned char*>(p);
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    selz[j] = 0;
    ug[j] = u0[(size_t)b * N + j];  // the gains in shared memory: select_pool reads them often
    if (tv.base) tv.gains(b, 0, N)[j] = ug[j];
  }
  for (int h = threadIdx.x; h < sel::HBINS; h += blockDim.x) w.hist[h] = 0;
  if (threadIdx.x < sel::CBINS) w.coarse[threadIdx.x] = 0;
  __syncthreads();
  if (I > 1) {
    // several images: the first round only seeds S with each image's token of
    // largest singleton gain (ties to the lower index), one warp per image;
    // the filter takes them as its batch
    const int lane = threadIdx.x & 31, Ng = N / I;
    for (int k = threadIdx.x >> 5; k < I; k += blockDim.x >> 5) {
      long long bv = -1;
      int bj = 0x7fffffff;
      for (int j = k * Ng + lane; j < (k + 1) * Ng; j += 32)
        if (ug[j] > bv) {  // j ascending within a lane: the first maximum is kept
          bv = ug[j];
          bj = j;
        }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long ov = __shfl_xor_sync(FULL, bv, o);
        const int oj = __shfl_xor_sync(FULL, bj, o);
        if (ov > bv || (ov == bv && oj < bj)) {
          bv = ov;
          bj = oj;
        }
      }
      if (lane == 0) pool0[(size_t)b * P + k] = bj;
    }
    for (int k = I + threadIdx.x; k < P; k += blockDim.x) pool0[(size_t)b * P + k] = -1;
    if (threadIdx.x == 0) info[b * INFO_W] = I;
    return;
  }
  int bstar = -1;
  const int Pt = sel::select_pool(ug, selz, N, P, w, pool, nullptr, nullptr, &bstar);
  for (int k = threadIdx.x; k < P; k += blockDim.x) pool0[(size_t)b * P + k] = k < Pt ? pool[k] : -1;
  if (threadIdx.x == 0) {
    info[b * INFO_W] = Pt;
    info[b * INFO_W + 5] = bstar;
  }
}

// A lane keeps the sums of its pool slots in registers over the warp's rows; the
// warps are added in shared memory once (8 warps adding every row's 64 scores to
// the same shared words took a batch of 32 images 115 us, 108 us now).
template <int ROWS>
__global__ void __launch_bounds__(32 * ROWS) k_r0_rho(
    const float* __restrict__ C, int B, int N, int Mstride, int H, int L2, const int32_t* toff,
    int Tmax, int uniform_rows, const int32_t* __restrict__ pool0, const int32_t* __restrict__ info,
    int P, float resp_temp, float resp_eps, int fx_exp, const int32_t* fexp, int I, int rpw,
    long long* s0) {
  grid_dep_wait();
  if (I > 1) return;  // a seed round: no responsibilities
  constexpr int U = GMC_MAX_POOL / 32;
  __shared__ unsigned long long sblk[ROWS][GMC_MAX_POOL];
  const int b = blockIdx.y;
  const int Pt = info[b * INFO_W];
  if (Pt == 0) return;
  int Mb = Mstride;
  if (!uniform_rows) Mb = H * text_geom(toff, b, B, Tmax, nullptr).T + N + L2;
  const int m0 = blockIdx.x * ROWS * rpw;
  if (m0 >= Mb) return;
  const float fxs = ldexpf(1.f, fexp ? fexp[b] : fx_exp);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int pool[U];
  unsigned long long acc[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int k = lane + 32 * u;
    pool[u] = k < Pt ? pool0[(size_t)b * P + k] : -1;
    acc[u] = 0;
  }
  const int mw = m0 + w * rpw, nr = min(rpw, Mb - mw);  // this warp's rows
  const float* row = C + ((size_t)b * Mstride + mw) * N;
  float next[U];
#pragma unroll
  for (int u = 0; u < U; ++u) next[u] = nr > 0 && pool[u] >= 0 ? row[pool[u]] : 0.f;
  for (int ir = 0; ir < nr; ++ir) {
    float Rd[U];
    row += N;
#pragma unroll
    for (int u = 0; u < U; ++u) {  // b = 0: the residual is the client value
      Rd[u] = next[u];
      next[u] = ir + 1 < nr && pool[u] >= 0 ? row[pool[u]] : 0.f;
    }
    float rmax = 0.f;
    int npool = 0;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (Rd[u] > 0.f) { rmax = fmaxf(rmax, Rd[u]); ++npool; }
    rmax = warp_max(rmax);
    npool = warp_sum_int(npool);
    if (npool > 0) {
      // softmax of R / tau shifted by its largest logit rmax / tau: every
      // exponential is at most 1, whatever resp_temp
      const float tau = resp_temp * rmax + resp_eps;
      const float e0 = expf(-rmax / tau);  // a pool token with R = 0
      float ex[U], z = 0.f;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        ex[u] = Rd[u] > 0.f ? expf((Rd[u] - rmax) / tau) : 0.f;
        z += ex[u];
      }
      z = warp_sum(z) + (float)(Pt - npool) * e0;
      const float invz = 1.f / z;
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (Rd[u] > 0.f) acc[u] += (unsigned long long)to_fix(ex[u] * invz * Rd[u], fxs);
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) sblk[w][lane + 32 * u] = acc[u];
  __syncthreads();
  for (int k = threadIdx.x; k < Pt; k += blockDim.x) {
    unsigned long long v = 0;
#pragma unroll
    for (int q = 0; q < ROWS; ++q) v += sblk[q][k];
    if (v) atomicAdd((unsigned long long*)&s0[(size_t)b * P + k], v);
  }
}

template <int ROWS>
__global__ void __launch_bounds__(32 * ROWS) k_r0_filter(
    float* C, uint16_t* scol, int B, int N, int K, int Mstride, int H, int L2,
    const int32_t* toff, int Tmax, int uniform_rows, const int32_t* __restrict__ pool0,
    int32_t* info, const long long* __restrict__ s0, int P, int bsz, int fx_exp,
    const int32_t* fexp, long long* u1, float* bcov, int32_t* cnt, long long* fv,
    int32_t* order, int rpw, int I, TraceView tv) {
  grid_dep_wait();
  __shared__ int pool[GMC_MAX_POOL];
  __shared__ long long sc[GMC_MAX_POOL];
  __shared__ int batch[GMC_MAX_POOL];
  __shared__ long long fb[3];
  // the warps' tiles, then the block's contributions to the next gains (N <= 8,192),
  // one global addition per column at the end
  extern __shared__ float4 sm_r0f[];
  const int b = blockIdx.y;
  const int Pt = info[b * INFO_W];
  if (Pt == 0) return;
  int Mb = Mstride, MG = Mstride;
  if (!uniform_rows) {
    MG = H * text_geom(toff, b, B, Tmax, nullptr).T;
    Mb = MG + N + L2;
  }
  const int m0 = blockIdx.x * ROWS * rpw;
  if (m0 >= Mb) return;
  const float fxs = ldexpf(1.f, fexp ? fexp[b] : fx_exp);
  const int nb = I > 1 ? Pt : min(bsz, min(Pt, K));  // a seed round takes its whole pool
  for (int k = threadIdx.x; k < Pt; k += blockDim.x) {
    pool[k] = pool0[(size_t)b * P + k];
    sc[k] = s0[(size_t)b * P + k];
  }
  if (threadIdx.x < 3) fb[threadIdx.x] = 0;
  constexpr int TILE = sel::ROW_STEP / 4;
  const sel::GainSums<true> sums{reinterpret_cast<uint32_t*>(sm_r0f + ROWS * TILE), N};
  sums.clear();
  __syncthreads();
  {
    const int lane = threadIdx.x & 31, gl = lane & 7;
    const unsigned gm = 0xFFu << (lane & 24);
    for (int k = threadIdx.x >> 3; k < Pt; k += blockDim.x >> 3) {  // 8 lanes per pool token
      const int rank = I > 1 ? k : sel::group_score_rank(sc, pool, Pt, k, gl, gm);
      if (gl == 0 && rank < nb) batch[rank] = pool[k];
    }
  }
  __syncthreads();
  if (blockIdx.x == 0) {  // record the first batch once per image
    for (int q = threadIdx.x; q < nb; q += blockDim.x) order[(size_t)b * K + q] = batch[q];
    if (threadIdx.x == 0) {
      info[b * INFO_W + 1] = nb;  // selected so far
      info[b * INFO_W + 2] = 1;   // rounds done
    }
    if (tv.base) {
      int32_t* tp = tv.at<int32_t>(b, tv.off_pool);
      for (int k = threadIdx.x; k < tv.pool_size; k += blockDim.x) tp[k] = k < Pt ? pool[k] : -1;
      if (threadIdx.x == 0) tv.at<int32_t>(b, tv.off_round_end)[0] = nb;
    }
  }
  const int lane = threadIdx.x & 31;
  for (int ir = 0; ir < rpw; ++ir) {
    const int m = m0 + (threadIdx.x >> 5) * rpw + ir;
    if (m >= Mb) break;
    float* vals = C + ((size_t)b * Mstride + m) * N;
    uint16_t* cols = scol + ((size_t)b * Mstride + m) * N;
    float bnew = 0.f;
    for (int t = lane; t < nb; t += 32) bnew = fmaxf(bnew, vals[batch[t]]);
    bnew = warp_max(bnew);
    const long long fb_new = to_fix(bnew, fxs);
    float4* tile = sm_r0f + (threadIdx.x >> 5) * TILE;
    float rowmax = 0.f;  // only the trace reports F(V)
    const int w =
        tv.base ? sel::filter_dense_row<true, ROWS == 16>(vals, cols, N, bnew, fb_new, fxs, sums, tile, &rowmax)
                : sel::filter_dense_row<false, ROWS == 16>(vals, cols, N, bnew, fb_new, fxs, sums, tile, &rowmax);
    if (lane == 0) {
      bcov[(size_t)b * Mstride + m] = bnew;
      cnt[(size_t)b * Mstride + m] = w;
      if (tv.base) {
        const int bank = m < MG ? 0 : (m < MG + N ? 1 : 2);
        atomicAdd((unsigned long long*)&fb[bank], (unsigned long long)to_fix(rowmax, fxs));
        atomicAdd(tv.cover(b, 0), (unsigned long long)fb_new);  // F after the round
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < 3 && fb[threadIdx.x])
    atomicAdd((unsigned long long*)&fv[(size_t)b * 4 + threadIdx.x], (unsigned long long)fb[threadIdx.x]);
  sums.flush(reinterpret_cast<unsigned long long*>(u1 + (size_t)b * N), false);
}

// ---- sparse rounds on the whole GPU -------------------------------------------

// One block per image: a chain of memory round trips and barriers.  The gains are read
// once, into shared memory and into the buffer the filter adds its changes to, and
// nothing says which tokens are selected: their entries are all dead, so their gains are
// exactly zero and they are no candidates.  Two reads of the gains and one of the
// selected tokens took N = 1,296 7.0 us, 2,592 8.2, 4,096 9.4; now 6.7, 6.6 and 7.3.
__global__ void __launch_bounds__(POOL_THREADS, 1) k_rg_pool(const long long* __restrict__ ucur,
                                                          long long* unext, int B, int N, int K,
                                                          int P, const int32_t* toff, int Tmax,
                                                          int32_t* pool0, int32_t* info,
                                                          long long* sc, TraceView tv) {
  grid_dep_wait();
  extern __shared__ __align__(16) char sm_rgp[];
  const int b = blockIdx.x;
  const int S = info[b * INFO_W + 1], rd = info[b * INFO_W + 2];
  int hint = info[b * INFO_W + 5];
  for (int k = threadIdx.x; k < P; k += blockDim.x) sc[(size_t)b * P + k] = 0;
  // the next gains start from these: the filter adds only the changes of the
  // rows whose coverage grows
  const long long* ub = ucur + (size_t)b * N;
  long long* un = unext + (size_t)b * N;
  // nothing to do here once the budget is met or when the first round found
  // no gain: the cluster kernel handles those cases
  const bool skip = (toff && text_geom(toff, b, B, Tmax, nullptr).T == 0) || rd == 0 || S >= K;
  if (skip) {
    for (int j = threadIdx.x; j < N; j += blockDim.x) un[j] = ub[j];
    if (threadIdx.x == 0) info[b * INFO_W] = 0;
    return;
  }
  sel::PoolScratch w{};  // gains in shared memory: no boundary staging
  char* p = sm_rgp;
  sel::WindowScratch ws;
  ws.win = reinterpret_cast<int*>(p);       p += sizeof(int) * (sel::WBINS + 4);
  ws.cu = reinterpret_cast<long long*>(p);  p += sizeof(long long) * sel::WCAP;
  ws.cj = reinterpret_cast<int*>(p);        p += sizeof(int) * sel::WCAP;
  long long* ug = reinterpret_cast<long long*>(p);  p += sizeof(long long) * (size_t)N;
  w.hist = reinterpret_cast<int*>(p);       p += sizeof(int) * sel::HBINS;
  w.bnd = reinterpret_cast<int*>(p);        p += sizeof(int) * N;
  w.wsum = reinterpret_cast<int*>(p);       p += sizeof(int) * 32;
  w.scal = reinterpret_cast<int*>(p);       p += sizeof(int) * 8;
  w.coarse = reinterpret_cast<int*>(p);     p += sizeof(int) * sel::CBINS;
  int* pool = reinterpret_cast<int*>(p);    p += sizeof(int) * P;
  w.key = reinterpret_cast<short*>(p);     p += sizeof(short) * (size_t)N;
  w.pk = reinterpret_cast<unsigned char*>(p); p += (size_t)N;
  unsigned char* none = reinterpret_cast<unsigned char*>(p);
  // the gains in shared memory (select_pool reads them often): copied here
  // without a boundary hint, else by the window pool's first pass
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    none[j] = 0;
    if (hint < 0) un[j] = ug[j] = ub[j];
  }
  for (int h = threadIdx.x; h < sel::HBINS; h += blockDim.x) w.hist[h] = 0;
  if (threadIdx.x < sel::CBINS) w.coarse[threadIdx.x] = 0;
  for (int q = threadIdx.x; q < sel::WBINS + 4; q += blockDim.x) ws.win[q] = 0;
  __syncthreads();
  int Pt = sel::select_pool_window([&](int j) { return un[j] = ub[j]; }, ug, none, N, P, ws, pool,
                                   nullptr, &hint);
  if (Pt < 0) Pt = sel::select_pool(ug, none, N, P, w, pool, nullptr, nullptr, &hint);
  if (tv.base)
    for (int j = threadIdx.x; j < N; j += blockDim.x) tv.gains(b, rd, N)[j] = ug[j];
  for (int k = threadIdx.x; k < P; k += blockDim.x) pool0[(size_t)b * P + k] = k < Pt ? pool[k] : -1;
  if (threadIdx.x == 0) {
    info[b * INFO_W + 5] = hint;
    info[b * INFO_W] = Pt;
    info[b * INFO_W + 3] = S;
    info[b * INFO_W + 4] = rd;
  }
  if (tv.base && Pt > 0) {
    int32_t* tp = tv.at<int32_t>(b, tv.off_pool) + (size_t)rd * tv.pool_size;
    for (int k = threadIdx.x; k < tv.pool_size; k += blockDim.x) tp[k] = k < Pt ? pool[k] : -1;
  }
}

template <int ROWS>
__global__ void __launch_bounds__(32 * ROWS, ROWS == 16 ? 4 : 5) k_rg_rho(
    const float* __restrict__ C, const uint16_t* __restrict__ scol,
    const float* __restrict__ bcov, const int32_t* __restrict__ cnt, int B, int N, int Mstride,
    int H, int L2, const int32_t* toff, int Tmax, int uniform_rows,
    const int32_t* __restrict__ pool0, const int32_t* __restrict__ info, int P, float resp_temp,
    float resp_eps, int fx_exp, const int32_t* fexp, int rpw, long long* sc) {
  grid_dep_wait();
  __shared__ uint32_t sblk[3 * GMC_MAX_POOL];  // limbs: at most ROWS * rpw additions per slot
  __shared__ int fslot[ROWS][GMC_MAX_POOL];  // a row's pool entries: slot and residual
  __shared__ float fres[ROWS][GMC_MAX_POOL];
  extern __shared__ short pslot[];              // [N] pool slot of every token or -1
  const int b = blockIdx.y;
  const int Pt = info[b * INFO_W];
  if (Pt == 0) return;
  int Mb = Mstride;
  if (!uniform_rows) Mb = H * text_geom(toff, b, B, Tmax, nullptr).T + N + L2;
  const int m0 = blockIdx.x * ROWS * rpw;
  if (m0 >= Mb) return;
  const float fxs = ldexpf(1.f, fexp ? fexp[b] : fx_exp);
  for (int j = threadIdx.x; j < N; j += blockDim.x) pslot[j] = -1;
  for (int k = threadIdx.x; k < 3 * GMC_MAX_POOL; k += blockDim.x) sblk[k] = 0;
  __syncthreads();
  for (int k = threadIdx.x; k < Pt; k += blockDim.x) pslot[pool0[(size_t)b * P + k]] = (short)k;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int mw = m0 + w * rpw, nr = min(rpw, Mb - mw);  // this warp's rows (rpw <= 32)
  const size_t row0 = (size_t)b * Mstride + mw;
  constexpr bool AHEAD = ROWS == 8;
  using Head = RowHead<AHEAD>;
  Head next;
  int cnts = 0;  // AHEAD: the rows' counts and coverages, one per lane
  float covs = 0.f;
  if constexpr (AHEAD) {
    if (lane < nr) {
      cnts = cnt[row0 + lane];
      covs = bcov[row0 + lane];
    }
    next.load(C + row0 * N, scol + row0 * N, __shfl_sync(FULL, cnts, 0), lane);
  }
  const unsigned lt = sel::lanemask_lt();
  for (int ir = 0; ir < nr; ++ir) {
    const size_t row = row0 + ir;
    const int n = AHEAD ? __shfl_sync(FULL, cnts, ir) : cnt[row];
    const float bm = AHEAD ? __shfl_sync(FULL, covs, ir) : bcov[row];
    const float* vals = C + row * N;
    const uint16_t* cols = scol + row * N;
    const Head head = next;
    if constexpr (AHEAD) {
      const int n1 = __shfl_sync(FULL, cnts, min(ir + 1, 31));
      next.load(vals + N, cols + N, ir + 1 < nr ? n1 : 0, lane);
    }
    int nf = 0;
    float rmax = 0.f;
    auto take = [&](int ps, float R) {  // a pool entry of the row: its slot and residual
      const unsigned bal = __ballot_sync(FULL, ps >= 0);
      if (ps >= 0) {
        const int at = nf + __popc(bal & lt);
        fslot[w][at] = ps;
        fres[w][at] = R;
        rmax = fmaxf(rmax, R);
      }
      nf += __popc(bal);
    };
#pragma unroll
    for (int u = 0; u < Head::U; ++u)
      if (32 * u < n) take(head.j[u] >= 0 ? (int)pslot[head.j[u]] : -1, head.v[u] - bm);
    constexpr int RU = 4;  // chunks of 32 entries whose loads are in flight together
    for (int e00 = 32 * Head::U; e00 < n; e00 += 32 * RU) {
      int ps[RU];
      float R[RU];
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        const int e = e00 + 32 * u + lane;
        ps[u] = e < n ? (int)cols[e] : -1;
      }
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        if (ps[u] >= 0) ps[u] = pslot[ps[u]];
        R[u] = ps[u] >= 0 ? vals[e00 + 32 * u + lane] - bm : 0.f;  // > 0: exceeds its coverage
      }
#pragma unroll
      for (int u = 0; u < RU; ++u) take(ps[u], R[u]);
    }
    rmax = warp_max(rmax);
    __syncwarp();
    if (nf > 0) {
      // softmax shifted by the largest logit (exponentials at most 1)
      const float tau = resp_temp * rmax + resp_eps;
      const float e0 = expf(-rmax / tau);  // pool tokens without a survivor here: R = 0
      float z = 0.f;
      for (int q = lane; q < nf; q += 32) z += expf((fres[w][q] - rmax) / tau);
      z = warp_sum(z) + (float)(Pt - nf) * e0;
      const float invz = 1.f / z;
      for (int q = lane; q < nf; q += 32) {
        const float R = fres[w][q];
        sel::limb_add(&sblk[fslot[w][q]], GMC_MAX_POOL,
                      (unsigned long long)to_fix(expf((R - rmax) / tau) * invz * R, fxs));
      }
      __syncwarp();  // the next row refills the warp's entries
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < Pt; k += blockDim.x) {
    const unsigned long long v = sel::limb_value(sblk + k, GMC_MAX_POOL);
    if (v) atomicAdd((unsigned long long*)&sc[(size_t)b * P + k], v);
  }
}

template <int ROWS>
__global__ void __launch_bounds__(32 * ROWS, ROWS == 16 ? 3 : 4) k_rg_filter(
    float* C, uint16_t* scol, int B, int N, int K, int Mstride, int H, int L2,
    const int32_t* toff, int Tmax, int uniform_rows, const int32_t* __restrict__ pool0,
    int32_t* info, const long long* __restrict__ sc0, int P, int bsz, int fx_exp,
    const int32_t* fexp, long long* unext, float* bcov, int32_t* cnt, int32_t* order, int rpw,
    TraceView tv) {
  grid_dep_wait();
  __shared__ int pool[GMC_MAX_POOL];
  __shared__ long long sc[GMC_MAX_POOL];
  __shared__ int batch[GMC_MAX_POOL];
  extern __shared__ __align__(16) char sm_rgf[];  // the falls of the gains, then the batch flags [N]
  const sel::GainSums<true> sums{reinterpret_cast<uint32_t*>(sm_rgf), N};
  unsigned char* inb = reinterpret_cast<unsigned char*>(sm_rgf) + sel::gain_sums_bytes<true>(N);
  const int b = blockIdx.y;
  const int Pt = info[b * INFO_W];
  if (Pt == 0) return;
  int Mb = Mstride;
  if (!uniform_rows) Mb = H * text_geom(toff, b, B, Tmax, nullptr).T + N + L2;
  const int m0 = blockIdx.x * ROWS * rpw;
  if (m0 >= Mb) return;
  const int S = info[b * INFO_W + 3], rd = info[b * INFO_W + 4];
  const float fxs = ldexpf(1.f, fexp ? fexp[b] : fx_exp);
  const int nb = min(bsz, min(Pt, K - S));
  for (int k = threadIdx.x; k < Pt; k += blockDim.x) {
    pool[k] = pool0[(size_t)b * P + k];
    sc[k] = sc0[(size_t)b * P + k];
  }
  sums.clear();
  for (int j = threadIdx.x; j < N; j += blockDim.x) inb[j] = 0;
  __syncthreads();
  {
    const int lane = threadIdx.x & 31, gl = lane & 7;
    const unsigned gm = 0xFFu << (lane & 24);
    for (int k = threadIdx.x >> 3; k < Pt; k += blockDim.x >> 3) {  // 8 lanes per pool token
      const int rank = sel::group_score_rank(sc, pool, Pt, k, gl, gm);
      if (gl == 0 && rank < nb) batch[rank] = pool[k];
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < nb; q += blockDim.x) inb[batch[q]] = 1;
  if (blockIdx.x == 0) {  // record the batch once per image
    for (int q = threadIdx.x; q < nb; q += blockDim.x) order[(size_t)b * K + S + q] = batch[q];
    if (threadIdx.x == 0) {
      info[b * INFO_W + 1] = S + nb;
      info[b * INFO_W + 2] = rd + 1;
      if (tv.base) tv.at<int32_t>(b, tv.off_round_end)[rd] = S + nb;
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int mw = m0 + (threadIdx.x >> 5) * rpw, nr = min(rpw, Mb - mw);  // this warp's rows
  const size_t row0 = (size_t)b * Mstride + mw;
  constexpr bool AHEAD = ROWS == 8;
  using Head = RowHead<AHEAD>;
  Head next;
  int cnts = 0;  // AHEAD: the rows' counts and coverages, one per lane
  float covs = 0.f;
  if constexpr (AHEAD) {
    if (lane < nr) {
      cnts = cnt[row0 + lane];
      covs = bcov[row0 + lane];
    }
    next.load(C + row0 * N, scol + row0 * N, __shfl_sync(FULL, cnts, 0), lane);
  }
  const unsigned lt = sel::lanemask_lt();
  for (int ir = 0; ir < nr; ++ir) {
    const size_t row = row0 + ir;
    const int n = AHEAD ? __shfl_sync(FULL, cnts, ir) : cnt[row];
    const float bold = AHEAD ? __shfl_sync(FULL, covs, ir) : bcov[row];
    float* vals = C + row * N;
    uint16_t* cols = scol + row * N;
    const Head head = next;
    if constexpr (AHEAD) {
      const int n1 = __shfl_sync(FULL, cnts, min(ir + 1, 31));
      next.load(vals + N, cols + N, ir + 1 < nr ? n1 : 0, lane);
    }
    // The list is walked FU chunks of 32 entries at a time, every load of the
    // chunks issued before the first use (and, below, before any survivor is
    // written back in place: a chunk's survivors land below its end).
    constexpr int FU = 4;
    float bnew = bold;
#pragma unroll
    for (int u = 0; u < Head::U; ++u)
      if (head.j[u] >= 0 && inb[head.j[u]]) bnew = fmaxf(bnew, head.v[u]);
    for (int e00 = 32 * Head::U; e00 < n; e00 += 32 * FU) {
      int jj[FU];
#pragma unroll
      for (int u = 0; u < FU; ++u) {
        const int e = e00 + 32 * u + lane;
        jj[u] = e < n ? (int)cols[e] : -1;
      }
#pragma unroll
      for (int u = 0; u < FU; ++u)
        if (jj[u] >= 0 && inb[jj[u]]) bnew = fmaxf(bnew, vals[e00 + 32 * u + lane]);
    }
    bnew = warp_max(bnew);
    const long long fb_new = to_fix(bnew, fxs);
    if (!(bnew > bold)) {  // no batch entry above the coverage: row and gains unchanged
      if (lane == 0 && tv.base) atomicAdd(tv.cover(b, rd), (unsigned long long)fb_new);
      continue;
    }
    const long long fb_old = to_fix(bold, fxs);
    int wr = 0;
    // an entry's residual moves from C - b_old to C - b_new, or to zero (exact:
    // integers modulo 2^64); survivors move down in order
    auto settle = [&](bool in, int j, float c) {
      const bool keep = in && c > bnew;
      const unsigned bal = __ballot_sync(FULL, keep);
      if (in) sums.add(j, (unsigned long long)((keep ? fb_new : to_fix(c, fxs)) - fb_old));
      if (keep) {
        const int pos = wr + __popc(bal & lt);
        vals[pos] = c;
        cols[pos] = (uint16_t)j;
      }
      wr += __popc(bal);
    };
#pragma unroll
    for (int u = 0; u < Head::U; ++u)
      if (32 * u < n) settle(head.j[u] >= 0, head.j[u], head.v[u]);
    for (int e00 = 32 * Head::U; e00 < n; e00 += 32 * FU) {
      float cc[FU];
      int jj[FU];
#pragma unroll
      for (int u = 0; u < FU; ++u) {
        const int e = e00 + 32 * u + lane;
        cc[u] = 0.f;
        jj[u] = 0;
        if (e < n) {
          cc[u] = vals[e];
          jj[u] = cols[e];
        }
      }
      __syncwarp();  // the chunks are read before any survivor moves down into them
#pragma unroll
      for (int u = 0; u < FU; ++u) settle(e00 + 32 * u + lane < n, jj[u], cc[u]);
    }
    if (lane == 0) {
      bcov[row] = bnew;
      cnt[row] = wr;
      if (tv.base) atomicAdd(tv.cover(b, rd), (unsigned long long)fb_new);  // F after the round
    }
  }
  __syncthreads();
  sums.flush(reinterpret_cast<unsigned long long*>(unext + (size_t)b * N), true);
}

// The responsibility and filter launches of every whole-GPU round, ROWS warps per block.
template <int ROWS>
static cudaError_t launch_rounds_rows(const R0State& r0, int B, int N, int K, int M,
                                      const int32_t* toff, int H, int T, int L2,
                                      const gmc_params& p, int fx_exp, const int32_t* fexp,
                                      float* C, uint16_t* scol, int32_t* order, const TraceView& tv,
                                      cudaStream_t st, int I, size_t smem) {
  const int P = p.pool_mult * p.batch_b;
  const int uniform = (H == 0);
  cudaError_t e;
  const int rpw = rows_per_warp(B, M, ROWS);
  const dim3 grid(ceil_div(M, ROWS * rpw), B);
  launch_k(k_r0_rho<ROWS>, grid, 32 * ROWS, 0, st, 1, C, B, N, M, H, L2, toff, T, uniform, r0.pool,
           r0.info, P, p.resp_temp, p.resp_eps, fx_exp, fexp, I, rpw, r0.s0);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t fsm = sizeof(float) * ROWS * sel::ROW_STEP + sel::gain_sums_bytes<true>(N);
  if ((e = set_smem_limit((const void*)k_r0_filter<ROWS>, fsm)) != cudaSuccess) return e;
  launch_k(k_r0_filter<ROWS>, grid, 32 * ROWS, fsm, st, 1, C, scol, B, N, K, M, H, L2, toff,
           T, uniform, r0.pool, r0.info, r0.s0, P, p.batch_b, fx_exp, fexp, r0.u1, r0.bcov, r0.cnt,
           r0.fv, order, rpw, I, tv);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // sparse rounds: gains alternate between u1 and u2
  // the pool kernel's layout is round 0's after the window scratch
  const size_t psm = smem + sizeof(int) * (sel::WBINS + 4) + 12 * (size_t)sel::WCAP;
  if ((e = set_smem_limit((const void*)k_rg_pool, psm)) != cudaSuccess) return e;
  const size_t rsm = sizeof(short) * (size_t)N;
  if ((e = set_smem_limit((const void*)k_rg_rho<ROWS>, rsm)) != cudaSuccess) return e;
  const size_t gsm = sel::gain_sums_bytes<true>(N) + (size_t)N;
  if ((e = set_smem_limit((const void*)k_rg_filter<ROWS>, gsm)) != cudaSuccess) return e;
  const int rounds = sparse_gpu_rounds(B, N, M, H, T, L2, p, K, I);
  for (int rr = 1; rr <= rounds; ++rr) {
    long long* ucur = rr % 2 == 1 ? r0.u1 : r0.u2;
    long long* unext = rr % 2 == 1 ? r0.u2 : r0.u1;
    launch_k(k_rg_pool, B, pool_threads(N), psm, st, 1, (const long long*)ucur, unext, B, N, K, P,
             uniform ? nullptr : toff, T, r0.pool, r0.info, r0.s0, tv);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_k(k_rg_rho<ROWS>, grid, 32 * ROWS, rsm, st, 1, (const float*)C, (const uint16_t*)scol,
             (const float*)r0.bcov, (const int32_t*)r0.cnt, B, N, M, H, L2, toff, T, uniform,
             (const int32_t*)r0.pool, (const int32_t*)r0.info, P, p.resp_temp, p.resp_eps, fx_exp,
             fexp, rpw, r0.s0);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_k(k_rg_filter<ROWS>, grid, 32 * ROWS, gsm, st, 1, C, scol, B, N, K, M, H, L2, toff,
             T, uniform, (const int32_t*)r0.pool, r0.info, (const long long*)r0.s0, P, p.batch_b,
             fx_exp, fexp, unext, r0.bcov, r0.cnt, order, rpw, tv);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_round0(R0State& r0, int B, int N, int K, int M, const int32_t* toff,
                          int H, int T, int L2, const gmc_params& p, int fx_exp,
                          const int32_t* fexp, float* C, uint16_t* scol, const long long* u0,
                          int32_t* order, uint32_t* status, const TraceView& tv,
                          cudaStream_t st, int I) {
  const int P = p.pool_mult * p.batch_b;
  r0.ugain = sparse_gpu_rounds(B, N, M, H, T, L2, p, K, I) % 2 == 0 ? r0.u1 : r0.u2;
  cudaError_t e;
  const size_t smem =
      sizeof(long long) * (size_t)N + sizeof(int) * (sel::HBINS + N + 32 + 8 + sel::CBINS + P) +
      4 * (size_t)N + 64;
  if ((e = set_smem_limit((const void*)k_r0_pool, smem)) != cudaSuccess) return e;
  const int uniform = (H == 0);
  launch_k(k_r0_pool, B, 512, smem, st, 1, u0, B, N, P, uniform ? nullptr : toff, T, I, r0.pool, r0.info,
                                  r0.s0, r0.u1, r0.fv, status, tv);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // one image: 16 warps per block (fewer, larger blocks finish the rounds sooner); a
  // batch: 8
  return (B == 1 ? launch_rounds_rows<16> : launch_rounds_rows<8>)(
      r0, B, N, K, M, toff, H, T, L2, p, fx_exp, fexp, C, scol, order, tv, st, I, smem);
}

}  // namespace gmc
