// Wide selection: the batched responsibility solver (Sec. 3.3, Eq. (4);
// appendix Eq. (cond-responsibility) and its totality rule) with every round
// on the whole GPU, for candidate pools above GMC_MAX_POOL and visual counts
// above GMC_MAX_N: the long-prefix path (b = 512, pool 4b = 2048, N = 15,876;
// Table "Shared GMC configuration", long-prefix row), whose gains the paper
// evaluates in chunks over the whole M x N client matrix.
//
// Round t (support S_t, coverage b_m = max_{j in S_t} Cbar_mj, 0 for S empty):
//   R_mi = [Cbar_mi - b_m]_+,  u_i = sum_m R_mi
//   pool = the min(4b, #{u_i > 0}) unselected tokens of largest u (ties: lower index)
//   rho_m. = softmax over the pool of R_m. / (resp_temp * max_pool R_m. + resp_eps)
//   s_i = sum_m rho_mi R_mi; the top min(b, |pool|, K - |S|) pool tokens by s
//   enter S (ties: lower index); an empty pool fills the budget in ascending
//   index order.
// Four kernels per round:
//   k_w_pool    one block per image: the pool of the current gains (the
//               histogram selection of select_common.cuh, gains read from
//               global memory);
//   k_w_rho     the rows' responsibilities over the pool, summed into the scores
//               in 64-bit fixed point: k_w_rho_dense in the first round (a block
//               per row at a time), then a warp per row that walks its survivor
//               list three times (max, normaliser, scores: the temperature
//               depends on the row's max);
//   k_w_batch   one block per image: the best of the pool by (score desc, token
//               asc), found as the pool is; a bitonic sort where fewer than a
//               batch of them have a positive score;
//   k_w_filter  warp per client row: the new coverage b_m, the row's
//               survivors {i : Cbar_mi > b_m} compacted in place (values over
//               Cbar, tokens in scol), the next round's gains summed per block
//               in shared memory and added with one 64-bit atomic per column.
// Entries with Cbar_mi <= b_m have zero residual for the rest of the solve, so
// dropping them is exact.  Every sum is an integer (fixed point), so the
// result does not depend on the order blocks run in.  ceil(K / b) rounds are
// launched; a round whose pool is empty, or that starts with the budget met,
// does nothing.  k_w_final then fills the budget in ascending order if needed,
// writes the ascending support and the diagnostics.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "select_common.cuh"

namespace gmc {

namespace {
constexpr int DTHREADS = 512; // threads of a block of the dense responsibilities
constexpr int DROWS = 3;      // client rows it has in shared memory
constexpr int SROWS = 16;     // warps (client rows) per block of the later rounds'
constexpr int FROWS = 32;     // most warps of a filter block (one block per SM: the next gains
                              // of N tokens take 8 N bytes of shared memory)
constexpr int WP_THREADS = 1024;
constexpr int W_BCAP = 4096;  // boundary-bucket gains the pool kernel stages in shared memory

// Rows of image b: grounded [0, MG), appearance [MG, MG + MV), spatial after;
// 0 rows for an image whose text offsets are invalid.
__device__ __forceinline__ int wide_rows(const WideGeom& g, int b, int* MG) {
  if (g.uniform) {
    *MG = g.Mstride;
    return g.Mstride;
  }
  const TextGeom tg = text_geom(g.toff, b, g.B, g.Tmax, nullptr);
  if (tg.T == 0) {
    *MG = 0;
    return 0;
  }
  *MG = g.HV * tg.T;
  return *MG + g.MV + g.L2;
}

__device__ __forceinline__ int bank_of(int m, int MG, int MV) {
  return m < MG ? 0 : (m < MG + MV ? 1 : 2);
}

// gains read and written by round rnd: round 0 reads the column sums u0
__device__ __forceinline__ const long long* gains_in(const WideState& w, const long long* u0,
                                                     int rnd) {
  return rnd == 0 ? u0 : (rnd % 2 == 1 ? w.u1 : w.u2);
}
__device__ __forceinline__ long long* gains_out(const WideState& w, int rnd) {
  return rnd % 2 == 0 ? w.u1 : w.u2;
}
}  // namespace

// ---- pool ------------------------------------------------------------------------
// WIN: pools of at most WCAP / 2 tokens take the window pool (the boundary
// bucket of a round lies at or below the last one), with the gains staged in
// shared memory; the full histogram pool runs in round 0, when the window
// misses, and for larger pools (a separate instance, without the window's
// registers).  One block, bound by its chain of memory round trips, shared-memory
// additions and barriers: P = 2,048 of N = 15,876 took 30 us a round with a sorted
// boundary bucket, exponents matched across warps and a list of the selected
// tokens; 18 without.
template <bool WIN>
__global__ void __launch_bounds__(WP_THREADS, 1) k_w_pool(WideState w, WideGeom g, int P, int rnd,
                                                       const long long* __restrict__ u0,
                                                       TraceView tv) {
  constexpr bool win = WIN;
  grid_dep_wait();
  extern __shared__ __align__(16) char sm_wp[];
  const int b = blockIdx.x, N = g.N, K = g.K;
  const long long* ucur = gains_in(w, u0, rnd) + (size_t)b * N;
  long long* unext = gains_out(w, rnd) + (size_t)b * N;
  int32_t* info = w.info + b * INFO_W;
  // the scores and next gains of this round start at zero
  for (int k = threadIdx.x; k < P; k += blockDim.x) w.sc[(size_t)b * P + k] = 0;
  for (int j = threadIdx.x; j < N; j += blockDim.x) unext[j] = 0;
  if (rnd == 0) {
    for (int j = threadIdx.x; j < N; j += blockDim.x) w.stamp[(size_t)b * N + j] = 0;
    if (threadIdx.x < 4) w.fv[(size_t)b * 4 + threadIdx.x] = 0;
  }
  int MG;
  const int Mb = wide_rows(g, b, &MG);
  const int S = rnd == 0 ? 0 : info[1], rd = rnd == 0 ? 0 : info[2];
  int hint = rnd == 0 || !win ? -1 : info[5];  // the last round's boundary bucket
  __syncthreads();  // every thread has read info before thread 0 rewrites it
  if (rnd == 0 && threadIdx.x == 0) {
    info[1] = 0;
    info[2] = 0;
  }
  // nothing to do once the budget is met, after a round with an empty pool,
  // or for an invalid image
  if (Mb == 0 || S >= K || rd < rnd) {
    if (threadIdx.x == 0) info[0] = 0;
    return;
  }
  sel::PoolScratch ps;
  char* p = sm_wp;
  sel::WindowScratch ws{};
  long long* ug = nullptr;  // win: the gains, staged for the pool's passes
  if (win) {  // first, where its 16-byte loads are aligned whatever N is
    ws.win = reinterpret_cast<int*>(p);       p += sizeof(int) * (sel::WBINS + 4);
    ws.cu = reinterpret_cast<long long*>(p);  p += sizeof(long long) * sel::WCAP;
    ws.cj = reinterpret_cast<int*>(p);        p += sizeof(int) * sel::WCAP;
    ug = reinterpret_cast<long long*>(p);     p += sizeof(long long) * (size_t)N;
    for (int q = threadIdx.x; q < sel::WBINS + 4; q += blockDim.x) ws.win[q] = 0;
  }
  ps.hist = reinterpret_cast<int*>(p);       p += sizeof(int) * sel::HBINS;
  ps.bnd = reinterpret_cast<int*>(p);        p += sizeof(int) * (size_t)N;
  ps.wsum = reinterpret_cast<int*>(p);       p += sizeof(int) * 32;
  ps.scal = reinterpret_cast<int*>(p);       p += sizeof(int) * 8;
  ps.coarse = reinterpret_cast<int*>(p);     p += sizeof(int) * sel::CBINS;
  int* pool = reinterpret_cast<int*>(p);     p += sizeof(int) * (size_t)P;
  ps.key = reinterpret_cast<short*>(p);      p += sizeof(short) * (size_t)N;
  ps.pk = reinterpret_cast<unsigned char*>(p); p += (size_t)N;
  unsigned char* none = reinterpret_cast<unsigned char*>(p); p += (size_t)N;
  p = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(p) + 15) & ~static_cast<uintptr_t>(15));
  ps.bval = reinterpret_cast<long long*>(p);  // the boundary bucket's gains
  ps.bcap = min(N, W_BCAP);
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    none[j] = 0;
    if (tv.base) tv.gains(b, rd, N)[j] = ucur[j];
    if (win && hint < 0) ug[j] = ucur[j];  // else the window pool's first pass stages them
  }
  for (int h = threadIdx.x; h < sel::HBINS; h += blockDim.x) ps.hist[h] = 0;
  if (threadIdx.x < sel::CBINS) ps.coarse[threadIdx.x] = 0;
  __syncthreads();
  int Pt = -1;  // a selected token's entries are all dead and its gain exactly zero
  if constexpr (WIN)
    Pt = sel::select_pool_window([&](int j) { return ucur[j]; }, ug, none, N, P, ws, pool, nullptr,
                                 &hint);
  if (Pt < 0) Pt = sel::select_pool<true>(win ? ug : ucur, none, N, P, ps, pool, nullptr, nullptr, &hint);
  for (int k = threadIdx.x; k < P; k += blockDim.x) w.pool[(size_t)b * P + k] = k < Pt ? pool[k] : -1;
  if (threadIdx.x == 0) {
    info[0] = Pt;
    info[3] = S;
    info[4] = rd;
    info[5] = hint;
  }
  if (tv.base && Pt > 0) {
    int32_t* tp = tv.at<int32_t>(b, tv.off_pool) + (size_t)rd * tv.pool_size;
    for (int k = threadIdx.x; k < tv.pool_size; k += blockDim.x) tp[k] = k < Pt ? pool[k] : -1;
  }
}

// ---- responsibilities ----------------------------------------------------------------
// The dense first round (b = 0: a residual is the client value): one block an SM,
// whole rows one after another.  A row comes to shared memory as it lies, DROWS - 1
// rows ahead (the pool is one token in eight, so its values touch two sectors in
// three: gathering them took as much memory traffic and many more requests); each
// thread then keeps its SLOTS pool slots in registers, values, exponentials and sums,
// so an exponential is taken once and the sums meet nobody until the end.  Bound by
// reading the rows: 7,936 of 15,876 values, P = 2,048: a warp a row, gathering, with
// 64-bit shared-memory additions 193 us, now 124 (4.1 TB/s).
template <int SLOTS, bool VEC>
__global__ void __launch_bounds__(DTHREADS, 1) k_w_rho_dense(WideState w, WideGeom g, int P,
                                                             const float* __restrict__ C,
                                                             float resp_temp, float resp_eps,
                                                             int fx_exp, const int32_t* fexp) {
  grid_dep_wait();
  extern __shared__ __align__(16) char sm_wd[];
  constexpr int NW = DTHREADS / 32;
  __shared__ float red_max[NW], red_z[NW];
  __shared__ int red_n[NW];
  const int b = blockIdx.y, N = g.N;
  const int Pt = w.info[b * INFO_W];
  if (Pt == 0) return;
  int MG;
  const int Mb = wide_rows(g, b, &MG);
  if ((int)blockIdx.x >= Mb) return;
  const float fxs = ldexpf(1.f, fexp ? fexp[b] : fx_exp);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const size_t pitch = ((size_t)N + 3) & ~(size_t)3;
  float* rows = reinterpret_cast<float*>(sm_wd);  // [DROWS][pitch]
  int tok[SLOTS];
  long long acc[SLOTS];
#pragma unroll
  for (int q = 0; q < SLOTS; ++q) {
    const int k = threadIdx.x + DTHREADS * q;
    tok[q] = k < Pt ? w.pool[(size_t)b * P + k] : -1;
    acc[q] = 0;
  }
  auto fetch = [&](int m, int slot) {
    if (m < Mb) {
      const float* src = C + ((size_t)b * g.Mstride + m) * N;
      float* dst = rows + slot * pitch;
      if (VEC) {
        for (int j = 4 * threadIdx.x; j < N; j += 4 * DTHREADS) cp_async16(dst + j, src + j);
      } else {
        for (int j = threadIdx.x; j < N; j += DTHREADS) cp_async4(dst + j, src + j, true);
      }
    }
    cp_async_commit();
  };
  for (int q = 0; q < DROWS - 1; ++q) fetch(blockIdx.x + q * gridDim.x, q);
  for (int m = blockIdx.x, i = 0; m < Mb; m += gridDim.x, ++i) {
    cp_async_wait<DROWS - 2>();
    __syncthreads();  // row i is here, and every thread is done with row i - 1
    fetch(m + (DROWS - 1) * gridDim.x, (i + DROWS - 1) % DROWS);
    const float* row = rows + (i % DROWS) * pitch;
    float R[SLOTS];
    float mx = 0.f;
    int n = 0;
#pragma unroll
    for (int q = 0; q < SLOTS; ++q) {
      R[q] = tok[q] >= 0 ? row[tok[q]] : 0.f;
      mx = fmaxf(mx, R[q]);
      n += R[q] > 0.f;
    }
    mx = warp_max(mx);
    n = warp_sum_int(n);
    if (lane == 0) {
      red_max[wid] = mx;
      red_n[wid] = n;
    }
    __syncthreads();
    const float rmax = warp_max(lane < NW ? red_max[lane] : 0.f);
    const int nf = warp_sum_int(lane < NW ? red_n[lane] : 0);
    if (nf == 0) continue;  // uniform over the block
    // softmax of R / tau shifted by its largest logit rmax / tau
    const float tau = resp_temp * rmax + resp_eps;
    float ex[SLOTS], z = 0.f;
#pragma unroll
    for (int q = 0; q < SLOTS; ++q) {
      ex[q] = R[q] > 0.f ? expf((R[q] - rmax) / tau) : 0.f;
      z += ex[q];
    }
    z = warp_sum(z);
    if (lane == 0) red_z[wid] = z;
    __syncthreads();
    z = warp_sum(lane < NW ? red_z[lane] : 0.f) +
        (float)(Pt - nf) * expf(-rmax / tau);  // a pool token with R = 0
    const float invz = 1.f / z;
#pragma unroll
    for (int q = 0; q < SLOTS; ++q)
      if (R[q] > 0.f) acc[q] += to_fix(ex[q] * invz * R[q], fxs);
  }
#pragma unroll
  for (int q = 0; q < SLOTS; ++q) {
    const int k = threadIdx.x + DTHREADS * q;
    if (acc[q]) atomicAdd((unsigned long long*)&w.sc[(size_t)b * P + k], (unsigned long long)acc[q]);
  }
}

// Later rounds: a warp per row, over its survivor list with coverage bcov.  The
// entries in the pool are few, and their sums are three native 32-bit additions
// (select_common.cuh); one block takes many rows, so the slot table is laid out and
// the sums are flushed once per block and not once per eight rows (7,936 rows:
// 15.7 us a round, now 10).
__global__ void __launch_bounds__(32 * SROWS) k_w_rho(WideState w, WideGeom g, int P,
                                                      const float* __restrict__ C,
                                                      const uint16_t* __restrict__ scol,
                                                      float resp_temp, float resp_eps, int fx_exp,
                                                      const int32_t* fexp) {
  grid_dep_wait();
  extern __shared__ __align__(16) char sm_wr[];
  const int b = blockIdx.y, N = g.N;
  const int Pt = w.info[b * INFO_W];
  if (Pt == 0) return;
  int MG;
  const int Mb = wide_rows(g, b, &MG);
  const float fxs = ldexpf(1.f, fexp ? fexp[b] : fx_exp);
  const int32_t* gpool = w.pool + (size_t)b * P;
  unsigned long long* sc = reinterpret_cast<unsigned long long*>(w.sc) + (size_t)b * P;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (blockIdx.x * SROWS >= Mb) return;
  uint32_t* sblk = reinterpret_cast<uint32_t*>(sm_wr);  // [3][P] limbs
  short* pslot = reinterpret_cast<short*>(sblk + 3 * (size_t)P);  // [N] pool slot or -1
  for (int k = threadIdx.x; k < 3 * P; k += blockDim.x) sblk[k] = 0;
  int* fill = reinterpret_cast<int*>(pslot);
  for (int j = threadIdx.x; j < (N + 1) / 2; j += blockDim.x) fill[j] = -1;
  __syncthreads();
  for (int k = threadIdx.x; k < Pt; k += blockDim.x) pslot[gpool[k]] = (short)k;
  __syncthreads();
  for (int m = blockIdx.x * SROWS + wid; m < Mb; m += gridDim.x * SROWS) {
    const size_t row = (size_t)b * g.Mstride + m;
    const int n = w.cnt[row];
    const float bm = w.bcov[row];
    const float* vals = C + row * N;
    const uint16_t* cols = scol + row * N;
    // pass 1: the largest pool residual and the number of pool entries
    float rmax = 0.f;
    int nf = 0;
#pragma unroll 4
    for (int e = lane; e < n; e += 32) {
      const int k = pslot[cols[e]];
      const float x = vals[e];
      if (k >= 0) {
        rmax = fmaxf(rmax, x - bm);
        ++nf;
      }
    }
    rmax = warp_max(rmax);
    nf = warp_sum_int(nf);
    if (nf > 0) {
      const float tau = resp_temp * rmax + resp_eps;
      const float e0 = expf(-rmax / tau);  // pool tokens without a survivor here: R = 0
      float z = 0.f;
#pragma unroll 4
      for (int e = lane; e < n; e += 32) {
        const int k = pslot[cols[e]];
        const float x = vals[e];
        if (k >= 0) z += expf((x - bm - rmax) / tau);
      }
      z = warp_sum(z) + (float)(Pt - nf) * e0;
      const float invz = 1.f / z;
#pragma unroll 4
      for (int e = lane; e < n; e += 32) {
        const int k = pslot[cols[e]];
        const float x = vals[e];
        if (k >= 0) {
          const float R = x - bm;
          sel::limb_add(&sblk[k], P,
                        (unsigned long long)to_fix(expf((R - rmax) / tau) * invz * R, fxs));
        }
      }
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < Pt; k += blockDim.x) {
    const unsigned long long v = sel::limb_value(&sblk[k], P);
    if (v) atomicAdd(&sc[k], v);
  }
}

// ---- batch -----------------------------------------------------------------------------
__global__ void __launch_bounds__(WP_THREADS, 1) k_w_batch(WideState w, WideGeom g, int P, int NP,
                                                        int bsz, int32_t* order, TraceView tv) {
  grid_dep_wait();
  extern __shared__ __align__(16) char sm_wb[];
  const int b = blockIdx.x, K = g.K;
  int32_t* info = w.info + b * INFO_W;
  const int Pt = info[0];
  if (Pt == 0) return;
  const int S = info[3], rd = info[4];
  const int nb = min(bsz, min(Pt, K - S));
  long long* ks = reinterpret_cast<long long*>(sm_wb);   // [NP] scores
  int* kj = reinterpret_cast<int*>(ks + NP);             // [NP] tokens
  if (Pt <= sel::WCAP) {
    // a small pool: every slot's exact rank by (score desc, token asc) is its
    // place in the batch (the order the histogram selection and the sort
    // below give)
    for (int k = threadIdx.x; k < Pt; k += blockDim.x) {
      ks[k] = w.sc[(size_t)b * P + k];
      kj[k] = w.pool[(size_t)b * P + k];
    }
    __syncthreads();
    for (int k = threadIdx.x; k < Pt; k += blockDim.x) {
      const long long sk = ks[k];
      const int jk = kj[k];
      int r = 0;
      for (int q = 0; q < Pt; ++q) r += sel::key_before(ks[q], kj[q], sk, jk);
      if (r < nb) {
        w.batch[(size_t)b * P + r] = jk;
        w.stamp[(size_t)b * g.N + jk] = rd + 1;
        order[(size_t)b * K + S + r] = jk;
      }
    }
    if (threadIdx.x == 0) {
      info[1] = S + nb;
      info[2] = rd + 1;
      if (tv.base) tv.at<int32_t>(b, tv.off_round_end)[rd] = S + nb;
    }
    return;
  }
  // The batch is the top nb of the pool by (score desc, token asc): the
  // histogram selection over the pool slots with the tokens as tie-breakers.
  // Scores of zero are no candidates there; if fewer than nb are positive,
  // the bitonic sort below orders the whole pool instead.
  {
    char* p = reinterpret_cast<char*>(kj + NP);
    sel::PoolScratch ps{};
    ps.hist = reinterpret_cast<int*>(p);       p += sizeof(int) * sel::HBINS;
    ps.bnd = reinterpret_cast<int*>(p);        p += sizeof(int) * (size_t)NP;
    ps.wsum = reinterpret_cast<int*>(p);       p += sizeof(int) * 32;
    ps.scal = reinterpret_cast<int*>(p);       p += sizeof(int) * 8;
    ps.coarse = reinterpret_cast<int*>(p);     p += sizeof(int) * sel::CBINS;
    int* top = reinterpret_cast<int*>(p);      p += sizeof(int) * (size_t)NP;
    ps.key = reinterpret_cast<short*>(p);      p += sizeof(short) * (size_t)NP;
    ps.pk = reinterpret_cast<unsigned char*>(p); p += (size_t)NP;
    unsigned char* none = reinterpret_cast<unsigned char*>(p);
    for (int k = threadIdx.x; k < Pt; k += blockDim.x) {
      ks[k] = w.sc[(size_t)b * P + k];
      kj[k] = w.pool[(size_t)b * P + k];
      none[k] = 0;
    }
    for (int h = threadIdx.x; h < sel::HBINS; h += blockDim.x) ps.hist[h] = 0;
    if (threadIdx.x < sel::CBINS) ps.coarse[threadIdx.x] = 0;
    __syncthreads();
    const int got = sel::select_pool<true>(ks, none, Pt, nb, ps, top, nullptr, kj);
    if (got == nb) {  // uniform over the block
      for (int q = threadIdx.x; q < nb; q += blockDim.x) {
        const int j = kj[top[q]];
        w.batch[(size_t)b * P + q] = j;
        w.stamp[(size_t)b * g.N + j] = rd + 1;
        order[(size_t)b * K + S + q] = j;
      }
      if (threadIdx.x == 0) {
        info[1] = S + nb;
        info[2] = rd + 1;
        if (tv.base) tv.at<int32_t>(b, tv.off_round_end)[rd] = S + nb;
      }
      return;
    }
    __syncthreads();
  }
  for (int k = threadIdx.x; k < NP; k += blockDim.x) {
    const bool in = k < Pt;
    ks[k] = in ? w.sc[(size_t)b * P + k] : -1;  // padding sorts after every pool entry
    kj[k] = in ? w.pool[(size_t)b * P + k] : 0x7fffffff;
  }
  __syncthreads();
  // bitonic sort into (score desc, token asc); NP is a power of two
  for (int size = 2; size <= NP; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int t = threadIdx.x; t < NP / 2; t += blockDim.x) {
        const int lo = 2 * t - (t & (stride - 1));  // first index of the pair
        const int hi = lo + stride;
        const bool desc_block = (lo & size) == 0;   // this run sorts in key order
        const long long sa = ks[lo], sb = ks[hi];
        const int ja = kj[lo], jb = kj[hi];
        const bool b_first = sel::key_before(sb, jb, sa, ja);
        if (b_first == desc_block) {
          ks[lo] = sb; ks[hi] = sa;
          kj[lo] = jb; kj[hi] = ja;
        }
      }
      __syncthreads();
    }
  }
  for (int q = threadIdx.x; q < nb; q += blockDim.x) {
    const int j = kj[q];
    w.batch[(size_t)b * P + q] = j;
    w.stamp[(size_t)b * g.N + j] = rd + 1;
    order[(size_t)b * K + S + q] = j;
  }
  if (threadIdx.x == 0) {
    info[1] = S + nb;
    info[2] = rd + 1;
    if (tv.base) tv.at<int32_t>(b, tv.off_round_end)[rd] = S + nb;
  }
}

// ---- coverage update, survivor compaction, next gains ---------------------------------
// One block an SM (the next gains of N tokens are in its shared memory), of as
// many warps as give its rows to them evenly (launch_wide_select): the sums are
// cleared and flushed once per SM, and no SM waits for one warp's extra row.
// Blocks flush from different columns on, so that they do not all add to the same
// ones at once.  7,936 rows of 15,876: first round 205 us, now 139; a later
// round 15 us, now 11.
template <bool DENSE>
__global__ void __launch_bounds__(32 * FROWS) k_w_filter(WideState w, WideGeom g, int P, int rnd,
                                                         float* C, uint16_t* scol, int fx_exp,
                                                         const int32_t* fexp, TraceView tv) {
  grid_dep_wait();
  extern __shared__ __align__(16) char sm_wf[];
  const int b = blockIdx.y, N = g.N;
  const int32_t* info = w.info + b * INFO_W;
  const int Pt = info[0];
  if (Pt == 0) return;
  int MG;
  const int Mb = wide_rows(g, b, &MG);
  const int nw = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((int)blockIdx.x * nw >= Mb) return;
  // the warps' row tiles, then this block's part of the next gains
  float4* tile = reinterpret_cast<float4*>(sm_wf) + (DENSE ? wid * (sel::ROW_STEP / 4) : 0);
  const sel::GainSums<false> uacc{
      reinterpret_cast<uint32_t*>(sm_wf + (DENSE ? sizeof(float) * sel::ROW_STEP * nw : 0)), N};
  const int S = info[3], rd = info[4];
  const int nb = info[1] - S;  // the batch kernel has run: info[1] = S + nb
  const float fxs = ldexpf(1.f, fexp ? fexp[b] : fx_exp);
  const int32_t* batch = w.batch + (size_t)b * P;
  const int32_t* stamp = w.stamp + (size_t)b * N;
  __shared__ long long fb[3];
  if (threadIdx.x < 3) fb[threadIdx.x] = 0;
  uacc.clear();
  __syncthreads();
  const unsigned lt = sel::lanemask_lt();
  for (int m = blockIdx.x * nw + wid; m < Mb; m += gridDim.x * nw) {
    const size_t row = (size_t)b * g.Mstride + m;
    float* vals = C + row * N;
    uint16_t* cols = scol + row * N;
    int wr = 0;
    float bnew;
    if (DENSE) {
      bnew = 0.f;
#pragma unroll 8
      for (int t = lane; t < nb; t += 32) bnew = fmaxf(bnew, vals[batch[t]]);
      bnew = warp_max(bnew);
      const long long fb_new = to_fix(bnew, fxs);
      float rowmax;
      wr = sel::filter_dense_row<true, true>(vals, cols, N, bnew, fb_new, fxs, uacc, tile, &rowmax);
      if (lane == 0) {
        atomicAdd((unsigned long long*)&fb[bank_of(m, MG, g.MV)],
                  (unsigned long long)to_fix(rowmax, fxs));
        if (tv.base) atomicAdd(tv.cover(b, rd), (unsigned long long)fb_new);
      }
    } else {
      const int n = w.cnt[row];
      bnew = w.bcov[row];
#pragma unroll 4
      for (int e = lane; e < n; e += 32) {
        const float x = vals[e];
        if (stamp[cols[e]] == rd + 1) bnew = fmaxf(bnew, x);
      }
      bnew = warp_max(bnew);
      const long long fb_new = to_fix(bnew, fxs);
      constexpr int FU = 4;  // chunks of 32 entries loaded before any is written back
      for (int e00 = 0; e00 < n; e00 += 32 * FU) {
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
        __syncwarp();
#pragma unroll
        for (int u = 0; u < FU; ++u) {
          const bool keep = e00 + 32 * u + lane < n && cc[u] > bnew;
          const unsigned bal = __ballot_sync(FULL, keep);
          if (keep) {
            const int pos = wr + __popc(bal & lt);
            vals[pos] = cc[u];
            cols[pos] = (uint16_t)jj[u];
            uacc.add(jj[u], (unsigned long long)(to_fix(cc[u], fxs) - fb_new));
          }
          wr += __popc(bal);
        }
      }
      if (lane == 0 && tv.base) atomicAdd(tv.cover(b, rd), (unsigned long long)fb_new);
    }
    if (lane == 0) {
      w.bcov[row] = bnew;
      w.cnt[row] = wr;
    }
  }
  __syncthreads();
  if (DENSE && threadIdx.x < 3 && fb[threadIdx.x])
    atomicAdd((unsigned long long*)&w.fv[(size_t)b * 4 + threadIdx.x], (unsigned long long)fb[threadIdx.x]);
  uacc.flush(reinterpret_cast<unsigned long long*>(gains_out(w, rnd) + (size_t)b * N), false,
             (int)((long long)N * blockIdx.x / gridDim.x));
}

// ---- fill, ascending support, diagnostics ------------------------------------------------
__global__ void __launch_bounds__(WP_THREADS) k_w_final(WideState w, WideGeom g, int fx_exp,
                                                        const int32_t* fexp, int32_t* order,
                                                        int32_t* support, int32_t* slot,
                                                        int32_t* out_idx, uint32_t* status,
                                                        TraceView tv) {
  grid_dep_wait();
  constexpr int WORDS = GMC_MAX_N_LONG / 32;
  static_assert(WORDS <= WP_THREADS, "a thread per word");
  __shared__ uint32_t selw[WORDS];  // the selected tokens, a bit each
  __shared__ int wpre[WORDS];       // selected tokens before each word
  __shared__ int wsum[32];
  __shared__ long long fb[3];
  const int b = blockIdx.x, N = g.N, K = g.K;
  int MG;
  const int Mb = wide_rows(g, b, &MG);
  if (Mb == 0) return;
  const int32_t* info = w.info + b * INFO_W;
  const int S = info[1], rd = info[2];
  const int nwords = (N + 31) >> 5, k = threadIdx.x;
  if (k < nwords) selw[k] = 0;
  if (threadIdx.x < 3) fb[threadIdx.x] = 0;
  __syncthreads();
  for (int q = threadIdx.x; q < S; q += blockDim.x) {
    const int j = order[(size_t)b * K + q];
    atomicOr(&selw[j >> 5], 1u << (j & 31));
  }
  __syncthreads();
  const int filled = S < K ? K - S : 0;
  if (filled > 0) {  // zero-gain fill: the first K - S unselected tokens, ascending
    uint32_t open = k < nwords ? ~selw[k] : 0u;
    if (k == nwords - 1 && (N & 31)) open &= (1u << (N & 31)) - 1u;
    int pos = sel::block_exclusive_scan(__popc(open), wsum, nullptr);
    for (; open && pos < filled; open &= open - 1u, ++pos) {
      const int bit = __ffs(open) - 1;
      order[(size_t)b * K + S + pos] = 32 * k + bit;
      selw[k] |= 1u << bit;
    }
    __syncthreads();
  }
  {  // the support in ascending token order (whole lines of slots: a run of tokens a
     // thread, each writing its own, took 14.5 us at N = 15,876, now 6.9)
    int cnt = 0;
    const int pos = sel::block_exclusive_scan(k < nwords ? __popc(selw[k]) : 0, wsum, &cnt);
    if (k < nwords) wpre[k] = pos;
    __syncthreads();
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
      const uint32_t word = selw[j >> 5], bit = 1u << (j & 31);
      const int at = (word & bit) ? wpre[j >> 5] + __popc(word & (bit - 1u)) : -1;
      slot[(size_t)b * N + j] = at;
      if (at >= 0 && at < K) {
        support[(size_t)b * K + at] = j;
        if (out_idx) out_idx[(size_t)b * K + at] = j;
      }
    }
    if (threadIdx.x == 0 && cnt != K) set_status(status, GMC_STATUS_INTERNAL);
  }
  if (!tv.base) return;
  const int e = fexp ? fexp[b] : fx_exp;
  const float fxs = ldexpf(1.f, e);
  if (rd > 0) {  // F_b(S) from the final coverage of every row (the fill adds nothing)
    long long f[3] = {0, 0, 0};
    for (int m = threadIdx.x; m < Mb; m += blockDim.x)
      f[bank_of(m, MG, g.MV)] += to_fix(w.bcov[(size_t)b * g.Mstride + m], fxs);
    for (int q = 0; q < 3; ++q)
      if (f[q]) atomicAdd((unsigned long long*)&fb[q], (unsigned long long)f[q]);
  }
  __syncthreads();
  const int rounds = rd + (filled > 0 ? 1 : 0);
  if (threadIdx.x == 0) {
    gmc_trace_header* hd = tv.header(b);
    hd->K = K;
    hd->rounds = rounds;
    hd->filled = filled;
    const double inv = ldexp(1.0, -e);
    for (int q = 0; q < 3; ++q) {
      hd->F_S[q] = (float)((double)fb[q] * inv);
      hd->F_V[q] = (float)((double)w.fv[(size_t)b * 4 + q] * inv);
    }
  }
  int32_t* to = tv.at<int32_t>(b, tv.off_order);
  for (int q = threadIdx.x; q < K; q += blockDim.x) to[q] = order[(size_t)b * K + q];
  int32_t* te = tv.at<int32_t>(b, tv.off_round_end);
  for (int q = rd + threadIdx.x; q < tv.rounds_max; q += blockDim.x) te[q] = K;
  int32_t* tp = tv.at<int32_t>(b, tv.off_pool);
  for (size_t q = (size_t)rd * tv.pool_size + threadIdx.x; q < (size_t)tv.rounds_max * tv.pool_size;
       q += blockDim.x)
    tp[q] = -1;
}

// ---------------------------------------------------------------------------------------
int wide_rounds(int K, const gmc_params& p) { return (K + p.batch_b - 1) / p.batch_b; }

cudaError_t launch_wide_select(const WideState& w, const WideGeom& g, const gmc_params& p,
                               int fx_exp, const int32_t* fexp, float* C, uint16_t* scol,
                               const long long* u0, int32_t* order, int32_t* support,
                               int32_t* slot, int32_t* out_idx, uint32_t* status,
                               const TraceView& tv, cudaStream_t st) {
  static int sms = 0;
  cudaError_t e;
  if (sms == 0) {
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
      return e;
  }
  const int P = p.pool_mult * p.batch_b, N = g.N;
  int NP = 1;
  while (NP < P) NP <<= 1;
  const size_t psm = sizeof(int) * (sel::HBINS + (size_t)N + 32 + 8 + sel::CBINS + P) +
                     sizeof(short) * (size_t)N + 2 * (size_t)N + 16 +
                     sizeof(long long) * (size_t)std::min(N, W_BCAP) + 64;
  const size_t rsm_dense = sizeof(float) * DROWS * (((size_t)N + 3) & ~(size_t)3);
  const size_t rsm_sparse = 3 * sizeof(uint32_t) * (size_t)P + sizeof(short) * ((size_t)N + 1);
  const size_t bsm = (sizeof(long long) + sizeof(int)) * (size_t)NP +
                     sizeof(int) * (sel::HBINS + 2 * (size_t)NP + 32 + 8 + sel::CBINS) +
                     sizeof(short) * (size_t)NP + 2 * (size_t)NP + 80;
  // rows: the blocks that are on the GPU together take every row between them.  A filter
  // block has the fewest warps that do its rows in the same number of turns (33 rows: two
  // turns of 17 warps, not one and a part of 32).  A slot's limbs take LIMB_ADDS rows.
  const int per_image = std::max(1, sms / g.B);
  const int fblocks = std::min(per_image, (int)ceil_div(g.Mstride, 4));
  const int frows = (int)ceil_div(g.Mstride, fblocks);
  const int fwarps = (int)ceil_div(frows, ceil_div(frows, FROWS));
  const size_t fsm = sel::gain_sums_bytes<false>(N);
  const size_t fsm_dense = fsm + sizeof(float) * sel::ROW_STEP * (size_t)fwarps;
  // the window pool's extra shared memory: the staged gains and its scratch
  const size_t wsm = sizeof(long long) * ((size_t)N + sel::WCAP) + sizeof(int) * sel::WCAP +
                     sizeof(int) * (sel::WBINS + 4);
  const int win = P <= sel::WCAP / 2 && psm + wsm <= 227 * 1024 ? 1 : 0;
  const size_t psm_w = psm + (win ? wsm : 0);
  const void* kpool = win ? (const void*)k_w_pool<true> : (const void*)k_w_pool<false>;
  if ((e = set_smem_limit(kpool, psm_w)) != cudaSuccess) return e;
  // pool slots a thread: GMC_MAX_POOL_WIDE in all; rows on 16 bytes where N is a multiple of 4
  const bool vec = N % 4 == 0;
  auto* krho = P <= DTHREADS       ? (vec ? k_w_rho_dense<1, true> : k_w_rho_dense<1, false>)
               : P <= 4 * DTHREADS ? (vec ? k_w_rho_dense<4, true> : k_w_rho_dense<4, false>)
                                   : (vec ? k_w_rho_dense<8, true> : k_w_rho_dense<8, false>);
  static_assert(8 * DTHREADS >= GMC_MAX_POOL_WIDE, "a thread's slots hold the widest pool");
  if ((e = set_smem_limit((const void*)krho, rsm_dense)) != cudaSuccess) return e;
  if ((e = set_smem_limit((const void*)k_w_rho, rsm_sparse)) != cudaSuccess) return e;
  if ((e = set_smem_limit((const void*)k_w_batch, bsm)) != cudaSuccess) return e;
  if ((e = set_smem_limit((const void*)k_w_filter<true>, fsm_dense)) != cudaSuccess) return e;
  if ((e = set_smem_limit((const void*)k_w_filter<false>, fsm)) != cudaSuccess) return e;
  const dim3 rgrid(std::min(g.Mstride, per_image), g.B);
  const dim3 sgrid(std::max(std::min((int)ceil_div(g.Mstride, SROWS), 2 * per_image),
                            (int)ceil_div(g.Mstride, sel::LIMB_ADDS - SROWS)), g.B);
  const dim3 fgrid(fblocks, g.B);
  const int R = wide_rounds(g.K, p);
  for (int rnd = 0; rnd < R; ++rnd) {
    if (win)
      launch_k(k_w_pool<true>, g.B, WP_THREADS, psm_w, st, 1, w, g, P, rnd, u0, tv);
    else
      launch_k(k_w_pool<false>, g.B, WP_THREADS, psm_w, st, 1, w, g, P, rnd, u0, tv);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (rnd == 0)
      launch_k(krho, rgrid, DTHREADS, rsm_dense, st, 1, w, g, P, (const float*)C, p.resp_temp,
               p.resp_eps, fx_exp, fexp);
    else
      launch_k(k_w_rho, sgrid, 32 * SROWS, rsm_sparse, st, 1, w, g, P, (const float*)C,
               (const uint16_t*)scol, p.resp_temp, p.resp_eps, fx_exp, fexp);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_k(k_w_batch, g.B, WP_THREADS, bsm, st, 1, w, g, P, NP, p.batch_b, order, tv);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (rnd == 0)
      launch_k(k_w_filter<true>, fgrid, 32 * fwarps, fsm_dense, st, 1, w, g, P, rnd, C, scol,
               fx_exp, fexp, tv);
    else
      launch_k(k_w_filter<false>, fgrid, 32 * fwarps, fsm, st, 1, w, g, P, rnd, C, scol, fx_exp,
               fexp, tv);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  launch_k(k_w_final, g.B, WP_THREADS, 0, st, 1, w, g, fx_exp, fexp, order, support, slot,
           out_idx, status, tv);
  return cudaGetLastError();
}

}  // namespace gmc
