// Device pieces shared by the selection kernels (k_select.cu, k_round0.cu):
// the pool choice of Eq. (4) and deterministic block scans.
#pragma once

#include "common.cuh"

namespace gmc {
namespace sel {

constexpr int HBINS = 2048;

__device__ __forceinline__ bool key_before(long long ua, int ja, long long ub, int jb) {
  return ua > ub || (ua == ub && ja < jb);
}

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// 64-bit sums in shared memory as three 32-bit limbs of LIMB bits.  A 64-bit
// shared-memory addition is a compare-and-swap loop that retries once for every
// other thread on the same word, and popular tokens are on many rows; 32-bit
// additions without a result are native.  A word takes up to LIMB_ADDS values
// below 2^63 before its limbs are put together.
constexpr int LIMB = 21;
constexpr int LIMB_ADDS = (1 << (32 - LIMB)) - 1;
__device__ __forceinline__ void limb_add(uint32_t* w, int stride, unsigned long long v) {
  constexpr unsigned M = (1u << LIMB) - 1;
  atomicAdd(w, (unsigned)v & M);
  atomicAdd(w + stride, (unsigned)(v >> LIMB) & M);
  atomicAdd(w + 2 * stride, (unsigned)(v >> (2 * LIMB)));
}
__device__ __forceinline__ unsigned long long limb_value(const uint32_t* w, int stride) {
  return (unsigned long long)w[0] + ((unsigned long long)w[stride] << LIMB) +
         ((unsigned long long)w[2 * stride] << (2 * LIMB));
}

// Sums of a block's changes of the gains, one per token: limbs in the rounds of the
// standard path (N <= GMC_MAX_N: 96 KB at most), 64-bit words in the wide solver, whose
// N tokens would take 192 KB of limbs.
template <bool LIMBS>
__host__ __device__ inline size_t gain_sums_bytes(int N) {
  return (LIMBS ? 3 * sizeof(uint32_t) : sizeof(unsigned long long)) * (size_t)N;
}
template <bool LIMBS>
struct GainSums {
  uint32_t* w;
  int N;
  __device__ __forceinline__ void clear() const {
    for (int k = threadIdx.x; k < (LIMBS ? 3 : 2) * N; k += blockDim.x) w[k] = 0;
  }
  __device__ __forceinline__ void add(int j, unsigned long long v) const {
    if constexpr (LIMBS) limb_add(w + j, N, v);
    else atomicAdd(reinterpret_cast<unsigned long long*>(w) + j, v);
  }
  // every nonzero sum, its sign applied, into the global gains; from token `first` on, around
  __device__ __forceinline__ void flush(unsigned long long* gains, bool negative,
                                        int first = 0) const {
    for (int q = threadIdx.x; q < N; q += blockDim.x) {
      const int j = first + q < N ? first + q : first + q - N;
      unsigned long long v;
      if constexpr (LIMBS) v = limb_value(w + j, N);
      else v = reinterpret_cast<const unsigned long long*>(w)[j];
      if (v) atomicAdd(&gains[j], negative ? 0ull - v : v);
    }
  }
};

// One dense client row of N values, by one warp: the entries above `cover`
// (residual survivors) move to the front of the row in place, with their tokens
// in cols; their residuals are added to `sums`.  Returns the survivors; *rowmax
// (MAX) the row's largest value in every lane.
//
// A warp takes ROW_STEP values a step: 16 per lane, compared into a bit mask; one
// scan of the counts places every lane's survivors (lane by lane, ascending within
// a lane), and only they take the slow part, one per lane and turn, read back from
// the warp's tile in shared memory.
// With one survivor in sixteen, doing that part at every position instead cost a
// warp about four times the instructions.
// AHEAD: the next step's values are loaded before this step's are looked at, for
// blocks whose warps are few on an SM; 16 registers more, which cost a block
// where several share it (32 images: 251 us, 281 ahead; one image of N = 4,096:
// 43 us, 40 ahead).
constexpr int ROW_STEP = 512;  // values a step (2 KB of tile per warp)
constexpr int ROW_U = ROW_STEP / 128;  // 16-byte loads in flight per lane
template <bool MAX, bool AHEAD, class Sums>
__device__ __forceinline__ int filter_dense_row(float* vals, uint16_t* cols, int N, float cover,
                                                long long cover_fix, float fxs, const Sums& sums,
                                                float4* tile, float* rowmax) {
  const int lane = threadIdx.x & 31;
  const bool vec = (N & 3) == 0;  // rows start on 16 bytes
  float mx = 0.f;
  int w = 0;
  float4 buf[ROW_U];
  auto load = [&](int base) {
#pragma unroll
    for (int u = 0; u < ROW_U; ++u) {
      const int k = base + 4 * (u * 32 + lane);
      buf[u] = k < N ? *reinterpret_cast<const float4*>(vals + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  if (AHEAD && vec) load(0);
  for (int base = 0; base < N; base += ROW_STEP) {
    if (vec) {
      if (!AHEAD) load(base);
      __syncwarp();  // the last step's survivors are out of the tile
#pragma unroll
      for (int u = 0; u < ROW_U; ++u) tile[u * 32 + lane] = buf[u];
      if (AHEAD) load(base + ROW_STEP);  // the next step's, past every survivor this one writes
    } else {
      float b1[8];
      __syncwarp();
#pragma unroll
      for (int h = 0; h < ROW_STEP / 256; ++h) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int k = base + (h * 8 + u) * 32 + lane;
          b1[u] = k < N ? vals[k] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
          reinterpret_cast<float*>(tile)[(h * 8 + u) * 32 + lane] = b1[u];
      }
    }
    __syncwarp();
    unsigned mask = 0;
#pragma unroll
    for (int u = 0; u < ROW_U; ++u) {  // values past N are zero: never above a coverage
      const float4 x = tile[u * 32 + lane];
      mask |= (x.x > cover ? 1u : 0u) << (4 * u) | (x.y > cover ? 2u : 0u) << (4 * u) |
              (x.z > cover ? 4u : 0u) << (4 * u) | (x.w > cover ? 8u : 0u) << (4 * u);
      if (MAX) mx = fmaxf(fmaxf(mx, fmaxf(x.x, x.y)), fmaxf(x.z, x.w));
    }
    const int c = __popc(mask);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += y;
    }
    int pos = w + incl - c;
    w += __shfl_sync(FULL, incl, 31);
    while (mask) {
      const int bit = __ffs(mask) - 1;
      mask &= mask - 1;
      const int at = 4 * ((bit >> 2) * 32 + lane) + (bit & 3);
      const float x = reinterpret_cast<const float*>(tile)[at];
      vals[pos] = x;  // at or below the step's last value, which every lane has read
      cols[pos] = (uint16_t)(base + at);
      ++pos;
      sums.add(base + at, (unsigned long long)(to_fix(x, fxs) - cover_fix));
    }
  }
  if (MAX) *rowmax = warp_max(mx);
  __syncwarp();  // the next row reuses the tile
  return w;
}

// Monotone 11-bit bucket of a positive 64-bit gain: exponent and 5 mantissa bits.
__device__ __forceinline__ int gain_bucket(long long u) {
  const int lz = __clzll(u);                                      // 1..63 for 0 < u < 2^63
  const unsigned long long top = (unsigned long long)u << lz;     // leading one at bit 63
  return (63 - lz) * 32 + (int)((top >> 58) & 31);
}
// Block-wide exclusive scan of one int per thread (deterministic).  Every
// thread of the block must call it.
__device__ inline int block_exclusive_scan(int v, int* wsum, int* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(FULL, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  if (w == 0) {
    int t = lane < nw ? wsum[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, t, o);
      if (lane >= o) t += y;
    }
    if (lane < nw) wsum[lane] = t;  // inclusive prefix of warp totals
  }
  __syncthreads();
  const int before = (w > 0 ? wsum[w - 1] : 0) + x - v;
  const int tot = wsum[nw - 1];
  __syncthreads();
  if (total) *total = tot;
  return before;
}

// Shared-memory scratch of select_pool.
constexpr int CBINS = 64;       // coarse bins: the binary exponent of a gain
struct PoolScratch {
  int* hist;           // [HBINS] fine bins, all zero on entry and on return
  int* coarse;         // [CBINS] coarse bins
  int* bnd;            // [N]  tokens of the boundary bin, ascending
  short* key;          // [N]  bucket of every token (-1: not a candidate)
  unsigned char* pk;   // [N]  boundary tokens that enter the pool
  int* wsum;           // [32]
  int* scal;           // [8]
  long long* bval;     // optional [bcap]: the boundary bucket's gains, staged when the
                       // gains are in global memory (nullptr: read them in place)
  int bcap;
};

// Warp-aggregated append: every lane with `want` gets a distinct index from
// *counter (order within the warp by lane).  All lanes of the warp call it.
__device__ __forceinline__ int warp_append(bool want, int* counter) {
  const unsigned m = __ballot_sync(FULL, want);
  const int leader = m ? __ffs(m) - 1 : 0;  // lowest appending lane
  int base = 0;
  if (m && (int)(threadIdx.x & 31) == leader) base = atomicAdd(counter, __popc(m));
  base = __shfl_sync(FULL, base, leader);
  return base + __popc(m & lanemask_lt());
}

constexpr int RANK_MAX = 128;  // boundary tokens ranked exactly, 8 lanes each
constexpr int ID_BITS = 15;    // token and slot indices are below GMC_MAX_N_LONG = 2^14

// Pool of one round: the min(P, #{u_i > 0}) tokens with sel[i] == 0 of largest
// gain u (fixed point), ties to the lower index.  pool[0..Pt) lists the tokens
// above the boundary bucket (below) by index, then the boundary bucket's
// entering tokens by index; poolslot (optional) receives the slot of every
// pool token.  The slots are a deterministic function of the gains, the same
// in every block that calls this with the same data.  Returns Pt.
//
// Every gain gets an 11-bit bucket (exponent, 5 mantissa bits; monotone in u).
// One pass counts the buckets, their sums per exponent are 64 coarse bins; every warp then finds the boundary bucket
// holding the P-th largest gain from the coarse bins and the 32 fine bins of
// one exponent.  Warp w owns 32-token chunks [w * nc, (w + 1) * nc) (lane =
// token within a chunk, so every shared access is conflict-free); ballots
// order the tokens above the boundary bucket and those inside it by index,
// and one scan of the per-warp counts places them: no shared counter,
// nothing that depends on thread scheduling.  Tokens inside the boundary
// bucket are ranked exactly by (u desc, index asc).
// ids (optional): ties are broken by the lower ids[j] instead of the lower j
// (the batch kernel ranks pool slots by (score desc, token asc)).  REFINE
// (the wide solver's long prefixes) narrows a large boundary bucket digit by
// digit (below); the standard solvers, whose buckets are small, leave it out:
// it costs them registers.
// Every thread of the block must call it; blockDim is a multiple of 32.
// bstar_out (optional): the boundary bucket, or -1 when every candidate entered.
template <bool REFINE = false>
__device__ inline int select_pool(const long long* u, const unsigned char* sel, int N, int P,
                                  PoolScratch w, int* pool, short* poolslot,
                                  const int* ids = nullptr, int* bstar_out = nullptr) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int nc = (N + 32 * nw - 1) / (32 * nw);  // chunks per warp
  const unsigned lt = lanemask_lt();
  // 1. bucket of every candidate (-1: selected or zero gain), histograms; the
  //    gains of four chunks are loaded before any of their atomics
  for (int c0 = 0; c0 < nc; c0 += 4) {
    long long vv[4];
    bool cand[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int j = (wid * nc + c0 + t) * 32 + lane;
      const bool in = c0 + t < nc && j < N;
      vv[t] = in ? u[j] : 0;
      cand[t] = in && !sel[j];
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (c0 + t >= nc) break;  // uniform over the warp
      const int j = (wid * nc + c0 + t) * 32 + lane;
      int kb = -1;
      if (j < N) {
        if (cand[t] && vv[t] > 0) {
          kb = gain_bucket(vv[t]);
          atomicAdd(&w.hist[kb], 1);
        }
        w.key[j] = (short)kb;
      }
    }
  }
  __syncthreads();
  for (int e = wid; e < CBINS; e += nw) {  // an exponent's 32 buckets
    const int c = __reduce_add_sync(FULL, w.hist[e * 32 + lane]);
    if (lane == 0) w.coarse[e] = c;
  }
  __syncthreads();
  // 2. boundary bucket, found by every warp alike: coarse bins from the top,
  //    then the fine bins of the boundary exponent
  int bstar, above, Pt;
  {
    const int hi = CBINS - 1 - 2 * lane;  // this lane's two coarse bins: hi, hi - 1
    const int c0 = w.coarse[hi], c1 = w.coarse[hi - 1];
    int incl = c0 + c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += y;
    }
    const int npos = __shfl_sync(FULL, incl, 31);
    if (npos <= P) {
      bstar = -1;    // every candidate is in the pool
      above = npos;  // tokens above the boundary bucket
      Pt = npos;
    } else {
      const unsigned reach = __ballot_sync(FULL, incl >= P);
      const int L = __ffs(reach) - 1;  // first lane whose prefix reaches P
      int excl = __shfl_sync(FULL, incl - c0 - c1, L);
      const int l0 = __shfl_sync(FULL, c0, L);
      int cb = CBINS - 1 - 2 * L;
      if (excl + l0 < P) {
        excl += l0;
        cb -= 1;
      }
      const int f = cb * 32 + 31 - lane;  // fine bins of that exponent, top first
      const int fc = w.hist[f];
      int fi = fc;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, fi, o);
        if (lane >= o) fi += y;
      }
      const int Lf = __ffs(__ballot_sync(FULL, excl + fi >= P)) - 1;
      bstar = __shfl_sync(FULL, f, Lf);               // boundary bucket
      above = __shfl_sync(FULL, excl + fi - fc, Lf);  // tokens in higher buckets
      Pt = P;
    }
  }
  // 3. tokens above / inside the boundary bucket, by index: per-warp counts,
  //    one scan, then the placements (tmp: above, bnd: boundary bucket)
  int cu = 0, ca = 0;
  for (int c = 0; c < nc; ++c) {
    const int j = (wid * nc + c) * 32 + lane;
    const int kb = j < N ? w.key[j] : -1;
    cu += __popc(__ballot_sync(FULL, kb > bstar));
    ca += __popc(__ballot_sync(FULL, kb >= 0 && kb == bstar));
  }
  if (lane == 0) w.wsum[wid] = (cu << 16) | ca;  // cu, ca <= N <= 2^14
  __syncthreads();
  // every warp has read the histograms: clear the bins this thread counted
  for (int c = 0; c < nc; ++c) {
    const int j = (wid * nc + c) * 32 + lane;
    const int kb = j < N ? w.key[j] : -1;
    if (kb >= 0) w.hist[kb] = 0;
  }
  int pre, nb;
  {
    const int x = lane < nw ? w.wsum[lane] : 0;
    int incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += y;
    }
    pre = __shfl_sync(FULL, incl - x, wid);  // this warp's offsets (packed)
    nb = __shfl_sync(FULL, incl, 31) & 0xFFFF;
  }
  int pu = pre >> 16, pa = pre & 0xFFFF;
  for (int c = 0; c < nc; ++c) {
    const int j = (wid * nc + c) * 32 + lane;
    const int kb = j < N ? w.key[j] : -1;
    const bool up = kb > bstar, at = kb >= 0 && kb == bstar;
    const unsigned bu = __ballot_sync(FULL, up), ba = __ballot_sync(FULL, at);
    if (up) {
      const int slot = pu + __popc(bu & lt);
      pool[slot] = j;
      if (poolslot) poolslot[j] = (short)slot;
    }
    if (at) w.bnd[pa + __popc(ba & lt)] = j;
    pu += __popc(bu);
    pa += __popc(ba);
  }
  if (bstar >= 0) {
    __syncthreads();
    // 4. the boundary bucket's tokens that enter, ranked exactly by (u desc,
    //    index asc); they take the slots after the tokens above, by index
    int need = Pt - above;
    const bool staged = w.bval && nb <= w.bcap;  // uniform over the block
    if (staged) {
      for (int q = threadIdx.x; q < nb; q += blockDim.x) w.bval[q] = u[w.bnd[q]];
      __syncthreads();
    }
    // REFINE: the bucket (or the whole pool, when the gains are near-equal: up to N
    // tokens) is narrowed digit by digit, 11 bits at a time: the mantissa bits the
    // bucket left out, then the id (the lower one first).  A digit's histogram says
    // which tokens enter, which do not, and which are undecided (pk 1, 0, 2), until
    // at most RANK_MAX are left to rank exactly.  A bitonic sort of the bucket took
    // 78 block barriers at 4,096 gains; a digit takes six.
    int und = nb;  // uniform over the block
    if constexpr (REFINE) {
      for (int q = threadIdx.x; q < nb; q += blockDim.x) w.pk[q] = 2;
      const int mant = max((bstar >> 5) - 5, 0);  // gain bits below the bucket's
      int done = 0;                               // bits of (gain rest, id) consumed
      while (und > RANK_MAX && done < mant + ID_BITS) {
        const bool of_gain = done < mant;
        const int left = of_gain ? mant - done : mant + ID_BITS - done;
        const int bits = min(left, 11), lo = left - bits;
        const int dmask = (1 << bits) - 1;
        // the digit of boundary token q, monotone in (gain desc, id asc) order
        auto digit = [&](int q) {
          const int j = w.bnd[q];
          if (of_gain) return (int)((staged ? w.bval[q] : u[j]) >> lo) & dmask;
          return dmask - (((ids ? ids[j] : j) >> lo) & dmask);
        };
        __syncthreads();  // the histogram is clear, pk is complete
        for (int q = threadIdx.x; q < nb; q += blockDim.x)
          if (w.pk[q] == 2) atomicAdd(&w.hist[digit(q)], 1);
        __syncthreads();
        {  // a run of bins per thread, top digit first: the one holding the need-th token
          const int per = (HBINS + (int)blockDim.x - 1) / (int)blockDim.x;
          const int h0 = min(HBINS, (int)threadIdx.x * per), h1 = min(HBINS, h0 + per);
          int c = 0;
          for (int h = h0; h < h1; ++h) c += w.hist[HBINS - 1 - h];
          int before = block_exclusive_scan(c, w.wsum, nullptr);
          for (int h = h0; h < h1; ++h) {
            const int x = w.hist[HBINS - 1 - h];
            w.hist[HBINS - 1 - h] = 0;
            if (before < need && before + x >= need) {  // one bin of one thread
              w.scal[0] = HBINS - 1 - h;  // the boundary digit
              w.scal[1] = before;         // tokens of higher digits
              w.scal[2] = x;              // undecided ones
            }
            before += x;
          }
        }
        __syncthreads();
        const int db = w.scal[0];
        for (int q = threadIdx.x; q < nb; q += blockDim.x)
          if (w.pk[q] == 2) {
            const int dg = digit(q);
            w.pk[q] = dg > db ? 1 : (dg == db ? 2 : 0);
          }
        need -= w.scal[1];
        und = w.scal[2];
        done += bits;
      }
      __syncthreads();  // pk is complete, scal has been read
      if (threadIdx.x == 0) w.scal[0] = 0;
      __syncthreads();
      for (int q0 = 0; q0 < nb; q0 += blockDim.x) {  // the undecided ones, in any order
        const int q = q0 + threadIdx.x;
        const bool in = q < nb && w.pk[q] == 2;
        const int at = warp_append(in, &w.scal[0]);
        if (in) w.hist[at] = q;
      }
      __syncthreads();
      const int gl = threadIdx.x & 7;
      const unsigned gm = 0xFFu << (lane & 24);
      for (int i = threadIdx.x >> 3; i < und; i += blockDim.x >> 3) {
        const int q = w.hist[i], j = w.bnd[q];
        const long long v = staged ? w.bval[q] : u[j];
        const int id = ids ? ids[j] : j;
        int rank = 0;
        for (int i2 = gl; i2 < und; i2 += 8) {
          const int q2 = w.hist[i2], j2 = w.bnd[q2];
          rank += key_before(staged ? w.bval[q2] : u[j2], ids ? ids[j2] : j2, v, id);
        }
        rank += __shfl_xor_sync(gm, rank, 1);
        rank += __shfl_xor_sync(gm, rank, 2);
        rank += __shfl_xor_sync(gm, rank, 4);
        if (gl == 0) w.pk[q] = rank < need;
      }
      __syncthreads();
      for (int i = threadIdx.x; i < und; i += blockDim.x) w.hist[i] = 0;
      __syncthreads();
    } else {
      for (int q = threadIdx.x; q < nb; q += blockDim.x) {
        const int j = w.bnd[q];
        const long long v = staged ? w.bval[q] : u[j];
        const int id = ids ? ids[j] : j;
        int rank = 0;
        for (int q2 = 0; q2 < nb; ++q2) {
          const int j2 = w.bnd[q2];
          rank += key_before(staged ? w.bval[q2] : u[j2], ids ? ids[j2] : j2, v, id);
        }
        w.pk[q] = rank < need;
      }
      __syncthreads();
    }
    // slots in index order: each entering token counts the entering ones
    // before it (a small bucket), or a block scan of the entering flags over
    // contiguous ranges (a large one: its barriers cost less than the counts)
    if (nb <= 256) {
      for (int q = threadIdx.x; q < nb; q += blockDim.x) {
        if (!w.pk[q]) continue;
        int before = 0;
        for (int q2 = 0; q2 < q; ++q2) before += w.pk[q2];
        const int j = w.bnd[q];
        pool[above + before] = j;
        if (poolslot) poolslot[j] = (short)(above + before);
      }
    } else {
      const int per = (nb + (int)blockDim.x - 1) / (int)blockDim.x;
      const int q0 = min(nb, (int)threadIdx.x * per), q1 = min(nb, q0 + per);
      int c = 0;
      for (int q = q0; q < q1; ++q) c += w.pk[q];
      int before = block_exclusive_scan(c, w.wsum, nullptr);
      for (int q = q0; q < q1; ++q) {
        if (!w.pk[q]) continue;
        const int j = w.bnd[q];
        pool[above + before] = j;
        if (poolslot) poolslot[j] = (short)(above + before);
        ++before;
      }
    }
  }
  __syncthreads();
  if (bstar_out) *bstar_out = bstar;
  return Pt;
}

// Pool of a later round from a window of buckets below the previous boundary.
//
// A round takes its batch out of the candidates and can only lower the other
// gains (the coverage b_m grows), so the P-th largest gain of the next round is
// at most the P-th largest of this one: its bucket lies at or below the last
// boundary bucket `hint`.  One pass loads the gains (load(j), stored into u[j]
// for later readers), counts the candidates above a window of WBINS buckets
// that ends WTOP buckets above the hint and histograms the ones inside it;
// every warp finds the boundary bucket from the window alone.  The tokens in
// or above the boundary bucket (at most WCAP) are listed in any order and
// ranked exactly by (u desc, index asc); a pool token's slot is its rank, so
// the pool is the same in every block that calls this with the same gains and
// hint.  Three block barriers; a thread's loads of a pass are all issued before
// its atomics.
//
// Returns Pt and sets *hint to the new boundary bucket (-1 once every
// candidate enters); returns -1 when the boundary is not inside the window or
// more than WCAP tokens reach it (the caller then runs select_pool on u, which
// is complete on return).  With *hint < 0 it returns -1 at once and loads
// nothing.  Every thread gets the same answer.  Every thread of the block must
// call it.
constexpr int WBINS = 128;  // window buckets: 4 per lane of one warp
constexpr int WTOP = 8;     // window buckets above the hint
constexpr int WCAP = 256;   // candidates ranked exactly
constexpr int WU = 4;       // tokens a thread handles per pass step
struct WindowScratch {
  int* win;        // [WBINS + 4] window bins (top bucket first) and 4 counters, on 16
                   // bytes (read four bins a load); all zero on entry and on return
  long long* cu;   // [WCAP] candidates' gains
  int* cj;         // [WCAP] candidates' tokens
};

template <class Load>
__device__ inline int select_pool_window(Load load, long long* u, const unsigned char* sel, int N,
                                         int P, WindowScratch w, int* pool, short* poolslot,
                                         int* hint) {
  const int lane = threadIdx.x & 31;
  const int h = *hint;
  if (h < 0) return -1;  // uniform: every thread holds the same hint
  const int top = h + WTOP;             // highest window bucket (bin 0)
  int* cnt = w.win + WBINS;             // 0: above the window, 1: positive, 2: listed
  const int step = (int)blockDim.x;
  // 1. gains, window histogram, counts above the window and of positive candidates
  int npos_w = 0, nabove_w = 0;
  for (int j0 = (int)threadIdx.x - lane; j0 < N; j0 += WU * step) {  // warp-uniform
    long long v[WU];
    unsigned char sl[WU];
#pragma unroll
    for (int t = 0; t < WU; ++t) {
      const int j = j0 + t * step + lane;
      v[t] = j < N ? load(j) : 0;
      sl[t] = j < N ? sel[j] : 1;
    }
#pragma unroll
    for (int t = 0; t < WU; ++t) {
      const int j = j0 + t * step + lane;
      if (j < N) u[j] = v[t];
      const int kb = !sl[t] && v[t] > 0 ? gain_bucket(v[t]) : -1;
      const int bin = top - kb;
      if (kb >= 0 && bin >= 0 && bin < WBINS) atomicAdd(&w.win[bin], 1);
      npos_w += __popc(__ballot_sync(FULL, kb >= 0));
      nabove_w += __popc(__ballot_sync(FULL, kb > top));
    }
  }
  if (lane == 0) {
    if (nabove_w) atomicAdd(&cnt[0], nabove_w);
    if (npos_w) atomicAdd(&cnt[1], npos_w);
  }
  __syncthreads();
  // 2. boundary bucket, found by every warp alike
  const int npos = cnt[1], nabove = cnt[0];
  int bstar = -1, ncand = npos, Pt = npos;
  bool miss = false;
  if (npos > P) {
    Pt = P;
    if (nabove >= P) {
      miss = true;  // the boundary is above the window
    } else {
      const int4 c4 = reinterpret_cast<const int4*>(w.win)[lane];  // bins 4 lane .. 4 lane + 3
      const int s4 = c4.x + c4.y + c4.z + c4.w;
      int incl = s4;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
      }
      const int need = P - nabove;
      const unsigned reach = __ballot_sync(FULL, incl >= need);
      if (!reach) {
        miss = true;  // the boundary is below the window
      } else {
        const int L = __ffs(reach) - 1;
        int acc = __shfl_sync(FULL, incl - s4, L);
        const int b0 = __shfl_sync(FULL, c4.x, L), b1 = __shfl_sync(FULL, c4.y, L);
        const int b2 = __shfl_sync(FULL, c4.z, L), b3 = __shfl_sync(FULL, c4.w, L);
        int t = 0;
        if (acc + b0 < need) {
          acc += b0;
          t = 1;
          if (acc + b1 < need) {
            acc += b1;
            t = 2;
            if (acc + b2 < need) {
              acc += b2;
              t = 3;
            }
          }
        }
        const int bt = t == 0 ? b0 : t == 1 ? b1 : t == 2 ? b2 : b3;
        bstar = top - (4 * L + t);
        ncand = nabove + acc + bt;  // every candidate in or above the boundary bucket
        miss = ncand > WCAP;
      }
    }
  } else {
    miss = npos > WCAP;
  }
  if (miss) {
    __syncthreads();  // every warp has read the bins
    for (int q = threadIdx.x; q < WBINS + 4; q += blockDim.x) w.win[q] = 0;
    __syncthreads();
    return -1;
  }
  // 3. list the candidates in or above the boundary bucket (any order); a
  //    thread reads back only the gains it stored itself
  for (int j0 = (int)threadIdx.x - lane; j0 < N; j0 += WU * step) {
    long long v[WU];
    unsigned want = 0;
#pragma unroll
    for (int t = 0; t < WU; ++t) {
      const int j = j0 + t * step + lane;
      v[t] = j < N ? u[j] : 0;
      if (j < N && !sel[j] && v[t] > 0 && gain_bucket(v[t]) >= bstar) want |= 1u << t;
    }
    unsigned bal[WU];
    int tot = 0;
#pragma unroll
    for (int t = 0; t < WU; ++t) {
      bal[t] = __ballot_sync(FULL, (want >> t) & 1u);
      tot += __popc(bal[t]);
    }
    if (tot) {  // warp-uniform: one atomic per warp and step
      int base = 0;
      if (lane == 0) base = atomicAdd(&cnt[2], tot);
      base = __shfl_sync(FULL, base, 0);
      const unsigned lt = lanemask_lt();
#pragma unroll
      for (int t = 0; t < WU; ++t) {
        if ((want >> t) & 1u) {
          const int at = base + __popc(bal[t] & lt);
          w.cu[at] = v[t];
          w.cj[at] = j0 + t * step + lane;
        }
        base += __popc(bal[t]);
      }
    }
  }
  __syncthreads();
  // 4. rank every candidate among them (4 lanes each); slot = rank
  for (int q = threadIdx.x; q < WBINS + 4; q += blockDim.x) w.win[q] = 0;
  for (int base = ((int)threadIdx.x - lane) >> 2; base < ncand; base += blockDim.x >> 2) {
    const int q = base + (lane >> 2), gl = lane & 3;
    int rank = 0;
    long long v = 0;
    int jq = 0;
    if (q < ncand) {
      v = w.cu[q];
      jq = w.cj[q];
#pragma unroll 4
      for (int q2 = gl; q2 < ncand; q2 += 4) rank += key_before(w.cu[q2], w.cj[q2], v, jq);
    }
    rank += __shfl_xor_sync(FULL, rank, 1);
    rank += __shfl_xor_sync(FULL, rank, 2);
    if (q < ncand && gl == 0 && rank < Pt) {
      pool[rank] = jq;
      if (poolslot) poolslot[jq] = (short)rank;
    }
  }
  __syncthreads();
  *hint = Pt == P ? bstar : -1;
  return Pt;
}

// Rank of pool slot k among the Pt slots by (score desc, token asc), counted by
// the 8 lanes of an aligned group (mask gm).
__device__ __forceinline__ int group_score_rank(const long long* s, const int* pool, int Pt, int k,
                                                int gl, unsigned gm) {
  const long long sk = s[k];
  const int jk = pool[k];
  int rank = 0;
  for (int q = gl; q < Pt; q += 8) rank += key_before(s[q], pool[q], sk, jk);
  rank += __shfl_xor_sync(gm, rank, 1);
  rank += __shfl_xor_sync(gm, rank, 2);
  rank += __shfl_xor_sync(gm, rank, 4);
  return rank;
}

}  // namespace sel
}  // namespace gmc
