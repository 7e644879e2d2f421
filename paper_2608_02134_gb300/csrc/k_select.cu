// Batched responsibility selection (Sec. 3.3, Eq. (4); appendix Eq.
// (cond-responsibility) and its totality rule), one thread-block cluster per image.
//
// Round t with support S_t and coverage b_m = max_{j in S_t} Cbar_mj (0 for S empty):
//   R_mi = [Cbar_mi - b_m]_+,  u_i = sum_m R_mi
//   pool = the min(pool_size, #{u_i > 0}) unselected tokens of largest u (ties: lower index)
//   rho_m. = softmax over the pool of R_m. / (resp_temp * max_pool R_m. + resp_eps)
//   s_i = sum_m rho_mi R_mi; the top min(b, |pool|, K - |S|) pool tokens by s enter S
//   (ties: lower index); an empty pool fills the budget in ascending index order.
//
// Work-efficient residual form.  An entry with Cbar_mi <= b_m has R_mi = 0 now
// and in every later round (b only grows), so it never contributes to a gain,
// a responsibility or a coverage update again.  After the first (dense) round
// each client row keeps only its "survivors" {i : Cbar_mi > b_m}, and later
// rounds touch only those.  This is exact, not an approximation: the skipped
// entries are exactly the zero residuals.  (A pool member with R_mi = 0 still
// counts in row m's softmax denominator; the kernel adds those terms
// explicitly.  Every softmax is shifted by its row's largest logit, so no
// exponential exceeds 1 for any temperature.)
//
// The first rounds run over the whole GPU (k_round0.cu); this kernel continues
// with the survivor lists they left in global memory.  As soon as a CTA's lists
// fit in its shared memory they move there ("flat mode") under two indexes:
//   by row   (value, token): the gain update walks the rows whose coverage
//            grew, and no others;
//   by token (row, place of the entry in the row order): the responsibilities
//            and the coverage update read the pool's and the batch's tokens.
// An entry is dead when its value is at most its row's coverage; nothing is
// marked or compacted, so a round costs what its pool and its changed rows
// cost, not what the lists hold.  Lists that do not fit yet are walked in place
// in global memory by 8-lane groups ("global mode").
//
// Parallel layout.  The CS CTAs of a cluster split the client rows; each CTA
// keeps its rows' coverage and lists.  Gains and scores are summed in 64-bit
// fixed point, so every reduction is exact and order-independent: the solver
// is deterministic.  Per round:
//   pool:   every CTA reads the gains from their owners (token j belongs to CTA
//           j / SL) and selects the same pool: the tokens of at least the
//           threshold `lo` are listed, a long list cut, and ranked exactly; when
//           the guess lists too few, a lower one follows, and when that misses too
//           or lists too many, a radix search finds the threshold;
//   scores: every CTA stores its rows' responsibility-weighted residuals into
//           its own row in every CTA of the cluster; every CTA adds the rows
//           and picks the same batch;
//   gains:  the changes of the residuals of the rows whose coverage grew are
//           added at the tokens' owners (remote 64-bit integer additions).
// Two cluster barriers per round; all control decisions are derived from data
// every CTA holds identically, so all CTAs run the same barriers.  A round is a
// chain of shared-memory round trips and barriers: bound by how many dependent
// instructions its slowest warp executes (9 cycles each on average), not by
// bandwidth.  Hence thread-per-slot sums, keys of 32 bits instead of 64-bit
// comparisons, and no 64-bit shared-memory additions on contended words.
// A late round takes 17,000-18,500 cycles (8.5-9 us) at N = 1,296 and 4,096; the
// previous layout, which marked and compacted one token-sorted list and found
// the pool by a histogram, took 11.8 us at N = 1,296 and 20 us at N = 4,096,
// where its lists did not fit.
#include <cooperative_groups.h>
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "select_common.cuh"

namespace cg = cooperative_groups;

namespace gmc {

namespace {
constexpr int SEL_THREADS = 512;
constexpr int SEL_WARPS = SEL_THREADS / 32;
constexpr int SEL_MAX_CS = 16;
constexpr int HBINS = sel::HBINS;
constexpr int UNR = 4;     // global mode: entries in flight per lane in a sweep
constexpr int PCL = 8;     // global mode: pool entries a lane keeps in registers
constexpr int LCAP = SEL_THREADS;  // candidates ranked exactly in a round's pool
constexpr int EC = 2;      // flat mode: entries of a pool token a lane keeps in registers
constexpr size_t SMEM_LIMIT = 227 * 1024;
constexpr int ENTRY_BYTES = 10;  // flat mode: value 4, token 2, row 2, place 2
// Images of up to this many tokens sum a CTA's gain changes in its own shared
// memory and send one remote addition per token, whole warps to one owner;
// scattered remote additions cost about 4 cycles each.  Larger images send them
// one by one: their sums would take the room of a fifth of the entries, and the
// hand-over comes later.  Whole calls with the sums against without: N = 1,296
// 280.7 us / 290.5, 2,025 432 / 430, 3,025 556 / 566, 3,844 (T = 128) 755 / 834,
// 4,096 (T = 128) 744 / 719; above the line, 5,040 978 / 968, 6,400 1,619 / 1,423.
constexpr int AGG_MAX_N = 4096;
__host__ __device__ inline bool aggregates(int N, int R) {
  return N <= AGG_MAX_N && R <= sel::LIMB_ADDS;  // a row adds to a token at most once
}
__host__ __device__ inline int sel_pool_stride(int P) { return ((P + 1) & ~1) + 2; }

struct SelArgs {
  int B, N, K, Mstride, H, Tmax, L2;
  const int32_t* toff;  // compress path: per-image text lengths; select path: nullptr
  int uniform_rows;     // select path: every image has Mstride rows, all in bank 0
  int P, bsz;
  float resp_temp, resp_eps;
  int fx_exp;
  const int32_t* fexp;  // per-image fixed-point exponents (select path) or nullptr
  float* C;
  uint16_t* scol;
  const long long* u0;
  int32_t* order;
  int32_t* support;
  int32_t* slot;
  int32_t* out_idx;
  uint32_t* status;
  TraceView tv;
  int images;           // images per prompt (> 1: the first round seeded one token per image)
  R0State r0;           // state after the first rounds
};

struct SelSmem {
  unsigned long long* gacc;   // [SL] gains of the tokens this CTA owns: every CTA of the
                              // cluster adds the changes of its rows (read in a round's
                              // pool and changed after that round's score barrier)
  unsigned long long* sown;   // [SP] this CTA's scores
  unsigned long long* spart;  // [CS][SP] every CTA's scores (SP: P padded, sel_pool_stride)
  long long* s_acc;           // [P padded to 4] their sums
  uint32_t* zlo;              // [R] softmax denominator of a row, fixed point 2^40: low 24 bits
  uint32_t* zhi;              // [R] high bits, and the row's pool entries from bit 24
  long long* fb;              // [8] F_S[3] (fixed point), FB_LO
  uint32_t* ck;               // [LCAP] pool candidates' keys (gain_key), zero past the listed ones
  int* cj;                    // [LCAP] pool candidates' tokens
  uint32_t* selw;             // [ceil(N/32)] selected tokens, one bit each
  int* wpre;                  // [ceil(N/32)] counts before a word (final ordering)
  int* pool;                  // [P]
  int* wsum;                  // [32] scan scratch
  int* scal;                  // [16]
  int* hist;                  // [HBINS] radix search, zero between uses
  float* bcov;                // [R] coverage b_m
  int* rmaxb;                 // [R] bits of the row's largest pool residual
  int* bnb;                   // [R] bits of the row's largest batch value above its coverage
  uint16_t* rptr;             // [R + 1] flat: first entry of a row; global: survivors (count)
  uint16_t* chg;              // [R] rows whose coverage grew
  uint32_t* uloc;             // [3][N] this CTA's falls of the gains, in limbs (N <= AGG_MAX_N)
  uint32_t* sk;               // [SP] the scores' keys
  // the rest of the shared memory, by mode
  int* cs;                    // flat: [N + 1] first entry of a token
  float* rval;                // flat: [cap] by row: value
  uint16_t* rtok;             //             token
  uint16_t* crow;             // flat: [cap] by token: row
  uint16_t* cpos;             //             place in the row order
  short* poolslot;            // global: [N] pool slot of a token or -1
  int* inb;                   // global: [P] pool slot enters the batch
  unsigned long long* sw;     // global: [SEL_WARPS][P] per-warp partial scores
};

// SC_N0, SC_N1 count the listed candidates and SC_R0, SC_R1 add up their ranks, by
// the parity of the round; SC_KEY: key of the pool's last token
enum { SC_N0 = 0, SC_N1, SC_R0, SC_R1, SC_GLOBAL, SC_NCHG, SC_KEY, SC_BIN, SC_ABOVE, SC_COUNT };
enum { FB_LO = 4 };  // 64-bit word of fb: the next pool's threshold

// Byte offsets of the arrays in a CTA's shared memory.
struct SelOff {
  uint32_t gacc, sown, spart, s_acc, fb, ck, cj, selw, wpre, pool, wsum, scal, hist, bcov, rmaxb,
      zlo, zhi, bnb, rptr, chg, uloc, sk, cs, rval, rtok, crow, cpos, sw, inb, poolslot;
};
struct Layout {
  SelOff o;
  uint32_t fixed;  // bytes before the mode-dependent rest (above SMEM_LIMIT: does not fit)
  int cap;         // flat-mode entries that fit
};

// Shared-memory layout for R rows per CTA and SL owned tokens.
__host__ __device__ inline Layout sel_layout(int N, int P, int CS, int SL, int R) {
  uint32_t off = 0;
  auto take = [&](size_t bytes) {
    const uint32_t at = off;
    off += (uint32_t)((bytes + 15) & ~(size_t)15);
    return at;
  };
  const int nw = (N + 31) / 32;
  Layout L;
  SelOff& s = L.o;
  s.gacc = take(8 * (size_t)SL);
  s.sown = take(8 * (size_t)sel_pool_stride(P));
  s.spart = take(8 * (size_t)sel_pool_stride(P) * CS);
  s.s_acc = take(8 * (size_t)((P + 3) & ~3));
  s.fb = take(8 * 8);
  s.ck = take(4 * (size_t)LCAP);
  s.cj = take(4 * (size_t)LCAP);
  s.selw = take(4 * (size_t)nw);
  s.wpre = take(4 * (size_t)nw);
  s.pool = take(4 * (size_t)P);
  s.wsum = take(4 * 32);
  s.scal = take(4 * 16);
  s.hist = take(4 * (size_t)HBINS);
  s.bcov = take(4 * (size_t)R);
  s.rmaxb = take(4 * (size_t)R);
  s.zlo = take(4 * (size_t)R);
  s.zhi = take(4 * (size_t)R);
  s.bnb = take(4 * (size_t)R);
  s.rptr = take(2 * (size_t)(R + 1));
  s.chg = take(2 * (size_t)R);
  s.uloc = take(aggregates(N, R) ? 12 * (size_t)N : 0);
  s.sk = take(4 * (size_t)((sel_pool_stride(P) + 3) & ~3));
  L.fixed = off;
  // flat mode
  s.cs = take(4 * (size_t)(N + 1));
  const long long room = (long long)SMEM_LIMIT - (long long)off - 64;
  L.cap = room > 0 ? (int)(room / ENTRY_BYTES) & ~7 : -1;  // -1: never flat
  if (L.cap > 65528) L.cap = 65528;  // places are 16 bits
  const size_t cap = L.cap > 0 ? (size_t)L.cap : 0;
  s.rval = take(4 * cap);
  s.rtok = take(2 * cap);
  s.crow = take(2 * cap);
  s.cpos = take(2 * cap);
  // global mode, over the same bytes
  off = L.fixed;
  s.sw = take(8 * (size_t)SEL_WARPS * P);
  s.inb = take(4 * (size_t)P);
  s.poolslot = take(2 * (size_t)N);
  if (off > SMEM_LIMIT) L.fixed = SMEM_LIMIT + 1;  // does not fit
  return L;
}

// Address of local shared-memory address `local` in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void* local, int rank) {
  const uint32_t la = (uint32_t)__cvta_generic_to_shared(local);
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(la), "r"(rank));
  return ra;
}
// Fire-and-forget 64-bit add (no value is returned, so the issuing thread does
// not wait for the remote round trip; the next cluster barrier orders it before
// every later read).
__device__ __forceinline__ void red_add_cluster(uint32_t at, unsigned long long v) {
  asm volatile("red.shared::cluster.add.u64 [%0], %1;" ::"r"(at), "l"(v) : "memory");
}
__device__ __forceinline__ void store2_cluster(uint32_t at, unsigned long long v0,
                                               unsigned long long v1) {
  asm volatile("st.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(at), "l"(v0), "l"(v1) : "memory");
}
__device__ __forceinline__ unsigned long long load_cluster(uint32_t at) {
  unsigned long long v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(at) : "memory");
  return v;
}
// Exponent and 26 mantissa bits of a positive gain: monotone, 32 bits.
__device__ __forceinline__ uint32_t gain_key(unsigned long long v) {
  const int lz = __clzll((long long)v);
  return ((uint32_t)(63 - lz) << 26) | (uint32_t)(((v << lz) >> 37) & 0x3ffffffu);
}

using sel::block_exclusive_scan;
using sel::key_before;
using sel::lanemask_lt;

// Reductions inside an aligned group of G = 8 lanes (mask `gm`).
constexpr int G = 8;
__device__ __forceinline__ float group_max(float v, unsigned gm) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(gm, v, o));
  return v;
}
template <typename T>
__device__ __forceinline__ T group_sum(T v, unsigned gm) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(gm, v, o);
  return v;
}

// The smallest gain whose bucket (exponent, `bits` mantissa bits) is that of
// prefix p (leading one and `bits` bits) at exponent e.
__device__ __forceinline__ unsigned long long prefix_edge(int e, int bits, unsigned long long p) {
  return (p << (63 - bits)) >> (63 - e);
}

// The gain that gain_key made a key of, to its 27 bits.
__device__ __forceinline__ float key_gain(uint32_t k) {
  return ldexpf((float)(0x4000000u | (k & 0x3ffffffu)), (int)(k >> 26) - 26);
}
// x / d for d > 0 with r = 1 / d at hand: one correction of the quotient by its
// remainder (Markstein's division); a d near the ends of the range is divided by.
__device__ __forceinline__ float div_by(float x, float d, float r) {
  if (!(d > 1e-30f && d < 1e30f)) return x / d;
  const float q = x * r;
  return fmaf(fmaf(-q, d, x), r, q);
}

// Lists the tokens of gain >= lo >= 1 (key in ck, token in cj, any order; at most
// LCAP are kept) and counts them in *cnt (zero on entry).  A selected token's
// entries are all dead, so its gain is exactly zero and it is never listed.  Gains are
// signed, as in the rounds before: sums of invalid clients (negative or infinite ones,
// reported in the status) may have wrapped, and are then no candidates.
// addr(j): where token j's gain is; ga: that of the thread's first GA tokens.
// Every thread calls it; a barrier follows at the caller.
constexpr int GA = 4;
template <class Addr>
__device__ __forceinline__ void list_candidates(Addr addr, const uint32_t* ga, const SelSmem& s,
                                                int N, unsigned long long lo, int* cnt) {
  constexpr int U = GA;  // gains in flight per thread
  const int lane = threadIdx.x & 31;
  const unsigned lt = lanemask_lt();
  for (int j0 = (int)threadIdx.x - lane; j0 < N; j0 += U * SEL_THREADS) {
    unsigned long long v[U];
    if (j0 < SEL_THREADS) {  // the first tokens (ga: inside the tokens whatever t)
#pragma unroll
      for (int t = 0; t < U; ++t) v[t] = j0 + t * SEL_THREADS < N ? load_cluster(ga[t]) : 0ull;
    } else {
#pragma unroll
      for (int t = 0; t < U; ++t) v[t] = load_cluster(addr(min(N - 1, j0 + t * SEL_THREADS + lane)));
    }
#pragma unroll
    for (int t = 0; t < U; ++t)
      if (j0 + t * SEL_THREADS + lane >= N) v[t] = 0;
    unsigned bal[U], mine = 0;
    int tot = 0;
#pragma unroll
    for (int t = 0; t < U; ++t) {
      const bool at = (long long)v[t] >= (long long)lo;
      bal[t] = __ballot_sync(FULL, at);
      mine |= at ? 1u << t : 0u;
      tot += __popc(bal[t]);
    }
    if (!tot) continue;  // warp-uniform
    int at = 0;
    if (lane == 0) at = atomicAdd(cnt, tot);
    at = __shfl_sync(FULL, at, 0);
    while (mine) {  // a lane seldom has two
      const int t = __ffs(mine) - 1;
      mine &= mine - 1;
      unsigned long long x = v[0];
      unsigned bt = bal[0];
      int before = 0;
#pragma unroll
      for (int u = 1; u < U; ++u)
        if (t >= u) {
          before += __popc(bal[u - 1]);
          x = v[u];
          bt = bal[u];
        }
      const int k = at + before + __popc(bt & lt);
      if (k < LCAP) {
        s.ck[k] = gain_key(x);
        s.cj[k] = j0 + t * SEL_THREADS + lane;
      }
    }
  }
}

// Exact threshold of the pool by a radix search over the gains (the guess of
// the caller listed too few or too many).  On return ck / cj list every token the
// pool can hold (n of them, returned, at most LCAP): the tokens of at least the
// P-th largest gain's bucket, its mantissa refined 11 bits at a time until the
// list fits; if even equal gains overflow it, the lowest tokens among them.
// *cnt and the keys are zero on entry.  Every thread calls it and gets the same
// n and threshold.
template <class Addr>
__device__ int pool_search(Addr addr, const uint32_t* ga, const SelSmem& s, int N, int P, int* cnt,
                           unsigned long long* lo) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int e = -1, bits = 5;           // boundary exponent, mantissa bits of the prefix
  unsigned long long pre = 0;     // boundary prefix: leading one and `bits` bits
  int above = 0;                  // tokens above the boundary prefix
  for (int level = 0;; ++level) {
    // histogram of the next digit: (exponent, 5 bits), then 11 bits of the
    // tokens that share the boundary prefix
    const int nbits = level == 0 ? 5 : min(bits + 11, 63);
    for (int j = threadIdx.x; j < N; j += SEL_THREADS) {
      const long long v = (long long)load_cluster(addr(j));
      if (v <= 0) continue;
      const int lz = __clzll(v);
      const unsigned long long m = (unsigned long long)v << lz;
      int bin;
      if (level == 0) {
        bin = sel::gain_bucket(v);
      } else {
        if (63 - lz != e || (m >> (63 - bits)) != pre) continue;
        bin = (int)((m >> (63 - nbits)) & ((1ull << (nbits - bits)) - 1));
      }
      atomicAdd(&s.hist[bin], 1);
    }
    __syncthreads();
    if (wid == 0) {  // the bin holding the P-th largest: 64 bins per lane, top first
      int c = 0;
      for (int t = 0; t < HBINS / 32; ++t) c += s.hist[HBINS - 1 - (lane * (HBINS / 32) + t)];
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
      }
      const int need = P - above;
      const unsigned reach = __ballot_sync(FULL, incl >= need);
      if (lane == 0) s.scal[SC_BIN] = -1;
      __syncwarp();
      if (reach && lane == __ffs(reach) - 1) {
        int acc = incl - c, b = HBINS - 1 - lane * (HBINS / 32);
        while (acc + s.hist[b] < need) acc += s.hist[b--];
        s.scal[SC_BIN] = b;
        s.scal[SC_ABOVE] = acc;
        s.scal[SC_COUNT] = s.hist[b];
      }
    }
    __syncthreads();
    for (int h = threadIdx.x; h < HBINS; h += SEL_THREADS) s.hist[h] = 0;
    const int bin = s.scal[SC_BIN], in = s.scal[SC_COUNT], ab = s.scal[SC_ABOVE];
    __syncthreads();
    if (bin < 0) {  // level 0 only: every positive token enters (fewer than P)
      *lo = 1;
      list_candidates(addr, ga, s, N, 1ull, cnt);
      __syncthreads();
      return *cnt;
    }
    if (level == 0) {
      e = bin >> 5;
      pre = 32ull | (unsigned)(bin & 31);
    } else {
      pre = (pre << (nbits - bits)) | (unsigned)bin;
      bits = nbits;
    }
    above += ab;
    if (above + in <= LCAP) {
      *lo = prefix_edge(e, bits, pre);
      list_candidates(addr, ga, s, N, *lo, cnt);
      __syncthreads();
      return *cnt;
    }
    if (bits == 63) break;  // equal gains
  }
  // the tokens above the boundary gain, then the lowest of the equal ones
  const unsigned long long v0 = prefix_edge(e, 63, pre);
  *lo = v0;
  list_candidates(addr, ga, s, N, v0 + 1, cnt);
  __syncthreads();
  const int base = *cnt, need = P - base;
  const int per = (N + SEL_THREADS - 1) / SEL_THREADS;
  const int j0 = min(N, (int)threadIdx.x * per), j1 = min(N, j0 + per);
  auto equal = [&](int j) { return load_cluster(addr(j)) == v0; };
  int c = 0;
  for (int j = j0; j < j1; ++j) c += equal(j);
  int at = block_exclusive_scan(c, s.wsum, nullptr);
  for (int j = j0; j < j1 && at < need; ++j)
    if (equal(j)) {
      s.ck[base + at] = gain_key(v0);
      s.cj[base + at] = j;
      ++at;
    }
  __syncthreads();
  if (threadIdx.x == 0) *cnt = P;
  __syncthreads();
  return P;
}

}  // namespace

__global__ void __launch_bounds__(SEL_THREADS, 1) k_select(SelArgs a) {
  grid_dep_wait();
  extern __shared__ __align__(16) char sm_sel[];
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks();
  const int r = (int)cluster.block_rank();
  const int b = blockIdx.x / CS;
  const int N = a.N, P = a.P, K = a.K;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;

  // Image geometry: rows [0, MG) grounded, [MG, MG+N) appearance, rest spatial.
  int Mb, MG;
  bool valid = true;
  if (a.uniform_rows) {
    Mb = a.Mstride;
    MG = Mb;  // everything reported as bank 0
  } else {
    const TextGeom tg = text_geom(a.toff, b, a.B, a.Tmax, nullptr);
    valid = tg.T > 0;
    MG = a.H * tg.T;
    Mb = MG + N + a.L2;
  }
  // token j's gain is kept by CTA j / SL: whole warps of consecutive tokens
  const int SL = ((N + CS - 1) / CS + 31) & ~31;
  const unsigned slm = (unsigned)(0x100000000ull / (unsigned)SL) + 1u;  // j / SL, j < 2^16
  auto owner = [&](int j) { return (int)__umulhi((unsigned)j, slm); };
  // Rows are dealt to the CTAs in turn (CTA r holds rows r, r + CS, ...):
  // every CTA gets the same mix of grounded, appearance and spatial rows and
  // of the image's regions, so the work of every phase is about even.  The
  // layout is the same in every CTA of the cluster (remote addresses).
  const int R = (Mb + CS - 1) / CS;
  const int nrows = Mb > r ? (Mb - r + CS - 1) / CS : 0;
  auto grow = [&](int q) { return q * CS + r; };  // client row of local row q
  const Layout lay = sel_layout(N, P, CS, SL, R);
  SelSmem s;  // pointers formed here, from the shared array itself: shared-space accesses
  s.gacc = reinterpret_cast<unsigned long long*>(sm_sel + lay.o.gacc);
  s.sown = reinterpret_cast<unsigned long long*>(sm_sel + lay.o.sown);
  s.spart = reinterpret_cast<unsigned long long*>(sm_sel + lay.o.spart);
  s.s_acc = reinterpret_cast<long long*>(sm_sel + lay.o.s_acc);
  s.fb = reinterpret_cast<long long*>(sm_sel + lay.o.fb);
  s.ck = reinterpret_cast<uint32_t*>(sm_sel + lay.o.ck);
  s.cj = reinterpret_cast<int*>(sm_sel + lay.o.cj);
  s.selw = reinterpret_cast<uint32_t*>(sm_sel + lay.o.selw);
  s.wpre = reinterpret_cast<int*>(sm_sel + lay.o.wpre);
  s.pool = reinterpret_cast<int*>(sm_sel + lay.o.pool);
  s.wsum = reinterpret_cast<int*>(sm_sel + lay.o.wsum);
  s.scal = reinterpret_cast<int*>(sm_sel + lay.o.scal);
  s.hist = reinterpret_cast<int*>(sm_sel + lay.o.hist);
  s.bcov = reinterpret_cast<float*>(sm_sel + lay.o.bcov);
  s.rmaxb = reinterpret_cast<int*>(sm_sel + lay.o.rmaxb);
  s.zlo = reinterpret_cast<uint32_t*>(sm_sel + lay.o.zlo);
  s.zhi = reinterpret_cast<uint32_t*>(sm_sel + lay.o.zhi);
  s.bnb = reinterpret_cast<int*>(sm_sel + lay.o.bnb);
  s.rptr = reinterpret_cast<uint16_t*>(sm_sel + lay.o.rptr);
  s.chg = reinterpret_cast<uint16_t*>(sm_sel + lay.o.chg);
  s.uloc = reinterpret_cast<uint32_t*>(sm_sel + lay.o.uloc);
  s.sk = reinterpret_cast<uint32_t*>(sm_sel + lay.o.sk);
  s.cs = reinterpret_cast<int*>(sm_sel + lay.o.cs);
  s.rval = reinterpret_cast<float*>(sm_sel + lay.o.rval);
  s.rtok = reinterpret_cast<uint16_t*>(sm_sel + lay.o.rtok);
  s.crow = reinterpret_cast<uint16_t*>(sm_sel + lay.o.crow);
  s.cpos = reinterpret_cast<uint16_t*>(sm_sel + lay.o.cpos);
  s.sw = reinterpret_cast<unsigned long long*>(sm_sel + lay.o.sw);
  s.inb = reinterpret_cast<int*>(sm_sel + lay.o.inb);
  s.poolslot = reinterpret_cast<short*>(sm_sel + lay.o.poolslot);
  const int e = a.fexp ? a.fexp[b] : a.fx_exp;
  const float fxs = ldexpf(1.f, e);
  float* Cimg = a.C + (size_t)b * a.Mstride * N;
  uint16_t* Simg = a.scol + (size_t)b * a.Mstride * N;
  const int nwords = (N + 31) >> 5;
  const int SP = sel_pool_stride(P);

  // state after the rounds run on the whole GPU (k_round0.cu); a first round
  // with an empty pool leaves the gains of the empty support and nothing
  // selected
  const int rd0 = valid ? a.r0.info[b * INFO_W + 2] : 0;    // rounds done
  const int nb0 = rd0 > 0 ? a.r0.info[b * INFO_W + 1] : 0;  // tokens selected so far
  // pool threshold: below the boundary bucket of the last pool (-1: every
  // candidate entered it)
  unsigned long long lo = 1;
  {
    const int hint = rd0 > 0 ? a.r0.info[b * INFO_W + 5] : -1;
    if (hint >= 0) {
      lo = prefix_edge(hint >> 5, 5, 32ull | (unsigned)(hint & 31));
      lo -= lo >> 2;
    }
    if (lo == 0) lo = 1;
  }
  const long long* ug = rd0 > 0 ? a.r0.ugain : a.u0;
  for (int q = threadIdx.x; q < SL; q += SEL_THREADS) {  // the gains of the tokens this CTA owns
    const int j = r * SL + q;
    s.gacc[q] = j < N ? (unsigned long long)ug[(size_t)b * N + j] : 0ull;
  }
  for (int q = threadIdx.x; q < nwords; q += SEL_THREADS)
    s.selw[q] = q == nwords - 1 && (N & 31) ? ~0u << (N & 31) : 0u;  // past N: taken
  for (int h = threadIdx.x; h < HBINS; h += SEL_THREADS) s.hist[h] = 0;
  for (int j = threadIdx.x; j < N; j += SEL_THREADS) s.poolslot[j] = -1;
  const bool agg = aggregates(N, R);
  if (agg)
    for (int j = threadIdx.x; j < 3 * N; j += SEL_THREADS) s.uloc[j] = 0;
  for (int k = threadIdx.x; k < ((SP + 3) & ~3); k += SEL_THREADS) s.sk[k] = 0;
  for (int q = threadIdx.x; q < LCAP; q += SEL_THREADS) s.ck[q] = 0;
  if (threadIdx.x < 8) s.fb[threadIdx.x] = threadIdx.x == FB_LO ? (long long)lo : 0;
  if (threadIdx.x < 16) s.scal[threadIdx.x] = threadIdx.x == SC_GLOBAL;
  for (int q = threadIdx.x; q < nrows; q += SEL_THREADS) {
    const bool have = rd0 > 0;
    s.bcov[q] = have ? a.r0.bcov[(size_t)b * a.Mstride + grow(q)] : 0.f;
    s.rptr[q] = have ? (uint16_t)a.r0.cnt[(size_t)b * a.Mstride + grow(q)] : 0;
    s.rmaxb[q] = 0;
    s.zlo[q] = 0;
    s.zhi[q] = 0;
    s.bnb[q] = 0;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < nb0; q += SEL_THREADS) {
    const int j = a.order[(size_t)b * K + q];
    atomicOr(&s.selw[j >> 5], 1u << (j & 31));
  }
  cluster.sync();
  if (!valid) return;  // uniform across the cluster

  const int sub = lane / G, gl = lane % G;
  const int gid = wid * (32 / G) + sub, ngrp = SEL_WARPS * (32 / G);  // 8-lane groups
  const unsigned gm = 0xFFu << (sub * G);
  const unsigned lt = lanemask_lt() & gm;

  // Move this CTA's survivor lists from global into shared memory once they
  // all fit: copied row by row, then indexed by token with a counting sort.  The
  // order inside a token's segment depends on the schedule; nothing computed
  // from it does (integer and max reductions).
  auto migrate = [&]() {
    if (!s.scal[SC_GLOBAL] || nrows > 65535) return;  // row ids are stored in 16 bits
    const int rper = (nrows + SEL_THREADS - 1) / SEL_THREADS;
    const int q0 = min(nrows, (int)threadIdx.x * rper), q1 = min(nrows, q0 + rper);
    int mine = 0;
    for (int q = q0; q < q1; ++q) mine += s.rptr[q];
    int tot = 0;
    int at = block_exclusive_scan(mine, s.wsum, &tot);
    if (tot > lay.cap) return;  // uniform over the block; below 2^16: positions are 16 bits
    for (int q = q0; q < q1; ++q) {
      const int n = s.rptr[q];
      s.rptr[q] = (uint16_t)at;
      at += n;
    }
    if (threadIdx.x == 0) s.rptr[nrows] = (uint16_t)tot;
    for (int j = threadIdx.x; j <= N; j += SEL_THREADS) s.cs[j] = 0;
    __syncthreads();
    // every entry by one thread, MU loads in flight (rows are very uneven); tokens
    // counted in cs[j + 1].  Its row: the row of its 32 entries' first one, from a table
    // (a binary search of the rows' offsets for each, kept in the histogram's bins), then a
    // step or two; a search for every entry was most of the time before the first round (21
    // us at N = 1,296, now 12).
    for (int c = threadIdx.x; 32 * c < tot; c += SEL_THREADS) {
      int lo2 = 0, hi2 = nrows;  // rptr[lo2] <= p < rptr[hi2]
      while (hi2 - lo2 > 1) {
        const int mid = (lo2 + hi2) >> 1;
        if (s.rptr[mid] <= 32 * c) lo2 = mid; else hi2 = mid;
      }
      s.hist[c] = lo2;
    }
    __syncthreads();
    auto row_of = [&](int p) {
      int q = s.hist[p >> 5];
      while (s.rptr[q + 1] <= p) ++q;
      return q;
    };
    constexpr int MU = 8;
    for (int b0 = threadIdx.x; b0 < tot; b0 += MU * SEL_THREADS) {
      float v[MU];
      int j[MU];
#pragma unroll
      for (int u = 0; u < MU; ++u) {
        const int p = b0 + u * SEL_THREADS;
        v[u] = 0.f;
        j[u] = -1;
        if (p < tot) {
          const int q = row_of(p);
          const size_t g = (size_t)grow(q) * N + (p - s.rptr[q]);
          v[u] = Cimg[g];
          j[u] = Simg[g];
        }
      }
#pragma unroll
      for (int u = 0; u < MU; ++u)
        if (j[u] >= 0) {
          s.rval[b0 + u * SEL_THREADS] = v[u];
          s.rtok[b0 + u * SEL_THREADS] = (uint16_t)j[u];
          atomicAdd(&s.cs[j[u] + 1], 1);
        }
    }
    __syncthreads();
    {  // cs[j + 1] becomes the first entry of token j, then its fill cursor
      const int per = (N + SEL_THREADS - 1) / SEL_THREADS;
      const int j0 = min(N, (int)threadIdx.x * per), j1 = min(N, j0 + per);
      int c = 0;
      for (int j = j0; j < j1; ++j) c += s.cs[j + 1];
      int first = block_exclusive_scan(c, s.wsum, nullptr);
      for (int j = j0; j < j1; ++j) {
        const int n = s.cs[j + 1];
        s.cs[j + 1] = first;
        first += n;
      }
    }
    __syncthreads();
    for (int p = threadIdx.x; p < tot; p += SEL_THREADS) {
      const int d = atomicAdd(&s.cs[s.rtok[p] + 1], 1);
      s.crow[d] = (uint16_t)row_of(p);
      s.cpos[d] = (uint16_t)p;
    }
    __syncthreads();  // cs[j] is now the first entry of token j, cs[N] the total
    for (int c = threadIdx.x; 32 * c < tot; c += SEL_THREADS) s.hist[c] = 0;
    if (threadIdx.x == 0) s.scal[SC_GLOBAL] = 0;
    __syncthreads();
  };
  if (rd0 > 0) migrate();

  const int rounds_max = (K + a.bsz - 1) / a.bsz + 1 + (a.images > 1 ? 1 : 0);
  // where token j's gain is, and where those of this thread's first tokens are
  auto gain_addr = [&](int j) {
    const int o = owner(j);
    return cluster_addr(s.gacc + (j - o * SL), o);
  };
  uint32_t ga[GA];
#pragma unroll
  for (int t = 0; t < GA; ++t) ga[t] = gain_addr(min(N - 1, (int)threadIdx.x + t * SEL_THREADS));
  // add v to token j's gain at its owner (exact: 64-bit integer additions,
  // order-independent)
  auto gain_add = [&](int j, unsigned long long v) {
    red_add_cluster(gain_addr(j), v);
  };
  int S_count = nb0, rnd = rd0, filled = 0;
  // kept by the last thread: gain of the last pool's last token, its smoothed fall per
  // round, room left below the expected one
  float glast = 0.f, fall = 0.85f, room = 0.8f;
  while (S_count < K) {
    if (rnd >= rounds_max) {  // cannot happen (each round adds >= 1 token); guard the loop
      if (threadIdx.x == 0) set_status(a.status, GMC_STATUS_INTERNAL);
      break;
    }
    const bool flat = !s.scal[SC_GLOBAL];
    // ---- pool of this round ------------------------------------------------------
    // counters: zero; the other parity's are cleared below
    int* cnt = &s.scal[SC_N0 + (rnd & 1)];
    int* rsum = &s.scal[SC_R0 + (rnd & 1)];
    lo = (unsigned long long)s.fb[FB_LO];
    list_candidates(gain_addr, ga, s, N, lo, cnt);
    __syncthreads();
    int n = *cnt;
    const int guessed = n;
    int listed = n;
    if (n < P && lo > 1) {  // too few: once more from half the gain or a quarter of it
      __syncthreads();
      if (threadIdx.x == 0) *cnt = 0;
      s.ck[threadIdx.x] = 0;  // LCAP == SEL_THREADS
      lo = max(1ull, 4 * n < P ? lo >> 2 : lo >> 1);
      __syncthreads();
      list_candidates(gain_addr, ga, s, N, lo, cnt);
      __syncthreads();
      listed = n = *cnt;
    }
    if (n > LCAP || (n < P && lo > 1)) {  // the guess missed (uniform over the cluster)
      __syncthreads();
      if (threadIdx.x == 0) *cnt = 0;
      s.ck[threadIdx.x] = 0;  // LCAP == SEL_THREADS
      __syncthreads();
      listed = n = pool_search(gain_addr, ga, s, N, P, cnt, &lo);
    }
    const int Pt = min(n, P);
    // Ranking costs the square of the list: a long one is cut first, to those at or
    // above a key found by halving the keys' range (a barrier a step) that leaves P to
    // RANK_MAX of them (more where keys are equal).  405 candidates: 5 us, now 0.9.
    constexpr int RANK_MAX = SEL_THREADS / 4;  // ranked in one turn
    if (n > max(RANK_MAX, P)) {
      const uint32_t key = s.ck[threadIdx.x];  // LCAP == SEL_THREADS; past the list: 0
      const int jq = s.cj[threadIdx.x];
      const uint32_t top = __reduce_max_sync(FULL, key);
      if (lane == 0) s.wsum[wid] = (int)top;
      __syncthreads();
      uint32_t above = __reduce_max_sync(FULL, (uint32_t)s.wsum[lane & (SEL_WARPS - 1)]) + 1;
      uint32_t from = gain_key(lo);
      while (n > max(RANK_MAX, P) && above - from > 1) {  // n keys >= from, fewer than P >= above
        const uint32_t mid = from + ((above - from) >> 1);
        const int c = __syncthreads_count(key >= mid);
        if (c >= P) {
          from = mid;
          n = c;
        } else {
          above = mid;
        }
      }
      const bool in = (int)threadIdx.x < listed && key >= from;
      const unsigned bal = __ballot_sync(FULL, in);
      __syncthreads();  // every key and token is in a register, wsum has been read
      s.ck[threadIdx.x] = 0;
      if (lane == 0) s.wsum[wid] = __popc(bal);
      __syncthreads();
      const int before = __reduce_add_sync(FULL, lane < wid ? s.wsum[lane] : 0);
      if (in) {
        const int at = before + __popc(bal & lanemask_lt());
        s.ck[at] = key;
        s.cj[at] = jq;
      }
      __syncthreads();
    }
    // rank every candidate by its key among them (4 lanes each, four keys a load);
    // slot = rank
    {
      const uint4* k4 = reinterpret_cast<const uint4*>(s.ck);
      const int n4 = (n + 3) >> 2;
      for (int base = ((int)threadIdx.x - lane) >> 2; base < n; base += SEL_THREADS >> 2) {
        const int q = base + (lane >> 2);
        const uint32_t key = q < n ? s.ck[q] : 0xffffffffu;  // past the list: rank 0
        int gt = 0;
#pragma unroll 4
        for (int c = lane & 3; c < n4; c += 4) {
          const uint4 x = k4[c];
          gt += (x.x > key) + (x.y > key) + (x.z > key) + (x.w > key);
        }
        const int all = __reduce_add_sync(FULL, gt);
        if (lane == 0) atomicAdd(rsum, all);
        gt += __shfl_xor_sync(FULL, gt, 1);
        gt += __shfl_xor_sync(FULL, gt, 2);
        if (q < n && (lane & 3) == 0 && gt < Pt) {
          s.pool[gt] = s.cj[q];
          if (gt == Pt - 1) s.scal[SC_KEY] = (int)key;
        }
      }
    }
    if (!flat)
      for (int k = threadIdx.x; k < SEL_WARPS * Pt; k += SEL_THREADS) s.sw[k] = 0;
    if (r == 0 && a.tv.base)  // certificate input: the gains this round starts from
      for (int j = threadIdx.x; j < N; j += SEL_THREADS)
        a.tv.gains(b, rnd, N)[j] = (long long)load_cluster(gain_addr(j));
    __syncthreads();
    if (*rsum != n * (n - 1) / 2) {
      // equal keys: the ranks by (gain desc, token asc), gains read again
      __syncthreads();
      for (int q = threadIdx.x; q < n; q += SEL_THREADS) {
        const uint32_t key = s.ck[q];
        const int jq = s.cj[q];
        const long long v = (long long)load_cluster(gain_addr(jq));
        int rank = 0;
        for (int q2 = 0; q2 < n; ++q2) {
          const uint32_t k2 = s.ck[q2];
          rank += k2 > key ||
                  (k2 == key && q2 != q &&
                   key_before((long long)load_cluster(gain_addr(s.cj[q2])), s.cj[q2], v, jq));
        }
        if (rank < Pt) {
          s.pool[rank] = jq;
          if (rank == Pt - 1) s.scal[SC_KEY] = (int)key;
        }
      }
      __syncthreads();
    }
    if (Pt == 0) {
      // Zero-gain remainder: fill in ascending source order (F unchanged).
      const int need = K - S_count;
      int c = threadIdx.x < nwords ? __popc(~s.selw[threadIdx.x]) : 0;
      c = block_exclusive_scan(c, s.wsum, nullptr);  // nwords <= 256
      if (threadIdx.x < nwords) {
        uint32_t free_ = ~s.selw[threadIdx.x];
        while (free_ && c < need) {
          const int bit = __ffs(free_) - 1;
          free_ &= free_ - 1u;
          s.selw[threadIdx.x] |= 1u << bit;
          if (r == 0) a.order[(size_t)b * K + S_count + c] = 32 * (int)threadIdx.x + bit;
          ++c;
        }
      }
      if (r == 0 && a.tv.base && threadIdx.x == 0) {
        int32_t* tp = a.tv.at<int32_t>(b, a.tv.off_pool) + (size_t)rnd * a.tv.pool_size;
        for (int k = 0; k < a.tv.pool_size; ++k) tp[k] = -1;
        a.tv.at<int32_t>(b, a.tv.off_round_end)[rnd] = K;
      }
      filled = need;
      S_count = K;
      ++rnd;
      __syncthreads();
      break;
    }
    s.ck[threadIdx.x] = 0;  // LCAP == SEL_THREADS
    if (threadIdx.x == 0) {
      s.scal[SC_N0 + ((rnd + 1) & 1)] = 0;
      s.scal[SC_R0 + ((rnd + 1) & 1)] = 0;
      s.scal[SC_NCHG] = 0;
    }
    // Threshold of the next pool, by the last thread while others work: the gain g at
    // rank P, lowered by the smoothed fall of g per round and by a factor that the
    // lists' lengths steer to 3 P / 2 to 3 P candidates.
    auto next_threshold = [&]() {
      unsigned long long next = 1;
      if (Pt == P) {
        const float g = key_gain((uint32_t)s.scal[SC_KEY]);
        if (glast > 0.f) fall = 0.5f * (fall + fminf(1.f, fmaxf(0.4f, __fdividef(g, glast))));
        glast = g;
        room *= guessed > 6 * P ? 1.25f : guessed > 4 * P ? 1.12f : guessed > 3 * P ? 1.05f
                : guessed < P ? 0.85f : guessed < 3 * P / 2 ? 0.95f : 1.f;
        room = fminf(0.97f, fmaxf(0.3f, room));
        next = (unsigned long long)__float2ull_rz(g * fall * room);
        if (next == 0) next = 1;
      }
      s.fb[FB_LO] = (long long)next;
    };
    if (!flat) {  // uniform over the block
      for (int k = threadIdx.x; k < Pt; k += SEL_THREADS) s.poolslot[s.pool[k]] = (short)k;
      __syncthreads();
    }
    if (r == 0 && a.tv.base && threadIdx.x < a.tv.pool_size) {
      int32_t* tp = a.tv.at<int32_t>(b, a.tv.off_pool) + (size_t)rnd * a.tv.pool_size;
      tp[threadIdx.x] = threadIdx.x < Pt ? s.pool[threadIdx.x] : -1;
    }

    // ---- responsibilities and scores of this CTA's rows over the pool ----------------
    const float z_one = 1099511627776.f;  // 2^40: fixed-point scale of the softmax denominators
    const float z_inv = 1.f / z_one;
    const bool keep = flat && Pt <= ngrp;
    int kq[EC];
    float kV[EC] = {}, kR[EC] = {}, kE[EC], k0[EC];
    int p0 = 0, p1 = 0;  // the group's pool token: its entries not kept in registers
    if (flat) {
      // One 8-lane group per pool token reads the token's entries.  Per-row
      // values are order-independent (max of positive floats as integers,
      // fixed-point sums), so nothing depends on the schedule.  A lane keeps its
      // first EC entries in registers to the end of the round; longer segments
      // (and pools of more than ngrp tokens) are read again.
#pragma unroll
      for (int u = 0; u < EC; ++u) kq[u] = -1;
      // one entry: its row, value and residual (row -1: dead)
      auto entry = [&](int p, int& q, float& V, float& Rv) {
        q = s.crow[p];
        V = s.rval[s.cpos[p]];
        Rv = V - s.bcov[q];
        if (!(Rv > 0.f)) q = -1;
      };
      // step 1: largest pool residual and number of pool entries of a row
      auto step1 = [&](int q, float Rv) {
        atomicMax(&s.rmaxb[q], __float_as_int(Rv));
        atomicAdd(&s.zhi[q], 1u << 24);
      };
      // the row's largest residual, its temperature and the reciprocal of that
      auto row = [&](int q, float& rmax, float& t, float& rt) {
        rmax = __int_as_float(s.rmaxb[q]);
        t = a.resp_temp * rmax + a.resp_eps;
        rt = __frcp_rn(t);
      };
      // step 2: softmax denominators shifted by the row's largest logit (every term
      // at most 1, so at most 2^40 * pool size), exact in 2^-40
      auto add_z = [&](int q, float ex) {
        const unsigned long long z = (unsigned long long)to_fix(ex, z_one);
        atomicAdd(&s.zlo[q], (uint32_t)z & 0xffffffu);
        atomicAdd(&s.zhi[q], (uint32_t)(z >> 24));
      };
      // step 3: rho R, fixed point; pool tokens without an entry in row q have R = 0
      // and add e0 each to the row's denominator
      auto weigh = [&](int q, float Rv, float ex, float e0) {
        const uint32_t hi = s.zhi[q];
        const unsigned long long zf = ((unsigned long long)(hi & 0xffffffu) << 24) + s.zlo[q];
        const float z = fix_to_float(zf) * z_inv + (float)(Pt - (int)(hi >> 24)) * e0;
        return (unsigned long long)to_fix(ex / z * Rv, fxs);
      };
      for (int k = gid; k < Pt; k += ngrp) {
        const int j = s.pool[k];
        int p = s.cs[j] + gl;
        p1 = s.cs[j + 1];
        if (keep) {
#pragma unroll
          for (int u = 0; u < EC; ++u)
            if (p + u * G < p1) entry(p + u * G, kq[u], kV[u], kR[u]);
#pragma unroll
          for (int u = 0; u < EC; ++u)
            if (kq[u] >= 0) step1(kq[u], kR[u]);
          p += EC * G;
          p0 = p;
        }
        for (; p < p1; p += G) {
          int q;
          float V, Rv;
          entry(p, q, V, Rv);
          if (q >= 0) step1(q, Rv);
        }
      }
      __syncthreads();
      for (int k = gid; k < Pt; k += ngrp) {
        int p = p0;
        if (keep) {
          float rmax[EC], t[EC], rt[EC];
#pragma unroll
          for (int u = 0; u < EC; ++u) row(max(kq[u], 0), rmax[u], t[u], rt[u]);
#pragma unroll
          for (int u = 0; u < EC; ++u) {
            kE[u] = expf(div_by(kR[u] - rmax[u], t[u], rt[u]));
            k0[u] = expf(div_by(-rmax[u], t[u], rt[u]));
          }
#pragma unroll
          for (int u = 0; u < EC; ++u)
            if (kq[u] >= 0) add_z(kq[u], kE[u]);
        } else {
          p = s.cs[s.pool[k]] + gl;
          p1 = s.cs[s.pool[k] + 1];
        }
        for (; p < p1; p += G) {
          int q;
          float V, Rv;
          entry(p, q, V, Rv);
          if (q < 0) continue;
          float rmax, t, rt;
          row(q, rmax, t, rt);
          add_z(q, expf(div_by(Rv - rmax, t, rt)));
        }
      }
      __syncthreads();
      for (int k = gid; k < Pt; k += ngrp) {
        unsigned long long acc = 0;
        int p = p0;
        if (keep) {
#pragma unroll
          for (int u = 0; u < EC; ++u)
            if (kq[u] >= 0) acc += weigh(kq[u], kR[u], kE[u], k0[u]);
        } else {
          p = s.cs[s.pool[k]] + gl;
          p1 = s.cs[s.pool[k] + 1];
        }
        for (; p < p1; p += G) {
          int q;
          float V, Rv;
          entry(p, q, V, Rv);
          if (q < 0) continue;
          float rmax, t, rt;
          row(q, rmax, t, rt);
          acc += weigh(q, Rv, expf(div_by(Rv - rmax, t, rt)), expf(div_by(-rmax, t, rt)));
        }
        acc = group_sum(acc, gm);
        if (gl == 0) s.sown[k] = acc;
      }
    } else {
      // 8-lane group per row.  One sweep of the row finds its pool entries; each
      // lane keeps up to PCL of them in registers for the softmax (more: a
      // second sweep).
      for (int q0 = wid * (32 / G); q0 < nrows; q0 += SEL_WARPS * (32 / G)) {
        const int q = q0 + sub;
        const int n = q < nrows ? s.rptr[q] : 0;
        const float bm = q < nrows ? s.bcov[q] : 0.f;
        const float* vals = Cimg + (size_t)grow(q) * N;
        const uint16_t* cols = Simg + (size_t)grow(q) * N;
        float rmax = 0.f;
        int npool = 0, ncache = 0, mine = 0;  // mine: pool entries this lane saw
        float cv[PCL] = {};
        int cs[PCL] = {};
        bool spill = false;
        for (int k0 = gl; k0 < n; k0 += UNR * G) {
          int cc[UNR];
          float vv[UNR];
#pragma unroll
          for (int u = 0; u < UNR; ++u) {
            const int k = k0 + u * G;
            cc[u] = k < n ? (int)cols[k] : -1;
            vv[u] = k < n ? vals[k] : 0.f;
          }
#pragma unroll
          for (int u = 0; u < UNR; ++u) {
            const int ps = cc[u] >= 0 ? s.poolslot[cc[u]] : -1;
            if (ps >= 0) {
              rmax = fmaxf(rmax, vv[u] - bm);
#pragma unroll
              for (int t = 0; t < PCL; ++t)
                if (t == mine) {
                  cv[t] = vv[u];
                  cs[t] = ps;
                }
              spill |= mine >= PCL;
              ++mine;
            }
          }
        }
        rmax = group_max(rmax, gm);
        npool = group_sum(mine, gm);
        const bool any_spill = __any_sync(gm, spill);
        ncache = mine < PCL ? mine : PCL;
        if (npool > 0) {
          // softmax shifted by the row's largest logit (exponentials at most 1)
          const float tau = a.resp_temp * rmax + a.resp_eps;
          float z = 0.f;
          if (!any_spill) {
#pragma unroll
            for (int t = 0; t < PCL; ++t)
              if (t < ncache) z += expf(((cv[t] - bm) - rmax) / tau);
          } else {
            for (int k = gl; k < n; k += G)
              if (s.poolslot[cols[k]] >= 0) z += expf(((vals[k] - bm) - rmax) / tau);
          }
          z = group_sum(z, gm) + (float)(Pt - npool) * expf(-rmax / tau);  // R = 0 entries
          const float invz = 1.f / z;
          if (!any_spill) {
#pragma unroll
            for (int t = 0; t < PCL; ++t)
              if (t < ncache) {
                const float Rv = cv[t] - bm;
                atomicAdd(&s.sw[wid * Pt + cs[t]],
                          (unsigned long long)to_fix(expf((Rv - rmax) / tau) * invz * Rv, fxs));
              }
          } else {
            for (int k = gl; k < n; k += G) {
              const int ps = s.poolslot[cols[k]];
              if (ps >= 0) {
                const float Rv = vals[k] - bm;
                atomicAdd(&s.sw[wid * Pt + ps],
                          (unsigned long long)to_fix(expf((Rv - rmax) / tau) * invz * Rv, fxs));
              }
            }
          }
        }
      }
      __syncthreads();
      for (int k = threadIdx.x; k < Pt; k += SEL_THREADS) {
        unsigned long long v = 0;
        for (int w2 = 0; w2 < SEL_WARPS; ++w2) v += s.sw[w2 * Pt + k];
        s.sown[k] = v;
      }
    }
    __syncthreads();
    // this CTA's scores into its row of every CTA: one warp per target, whole lines
    for (int c = wid; c < CS; c += SEL_WARPS)
      for (int k = 2 * lane; k < Pt; k += 64)
        store2_cluster(cluster_addr(s.spart + (size_t)r * SP + k, c), s.sown[k], s.sown[k + 1]);
    // Barrier: every CTA's scores have reached every CTA, and every CTA has read this
    // round's gains.  Between arriving and waiting: the threshold, and the
    // responsibilities' row values back to zero.
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    if (threadIdx.x == SEL_THREADS - 1) next_threshold();
    if (flat)
      for (int q = threadIdx.x; q < nrows; q += SEL_THREADS) {
        s.rmaxb[q] = 0;
        s.zlo[q] = 0;
        s.zhi[q] = 0;
      }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

    // ---- batch: the slots' sums, ranked -------------------------------------------
    const int nb = min(a.bsz, min(Pt, K - S_count));
    if (threadIdx.x < ((Pt + 3) & ~3)) {  // at most P <= GMC_MAX_POOL slots: a thread each
      const int k = threadIdx.x;
      unsigned long long v = 0;
      if (k < Pt) {
#pragma unroll 8
        for (int c = 0; c < CS; ++c) v += s.spart[c * SP + k];
      }
      s.s_acc[k] = (long long)v;
      s.sk[k] = (long long)v > 0 ? gain_key(v) : 0u;  // past Pt: zero
    }
    __syncthreads();
    // 8 lanes rank each pool token by its score's key, four keys a load; tokens whose
    // key is not alone are ranked by (score desc, token asc)
    for (int k = gid; k < Pt; k += ngrp) {
      const uint32_t key = s.sk[k];
      const int jk = s.pool[k];
      const uint4* k4 = reinterpret_cast<const uint4*>(s.sk);
      int gt = 0, ge = 0;
#pragma unroll 2
      for (int c = gl; c < (Pt + 3) >> 2; c += G) {  // keys past Pt: zero
        const uint4 x = k4[c];
        gt += (x.x > key) + (x.y > key) + (x.z > key) + (x.w > key);
        ge += (x.x >= key) + (x.y >= key) + (x.z >= key) + (x.w >= key);
      }
      int rank = group_sum((ge << 16) | gt, gm);
      ge = rank >> 16;
      rank &= 0xffff;
      if (ge != rank + 1) rank = sel::group_score_rank(s.s_acc, s.pool, Pt, k, gl, gm);
      if (gl == 0) {
        if (!flat) s.inb[k] = rank < nb;
        if (rank < nb) {
          atomicOr(&s.selw[jk >> 5], 1u << (jk & 31));
          if (r == 0) a.order[(size_t)b * K + S_count + rank] = jk;
        }
      }
      if (flat && rank < nb) {
        // the batch token's entries: largest value above the coverage per row;
        // whoever raises a row first lists it
        auto raise = [&](int q, float V) {
          if (atomicMax(&s.bnb[q], __float_as_int(V)) == 0)
            s.chg[atomicAdd(&s.scal[SC_NCHG], 1)] = (uint16_t)q;
        };
        int p = p0, pe = p1;
        if (keep) {
          int old[EC], nf = 0;
#pragma unroll
          for (int u = 0; u < EC; ++u)
            old[u] = kq[u] >= 0 ? atomicMax(&s.bnb[kq[u]], __float_as_int(kV[u])) : 1;
#pragma unroll
          for (int u = 0; u < EC; ++u) nf += old[u] == 0;
          int at = nf ? atomicAdd(&s.scal[SC_NCHG], nf) : 0;
#pragma unroll
          for (int u = 0; u < EC; ++u)
            if (old[u] == 0) s.chg[at++] = (uint16_t)kq[u];
        } else {
          p = s.cs[jk] + gl;
          pe = s.cs[jk + 1];
        }
        for (; p < pe; p += G) {
          const int q = s.crow[p];
          const float V = s.rval[s.cpos[p]];
          if (V > s.bcov[q]) raise(q, V);
        }
      }
    }
    __syncthreads();
    if (r == 0 && a.tv.base && threadIdx.x == 0)
      a.tv.at<int32_t>(b, a.tv.off_round_end)[rnd] = S_count + nb;
    // ---- coverage update and the changes of the gains ------------------------------
    if (flat) {
      // an entry's residual moves from C - b_old to C - b_new, or to zero when it
      // dies (exact: integers modulo 2^64)
      const int nchg = s.scal[SC_NCHG];
      for (int c = wid; c < nchg; c += SEL_WARPS) {  // a warp per row: rows are very uneven
        const int q = s.chg[c], pe = s.rptr[q + 1];
        const float bo = s.bcov[q], bn = __int_as_float(s.bnb[q]);
        const long long fo = to_fix(bo, fxs), fn = to_fix(bn, fxs);
        for (int pb = s.rptr[q] + lane; pb < pe; pb += UNR * 32) {
          float v[UNR];
          int j[UNR];
#pragma unroll
          for (int u = 0; u < UNR; ++u) {
            const int p = pb + u * 32;
            v[u] = p < pe ? s.rval[p] : 0.f;  // 0: below every coverage
            j[u] = p < pe ? (int)s.rtok[p] : 0;
          }
#pragma unroll
          for (int u = 0; u < UNR; ++u)
            if (v[u] > bo) {
              const unsigned long long d =  // the fall of the gain
                  (unsigned long long)((v[u] > bn ? fn : to_fix(v[u], fxs)) - fo);
              if (agg) sel::limb_add(&s.uloc[j[u]], N, d); else gain_add(j[u], 0ull - d);
            }
        }
        __syncwarp();
        if (lane == 0) {
          s.bcov[q] = bn;
          s.bnb[q] = 0;
        }
      }
      if (agg) {
        __syncthreads();
#pragma unroll
        for (int t = 0; t < GA; ++t) {
          const int j = (int)threadIdx.x + t * SEL_THREADS;
          if (j >= N) break;
          const unsigned long long d = sel::limb_value(s.uloc + j, N);
          if (d) {
            red_add_cluster(ga[t], 0ull - d);
            s.uloc[j] = s.uloc[N + j] = s.uloc[2 * N + j] = 0;
          }
        }
        for (int j = threadIdx.x + GA * SEL_THREADS; j < N; j += SEL_THREADS) {
          const unsigned long long d = sel::limb_value(s.uloc + j, N);
          if (d) {
            gain_add(j, 0ull - d);
            s.uloc[j] = s.uloc[N + j] = s.uloc[2 * N + j] = 0;
          }
        }
      }
    } else {
      for (int q0 = wid * (32 / G); q0 < nrows; q0 += SEL_WARPS * (32 / G)) {
        const int q = q0 + sub;
        const int n = q < nrows ? s.rptr[q] : 0;
        const float bm = q < nrows ? s.bcov[q] : 0.f;
        float* vals = Cimg + (size_t)grow(q) * N;
        uint16_t* cols = Simg + (size_t)grow(q) * N;
        float bnew = bm;
        for (int k0 = gl; k0 < n; k0 += UNR * G) {
          int cc[UNR];
          float vv[UNR];
#pragma unroll
          for (int u = 0; u < UNR; ++u) {
            const int k = k0 + u * G;
            cc[u] = k < n ? (int)cols[k] : -1;
            vv[u] = k < n ? vals[k] : 0.f;
          }
#pragma unroll
          for (int u = 0; u < UNR; ++u) {
            const int ps = cc[u] >= 0 ? s.poolslot[cc[u]] : -1;
            if (ps >= 0 && s.inb[ps]) bnew = fmaxf(bnew, vv[u]);
          }
        }
        bnew = group_max(bnew, gm);
        const long long fb_new = to_fix(bnew, fxs), fb_old = to_fix(bm, fxs);
        // a row whose coverage stayed keeps its list and changes no gain; the
        // others are compacted in place
        const int nch = bnew > bm ? n : 0;  // uniform over the group
        int w = n - nch;
        for (int base = 0; base < nch; base += UNR * G) {
          float c[UNR];
          int jj[UNR];
#pragma unroll
          for (int u = 0; u < UNR; ++u) {
            const int k = base + u * G + gl;
            c[u] = k < n ? vals[k] : 0.f;
            jj[u] = k < n ? (int)cols[k] : 0;
          }
          __syncwarp(gm);  // the group has read all UNR*G entries before any overwrite
#pragma unroll
          for (int u = 0; u < UNR; ++u) {
            const int k = base + u * G + gl;
            const bool keep = k < n && c[u] > bnew;
            const unsigned msk = __ballot_sync(gm, keep);
            if (k < n) {
              const long long d = keep ? fb_old - fb_new : fb_old - to_fix(c[u], fxs);
              if (d) gain_add(jj[u], (unsigned long long)d);
            }
            if (keep) {
              const int pos = w + __popc(msk & lt);
              vals[pos] = c[u];
              cols[pos] = (uint16_t)jj[u];
            }
            w += __popc(msk);
          }
        }
        if (gl == 0 && q < nrows) {
          s.bcov[q] = bnew;
          s.rptr[q] = (uint16_t)w;
        }
      }
    }
    if (a.tv.base) {  // certificate input: F(S) after this round, this CTA's rows
      __syncthreads();
      long long f = 0;
      for (int q = threadIdx.x; q < nrows; q += SEL_THREADS) f += to_fix(s.bcov[q], fxs);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(FULL, f, o);
      if (lane == 0 && f) atomicAdd(a.tv.cover(b, rnd), (unsigned long long)f);
    }
    if (!flat) {
      __syncthreads();
      for (int k = threadIdx.x; k < Pt; k += SEL_THREADS) s.poolslot[s.pool[k]] = -1;
      __syncthreads();
      migrate();
    }
    S_count += nb;
    ++rnd;
    if (S_count >= K) break;
    cluster.sync();  // every change of the gains has reached its owner
  }

  // ---- final: coverage per bank, sorted support, trace ---------------------
  __syncthreads();
  {
    long long f0 = 0, f1 = 0, f2 = 0;
    for (int q = threadIdx.x; q < nrows; q += SEL_THREADS) {
      const int m = grow(q);
      const long long v = to_fix(s.bcov[q], fxs);
      if (m < MG) f0 += v; else if (m < MG + N) f1 += v; else f2 += v;
    }
    if (a.tv.base) {
      long long* fb0 = cluster.map_shared_rank(s.fb, 0);
      if (f0) atomicAdd((unsigned long long*)&fb0[0], (unsigned long long)f0);
      if (f1) atomicAdd((unsigned long long*)&fb0[1], (unsigned long long)f1);
      if (f2) atomicAdd((unsigned long long*)&fb0[2], (unsigned long long)f2);
    }
  }
  cluster.sync();
  if (r != 0) return;
  {  // the support in ascending token order: tokens selected before each word, one block scan
    const uint32_t last = (N & 31) ? ~0u << (N & 31) : 0u;  // bits past N
    int c = 0;
    if (threadIdx.x < nwords)
      c = __popc(s.selw[threadIdx.x] & ~((int)threadIdx.x == nwords - 1 ? last : 0u));
    int cnt = 0;
    c = block_exclusive_scan(c, s.wsum, &cnt);  // nwords <= 256
    if (threadIdx.x < nwords) s.wpre[threadIdx.x] = c;
    __syncthreads();
    for (int j = threadIdx.x; j < N; j += SEL_THREADS) {
      const uint32_t w = s.selw[j >> 5];
      const bool on = (w >> (j & 31)) & 1u;
      const int pos = s.wpre[j >> 5] + __popc(w & ((1u << (j & 31)) - 1u));
      a.slot[(size_t)b * N + j] = on ? pos : -1;
      if (on && pos < K) {
        a.support[(size_t)b * K + pos] = j;
        if (a.out_idx) a.out_idx[(size_t)b * K + pos] = j;
      }
    }
    if (threadIdx.x == 0 && cnt != K) set_status(a.status, GMC_STATUS_INTERNAL);
  }
  if (a.tv.base) {
    if (threadIdx.x == 0) {
      gmc_trace_header* hd = a.tv.header(b);
      hd->K = K;
      hd->rounds = rnd;
      hd->filled = filled;
      const double inv = ldexp(1.0, -e);
      for (int q = 0; q < 3; ++q) {
        hd->F_S[q] = (float)((double)s.fb[q] * inv);
        hd->F_V[q] = (float)((double)a.r0.fv[(size_t)b * 4 + q] * inv);
      }
    }
    int32_t* to = a.tv.at<int32_t>(b, a.tv.off_order);
    for (int q = threadIdx.x; q < K; q += SEL_THREADS) to[q] = a.order[(size_t)b * K + q];
    int32_t* te = a.tv.at<int32_t>(b, a.tv.off_round_end);
    for (int q = rnd + threadIdx.x; q < a.tv.rounds_max; q += SEL_THREADS) te[q] = K;
    int32_t* tp = a.tv.at<int32_t>(b, a.tv.off_pool);
    for (size_t q = (size_t)rnd * a.tv.pool_size + threadIdx.x;
         q < (size_t)a.tv.rounds_max * a.tv.pool_size; q += SEL_THREADS)
      tp[q] = -1;
  }
}

// Batched certificate (Sec. 4.1 Eq. (6); appendix Eq. (cond-batched-bound)),
// computed only for the diagnostics trace from what the solver recorded there:
// round t's gains u^t and F(S) after it.  U_t, the sum of the K largest gains
// of the tokens not selected before round t, comes from the K-th largest gain
// theta (binary search on the fixed-point value, counting on the whole
// block): U_t = sum_{u > theta} u + (K - #{u > theta}) theta, exactly.
// c_B = 1 - prod_t (1 - q_t) over the rounds with U_t > 0,
// q_t = (F_t - F_{t-1}) / U_t.  One block per image.
__global__ void __launch_bounds__(256) k_certificate(int N, int K, TraceView tv) {
  grid_dep_wait();
  extern __shared__ __align__(16) char sm_cert[];
  long long* g = reinterpret_cast<long long*>(sm_cert);               // [N]
  unsigned char* done = reinterpret_cast<unsigned char*>(g + N);      // [N] selected before t
  __shared__ long long red[8];
  __shared__ unsigned long long red2[8];
  const int b = blockIdx.x;
  gmc_trace_header* hd = tv.header(b);
  const int R = hd->rounds;
  const int32_t* order = tv.at<int32_t>(b, tv.off_order);
  const int32_t* rend = tv.at<int32_t>(b, tv.off_round_end);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int j = threadIdx.x; j < N; j += blockDim.x) done[j] = 0;
  // block sum of (count, value) over the unselected tokens with g > x (or >= x)
  auto count_ge = [&](long long x) {
    long long c = 0;
    for (int j = threadIdx.x; j < N; j += blockDim.x) c += (!done[j] && g[j] >= x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
    __syncthreads();
    if (lane == 0) red[wid] = c;
    __syncthreads();
    long long t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    return t;
  };
  double prod = 1.0, Fprev = 0.0;
  const double inv = 1.0;  // q_t is a ratio of two fixed-point values: the scale cancels
  for (int t = 0; t < R; ++t) {
    __syncthreads();
    const int before = t > 0 ? rend[t - 1] : 0;
    for (int q = threadIdx.x; q < before; q += blockDim.x) done[order[q]] = 1;
    const long long* gt = tv.gains(b, t, N);
    for (int j = threadIdx.x; j < N; j += blockDim.x) g[j] = gt[j] < 0 ? 0 : gt[j];
    __syncthreads();
    // theta = the largest x with #{u >= x} >= K (0 when fewer than K tokens
    // remain).  Every gain is at most the fixed-point total mass, below 2^62, so
    // the search range [0, 2^62] halves in at most 63 steps
    long long lo = 0, hi = 1LL << 62;
    if (count_ge(0) >= K) {
      for (int it = 0; it < 64 && lo < hi; ++it) {
        const long long mid = lo + (hi - lo + 1) / 2;
        if (count_ge(mid) >= K) lo = mid; else hi = mid - 1;
      }
    }
    const long long theta = lo;
    // sum and count of the gains above theta
    unsigned long long sv = 0;
    long long cv = 0;
    for (int j = threadIdx.x; j < N; j += blockDim.x)
      if (!done[j] && g[j] > theta) {
        sv += (unsigned long long)g[j];
        ++cv;
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sv += __shfl_xor_sync(FULL, sv, o);
      cv += __shfl_xor_sync(FULL, cv, o);
    }
    __syncthreads();
    if (lane == 0) {
      red2[wid] = sv;
      red[wid] = cv;
    }
    __syncthreads();
    unsigned long long S = 0;
    long long C = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      S += red2[w];
      C += red[w];
    }
    const long long remain = count_ge(0);
    const double U = remain >= K ? (double)S + (double)(K - C) * (double)theta : (double)S;
    const double F = (double)*tv.cover(b, t) * inv;
    if (U > 0.0) {
      prod *= 1.0 - (F - Fprev) / U;
      Fprev = F;
    }
  }
  if (threadIdx.x == 0) hd->c_B = (float)(1.0 - prod);
}

static int g_num_sms = 0;

static cudaError_t num_sms() {
  if (g_num_sms) return cudaSuccess;
  int dev = 0, n = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(k_select, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) !=
      cudaSuccess)
    return e;
  g_num_sms = n;
  return cudaSuccess;
}

// The largest cluster launch_select tries (images x CTAs within the SMs) has
// the smallest per-CTA state; the state of any smaller one is larger.
static int first_cluster_size(int B) {
  int CS = 1;
  while (CS * 2 <= SEL_MAX_CS && (long long)B * CS * 2 <= g_num_sms) CS *= 2;
  return CS;
}

// Until the survivor lists fit the cluster's shared memory a round costs 50 us and more
// in a cluster (they stay in global memory), 21 to 40 us on the whole GPU; after that 8
// to 11 us in a cluster.  How many rounds that takes follows from the load, the entries
// of a CTA's dense rows over what its shared memory holds of them, and from the tokens a
// round selects.  A grounded row counts a third in the load (attention is concentrated:
// few entries survive a round), a spatial one five times (its distances fall off slowly);
// gmc_select's rows have no kind.  Calls in us by sparse rounds on the GPU at b = 16:
//   N = 1,296, T = 64, K = 453   1: 379, 2: 368, 3: 362, 6: 379   (the rule: 1)
//   N = 1,296, T = 256, K = 77   1: 483, 2: 320, 3: 322, 6: 319   (2)
//   N = 2,304, T = 32, H = 4     2: 563, 3: 426, 4: 427, 8: 438   (3)
//   N = 3,025, T = 64            2: 599, 4: 489, 5: 493, 6: 501   (5)
//   N = 4,096, T = 128           4: 915, 6: 817, 8: 745, 10: 767  (8)
//   N = 6,400, T = 128           8: 1,606, 10: 1,525, 12: 1,439, 16: 1,469  (12)
// Over 134 shapes (N 144 to 7,568, T 8 to 256, one to 64 images, b 8 to 32) the rule is
// 1.4% above the best count in the mean, 8% at most; steps in N alone 6.2%, 58%.
int sparse_gpu_rounds(int B, int N, int M, int H, int T, int L2, const gmc_params& p, int K,
                      int images) {
  if (num_sms() != cudaSuccess) cudaGetLastError();
  const int CS = first_cluster_size(B), SL = ((N + CS - 1) / CS + 31) & ~31;
  const int cap = sel_layout(N, p.pool_mult * p.batch_b, CS, SL, (M + CS - 1) / CS).cap;
  const double ground = (double)H * T, rows = ground / 3 + (M - ground - L2) + 5.0 * L2;
  const double load = rows * N / CS / (cap > 0 ? cap : 1);
  const double rounds = std::max(1.0, (0.92 * sqrt(load) - 1.5) * sqrt(16.0 / p.batch_b));
  const int left = K - (images > 1 ? images : p.batch_b);  // no more than the budget has left
  const int most = left > 0 ? (left + p.batch_b - 1) / p.batch_b : 0;
  return (int)std::min(rounds, (double)most);
}

// Bytes per CTA that bound the problems given to the cluster solver: what an
// earlier layout of its state took.  The present one is smaller (sel_layout),
// but the line stays: multi-image prompts beyond it are refused, and single
// images beyond it (N above about 7,700 at H = 28, T = 128) keep more survivors
// than a cluster holds for most of their rounds, which the whole-GPU solver
// then runs faster than a cluster walking them in global memory.
static size_t cluster_bytes(size_t N, size_t P, size_t R, size_t gwords) {
  size_t off = 0;
  for (size_t bytes : {8 * gwords, 8 * N, (size_t)8192, (size_t)256, N, 2 * N, 4 * N, N, 2 * N, 4 * P,
                       8 * P, 128 * P, 4 * P, 4 * P, (size_t)128, 4 * R, 4 * R, 4 * R, 4 * R, 8 * R,
                       4 * R, 8 * R, 8 * R, 4 * N + 4, (size_t)528, (size_t)2048, (size_t)1024,
                       (size_t)64, (size_t)64})
    off += (bytes + 15) & ~(size_t)15;
  return off + 1024;
}

bool select_fits(int B, int N, int M, int P) {
  if (num_sms() != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const int CS = first_cluster_size(B);
  const int RPC = (M + CS - 1) / CS;
  const int gwords = (CS > 1 ? 2 : 1) * ((N + CS - 1) / CS);
  return cluster_bytes(N, P, RPC, gwords) <= SMEM_LIMIT;
}

cudaError_t launch_select(const R0State& r0, int B, int N, int K, int M, const int32_t* toff, int H, int T, int L2,
                          const gmc_params& p, int fx_exp, const int32_t* fexp, float* C,
                          uint16_t* scol, const long long* u0, int32_t* order, int32_t* support,
                          int32_t* slot, int32_t* out_idx, uint32_t* status, const TraceView& tv,
                          cudaStream_t st, int I) {
  cudaError_t e;
  if ((e = num_sms()) != cudaSuccess) return e;
  SelArgs a;
  a.B = B; a.N = N; a.K = K; a.Mstride = M; a.H = H; a.Tmax = T; a.L2 = L2;
  a.toff = toff;
  a.uniform_rows = (H == 0);
  a.P = p.pool_mult * p.batch_b;
  a.bsz = p.batch_b;
  a.resp_temp = p.resp_temp;
  a.resp_eps = p.resp_eps;
  a.fx_exp = fx_exp;
  a.fexp = fexp;
  a.C = C; a.scol = scol; a.u0 = u0;
  a.order = order; a.support = support; a.slot = slot; a.out_idx = out_idx;
  a.status = status;
  a.tv = tv;
  a.r0 = r0;
  a.images = I;
  for (int CS = first_cluster_size(B); CS >= 1; CS /= 2) {
    const int SL = ((N + CS - 1) / CS + 31) & ~31;
    if (sel_layout(N, a.P, CS, SL, (M + CS - 1) / CS).fixed > SMEM_LIMIT) continue;
    // every CTA takes all the shared memory it can: what its state leaves holds entries
    const size_t smem = SMEM_LIMIT;
    if ((e = set_smem_limit((const void*)k_select, smem)) != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(B * CS);
    cfg.blockDim = dim3(SEL_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    e = cudaOccupancyMaxActiveClusters(&nclusters, (void*)k_select, &cfg);
    if (e != cudaSuccess || nclusters < 1) {
      cudaGetLastError();
      continue;
    }
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see grid_dep_wait
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    if ((e = cudaLaunchKernelEx(&cfg, k_select, a)) != cudaSuccess || !tv.base) return e;
    // diagnostics trace: the batched certificate from the recorded rounds
    return launch_certificate(B, N, K, tv, st);
  }
  return cudaErrorInvalidConfiguration;
}

cudaError_t launch_certificate(int B, int N, int K, const TraceView& tv, cudaStream_t st) {
  const size_t csm = (sizeof(long long) + 1) * (size_t)N;
  cudaError_t e;
  if ((e = set_smem_limit((const void*)k_certificate, csm)) != cudaSuccess) return e;
  launch_k(k_certificate, B, 256, csm, st, 1, N, K, tv);
  return cudaGetLastError();
}

}  // namespace gmc
