// Population transport (Sec. 3.4, Eq. (5); appendix Eq. (cond-transport)) and
// physical compaction (Algorithm 1 step 6; appendix "Index map and physical
// token accounting").
//
// Carrier j = support[k] receives the cluster C_j = {i : pi(i) = j}:
//   M_j = sum_{i in C_j} m_i,  c_j = M_j^-1 sum_{i in C_j} m_i h_i   (fp32 accumulation)
//   h~_j = c_j * rms(h_j) / (rms(c_j) + eps)                          (one cast to the
//                                                                     output type, RNE)
// and is written to compact row k.  Members are summed in ascending source
// order, so the result does not depend on scheduling.  Text rows, K/V rows
// and position ids are gathered bit-exactly at the kept sequence rows
// [support ascending ; N .. N+T_b-1], and so are the K/V rows of the dense
// prefix layers when the caller passes them (the cached path).
#include "common.cuh"
#include "kernels.cuh"

#include <cooperative_groups.h>
#include <algorithm>

namespace gmc {
namespace cg = cooperative_groups;

constexpr int TR_VEC = 8;        // elements per thread and row (one 16-B bf16 chunk)
constexpr int TR_THREADS = 128;  // threads per CTA
constexpr int TR_MAXS = 8;       // CTAs per output row (portable cluster size)
constexpr int TR_LIST = 64;      // members a warp lists at a time
constexpr int TR_RING = 8;       // member rows in flight per thread
constexpr int TR_GRP = 4;        // rows copied and added together

// A thread's 8 elements of a row from its 16-byte units in shared memory (units
// `stride` apart).
template <typename Tin> struct Row8;
template <> struct Row8<__nv_bfloat16> {
  static __device__ __forceinline__ void to_f32(const uint4* p, int, float* v) {
    const uint4 r = *p;
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&r);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float2 f = __bfloat1622float2(h[q]);
      v[2 * q] = f.x;
      v[2 * q + 1] = f.y;
    }
  }
};
template <> struct Row8<float> {
  static __device__ __forceinline__ void to_f32(const uint4* p, int stride, float* v) {
    const uint4 a = p[0], c = p[stride];
    v[0] = __uint_as_float(a.x); v[1] = __uint_as_float(a.y);
    v[2] = __uint_as_float(a.z); v[3] = __uint_as_float(a.w);
    v[4] = __uint_as_float(c.x); v[5] = __uint_as_float(c.y);
    v[6] = __uint_as_float(c.z); v[7] = __uint_as_float(c.w);
  }
};

// Thread t's 8 elements into a slice of `cnt` threads' elements at p: its 16-byte units
// are t and cnt + t, so that a warp's accesses are whole lines in fp32 too.
template <typename Tin> struct Vec8;
template <> struct Vec8<__nv_bfloat16> {
  static __device__ __forceinline__ void store(__nv_bfloat16* p, int t, int, const float* v) {
    uint4 raw;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&raw);
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
    reinterpret_cast<uint4*>(p)[t] = raw;
  }
};
template <> struct Vec8<float> {
  static __device__ __forceinline__ void store(float* p, int t, int cnt, const float* v) {
    reinterpret_cast<float4*>(p)[t] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(p)[cnt + t] = make_float4(v[4], v[5], v[6], v[7]);
  }
};

// CTAs per output row: the row's D/8 chunks split so a CTA holds at most 128.
inline int transport_split(int D) {
  return std::min(TR_MAXS, std::max(1, ceil_div(D / TR_VEC, TR_THREADS)));
}

// A cluster of S CTAs per output row of an image (CTA rank = slice of D):
//   r < K:            carrier j = support[r]: its members (pi(i) = j, ascending
//                     source order), M_j, c_j over the CTA's slice, the slice's sum
//                     of squares sent to every CTA of the row through distributed
//                     shared memory (added in rank order, so every slice applies
//                     the same RMS scale), the compact hidden row r; plus the
//                     carrier's K/V rows, position ids and out_idx;
//   K <= r < K + T_b: text row N + r - K copied (hidden, K/V and position ids).
//
// Members: one 32-bit word per 32 tokens, read from the carrier's membership
// bitmap when the assignment kernel wrote one (mbits != nullptr), else built by
// ballots over the assignment.  Up to 4,096 tokens every warp reads the words (four
// per lane) and lists the members for itself, TR_LIST at a time (a scan of its
// lanes' counts places them in token order), so the warps meet only in the sum of
// squares; above (COOP, N <= 16,384) the warps take a quarter of the words each
// and share one list.
//
// A carrier's time is the chain words -> list -> member rows -> norm, and the
// longest list sets the end: most carriers have a handful of members, a few
// dozens, and a batch of rows in registers costs a memory round trip each.  So a
// thread copies its 16 bytes of TR_RING rows ahead into its own ring in shared
// memory (no barrier: it reads only what it copied), which also leaves registers
// for more CTAs; rings of 12 and 16 rows took more shared memory and gained
// nothing.  Against rows in registers, a block scan of the membership and text
// rows copied beside the carriers: 4 x (N = 2,295, K = 459, D = 3,584) from a
// caller's assignment 95.0 -> 63.2 us a call, N = 1,296, K = 257 13.3 -> 10.3 us,
// 32 such images 213 -> 202 us.  In fp32 a thread's two units lie a slice apart: side by
// side, each copy of a warp touched half of every 32-byte sector and the sectors were
// fetched twice (calls of N = 1,296, K = 257 23.8 us, now 20.8; 4,096, 400 48.3, now
// 40.1; 6,400, 640 69.9, now 58.2).
template <typename Tin, bool COOP>
__global__ void __launch_bounds__(TR_THREADS) k_transport(
    const Tin* __restrict__ hidden, const Tin* __restrict__ keys, const int32_t* __restrict__ pos,
    const int32_t* __restrict__ support, const int32_t* __restrict__ pi,
    const float* __restrict__ mass, const float* __restrict__ rmsh,
    const uint32_t* __restrict__ mbits, const int32_t* toff, int B, int N, int K, int Tmax, int D,
    int HD, int S, float rms_eps, int check, int32_t* out_idx, Tin* out_hidden, Tin* out_kv,
    int32_t* out_pos, uint32_t* status, PrefixKV pf) {
  grid_dep_wait();
  constexpr int NW = TR_THREADS / 32;
  constexpr int U = TR_VEC * (int)sizeof(Tin) / 16;  // 16-B units per chunk
  __shared__ uint16_t list[NW][TR_LIST];
  __shared__ float red[NW];
  __shared__ float ss_all[TR_MAXS];
  __shared__ uint4 ring[TR_RING][U][TR_THREADS];
  __shared__ int wcnt[NW];
  extern __shared__ uint32_t words[];  // [ceil(N / 32)] without a bitmap
  const int b = blockIdx.y, r = blockIdx.x / S, part = blockIdx.x % S;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int t0 = part * TR_THREADS + tid, nt = S * TR_THREADS;  // thread of the row
  const int nwd = (N + 31) >> 5;
  const bool car = r < K;
  const int j = car ? support[(size_t)b * K + r] : 0;
  const uint32_t* bits = mbits ? mbits + ((size_t)b * K + r) * nwd : words;
  // this lane's words: of the whole image (N <= 4,096), or of its warp's quarter
  constexpr int WL = 4;
  const int xl = COOP ? (w * 32 + lane) * WL : lane * WL;
  uint32_t wd[WL];
  auto load_words = [&]() {
#pragma unroll
    for (int q = 0; q < WL; ++q) wd[q] = xl + q < nwd ? bits[xl + q] : 0u;
  };
  if (car && mbits) load_words();
  const TextGeom tg = text_geom(toff, b, B, Tmax, status);
  if (tg.T == 0 || r >= K + tg.T) return;  // uniform over the cluster
  const SeqIdx sq(b, N, K, tg.off, tg.T);
  const int nkv = HD * (int)sizeof(Tin) / 16;
  const int src = car ? j : N + r - K;  // kept sequence row of output row r
  const uint4* ks = reinterpret_cast<const uint4*>(keys + sq.key_row(src, HD));
  const uint4* vs = reinterpret_cast<const uint4*>(keys + sq.value_row(src, HD));
  uint4* kd = reinterpret_cast<uint4*>(out_kv + sq.out_kv_row(0, r, HD));
  uint4* vd = reinterpret_cast<uint4*>(out_kv + sq.out_kv_row(1, r, HD));
  // the dense prefix layers' K/V rows; the loads of PL layers are in flight together
  auto copy_prefix = [&]() {
    constexpr int PL = 8;
    for (int l0 = 0; l0 < pf.n; l0 += PL)
      for (int q = t0; q < 2 * nkv; q += nt) {
        const int wv = q >= nkv, e = q - wv * nkv;
        const size_t ro = wv == 0 ? sq.key_row(src, HD) : sq.value_row(src, HD);
        const size_t wo = sq.out_kv_row(wv, r, HD);
        uint4 v[PL];
#pragma unroll
        for (int u = 0; u < PL; ++u)
          if (l0 + u < pf.n)
            v[u] = reinterpret_cast<const uint4*>(static_cast<const Tin*>(pf.keys[l0 + u]) + ro)[e];
#pragma unroll
        for (int u = 0; u < PL; ++u)
          if (l0 + u < pf.n) reinterpret_cast<uint4*>(static_cast<Tin*>(pf.out[l0 + u]) + wo)[e] = v[u];
      }
  };
  if (!car) {  // text row: bit-exact copies
    const uint4* hs = reinterpret_cast<const uint4*>(hidden + sq.hidden_row(src, D));
    uint4* hd = reinterpret_cast<uint4*>(out_hidden + sq.out_hidden_row(r, D));
    const int nh = D * (int)sizeof(Tin) / 16;
    for (int q = t0; q < nkv; q += nt) {
      const uint4 kk = ks[q], vv = vs[q];
      kd[q] = kk;
      vd[q] = vv;
    }
    for (int q = t0; q < nh; q += nt) hd[q] = hs[q];
    if (t0 < 3) out_pos[sq.out_pos(t0, r)] = pos[sq.pos(t0, src)];
    copy_prefix();
    return;
  }
  // the first K/V units and the position ids are in flight to the end
  uint4 kk = make_uint4(0, 0, 0, 0), vv = kk;
  if (t0 < nkv) {
    kk = ks[t0];
    vv = vs[t0];
  }
  const int pos3 = t0 < 3 ? pos[sq.pos(t0, src)] : 0;
  // first phase of the cluster barrier: every CTA of the row has started before any
  // writes into its shared memory (waited on just before that)
  if (S > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  const float rms_j = rmsh[(size_t)b * N + j];
  if (!mbits) {
    const int32_t* pb = pi + (size_t)b * N;
    constexpr int PU = 8;  // assignments in flight per lane
    for (int x0 = w; x0 < nwd; x0 += PU * NW) {
      int v[PU];
#pragma unroll
      for (int u = 0; u < PU; ++u) {
        const int i = (x0 + u * NW) * 32 + lane;
        v[u] = i < N ? pb[i] : -1;
      }
#pragma unroll
      for (int u = 0; u < PU; ++u) {
        const unsigned bal = __ballot_sync(FULL, v[u] == j);
        if (lane == 0 && x0 + u * NW < nwd) words[x0 + u * NW] = bal;
      }
    }
    __syncthreads();
    load_words();
  }
  // the CTA's slice of D: cnt threads take TR_VEC elements each (units tid and, in fp32,
  // cnt + tid)
  const int nch = D / TR_VEC, cper = ceil_div(nch, S), c0 = part * cper;
  const int cnt = max(0, min(cper, nch - c0));
  const bool active = tid < cnt;
  const Tin* hb = hidden + sq.hidden_row(0, D) + c0 * TR_VEC;
  const float* mb = mass + (size_t)b * N;
  float acc[TR_VEC];
#pragma unroll
  for (int q = 0; q < TR_VEC; ++q) acc[q] = 0.f;
  float Msum = 0.f;
  // members before this lane's words, and in all
  int c = 0;
#pragma unroll
  for (int q = 0; q < WL; ++q) c += __popc(wd[q]);
  int before = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(FULL, before, o);
    if (lane >= o) before += y;
  }
  int total = __shfl_sync(FULL, before, 31);
  before -= c;
  if (COOP) {
    if (lane == 0) wcnt[w] = total;
    __syncthreads();
    total = 0;
#pragma unroll
    for (int q = 0; q < NW; ++q) {
      before += q < w ? wcnt[q] : 0;
      total += wcnt[q];
    }
  }
  uint16_t* lst = COOP ? list[0] : list[w];
  for (int base = 0; base < total; base += TR_LIST) {
    int p = before - base;
    if (COOP) __syncthreads(); else __syncwarp();  // the last list has been read
    if (c && p < TR_LIST)
#pragma unroll
      for (int q = 0; q < WL; ++q) {
        uint32_t m = wd[q];
        while (m) {
          const int bit = __ffs(m) - 1;
          if (p >= 0 && p < TR_LIST) lst[p] = (uint16_t)(32 * (xl + q) + bit);
          ++p;
          m &= m - 1u;
        }
      }
    if (COOP) __syncthreads(); else __syncwarp();
    const int n = min(TR_LIST, total - base);
    auto copy = [&](int q0) {  // TR_GRP rows from q0 on, one group
#pragma unroll
      for (int u = 0; u < TR_GRP; ++u)
        if (q0 + u < n && active) {
          const uint4* row = reinterpret_cast<const uint4*>(hb + (size_t)lst[q0 + u] * D) + tid;
#pragma unroll
          for (int x = 0; x < U; ++x) cp_async16(&ring[(q0 + u) % TR_RING][x][tid], row + x * cnt);
        }
      cp_async_commit();
    };
#pragma unroll
    for (int q0 = 0; q0 < TR_RING; q0 += TR_GRP) copy(q0);
    // the list's weights, two per lane
    const float w0 = lane < n ? mb[lst[lane]] : 0.f;
    const float w1 = lane + 32 < n ? mb[lst[lane + 32]] : 0.f;
    for (int q0 = 0; q0 < n; q0 += TR_GRP) {  // ascending source order
      cp_async_wait<TR_RING / TR_GRP - 1>();
#pragma unroll
      for (int u = 0; u < TR_GRP; ++u) {
        const int q = q0 + u;
        const float wg = __shfl_sync(FULL, q < 32 ? w0 : w1, q & 31);
        if (q < n) {
          Msum += wg;
          if (active) {
            float v[TR_VEC];
            Row8<Tin>::to_f32(&ring[q % TR_RING][0][tid], TR_THREADS, v);
#pragma unroll
            for (int t = 0; t < TR_VEC; ++t) acc[t] = fmaf(wg, v[t], acc[t]);
          }
        }
      }
      copy(q0 + TR_RING);
    }
  }
  cp_async_wait<0>();
  const float invM = 1.f / Msum;
  float ss = 0.f;
#pragma unroll
  for (int t = 0; t < TR_VEC; ++t) {
    acc[t] *= invM;
    if (active) ss = fmaf(acc[t], acc[t], ss);
  }
  ss = warp_sum(ss);
  if (lane == 0) red[w] = ss;
  __syncthreads();
  ss = 0.f;
#pragma unroll
  for (int q = 0; q < NW; ++q) ss += red[q];
  if (S > 1) {
    // the slice sum goes to slot `part` of every CTA of the row; one barrier
    // phase publishes the stores, then each CTA adds the S slots in rank order
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    if (tid < S) *cg::this_cluster().map_shared_rank(&ss_all[part], tid) = ss;
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    ss = 0.f;
    for (int q = 0; q < S; ++q) ss += ss_all[q];
  }
  const float scale = rms_j / (sqrtf(ss / (float)D) + rms_eps);
  if (active) {
    float v[TR_VEC];
#pragma unroll
    for (int t = 0; t < TR_VEC; ++t) {
      v[t] = acc[t] * scale;
      if (check && !isfinite(v[t])) set_status(status, GMC_STATUS_NONFINITE);
    }
    Vec8<Tin>::store(out_hidden + sq.out_hidden_row(r, D) + c0 * TR_VEC, tid, cnt, v);
  }
  if (t0 < nkv) {
    kd[t0] = kk;
    vd[t0] = vv;
  }
  for (int q = t0 + nt; q < nkv; q += nt) {
    const uint4 k2 = ks[q], v2 = vs[q];
    kd[q] = k2;
    vd[q] = v2;
  }
  if (t0 < 3) out_pos[sq.out_pos(t0, r)] = pos3;
  if (t0 == 0) out_idx[(size_t)b * K + r] = j;
  copy_prefix();
}

template <typename T>
static cudaError_t launch_transport_t(const Dims& dm, const gmc_params& p, const void* hidden,
                                      const void* keys, const int32_t* pos, const int32_t* support,
                                      const int32_t* pi, const float* mass, const float* rmsh,
                                      const uint32_t* mbits, int32_t* out_idx, void* out_hidden,
                                      void* out_kv, int32_t* out_pos, uint32_t* status,
                                      cudaStream_t st, const PrefixKV& pf) {
  const int S = transport_split(dm.D);
  const bool small = dm.N <= 32 * 32 * 4;
  const int nwd = ceil_div(dm.N, 32);
  const size_t smem = mbits ? 0 : sizeof(uint32_t) * nwd;
  auto kern = small ? k_transport<T, false> : k_transport<T, true>;
  const cudaError_t e = set_smem_limit((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  launch_k(kern, dim3((dm.K + dm.T) * S, dm.B), TR_THREADS, smem, st, S, (const T*)hidden,
           (const T*)keys, pos, support, pi, mass, rmsh, mbits, dm.toff, dm.B, dm.N, dm.K, dm.T, dm.D,
           dm.Hkv * dm.d, S, p.rms_eps, p.check_mode, out_idx, (T*)out_hidden, (T*)out_kv, out_pos,
           status, pf);
  return cudaGetLastError();
}

cudaError_t launch_transport(const Dims& dm, const gmc_params& p, const void* hidden,
                             const void* keys, const int32_t* pos, const int32_t* support,
                             const int32_t* pi, const float* mass, const float* rmsh,
                             const uint32_t* mbits, int32_t* out_idx, void* out_hidden,
                             void* out_kv, int32_t* out_pos, uint32_t* status, cudaStream_t st,
                             const PrefixKV* prefix) {
  // mbits: the carrier membership bitmaps, or nullptr to scan the assignment
  return (dm.dtype == GMC_BF16 ? launch_transport_t<__nv_bfloat16> : launch_transport_t<float>)(
      dm, p, hidden, keys, pos, support, pi, mass, rmsh, mbits, out_idx, out_hidden, out_kv, out_pos,
      status, st, prefix ? *prefix : PrefixKV{});
}

}  // namespace gmc
