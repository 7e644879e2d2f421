// Head patterns, farthest-first head clusters, head weights and message energy
// (appendix Eq. (cond-head-pattern), (cond-head-weight), (cond-grounded-energy)).
//
// The pattern of head h stacks its atoms u_i^{h,t} = A[h,t,i] [Z_h[i]; sigma_h]
// over all (t, i), scaled to unit mean atom norm.  Only inner products of
// patterns are needed, and they factor per token:
//   <U_h, U_g> = sum_i (Z_h[i].Z_g[i] + sigma_h sigma_g) sum_t A[h,t,i] A[g,t,i]
// so the H x H Gram is accumulated token block by token block without ever
// forming the (T N (r+1))-long patterns.  The mean atom norm of head h is
// sum_t rs[h,t] / (T N) (rs from the message kernel).
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace gmc {

__device__ __forceinline__ float query_weight(int t, int Tb, float wq) {
  return (t == Tb - 1 ? wq : 1.f) / ((float)(Tb - 1) + wq);
}

// Sums n values over the warp's 32 lanes, halving the values each lane holds at
// every step (51 shuffles for 49 values instead of 5 each).  On return v[0],
// v[1] hold the totals number index(lane, 0) and index(lane, 1) of the n
// (LaneSum::index; -1: none).  A fixed tree: the same on every call.
template <int n, int o>
struct LaneSum {
  static constexpr int K = (n + 1) / 2;
  static __device__ __forceinline__ void run(float* v, int lane) {
    const bool up = lane & o;
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const float hi = K + q < n ? v[K + q] : 0.f;
      v[q] = (up ? hi : v[q]) + __shfl_xor_sync(FULL, up ? v[q] : hi, o);
    }
    if constexpr (o > 1) LaneSum<K, o / 2>::run(v, lane);
  }
  static __device__ __forceinline__ int index(int lane, int f) {
    int i;
    if constexpr (o > 1) i = LaneSum<K, o / 2>::index(lane, f);
    else i = f < K ? f : -1;
    if (i < 0) return -1;
    i += (lane & o) ? K : 0;
    return i < n ? i : -1;
  }
};

// a + x, *e its rounding error (Knuth's two-sum).
__device__ __forceinline__ float two_sum(float a, float x, float* e) {
  const float t = a + x, z = t - a;
  *e = (a - (t - z)) + (x - z);
  return t;
}

// A 16-byte shared load that is issued where it stands: the weights of a pair
// re-read their probe values instead of holding 2 HB of them in registers
// beside the sums.
__device__ __forceinline__ float4 lds4(unsigned a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a));
  return v;
}

constexpr int HS_WARPS = 10;  // warps per block: the 10 head-block pairs of 28 or 32 heads
constexpr int HS_TC = 8;      // queries of a stage per lane group (TT groups)
// Words between the staged rows of two queries: every head block padded to HB,
// and TT > 1 query groups of a warp on distinct banks.
__host__ __device__ constexpr int hs_stride(int H, int HB, int TT) {
  return (ceil_div(H, HB) * HB * (32 / TT) + 31) / 32 * 32 + (TT > 1 ? 32 / TT : 0);
}

// Pattern Gram and query-weighted squares of a group of tokens.
//
// Work split: a block takes TOK = 32 / TT consecutive tokens of an image; a
// warp takes one pair of head blocks (HB heads each) and keeps the HB x HB sums
// sum_t A[h,t,i] A[g,t,i] in registers, lane = (query t mod TT, token).  A
// passes once through shared memory (cp.async, two stages of TC queries), laid
// out [query][head][token], so a lane's 2 HB operands of a query lie at fixed
// offsets from one address and feed HB^2 FMAs.  Then every lane applies its
// token's weights Z_h . Z_g + sigma_h sigma_g and the lanes are added.  With fewer
// pairs than HS_WARPS the queries are dealt to `ts` slices of warps.
//
// Precision.  The squares W2 of a token are a lane's sum over the queries: every FOLD
// stages (32 queries of a lane, 16 with TT > 1) it goes into a total whose rounding
// errors are kept (Knuth's two-sum), in the lane's own words of shared memory.  Against
// 64 bits, root mean square over the tokens at T = 64, 128, 256, TT = 1: 6.8e-8, 5.3e-8,
// 4.3e-8 (one chain over all queries: 1.2e-7, 1.7e-7, 2.3e-7); it costs 2% of the kernel
// there.  A pair's Gram entry keeps its one chain: its errors average out over
// the tokens, and rounding the sum to fp32 is what is left (1.1e-8 to 2e-8 of the norms'
// product at T = 64 to 256, with chains of 32 as well).
// TT: 1 reads whole 128-byte lines; 2 and 4 make more, smaller blocks for a
// single small image (head_tokens).  Bound by the shared-memory and FMA issue
// of 14 loads against 49 FMAs and the two stages' barriers.  The 4 x 4 tiles
// over [head][query][token] stages that it replaced used half the threads and 8
// shared loads for 16 FMAs: 656 -> 299 us at 32 ragged images of N = 1,296 (T <=
// 256), 229 -> 110 us at N = 15,876, T = 128, 64 -> 32 us at N = 4,096, T = 128,
// 17.1 -> 13.6 us at N = 1,296, T = 64 (H = 28).
template <int HB, int TT>
__global__ void __launch_bounds__(32 * HS_WARPS, HB == 8 ? 1 : 2)
    k_head_stats(const float* __restrict__ A, const float* __restrict__ Z,
                 const float* __restrict__ sigma, const int32_t* toff, int B, int N, int Tmax,
                 int H, float wq, float* hgpart, int nHG, float* W2, int ts, uint32_t* status) {
  grid_dep_wait();
  constexpr int TOK = 32 / TT, NV = HB * HB, TC = HS_TC * TT, FOLD = TT == 1 ? 4 : 2;
  extern __shared__ __align__(16) float sm_hs[];  // [2][TC][stride], then Z [nb HB][TOK]
  __shared__ float sgm[GMC_MAX_HEADS + 8];       // sigma_h of the image
  __shared__ float part[HS_WARPS][NV];        // slices' sums of a pair (ts > 1)
  // query-weighted squares: a lane's total and its rounding errors, then (ts > 1)
  // the slices' sums
  __shared__ float w2s[HS_WARPS][HB][32], w2e[HS_WARPS][HB][32];
  const int b = blockIdx.y;
  const TextGeom tg = text_geom(toff, b, B, Tmax, status);
  if (tg.T == 0) return;
  const int Tb = tg.T;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nb = ceil_div(H, HB), npair = nb * (nb + 1) / 2;
  const int stride = hs_stride(H, HB, TT);
  const int i0 = blockIdx.x * TOK, tt = lane / TOK;
  const int i = i0 + lane % TOK;
  const bool tok = i < N;
  float* out = hgpart + ((size_t)b * nHG + blockIdx.x) * H * H;
  const float nu = 1.f / ((float)(Tb - 1) + wq);
  const float* Ab = A + (size_t)b * H * Tmax * N + i0;
  // rows of A start on 16 bytes when N % 4 == 0 (then four tokens are all
  // inside or all past the image); queries and tokens past the end are zero
  const bool vec = (N & 3) == 0;
  // thread's piece of a staged row (16 or 4 bytes) and its first (query, head) row;
  // a step moves `rstep` rows on, without a division
  const int pieces = vec ? TOK / 4 : TOK, pw = vec ? 4 : 1;
  const int pv = (int)threadIdx.x % pieces * pw, r0 = (int)threadIdx.x / pieces;
  const int rstep = 32 * HS_WARPS / pieces, dt = rstep / H, dh = rstep % H;
  const int rt = r0 / H, rh = r0 % H;
  const bool pin = i0 + pv < N;
  auto stage = [&](int t0, float* buf) {
    int t = rt, h = rh;
#pragma unroll 1
    while (t < TC) {
      const bool in = pin && t0 + t < Tb;
      const float* src = in ? Ab + ((size_t)h * Tmax + t0 + t) * N + pv : A;
      float* dst = buf + t * stride + h * TOK + pv;
      if (vec) cp_async16(dst, src, in);
      else cp_async4(dst, src, in);
      t += dt;
      h += dh;
      if (h >= H) {
        h -= H;
        ++t;
      }
    }
    cp_async_commit();
  };
  // the tokens' probe values and the heads' mass coordinates, beside the stages
  float4* zs = reinterpret_cast<float4*>(sm_hs + 2 * (size_t)TC * stride);
#pragma unroll 1
  for (int q = threadIdx.x; q < H * TOK; q += blockDim.x) {
    const int h = q / TOK, k = q % TOK;
    cp_async16(&zs[q],
               reinterpret_cast<const float4*>(Z) + ((size_t)b * H + h) * N + min(i0 + k, N - 1));
  }
  for (int h = threadIdx.x; h < H; h += blockDim.x) sgm[h] = sigma[(size_t)b * H + h];
  const int nst = ceil_div(Tb, TC);  // stages
  // ts slices of npair warps; ts == 1: the warps walk the pairs, in one pass
  // over the queries for every HS_WARPS pairs
  const int slice = ts > 1 ? w / npair : 0, wp = ts > 1 ? w % npair : w;
  const int npass = ts > 1 ? 1 : ceil_div(npair, HS_WARPS);
  for (int pass = 0; pass < npass; ++pass) {
    const int p = wp + pass * HS_WARPS;
    const bool mine = p < npair && slice < ts;
    int hb = 0, q = mine ? p : 0;  // pair p of the upper triangle, row by row
    while (q >= nb - hb) {
      q -= nb - hb;
      ++hb;
    }
    const int gb = hb + q, h0 = hb * HB, g0 = gb * HB;
    const bool diag = hb == gb;
    const int nh = min(HB, H - h0), ng = min(HB, H - g0);
    float acc[NV], w2[HB];
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] = 0.f;
#pragma unroll
    for (int u = 0; u < HB; ++u) w2[u] = 0.f;
    stage(0, sm_hs);
    for (int st = 0; st < nst; ++st) {
      if (st + 1 < nst) {
        stage((st + 1) * TC, sm_hs + (size_t)((st + 1) & 1) * TC * stride);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();
      if (mine) {
        const int tend = min(TC, Tb - st * TC);  // staged queries of the image
        const float* row = sm_hs + (size_t)(st & 1) * TC * stride + (slice * TT + tt) * stride +
                           lane % TOK;
        if (diag) {
#pragma unroll 1
          for (int t0 = slice * TT; t0 < tend; t0 += ts * TT, row += ts * TT * stride) {
            const float wt = st * TC + t0 + tt == Tb - 1 ? wq * nu : nu;
            float x[HB];
#pragma unroll
            for (int u = 0; u < HB; ++u) x[u] = row[(h0 + u) * TOK];
#pragma unroll
            for (int u = 0; u < HB; ++u) {
              w2[u] = fmaf(wt * x[u], x[u], w2[u]);
#pragma unroll
              for (int v = 0; v < HB; ++v) acc[u * HB + v] = fmaf(x[u], x[v], acc[u * HB + v]);
            }
          }
          if (st % FOLD == FOLD - 1 && st + 1 < nst) {
#pragma unroll
            for (int u = 0; u < HB; ++u) {
              float e = 0.f;
              w2s[w][u][lane] = st < FOLD ? w2[u] : two_sum(w2s[w][u][lane], w2[u], &e);
              w2e[w][u][lane] = st < FOLD ? 0.f : w2e[w][u][lane] + e;
              w2[u] = 0.f;
            }
          }
        } else {
#pragma unroll 1
          for (int t0 = slice * TT; t0 < tend; t0 += ts * TT, row += ts * TT * stride) {
            float x[HB], y[HB];
#pragma unroll
            for (int u = 0; u < HB; ++u) {
              x[u] = row[(h0 + u) * TOK];
              y[u] = row[(g0 + u) * TOK];
            }
#pragma unroll
            for (int u = 0; u < HB; ++u)
#pragma unroll
              for (int v = 0; v < HB; ++v) acc[u * HB + v] = fmaf(x[u], y[v], acc[u * HB + v]);
          }
        }
      }
      __syncthreads();  // the stage's buffer is free
    }
    if (!mine) continue;
    if (diag) {  // sum_t nu_t A[h,t,i]^2 of the block's heads
#pragma unroll
      for (int u = 0; u < HB; ++u) {
        if (nst > FOLD) {
          float e;
          const float t = two_sum(w2s[w][u][lane], w2[u], &e);
          w2[u] = t + (w2e[w][u][lane] + e);
        }
#pragma unroll
        for (int o = TOK; o < 32; o <<= 1) w2[u] += __shfl_xor_sync(FULL, w2[u], o);
        if (ts > 1) {
          if (tt == 0) w2s[w][u][lane % TOK] = w2[u];
        } else if (tt == 0 && tok && u < nh) {
          W2[((size_t)b * H + h0 + u) * N + i] = w2[u];
        }
      }
    }
    // the token's weights (heads past H: whatever the padding holds, never written)
    const unsigned zh0 = (unsigned)__cvta_generic_to_shared(zs + h0 * TOK + lane % TOK);
    const unsigned zg0 = (unsigned)__cvta_generic_to_shared(zs + g0 * TOK + lane % TOK);
#pragma unroll
    for (int v = 0; v < HB; ++v) {
      const float4 zg = lds4(zg0 + v * TOK * 16);
      const float sg = sgm[g0 + v];
#pragma unroll
      for (int u = 0; u < HB; ++u) {
        const float4 zh = lds4(zh0 + u * TOK * 16);
        const float wgt =
            fmaf(zh.x, zg.x, fmaf(zh.y, zg.y, fmaf(zh.z, zg.z, fmaf(zh.w, zg.w, sgm[h0 + u] * sg))));
        acc[u * HB + v] = tok ? wgt * acc[u * HB + v] : 0.f;
      }
    }
    LaneSum<NV, 16>::run(acc, lane);
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      const int k = LaneSum<NV, 16>::index(lane, f);
      if (k < 0) continue;
      const int u = k / HB, v = k % HB;
      if (u >= nh || v >= ng) continue;
      if (ts > 1) {
        part[w][k] = acc[f];
      } else {
        out[(h0 + u) * H + g0 + v] = acc[f];
        if (!diag) out[(g0 + v) * H + h0 + u] = acc[f];
      }
    }
  }
  if (ts == 1) return;
  // the slices in order
  __syncthreads();
  for (int e = threadIdx.x; e < npair * NV; e += blockDim.x) {
    const int p = e / NV, k = e % NV;
    int hb = 0, q = p;
    while (q >= nb - hb) {
      q -= nb - hb;
      ++hb;
    }
    const int h = hb * HB + k / HB, g = (hb + q) * HB + k % HB;
    if (h >= H || g >= H) continue;
    float s = 0.f;
    for (int x = 0; x < ts; ++x) s += part[x * npair + p][k];
    out[h * H + g] = s;
    if (q > 0) out[g * H + h] = s;
  }
  for (int e = threadIdx.x; e < nb * HB * TOK; e += blockDim.x) {
    const int hb = e / (HB * TOK), u = e / TOK % HB, k = e % TOK;
    const int h = hb * HB + u, tk = blockIdx.x * TOK + k;
    if (h >= H || tk >= N) continue;
    const int p = hb * nb - hb * (hb - 1) / 2;  // the diagonal pair of head block hb
    float s = 0.f;
    for (int x = 0; x < ts; ++x) s += w2s[x * npair + p][u][k];
    W2[((size_t)b * H + h) * N + tk] = s;
  }
}

// Ties: the first centre is the lowest-index largest pattern, each next centre
// the lowest-index head of smallest max-cosine, and a head joins the earliest
// centre among equally similar ones.
__device__ __forceinline__ void warp_argbest(float& v, int& idx, bool want_max) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(FULL, v, o);
    const int oi = __shfl_xor_sync(FULL, idx, o);
    const bool better = want_max ? (ov > v || (ov == v && oi < idx))
                                 : (ov < v || (ov == v && oi < idx));
    if (oi >= 0 && (idx < 0 || better)) { v = ov; idx = oi; }
  }
}

// Farthest-first head clusters and head weights of image b from its reduced
// pattern Gram (read past L1: other blocks wrote it).  The cosines, dispersions and weights are fp32: the weights enter as
// 1 / (dispersion + head_eps) with head_eps = 0.05 by default, far above the
// fp32 rounding of a cosine.  One block, one warp for the centres (two heads
// per lane, H <= 64).  A chain of short steps between barriers: with one view
// the Gram is read once into shared memory, all loads in flight together.
__device__ void cluster_heads(const float* hgb, int b, int T, int N, int H, int max_clusters,
                              float head_eps, float* omega, const TraceView& tv, float* sm,
                              const ViewGrams& vg) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float* cs = sm;                       // [H*H] pattern cosines
  float* pre = cs + H * H;              // [H]   pattern norm / mean atom norm
  float* dot = pre + H;                 // [H]   1/||U_h||, later h's cosine sum in its cluster
  float* inv = dot + H;                 // [H]   1 / (dispersion + eps)
  float* csum = inv + H;                // [GMC_MAX_HEADS] 1 / norm of a cluster's sum
  float* isum = csum + GMC_MAX_HEADS;   // [GMC_MAX_HEADS]
  int* asg = reinterpret_cast<int*>(isum + GMC_MAX_HEADS);  // [H] cluster of every head
  int* cent = asg + H;                  // [GMC_MAX_HEADS] centres
  int* ccnt = cent + GMC_MAX_HEADS;     // [GMC_MAX_HEADS] cluster sizes
  const float TN = (float)T * (float)N;
  if (vg.n > 1) {
    // patterns over the views (Eq. (cond-head-pattern)): with U_h^v the view's
    // atoms over their mean norm m_v[h] = sum_t rs_v[h,t] / (T N),
    // <u_h, u_g> = sum_v beta_v G_v[h][g] / (m_v[h] m_v[g])
    const int HE = H * H + H;
    for (int h = threadIdx.x; h < H; h += blockDim.x) {
      float a = 0.f;
      for (int v = 0; v < vg.n; ++v) {
        const float* hv = vg.HG[v] + (size_t)b * HE;
        const float m = __ldcg(&hv[H * H + h]) / TN;
        if (m > 0.f) a += vg.beta[v] * __ldcg(&hv[h * H + h]) / (m * m);
      }
      pre[h] = a > 0.f ? sqrtf(a) : 0.f;
      dot[h] = a > 0.f ? 1.f / sqrtf(a) : 0.f;
    }
    __syncthreads();
    for (int p = threadIdx.x; p < H * H; p += blockDim.x) {
      const int h = p / H, g = p % H;
      float x = 0.f;
      for (int v = 0; v < vg.n; ++v) {
        const float* hv = vg.HG[v] + (size_t)b * HE;
        const float mh = __ldcg(&hv[H * H + h]) / TN, mg = __ldcg(&hv[H * H + g]) / TN;
        if (mh > 0.f && mg > 0.f) x += vg.beta[v] * __ldcg(&hv[p]) / (mh * mg);
      }
      cs[p] = x * dot[h] * dot[g];
    }
    __syncthreads();
  } else {
    for (int p = threadIdx.x; p < H * H; p += blockDim.x) cs[p] = __ldcg(&hgb[p]);
    for (int h = threadIdx.x; h < H; h += blockDim.x) inv[h] = __ldcg(&hgb[H * H + h]);
    __syncthreads();
    for (int h = threadIdx.x; h < H; h += blockDim.x) {
      const float a = cs[h * H + h];
      const float mean = inv[h] / TN;  // sum_t rs / (T N)
      pre[h] = (mean > 0.f && a > 0.f) ? sqrtf(a) / mean : 0.f;
      dot[h] = a > 0.f ? 1.f / sqrtf(a) : 0.f;  // 1 / ||U_h||, 0 for a zero pattern
    }
    __syncthreads();
    for (int p = threadIdx.x; p < H * H; p += blockDim.x) cs[p] = cs[p] * dot[p / H] * dot[p % H];
    __syncthreads();
  }
  const int nc = min(max_clusters, H);
  if (wid == 0) {  // farthest-first centres, two heads per lane (H <= 64)
    const int h0 = lane, h1 = lane + 32;
    bool c0 = false, c1 = false;  // is h0 / h1 a centre
    float mc0 = -INFINITY, mc1 = -INFINITY;  // largest cosine of h0 / h1 to a centre
    int newest;                              // the latest centre (the same in every lane)
    {
      float v = -1.f;
      int idx = -1;
      if (h0 < H) { v = pre[h0]; idx = h0; }
      if (h1 < H && (idx < 0 || pre[h1] > v)) { v = pre[h1]; idx = h1; }
      warp_argbest(v, idx, true);
      if (lane == 0) cent[0] = idx;
      c0 = (h0 == idx);
      c1 = (h1 == idx);
      newest = idx;
    }
    for (int c = 1; c < nc; ++c) {
      if (h0 < H) mc0 = fmaxf(mc0, cs[h0 * H + newest]);
      if (h1 < H) mc1 = fmaxf(mc1, cs[h1 * H + newest]);
      float v = 0.f;
      int idx = -1;
      for (int q = 0; q < 2; ++q) {
        const int h = q ? h1 : h0;
        if (h >= H || (q ? c1 : c0)) continue;
        const float mc = q ? mc1 : mc0;
        if (idx < 0 || mc < v) { v = mc; idx = h; }
      }
      warp_argbest(v, idx, false);
      if (lane == 0) cent[c] = idx;
      c0 |= (h0 == idx);
      c1 |= (h1 == idx);
      newest = idx;
    }
  }
  __syncthreads();
  // each head joins its most similar centre (the earliest among equals)
  for (int h = threadIdx.x; h < H; h += blockDim.x) {
    int bk = 0;
    for (int k = 1; k < nc; ++k)
      if (cs[h * H + cent[k]] > cs[h * H + cent[bk]]) bk = k;
    asg[h] = bk;
  }
  __syncthreads();
  // sums over heads as warp trees (two heads per lane, fixed order)
  const int nw = blockDim.x >> 5;
  for (int h = wid; h < H; h += nw) {
    float d = 0.f;
    if (lane < H && asg[lane] == asg[h]) d += cs[h * H + lane];
    if (lane + 32 < H && asg[lane + 32] == asg[h]) d += cs[h * H + lane + 32];
    d = warp_sum(d);
    if (lane == 0) dot[h] = d;
  }
  __syncthreads();
  // ||sum_{g in k} u_g||^2 (in cosine units) = sum over the cluster's dot values
  for (int k = wid; k < nc; k += nw) {
    float sk = 0.f;
    int n = 0;
    if (lane < H && asg[lane] == k) { sk += dot[lane]; ++n; }
    if (lane + 32 < H && asg[lane + 32] == k) { sk += dot[lane + 32]; ++n; }
    sk = warp_sum(sk);
    n = warp_sum_int(n);
    if (lane == 0) {
      csum[k] = sk > 0.f ? rsqrtf(sk) : 0.f;  // 1 / ||sum_{g in k} u_g||
      ccnt[k] = n;
    }
  }
  __syncthreads();
  for (int h = threadIdx.x; h < H; h += blockDim.x) {
    const float dh = 1.f - dot[h] * csum[asg[h]];
    inv[h] = 1.f / (dh + head_eps);
  }
  __syncthreads();
  for (int k = wid; k < nc; k += nw) {
    float sk = 0.f;
    if (lane < H && asg[lane] == k) sk += inv[lane];
    if (lane + 32 < H && asg[lane + 32] == k) sk += inv[lane + 32];
    sk = warp_sum(sk);
    if (lane == 0) isum[k] = sk;
  }
  __syncthreads();
  int C = 0;
  for (int k = 0; k < nc; ++k) C += ccnt[k] > 0;
  for (int h = threadIdx.x; h < H; h += blockDim.x) {
    const float w = inv[h] / isum[asg[h]] / (float)C;
    omega[(size_t)b * H + h] = w;
    if (tv.base) {
      tv.at<int32_t>(b, tv.off_head_assign)[h] = asg[h];
      tv.at<float>(b, tv.off_omega)[h] = w;
    }
  }
  if (tv.base) {
    if (threadIdx.x == 0) tv.header(b)->n_clusters = C;
    int32_t* tc = tv.at<int32_t>(b, tv.off_centres);
    for (int k = threadIdx.x; k < max_clusters; k += blockDim.x) tc[k] = k < nc ? cent[k] : -1;
  }
}

// A sum of fp32 terms in three words: every addition's rounding error is kept in mid
// (Knuth's two-sum), and that sum's errors in lo: about 72 bits, all on the fp32 pipe.
// fp64 additions run at a small fraction of its rate on this GPU: the reduction below
// took 33 us longer with them in a batch of 32 images, 2 us at one (two words,
// about 48 bits: 1 us less than three).
struct Sum3 {
  float hi = 0.f, mid = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float x) {
    float e;
    hi = two_sum(hi, x, &e);
    mid = two_sum(mid, e, &e);
    lo += e;
  }
  __device__ __forceinline__ void add(const Sum3& o) {
    float e;
    add(o.hi);
    mid = two_sum(mid, o.mid, &e);
    lo += e + o.lo;
  }
  // the sum over the lanes that differ in the bits below `n` (a fixed tree)
  __device__ __forceinline__ void reduce(int n) {
    for (int o = n / 2; o > 0; o >>= 1) {
      Sum3 y;
      y.hi = __shfl_xor_sync(FULL, hi, o);
      y.mid = __shfl_xor_sync(FULL, mid, o);
      y.lo = __shfl_xor_sync(FULL, lo, o);
      add(y);
    }
  }
  // rounded to fp32 once; a sum past its range is infinite, and so are its errors not numbers
  __device__ __forceinline__ float value() const {
    return isfinite(hi) ? (float)((double)hi + ((double)mid + (double)lo)) : hi;
  }
};

// The pattern Gram of image blockIdx.y: the token blocks' partials added up.
// The first gridDim.x - nrb blocks take 32 Gram entries each, one per lane (a
// warp reads one line of a partial), and their warps every HR_WARPS-th partial,
// twelve loads in flight (one round trip for the 162 partials of N = 1,296).
// The last nrb blocks sum every head's atom norms sum_t rs[h,t] (rs in nRS
// parts per query), a warp per head.  HG[b] holds the H*H Gram followed by the
// H atom-norm totals.  The image's last block to finish (ticket zeroed with
// the status word) clusters the heads.
constexpr int HR_WARPS = 16;
__global__ void __launch_bounds__(32 * HR_WARPS)
    k_hg_reduce(const float* __restrict__ hgpart, int nHG, int B, int N, int H,
                const float* __restrict__ rs, int nRS, const int32_t* toff, int Tmax, float* HG,
                uint32_t* tick, int max_clusters, float head_eps, float* omega, TraceView tv,
                int cluster, const ViewGrams vg, int nrb, uint32_t* status) {
  grid_dep_wait();
  extern __shared__ float sm_hc[];
  __shared__ Sum3 psum[HR_WARPS][33];
  __shared__ int last;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, b = blockIdx.y;
  const int HH = H * H, HE = HH + H;
  const TextGeom tg = text_geom(toff, b, B, Tmax, status);
  if (tg.T == 0) return;  // uniform over the image
  const int ngb = gridDim.x - nrb;
  if ((int)blockIdx.x < ngb) {
    const int p = blockIdx.x * 32 + lane;
    const float* src = hgpart + (size_t)b * nHG * HH + p;
    Sum3 s;
    if (p < HH) {
      constexpr int U = 12;
      for (int k0 = w; k0 < nHG; k0 += U * HR_WARPS) {
        float v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int k = k0 + u * HR_WARPS;
          v[u] = k < nHG ? src[(size_t)k * HH] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) s.add(v[u]);
      }
    }
    psum[w][lane] = s;
    __syncthreads();
    // half-warp: one entry, lane = source warp
    const int pe = 2 * w + (lane >> 4), p2 = blockIdx.x * 32 + pe;
    Sum3 t = psum[lane & 15][pe];
    t.reduce(HR_WARPS);
    if ((lane & 15) == 0 && p2 < HH) HG[(size_t)b * HE + p2] = t.value();
  } else {
    const int h = (blockIdx.x - ngb) * HR_WARPS + w;
    if (h < H) {
      Sum3 s;
      const float* r = rs + ((size_t)b * H + h) * nRS * Tmax;
      const int n = nRS * tg.T;  // (part, query) pairs, eight per lane in flight
      for (int k0 = lane; k0 < n; k0 += 32 * 8) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int k = k0 + 32 * u;
          v[u] = k < n ? r[(size_t)(k / tg.T) * Tmax + k % tg.T] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) s.add(v[u]);
      }
      s.reduce(32);
      if (lane == 0) HG[(size_t)b * HE + HH + h] = s.value();
    }
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&tick[b], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last || !cluster) return;  // a historical view's Gram waits for the current view's call
  __threadfence();
  cluster_heads(HG + (size_t)b * HE, b, tg.T, N, H, max_clusters, head_eps, omega, tv, sm_hc, vg);
}

namespace {
// Heads per register block: the one that pads H least (28 -> 7, 32 -> 8), the
// larger among equals.
int head_block(int H) {
  int best = 8;
  for (int hb : {7, 4})
    if (ceil_div(H, hb) * hb < ceil_div(H, best) * best) best = hb;
  return best;
}
}  // namespace

// Tokens per head-statistics block.  32 (whole lines) once those blocks fill
// the SMs twice over; below that smaller blocks keep more SMs busy: at one
// image of N = 1,296 the 162 blocks of 8 tokens, at N = 4,096 the 256 of 16.
int head_tokens(int B, int N) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      sms = 152;
    }
  }
  for (int tok : {32, 16})
    if ((long long)B * ceil_div(N, tok) >= (tok == 32 ? 2LL : 1LL) * sms) return tok;
  return 8;
}

// The documented head limit of the library (include/gmc.h).
bool heads_supported(int H) { return H >= 1 && H <= 56; }

cudaError_t launch_heads(const Dims& dm, const gmc_params& p, Scratch& s, const TraceView& tv,
                         cudaStream_t st, int cluster, const ViewGrams* views) {
  const int H = dm.H;
  cudaError_t e;
  const int hb = head_block(H), nb = ceil_div(H, hb), npair = nb * (nb + 1) / 2;
  // few pairs of head blocks: the queries in slices, one per group of warps
  const int ts = std::max(1, HS_WARPS / npair);
  const int tt = 32 / s.hgtok;
  const size_t smem = sizeof(float) * 2 * (size_t)HS_TC * tt * hs_stride(H, hb, tt) +
                      sizeof(float4) * (size_t)nb * hb * s.hgtok;
  auto kern = [&]() {
    switch (hb) {
      case 7: return s.hgtok == 32 ? k_head_stats<7, 1> : s.hgtok == 16 ? k_head_stats<7, 2> : k_head_stats<7, 4>;
      case 4: return s.hgtok == 32 ? k_head_stats<4, 1> : s.hgtok == 16 ? k_head_stats<4, 2> : k_head_stats<4, 4>;
      default: return s.hgtok == 32 ? k_head_stats<8, 1> : s.hgtok == 16 ? k_head_stats<8, 2> : k_head_stats<8, 4>;
    }
  }();
  if ((e = set_smem_limit((const void*)kern, smem)) != cudaSuccess) return e;
  launch_k(kern, dim3(s.nHG, dm.B), 32 * HS_WARPS, smem, st, 1, s.A, s.Z, s.sigma, dm.toff, dm.B,
           dm.N, dm.T, H, p.terminal_q_weight, s.hgpart, s.nHG, s.W2, ts, s.status);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t smem2 = sizeof(float) * ((size_t)H * H + 3 * H + 2 * GMC_MAX_HEADS) +
                       sizeof(int) * (H + 2 * GMC_MAX_HEADS);
  if ((e = set_smem_limit((const void*)k_hg_reduce, smem2)) != cudaSuccess) return e;
  const int nrb = ceil_div(H, HR_WARPS);
  launch_k(k_hg_reduce, dim3(ceil_div(H * H, 32) + nrb, dm.B), 32 * HR_WARPS, smem2, st, 1,
           (const float*)s.hgpart, s.nHG, dm.B, dm.N, H, (const float*)s.rs, s.nRS, dm.toff, dm.T,
           s.HG, s.tick3, p.max_head_clusters, p.head_eps, s.omega, tv, cluster,
           views ? *views : ViewGrams{}, nrb, s.status);
  return cudaGetLastError();
}

}  // namespace gmc
