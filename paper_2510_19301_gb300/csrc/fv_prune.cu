// fv_prune.cu -- the exact forward engine with bounded candidate rows (exact
// decoding, dense transitions, 128 < K <= 4096).
//
// The max-plus step (Sec. III-A) needs, for every target j, the maximum over
// i of fl(delta[i] + A[i][j]).  Evaluating all K rows is bound by the FP32
// max (64 candidates per clock per SM), and most rows cannot win.  Here a
// column keeps the list of its M largest weights and a cutoff b_j, the
// largest weight outside the list.  A row i outside the list of j gives at
// most fl(delta[i] + b_j) (rounding is monotone), so once a target holds a
// candidate above that it needs no row with a smaller delta.  Per step a warp
//   1. forms the M listed candidates of its targets, and the candidates of
//      the rows with delta >= max(delta) - gap (its gap follows what its last
//      steps needed);
//   2. from the best candidates so far computes the smallest delta that could
//      still reach a target, and forms the candidates of the rows between
//      that and the first threshold.
// Only the maximum is kept: delta_t = fl(max + E_t) is exact on any input (an
// input that bounds badly only runs more rows), delta rows go to the
// workspace, and the backtrack recomputes the argmax of the path's own states
// (below), K candidates per step instead of K^2 backpointers.  A sequence that
// forms too many rows is handed to the other engines (prune_give).  On Dirichlet(1)
// weights with log-softmax normal emissions a step takes about 34 of 256 rows,
// 40 of 512, 61 of 1000.
//
// Measured (GB300): 1024 sequences of 500 .. 4000 steps, K = 256: 17.3 -> 7.6
// ms per decode against the slot engine of fv_dense.cu; 150 sequences of 200
// .. 1500 steps, K = 1000: 21.8 -> 7.0 ms; 8 sequences of 1500 steps, K = 4096:
// 31.7 -> 17.6 ms; one K = 512 sequence of 512 steps: 1.80 -> 1.37 ms.  Bound
// now: latency and shared-memory wavefronts (at K = 256, 730 wavefronts and
// 2270 warp instructions per job step), not the max.
#include <cuda_runtime.h>
#include <float.h>
#include <math_constants.h>
#include <stdint.h>

#include <atomic>

#include "fv_internal.cuh"
#include "fv_launch.h"

namespace fv {

constexpr int kGiveLevels = 31;  // votes on handing a sequence over (below)

// ------------------------------------------------------------------- prep
// Order-preserving key of a float (larger float, larger key); 0 is below
// every key of a number.
__device__ __forceinline__ uint32_t ord_key(float x) {
  const uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord_value(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Padded row copy of logA (stride KP, columns beyond K -inf), its
// column-major copy (rows K .. KD - 1 -inf) and, per column, the cutoff and the list of the rows above it, in ascending row
// order: the largest cutoff with at most M rows above it, found by bisecting
// the keys (a warp per column, VPL keys per lane in registers).
// One CTA takes 8 adjacent columns, staged column-major in shared memory so
// that global loads read whole 32-byte sectors.
template <int VPL>
__global__ void __launch_bounds__(256) prune_prep_kernel(const float* logA, int K, int KP, int M, float* Apad,
                                                         float* AT, float* lval, uint16_t* lrow, float* cut,
                                                         int32_t* stat) {
  extern __shared__ float scol[];  // [8][32 * VPL + 4]
  constexpr int ST = 32 * VPL + 4;
  const int j0 = blockIdx.x * 8, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (stat && blockIdx.x == 0 && tid < 2 * kGiveLevels) stat[tid] = 0;
  for (int x = tid; x < 8 * K; x += 256) {
    const int i = x >> 3, c = x & 7;
    const float v = j0 + c < K ? __ldg(logA + (int64_t)i * K + j0 + c) : -CUDART_INF_F;
    scol[c * ST + i] = v;
    Apad[(int64_t)i * KP + j0 + c] = v;
  }
  __syncthreads();
  const int j = j0 + warp;
  if (j < K) {
    const int KD = wide_lane_stride(K);
    for (int i = lane; i < KD; i += 32) AT[(int64_t)j * KD + i] = i < K ? scol[warp * ST + i] : -CUDART_INF_F;
  }
  uint32_t key[VPL];
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    const int i = 32 * k + lane;
    key[k] = (i < K && j < K) ? ord_key(scol[warp * ST + i]) : 0u;
  }
  uint32_t prefix = 0, lim = 0;  // the list: keys >= lim (lim 0: keys > prefix)
  for (int bit = 31; bit >= 0; --bit) {
    const uint32_t tr = prefix | (1u << bit);
    int c = 0;
#pragma unroll
    for (int k = 0; k < VPL; ++k) c += key[k] >= tr;
    c = __reduce_add_sync(0xffffffffu, c);
    if (c == M) {
      lim = tr;
      break;
    }
    if (c > M) prefix = tr;
  }
  if (!lim) lim = prefix + 1;
  uint32_t top = 0;
  int base = 0;
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    const bool in = key[k] >= lim && key[k] != 0u;
    if (!in && key[k] > top) top = key[k];
    const uint32_t m = __ballot_sync(0xffffffffu, in);
    const int p = base + __popc(m & ((1u << lane) - 1u));
    if (in && p < M) {
      lval[(int64_t)p * KP + j] = ord_value(key[k]);
      lrow[(int64_t)p * KP + j] = (uint16_t)(32 * k + lane);
    }
    base += __popc(m);
  }
  top = __reduce_max_sync(0xffffffffu, top);
  for (int p = base + lane; p < M; p += 32) {
    lval[(int64_t)p * KP + j] = -CUDART_INF_F;
    lrow[(int64_t)p * KP + j] = 0;
  }
  if (lane == 0) cut[j] = top ? ord_value(top) : -CUDART_INF_F;
}

// ----------------------------------------------------------------- engine
// (NaN operands are passed over)
__device__ __forceinline__ float warp_max_f32(float x) {
  float r;
  asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float warp_min_f32(float x) {
  float r;
  asm("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}
// A delta below the result gives fl(delta + b) < best: the margin of 2^-22
// of the magnitudes covers the roundings of the difference, of the margin
// and of the sum.  best = -inf gives -inf (every finite delta matters).
__device__ __forceinline__ float need_delta(float best, float b) {
  return __fmaf_rn(-2.384185791e-7f, __fadd_rn(fabsf(best), fabsf(b)), __fadd_rn(best, -b));
}
__device__ __forceinline__ float ld_stream(const float* p) {
  float v;
  asm volatile("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
template <int C>
__device__ __forceinline__ void ld_stream_vec(const float* p, float (&e)[C]) {
  if constexpr (C == 4)
    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(e[0]), "=f"(e[1]), "=f"(e[2]), "=f"(e[3])
                 : "l"(p));
  else if constexpr (C == 2)
    asm volatile("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(e[0]), "=f"(e[1]) : "l"(p));
}
// C adjacent weights of one row
template <int C>
struct Vec {
  float v[C];
  __device__ __forceinline__ void lds(const float* p) {
    if constexpr (C == 4) {
      const float4 x = *reinterpret_cast<const float4*>(p);
      v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else if constexpr (C == 2) {
      const float2 x = *reinterpret_cast<const float2*>(p);
      v[0] = x.x; v[1] = x.y;
    } else {
      v[0] = *p;
    }
  }
  __device__ __forceinline__ void ldg(const float* p) {
    if constexpr (C == 4) {
      const float4 x = __ldg(reinterpret_cast<const float4*>(p));
      v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else if constexpr (C == 2) {
      const float2 x = __ldg(reinterpret_cast<const float2*>(p));
      v[0] = x.x; v[1] = x.y;
    } else {
      v[0] = __ldg(p);
    }
  }
};

constexpr int kPruneAhead = 3;  // emission scores loaded this many steps ahead
// The first row pass takes delta >= max(delta) - share x gap, gap a moving
// mean of the depth that was needed: per warp (kGap), or for a common list
// the largest depth of the job's warps here (kGapCommon; the second common
// list reaches to kFarGap).  Measured: 0.75 / 0.85 / 1.0 / 1.15 of a warp's
// own depth, 1024 K = 256 sequences, 7.91 / 7.78 / 7.88 / 8.42 ms; 0.85 / 0.95
// / 1.05 of the largest, 150 K = 1000 sequences, 7.24 / 7.41 / 7.82 ms and 8 K
// = 4096 sequences 17.6 / 17.1 / 18.4 ms; 0.85 / 1.0 of the mean depth 8.13 /
// 7.62 and 18.6 / 17.4 ms.
constexpr float kGap = 0.85f, kGapCommon = 0.9f, kFarGap = 1.3f;

// KP = padded state count, CL = CTAs (a cluster) that split a job's columns,
// C = adjacent columns per lane (a job takes W = KP / (32 CL C) warps of each
// CTA), G = jobs side by side, RES = the CTA's columns of logA are resident
// in shared memory (else rows are read through L1 / L2), M = column list
// length, BEAM: a dynamic beam (Sec. V-C) instead of every state: delta is
// -inf outside the beam, the top-B of the candidates is taken at the start of
// the next step.
template <int KP, int CL, int C, int G, bool RES, int M, bool BEAM>
struct PruneCfg {
  static constexpr int KH = KP / CL, W = KH / (32 * C), NT = G * W * 32, NW = KP / 32;
  static constexpr int WB = NW < 8 ? NW : 8;  // words (of 32 rows) per list batch
  static constexpr int U = RES ? 4 : (C <= 2 ? 16 : 8);  // rows in flight (shared memory / L2 latency)
  // row list entries of a warp (a batch may add 32 WB to a list that is not yet full)
  static constexpr int CAP = (NW <= WB ? KP : 32 * WB + 128) + 2 * U;
  static constexpr size_t a_bytes = RES ? (size_t)KP * KH * 4 : 0;
  static constexpr size_t d_bytes = (size_t)G * 2 * KP * 4;  // delta, double buffered
  static constexpr size_t l_bytes = (size_t)G * W * CAP * 8;
  // COOP: the warps of a job build the first row list together, and a second
  // one of the rows the later pass is likely to want
  static constexpr bool COOP = W > 1 && (NW > 8 || BEAM);
  static constexpr int NL = KP + U;  // entries of a common list
  static constexpr size_t s_bytes = COOP ? (size_t)G * 2 * NL * 8 : 0;
  // STAGE: the columns that the bulk copies send, double buffered.  A beam
  // masks its delta at the start of the next step, when a copy may still be
  // reading; without a beam the copies read delta itself, which is written
  // again two steps later, once every CTA has the copy.
  static constexpr bool STAGE = BEAM && CL > 2;
  static constexpr size_t x_bytes = STAGE ? (size_t)2 * KH * 4 : 0;
  static constexpr size_t smem = a_bytes + d_bytes + l_bytes + s_bytes + x_bytes;
};
// bounded wait of the cluster exchange (~1 s at 2 GHz)
constexpr long long kPruneWaitCycles = 1ll << 31;

// Before steps t = 8, 16, 32, ... a job's warps, in all of its CTAs, tell each
// other how many rows per step they have formed since the last time (the most
// of any warp sets the step's time), and agree whether the sequence is handed
// over.  The launch's jobs add theirs up, and a sequence leaves where the steps
// left to it, at a + b rows each, take longer than all its steps there (unit:
// a step there) by the average of the time before, so that like sequences
// leave together and the other engine is not run beside half a launch; or
// where by its own rows they take kGiveAlone times as long.
constexpr float kGiveAlone = 2.5f;
__device__ __forceinline__ bool give_longer(float rows, float times, float ga, float gb, int t, int T) {
  return (float)(T - t) * __fmaf_rn(gb, rows, ga) > times * (float)T;
}
// A warp's word: its rows, and in the high half whether the launch's average
// says to leave.  (Not inlined: its registers are not the step loop's.)
__device__ __noinline__ uint32_t give_word(const int32_t* stat, uint32_t rows, float ga, float gb, int t, int T) {
  const volatile int32_t* s = stat + 2 * (30 - __clz(t));
  const int sum = s[0], n = s[1];
  const bool leave = n > 0 && give_longer((float)sum / (float)n, 1.f, ga, gb, t, T);
  return (rows < 0xffffu ? rows : 0xffffu) | (leave ? 0x10000u : 0u);
}
// The job's decision, from all words; `lead`: one thread of the job.
__device__ __forceinline__ bool give_decide(const uint32_t* words, int n, int32_t* stat, bool lead, float ga, float gb,
                                         int t, int T) {
  uint32_t most = 0, leave = 0;
#pragma unroll 1
  for (int x = 0; x < n; ++x) {
    const uint32_t w = words[x];
    most = max(most, w & 0xffffu);
    leave |= w >> 16;
  }
  if (lead) {
    int32_t* s = stat + 2 * (31 - __clz(t));
    atomicAdd(s, (int)most);
    atomicAdd(s + 1, 1);
  }
  return leave != 0 || give_longer((float)most, kGiveAlone, ga, gb, t, T);
}

template <int KP, int CL, int C, int G, bool RES, int M, bool BEAM>
__global__ void __launch_bounds__(PruneCfg<KP, CL, C, G, RES, M, BEAM>::NT, 1) prune_fwd_kernel(DenseArgs a) {
  using Cfg = PruneCfg<KP, CL, C, G, RES, M, BEAM>;
  constexpr int KH = Cfg::KH, W = Cfg::W, NT = Cfg::NT, NW = Cfg::NW, CAP = Cfg::CAP, WB = Cfg::WB, U = Cfg::U;
  constexpr bool COOP = Cfg::COOP;
  constexpr bool GIVE = !BEAM && KP > 256;  // sequences may be handed to the other engines
  // where the votes on that are taken: between runs of the step loop, or at
  // its top (by what the compiler makes of the loop: one K = 512 sequence 1.38
  // / 1.42 ms, 150 K = 1000 sequences 7.55 / 7.05, 8 K = 4096 ones 21.0 / 17.8)
  constexpr bool LOOK_OUT = GIVE && KP == 512;
  extern __shared__ __align__(16) char smem[];
  __shared__ __align__(8) uint64_t s_bar[G][2];
  __shared__ int s_abort;
  __shared__ uint32_t s_stop[CL];
  __shared__ __align__(8) uint64_t s_wbar[G];     // the words of a job's other CTAs are here
  __shared__ uint32_t s_votes[GIVE ? G : 1][W];     // exchanges of words so far, per warp
  __shared__ int s_rows[GIVE ? G : 1][W];           // rows formed since the last one, per warp
  __shared__ uint32_t s_word[GIVE ? G : 1][CL][W];  // what the warps say (give_word)
  __shared__ float s_max[G][W], s_need[G][2][W];  // COOP: per warp maxima and depths
  __shared__ int s_cnt[G][2][2];                  // COOP: entries of the common lists, by step parity
  // BEAM: candidates per bin (by step parity), those of the bin that holds
  // the B-th, winners per warp
  static_assert(!BEAM || (Cfg::COOP && G == 1), "beams: one job per CTA or cluster");
  constexpr int BT = BEAM ? 128 : 1;
  __shared__ __align__(16) int s_hist[BEAM ? 2 : 1][BEAM ? 256 : 4];
  __shared__ float2 s_tie[BT];
  __shared__ int s_ntie[2], s_win[W];
  const bool stop = a.hdr->status != 0;  // an earlier kernel recorded an error
  if (CL == 1 && stop) return;
  const int K = a.K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = warp / W, gw = warp % W, gt = gw * 32 + lane;  // job group, its warp and thread
  const uint32_t rank = CL > 1 ? cluster_ctarank() : 0u;
  const int col0 = (int)rank * KH + gt * C;
  const uint32_t lt = (1u << lane) - 1u;
  char* sA = smem + gt * C * 4;
  float* sd = reinterpret_cast<float*>(smem + Cfg::a_bytes) + grp * 2 * KP;
  float2* list = reinterpret_cast<float2*>(smem + Cfg::a_bytes + Cfg::d_bytes) + warp * CAP;
  float2* near = reinterpret_cast<float2*>(smem + Cfg::a_bytes + Cfg::d_bytes + Cfg::l_bytes) + grp * 2 * Cfg::NL;
  float2* far = near + Cfg::NL;
  // barrier of the job's warps here; true where any thread passes true
  auto group_any = [&](bool x) -> bool {
    if constexpr (W == 1) {
      __syncwarp();  // (a vote alone orders no memory between the lanes)
      return __any_sync(0xffffffffu, x);
    } else {
      uint32_t r;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, %2, %3, p;\n\t"
          "selp.u32 %0, 1, 0, q;\n\t}"
          : "=r"(r)
          : "r"((uint32_t)x), "r"(grp + 1), "n"(W * 32)
          : "memory");
      return r != 0;
    }
  };
  if constexpr (RES) {
    const float4* src = reinterpret_cast<const float4*>(a.pr_A);
    float4* dst = reinterpret_cast<float4*>(smem);
    for (int x = threadIdx.x; x < K * (KH / 4); x += NT)
      dst[x] = __ldg(src + (x / (KH / 4)) * (KP / 4) + rank * (KH / 4) + x % (KH / 4));
  }
  const char* __restrict__ gA = reinterpret_cast<const char*>(a.pr_A + col0);
  constexpr int RB = (RES ? KH : KP) * 4;  // bytes of a row of the copy that is read
  // the columns' lists stay in registers: values, row offsets (4 * row)
  float lv[M][C], cut[C];
  uint32_t lr[M][(C + 1) / 2];
#pragma unroll
  for (int x = 0; x < M; ++x)
#pragma unroll
    for (int c = 0; c < C; ++c) {
      lv[x][c] = __ldg(a.pr_val + x * KP + col0 + c);
      const uint32_t r = 4u * __ldg(a.pr_row + x * KP + col0 + c);
      lr[x][c / 2] = c % 2 ? (lr[x][c / 2] | (r << 16)) : r;
    }
#pragma unroll
  for (int c = 0; c < C; ++c) cut[c] = __ldg(a.pr_cut + col0 + c);
  uint32_t peer[2] = {0u, 0u};  // CL = 2: shared memory of either CTA
  const uint32_t self = smem_addr(smem);
  if (threadIdx.x == 0) s_abort = 0;
  if (GIVE && lane == 0) s_votes[grp][gw] = 0;
  if constexpr (CL > 1) {
    if constexpr (CL == 2) {
      peer[0] = dsmem_addr(smem, 0);
      peer[1] = dsmem_addr(smem, 1);
    }
    if (threadIdx.x < 2 * G) {
      mbar_init(smem_addr(&s_bar[0][0] + threadIdx.x), 1);
      if (threadIdx.x < G) mbar_init(smem_addr(&s_wbar[threadIdx.x]), 1);
      fence_mbar_init_cluster();
    }
    cluster_sync_all();  // every CTA of the cluster runs and its barriers are ready
    // the decision to stop is the cluster's: every CTA sees every flag
    if (threadIdx.x < CL) dsmem_st_u32(dsmem_addr(&s_stop[rank], threadIdx.x), stop ? 1u : 0u);
    cluster_sync_all();
    bool any = false;
#pragma unroll
    for (int r = 0; r < CL; ++r) any |= s_stop[r] != 0;
    if (any) return;
  } else {
    __syncthreads();
  }
  const int count = a.order_count;
  // job slots of the launch; a slot's jobs: longest first, rows of slots
  // forwards and backwards in turn, so every SM gets about the same steps
  // (every CTA of a cluster computes the same job without a message)
  const int ncl = (int)gridDim.x / CL, slots = ncl * G;
  const int cid = (int)blockIdx.x / CL;
  const int slot = grp * ncl + ((grp & 1) ? ncl - 1 - cid : cid);
  bool live = true, dead = false, gave = false;
  uint32_t ph = 0;  // steps run so far: buffer ph & 1, its (ph >> 1)-th use

  for (int round = 0;; ++round) {
    const int job = round * slots + ((round & 1) ? slots - 1 - slot : slot);
    if (round * slots >= count) break;
    if (job >= count) continue;
    const int b = a.order[a.order_begin + job];
    const Job jb = a.jobs[b];
    const int T = jb.T;
    const bool dense = a.emit == FV_EMIT_DENSE;
    // emission scores of the next kPruneAhead steps, oldest first; symbols
    // are read one step before the table entries they select
    float er[kPruneAhead][C];
    int xs = 0;
    const float* ep = dense ? a.E + jb.e_off + col0 : nullptr;  // row of the next load
    float* dt = a.pr_D + jb.aux_off + col0;                     // row of this step's delta
    const bool vec = dense && C > 1 && K % C == 0 && ((reinterpret_cast<uintptr_t>(ep) & (4 * C - 1)) == 0);
    auto load_e = [&](int t, float (&e)[C]) {
      if (vec) {
        // whole pieces of an aligned row
        if (t < T && col0 < K) ld_stream_vec<C>(ep, e);
        ep += K;
        return;
      }
      if (dense) {
#pragma unroll
        for (int c = 0; c < C; ++c)
          if (t < T && col0 + c < K) e[c] = ld_stream(ep + c);
        ep += K;
        return;
      }
#pragma unroll
      for (int c = 0; c < C; ++c)
        if (t < T && col0 + c < K) e[c] = __ldg(a.logB + (int64_t)(col0 + c) * a.V + xs);
      if (t + 1 < T) xs = __ldg(a.obs + jb.e_off + t + 1);
    };
    if (!dense) xs = __ldg(a.obs + jb.e_off);
#pragma unroll
    for (int k = 0; k < kPruneAhead; ++k) {
#pragma unroll
      for (int c = 0; c < C; ++c) er[k][c] = 0.f;
      load_e(k, er[k]);
    }
    float bref = 0.f, bscale = 32.f, bdepth = 4.f, binc = 0.f, bmax = 0.f;  // BEAM: bins of the top-B select
    if constexpr (BEAM) {
      for (int x = gt; x < 512; x += W * 32) s_hist[x >> 8][x & 255] = 0;
      if (gt < 2) s_ntie[gt] = 0;
      // (ordered by the barriers of the first step)
    }
    float gap = 0.f;  // how far below the maximum this warp's last steps had to look
    // hand the sequence over before step t?  (or, `live` false, a wait ran out)
    auto stop_before = [&](int t) -> bool {
      constexpr int g0 = GIVE ? 1 : 0;
      const uint32_t rows = (uint32_t)s_rows[g0 * grp][gw] / (uint32_t)(t == 8 ? 8 : t / 2);
      __syncwarp();
      if (lane == 0) s_rows[g0 * grp][gw] = 0;
      const uint32_t word = give_word(a.give_stat, rows, a.give_a, a.give_b, t, T);
      if (lane == 0) s_word[g0 * grp][rank][gw] = word;
      bool late = false;
      if constexpr (CL > 1) {
        const uint32_t bar = smem_addr(&s_wbar[grp]), par = s_votes[g0 * grp][gw] & 1u;
        if (gt == 0) mbar_arrive_expect_tx(bar, (CL - 1) * W * 4);
        if (lane < CL && lane != (int)rank)
          st_async_u32(dsmem_addr(&s_word[g0 * grp][rank][gw], lane), word, dsmem_addr(&s_wbar[grp], lane));
        const long long w0 = clock64();
        while (!late && !mbar_try_wait_cluster(bar, par))
          late = *(volatile int*)&s_abort || clock64() - w0 > kPruneWaitCycles;
      }
      __syncwarp();
      if (lane == 0) ++s_votes[g0 * grp][gw];
      if (group_any(late)) {
        // (as at the end of a step, below)
        set_status(a.hdr, FV_ETIMEOUT, 6);
        *(volatile int*)&s_abort = 1;
        const long long w0 = clock64();
        while (clock64() - w0 < (1ll << 18)) {
        }
        live = false;
        return true;
      }
      gave = give_decide(&s_word[g0 * grp][0][0], CL * W, a.give_stat, rank == 0 && gt == 0, a.give_a, a.give_b, t, T);
      return gave;
    };
    if (GIVE && lane == 0) s_rows[grp][gw] = 0;
    int t = 0, look = LOOK_OUT && a.give_b > 0.f && T > 8 ? 8 : T;
  steps:
    __attribute__((unused));
    for (; t < (LOOK_OUT ? look : T); ++t, ++ph) {
      if constexpr (GIVE && !LOOK_OUT) {
        if (t >= 8 && (t & (t - 1)) == 0 && a.give_b > 0.f && stop_before(t)) break;
      }
      const uint32_t cur = ph & 1u;  // buffer written by this step; cur ^ 1 is read
      float e[C];
#pragma unroll
      for (int c = 0; c < C; ++c) {
        e[c] = er[0][c];
#pragma unroll
        for (int k = 0; k + 1 < kPruneAhead; ++k) er[k][c] = er[k + 1][c];
      }
      load_e(t + kPruneAhead, er[kPruneAhead - 1]);
      float dval[C];
      const float* dl = sd + (cur ^ 1u) * KP;
      if (t == 0) {
        if (COOP && lane == 0) s_need[grp][cur][gw] = -1.f;
#pragma unroll
        for (int c = 0; c < C; ++c)
          dval[c] = col0 + c < K ? __fadd_rn(__ldg(a.log_pi + col0 + c), e[c]) : -CUDART_INF_F;
      } else {
        constexpr bool KEEP = NW <= 8 && !COOP;  // the deltas of this lane stay in registers
        constexpr int NK = COOP ? NW / W : NW;  // words this warp looks over for the maximum
        float dk[COOP && NK > WB ? NK : WB], dmax = -CUDART_INF_F;
#pragma unroll
        for (int k = 0; k < NK; ++k) {
          const float d = dl[32 * (COOP ? gw * NK + k : k) + lane];
          if constexpr (KEEP || COOP) dk[k] = d;
          dmax = fmaxf(dmax, d);
        }
        dmax = warp_max_f32(dmax);
        float lo, lo1 = 0.f;  // pass 0 takes delta >= lo; the second common list lo1 <= delta < lo
        int n = 0, n1 = 0;
        if constexpr (COOP) {
          int win = 0;  // BEAM: winners of the lower lanes' rows in this warp, then this lane's
          if constexpr (BEAM) {
            // ---- top-B of the K candidates under (score desc, id asc).  A
            // bin is a monotone function of the score, so whole bins above
            // the B-th candidate's are taken and only that bin is ranked.
            if (t == 1) {
              if (lane == 0) s_max[grp][gw] = dmax;
              group_any(false);
#pragma unroll
              for (int w = 0; w < W; ++w) dmax = fmaxf(dmax, s_max[grp][w]);
              bref = bmax = dmax > -CUDART_INF_F ? dmax : 0.f;
              group_any(false);
            }
            const int Wb = a.beam_B < K ? a.beam_B : K;
            bool take[NK], in[NK];  // winners; candidates still to be decided
#pragma unroll
            for (int k = 0; k < NK; ++k) {
              take[k] = false;
              in[k] = dk[k] > -CUDART_INF_F;
            }
            // the bin that holds the B-th candidate, the winners in it, its size
            int bb = 256, left = Wb, inb = 0, bb0 = 256;
            bool open = false;
#pragma unroll 1
            for (int shift = 32;; shift -= 8) {
              // bins of the score first; where more candidates share the bin
              // than can be ranked (a wrong guess of the scale, or ties),
              // radix passes over the ordered keys of those
              int bin[NK];
#pragma unroll
              for (int k = 0; k < NK; ++k) {
                if (shift == 32) {
                  const float x = __fadd_rn(bref, -dk[k]) * bscale;
                  bin[k] = x > 0.f ? (x < 255.f ? (int)x : 255) : 0;
                } else {
                  bin[k] = 255 - (int)((ord_key(__fadd_rn(dk[k], 0.f)) >> shift) & 0xffu);
                }
                if (in[k]) atomicAdd(&s_hist[cur][bin[k]], 1);
              }
              group_any(false);
              const int4 h0 = *reinterpret_cast<const int4*>(&s_hist[cur][8 * lane]);
              const int4 h1 = *reinterpret_cast<const int4*>(&s_hist[cur][8 * lane + 4]);
              const int h[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
              int sum = 0;
#pragma unroll
              for (int x = 0; x < 8; ++x) sum += h[x];
              int incl = sum;
#pragma unroll
              for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
              }
              const int total = __shfl_sync(0xffffffffu, incl, 31);
              bb = 256;
              if (total > left) {
                const int need = left;
                int acc = incl - sum;
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                  if (acc < need && need <= acc + h[x]) {
                    bb = 8 * lane + x;
                    left = need - acc;
                    inb = h[x];
                  }
                  acc += h[x];
                }
                const int src = __ffs(__ballot_sync(0xffffffffu, bb < 256)) - 1;
                bb = __shfl_sync(0xffffffffu, bb, src);
                left = __shfl_sync(0xffffffffu, left, src);
                inb = __shfl_sync(0xffffffffu, inb, src);
              } else if (total == 0) {
                dead = true;  // the beam emptied: no finite path (every CTA sees the same)
                break;
              }
              if (shift == 32) bb0 = bb;
              open = bb < 256 && left < inb;
#pragma unroll
              for (int k = 0; k < NK; ++k) {
                take[k] = take[k] || (in[k] && (bin[k] < bb || (bin[k] == bb && !open)));
                in[k] = in[k] && open && bin[k] == bb;
              }
              if (!open || inb <= BT || shift == 0) break;
              group_any(false);  // (the counts have been read)
              for (int x = gt; x < 256; x += W * 32) s_hist[cur][x] = 0;
              group_any(false);
            }
            if (dead) {
              if (rank == 0 && gt == 0) set_status(a.hdr, FV_EINFEASIBLE, (uint32_t)b);
              break;
            }
            for (int x = gt; x < 256; x += W * 32) s_hist[cur ^ 1u][x] = 0;
            if (gt == 0) s_ntie[cur ^ 1u] = 0;
            if (open && inb <= BT) {
#pragma unroll
              for (int k = 0; k < NK; ++k)
                if (in[k])
                  s_tie[atomicAdd(&s_ntie[cur], 1)] = make_float2(dk[k], __int_as_float(32 * (gw * NK + k) + lane));
              group_any(false);
              if (inb <= 32) {
                // a lane per candidate: the last winner among them, for all
                const float2 q = lane < inb ? s_tie[lane] : make_float2(-CUDART_INF_F, __int_as_float(0x7fffffff));
                const int qi = __float_as_int(q.y);
                int ahead = 0;
                for (int x = 0; x < inb; ++x) {
                  const float y = __shfl_sync(0xffffffffu, q.x, x);
                  const int yi = __shfl_sync(0xffffffffu, qi, x);
                  ahead += y > q.x || (y == q.x && yi < qi);
                }
                const int src = __ffs(__ballot_sync(0xffffffffu, lane < inb && ahead == left - 1)) - 1;
                const float tv = __shfl_sync(0xffffffffu, q.x, src & 31);
                const int ti = __shfl_sync(0xffffffffu, qi, src & 31);
#pragma unroll
                for (int k = 0; k < NK; ++k)
                  if (in[k]) take[k] = dk[k] > tv || (dk[k] == tv && 32 * (gw * NK + k) + lane <= ti);
              } else
#pragma unroll
              for (int k = 0; k < NK; ++k)
                if (in[k]) {
                  const int id = 32 * (gw * NK + k) + lane;
                  int ahead = 0;
                  for (int x = 0; x < inb; ++x) {
                    const float2 q = s_tie[x];
                    ahead += q.x > dk[k] || (q.x == dk[k] && __float_as_int(q.y) < id);
                  }
                  take[k] = ahead < left;
                }
            } else if (open) {
              // more equal scores than the list holds: the lowest ids of them
              int mine = 0;
#pragma unroll
              for (int k = 0; k < NK; ++k) mine += __popc(__ballot_sync(0xffffffffu, in[k]));
              if (lane == 0) s_win[gw] = mine;
              group_any(false);
              int ahead = 0;
#pragma unroll
              for (int w = 0; w < W; ++w) ahead += w < gw ? s_win[w] : 0;
#pragma unroll
              for (int k = 0; k < NK; ++k) {
                const uint32_t mk = __ballot_sync(0xffffffffu, in[k]);
                if (in[k]) take[k] = ahead + __popc(mk & lt) < left;
                ahead += __popc(mk);
              }
              group_any(false);  // (s_win is written again below)
            }
            // outside the beam: -inf, here and in the vector that is read
            float* dm = sd + (cur ^ 1u) * KP;
            dmax = -CUDART_INF_F;
            int mine = 0;
#pragma unroll
            for (int k = 0; k < NK; ++k) {
              if (!take[k]) {
                if (dk[k] > -CUDART_INF_F) dm[32 * (gw * NK + k) + lane] = -CUDART_INF_F;
                dk[k] = -CUDART_INF_F;
              }
              dmax = fmaxf(dmax, dk[k]);
              mine += take[k];
            }
            dmax = warp_max_f32(dmax);
            int x = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const int y = __shfl_up_sync(0xffffffffu, x, o);
              if (lane >= o) x += y;
            }
            win = x - mine;
            if (lane == 31) s_win[gw] = x;
            // the next step's bins: the B-th candidate near the middle
            if (bb0 < 256) {
              if (bb0 == 255) bdepth *= 1.5f;
              else bdepth = 0.75f * bdepth + 0.25f * (((float)bb0 + 0.5f) / bscale);
              bdepth = fmaxf(bdepth, fmaxf(0.25f * gap, 1e-30f));
            }
          }
          if (lane == 0) s_max[grp][gw] = dmax;
          if (gt < 2) s_cnt[grp][cur][gt] = 0;
          group_any(false);
          float most = -1.f;
#pragma unroll
          for (int w = 0; w < W; ++w) {
            dmax = fmaxf(dmax, s_max[grp][w]);
            const float x = s_need[grp][cur ^ 1u][w];
            most = fmaxf(most, x);
          }
          if constexpr (BEAM) {
            // this CTA's winners of step t - 1 to the table (any order)
            int pos = win, all = 0;
#pragma unroll
            for (int w = 0; w < W; ++w) {
              const int x = s_win[w];
              all += x;
              if (w < gw) pos += x;
            }
            const int64_t base = jb.aux_off + (int64_t)(t - 1) * a.beam_stride;
#pragma unroll
            for (int k = 0; k < NK; ++k)
              if (dk[k] > -CUDART_INF_F) {
                const int id = 32 * (gw * NK + k) + lane;
                if (CL == 1 || (id >= (int)rank * KH && id < ((int)rank + 1) * KH)) {
                  a.beam_id[base + pos] = id;
                  a.beam_val[base + pos] = dk[k];
                }
                ++pos;
              }
            for (int x = all + gt; x < a.beam_stride && rank == 0; x += W * 32) a.beam_id[base + x] = -1;
            const float g = __fadd_rn(dmax, -bmax);
            if (fabsf(g) < 1e30f) {
              binc = 0.9f * binc + 0.1f * g;
              bmax = dmax;
            }
            bref = __fadd_rn(bmax, binc);
            bscale = 160.f / bdepth;
          }
          if (most >= 0.f) gap = 0.75f * gap + 0.25f * most;
          lo = fmaxf(__fmaf_rn(-kGapCommon, gap, dmax), -FLT_MAX);  // (never rows at -inf)
          lo1 = fmaxf(__fmaf_rn(-kFarGap, gap, dmax), -FLT_MAX);
          // this lane's rows of either list (low and high half), their
          // places by a scan over the lanes and one add per warp and list
          uint32_t c = 0;
#pragma unroll
          for (int k = 0; k < NK; ++k) c += dk[k] >= lo ? 1u : (dk[k] >= lo1 ? 0x10000u : 0u);
          uint32_t x = c;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
          }
          uint32_t base = 0;
          const uint32_t tot = __shfl_sync(0xffffffffu, x, 31);
          if (lane >= 30) base = (uint32_t)atomicAdd(&s_cnt[grp][cur][lane - 30], (int)(lane == 30 ? tot & 0xffffu : tot >> 16));
          int p0 = (int)(__shfl_sync(0xffffffffu, base, 30) + ((x - c) & 0xffffu));
          int p1 = (int)(__shfl_sync(0xffffffffu, base, 31) + ((x - c) >> 16));
#pragma unroll
          for (int k = 0; k < NK; ++k) {
            const float2 ent = make_float2(dk[k], __int_as_float((32 * (gw * NK + k) + lane) * RB));
            const bool i0 = dk[k] >= lo, i1 = !i0 && dk[k] >= lo1;
            float2* to = i0 ? near + p0 : far + p1;
            if (i0 || i1) *to = ent;
            p0 += i0;
            p1 += i1;
          }
          group_any(false);
          n = s_cnt[grp][cur][0];
          n1 = s_cnt[grp][cur][1];
        } else {
          lo = fmaxf(__fmaf_rn(-kGap, gap, dmax), -FLT_MAX);  // (never rows at -inf)
        }
        float best[C];
#pragma unroll
        for (int c = 0; c < C; ++c) best[c] = -CUDART_INF_F;
        Vec<C> v[U];
        float d[U];
        // rows src[i .. i + U) into v, their deltas into d
        auto load_rows = [&](const float2* src, int i) {
#pragma unroll
          for (int u = 0; u < U / 2; ++u) {
            const float4 q = *reinterpret_cast<const float4*>(src + i + 2 * u);
            const char* base = RES ? sA : gA;
            const float* r0 = reinterpret_cast<const float*>(base + __float_as_int(q.y));
            const float* r1 = reinterpret_cast<const float*>(base + __float_as_int(q.w));
            if constexpr (RES) {
              v[2 * u].lds(r0);
              v[2 * u + 1].lds(r1);
            } else {
              v[2 * u].ldg(r0);
              v[2 * u + 1].ldg(r1);
            }
            d[2 * u] = q.x;
            d[2 * u + 1] = q.z;
          }
        };
        auto use_rows = [&]() {
#pragma unroll
          for (int u = 0; u < U; u += 2)
#pragma unroll
            for (int c = 0; c < C; ++c)
              best[c] = fmaxf(best[c], fmaxf(__fadd_rn(d[u], v[u].v[c]), __fadd_rn(d[u + 1], v[u + 1].v[c])));
        };
        // pads the list to whole groups with rows that give -inf
        auto close_list = [&](float2* src, int n) {
          if (lane < U) src[n + lane] = make_float2(-CUDART_INF_F, 0.f);
          __syncwarp();
        };
        // the listed rows (their order does not matter: only the maximum is kept)
        auto flush = [&](int n) {
          if (GIVE && lane == 0) s_rows[grp][gw] += n;
          close_list(list, n);
#pragma unroll 1
          for (int i = 0; i < n; i += U) {
            load_rows(list, i);
            use_rows();
          }
          __syncwarp();
        };
        // the rows of the words kb .. kb + WB with lo <= delta < hi, after
        // the n entries of the list; returns the new count
        auto list_words = [&](int kb, float lo, float hi, int n) -> int {
          if constexpr (!KEEP) {
#pragma unroll
            for (int k = 0; k < WB; ++k) dk[k] = dl[32 * (kb + k) + lane];
          }
#pragma unroll
          for (int k = 0; k < WB; ++k) {
            const bool in = dk[k] >= lo && dk[k] < hi;
            const uint32_t mk = __ballot_sync(0xffffffffu, in);
            if (in) list[n + __popc(mk & lt)] = make_float2(dk[k], __int_as_float((32 * (kb + k) + lane) * RB));
            n += __popc(mk);
          }
          return n;
        };
        // pass 0: rows with delta >= dmax - gap.  The first group's loads are
        // under way while the lists' candidates are formed.
        float2* const first = COOP ? near : list;
        if constexpr (!COOP) {
#pragma unroll 1
          for (int kb = 0; kb < NW; kb += WB) {
            n = list_words(kb, lo, CUDART_INF_F, n);
            if (kb + WB < NW && n > CAP - 2 * U - 32 * WB) {
              flush(n);
              n = 0;
            }
          }
        }
        if (GIVE && lane == 0) s_rows[grp][gw] += n;
        close_list(first, n);  // (every warp writes the same beyond a common list)
        load_rows(first, 0);
#pragma unroll
        for (int x = 0; x < M; ++x)
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const uint32_t o = c % 2 ? lr[x][c / 2] >> 16 : lr[x][c / 2] & 0xffffu;
            best[c] = fmaxf(best[c], __fadd_rn(*reinterpret_cast<const float*>(reinterpret_cast<const char*>(dl) + o),
                                               lv[x][c]));
          }
        use_rows();
#pragma unroll 1
        for (int i = U; i < n; i += U) {
          load_rows(first, i);
          use_rows();
        }
        // pass 1: the rows below that which could still reach a target of
        // this warp.  (A column without a finite weight outside its list
        // gives NaN, which the minimum passes over.)
        float th = CUDART_INF_F;
#pragma unroll
        for (int c = 0; c < C; ++c) th = fminf(th, need_delta(best[c], cut[c]));
        th = warp_min_f32(th);
        const float need = __fadd_rn(dmax, -th);
        const bool depth = need < CUDART_INF_F && need >= 0.f;
        if constexpr (COOP) {
          if (lane == 0) s_need[grp][cur][gw] = depth ? need : -1.f;
        } else {
          if (depth) gap = 0.75f * gap + 0.25f * need;
        }
        if (th < lo) {
          __syncwarp();
          if (COOP && th >= lo1) {
            // the second common list holds them
            n = 0;
#pragma unroll 1
            for (int i0 = 0; i0 < n1; i0 += 32) {
              const bool have = i0 + lane < n1;
              const float2 ent = far[have ? i0 + lane : 0];
              const bool in = have && ent.x >= th;
              const uint32_t mk = __ballot_sync(0xffffffffu, in);
              if (in) list[n + __popc(mk & lt)] = ent;
              n += __popc(mk);
              if (i0 + 32 >= n1 || n > CAP - 2 * U - 32) {
                flush(n);
                n = 0;
              }
            }
          } else {
            const float hi = lo;
            lo = fmaxf(th, -FLT_MAX);
            n = 0;
#pragma unroll 1
            for (int kb = 0; kb < NW; kb += WB) {
              n = list_words(kb, lo, hi, n);
              if (kb + WB >= NW || n > CAP - 2 * U - 32 * WB) {
                flush(n);
                n = 0;
              }
            }
          }
        }
        bool zero = false;
#pragma unroll
        for (int c = 0; c < C; ++c) {
          dval[c] = __fadd_rn(best[c], e[c]);  // (-inf beyond K)
          zero = zero || dval[c] == 0.f;
        }
        if (zero) {
          // a zero plus E = -0 has the sign of the kept candidate's zero,
          // the lowest maximising row's
#pragma unroll
          for (int c = 0; c < C; ++c)
            if (best[c] == 0.f && __float_as_uint(e[c]) == 0x80000000u && col0 + c < K)
              for (int i = 0; i < K; ++i) {
                const float x = __fadd_rn(dl[i], __ldg(a.pr_A + (int64_t)i * KP + col0 + c));
                if (x == 0.f) {
                  dval[c] = __fadd_rn(x, e[c]);
                  break;
                }
              }
        }
      }
      // ---- delta_t: shared memory (of every CTA of the cluster) and the table
      float* dn = sd + cur * KP + col0;
      if constexpr (C == 4) *reinterpret_cast<float4*>(dn) = make_float4(dval[0], dval[1], dval[2], dval[3]);
      else if constexpr (C == 2) *reinterpret_cast<float2*>(dn) = make_float2(dval[0], dval[1]);
      else dn[0] = dval[0];
      if constexpr (CL > 1) {
        const uint32_t bar = smem_addr(&s_bar[grp][cur]);
        // test hook: CTA 1 keeps its second step from the others
        const bool withhold = t == 1 && rank == 1 && a.wide_withhold;
        if (gt == 0) mbar_arrive_expect_tx(bar, (CL - 1) * KH * 4);
        if constexpr (CL == 2) {
          // 16 bytes per store: four lanes' columns where a lane has one
          uint4 v = make_uint4(__float_as_uint(dval[0]), 0, 0, 0);
          bool send = true;
          int c4 = col0;
          if constexpr (C == 4) {
            v = make_uint4(__float_as_uint(dval[0]), __float_as_uint(dval[1]), __float_as_uint(dval[2]),
                           __float_as_uint(dval[3]));
          } else {
            __syncwarp();
            send = lane < 8 * C;
            c4 = col0 - lane * C + 4 * (send ? lane : 0);
            v = *reinterpret_cast<const uint4*>(sd + cur * KP + c4);
          }
          if (send && !withhold) {
            const uint32_t off = smem_addr(sd + cur * KP + c4) - self, boff = bar - self;
            const uint32_t to = rank ? peer[0] : peer[1];
            st_async_v4(to + off, v, to + boff);
          }
        } else {
          // one copy of the CTA's columns to each of the others
          const float* own = sd + cur * KP + (int)rank * KH;
          if constexpr (Cfg::STAGE) {
            float* sx = reinterpret_cast<float*>(smem + Cfg::a_bytes + Cfg::d_bytes + Cfg::l_bytes + Cfg::s_bytes) +
                        cur * KH;
#pragma unroll
            for (int c = 0; c < C; ++c) sx[gt * C + c] = dval[c];
            own = sx;
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          group_any(false);
          if (gt < CL && gt != (int)rank && !withhold) {
            const uint32_t src = smem_addr(own), dst = smem_addr(sd + cur * KP + (int)rank * KH);
            const uint32_t to = dsmem_addr(smem, gt);
            asm volatile(
                "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    to + (dst - self)),
                "r"(src), "r"(KH * 4), "r"(to + (bar - self))
                : "memory");
          }
        }
      }
      if constexpr (BEAM) {
        // (the beam of this step goes to the table once it is known)
      } else if (C > 1 && K % C == 0) {
        if (col0 < K) {
          if constexpr (C == 4) __stcs(reinterpret_cast<float4*>(dt), make_float4(dval[0], dval[1], dval[2], dval[3]));
          if constexpr (C == 2) __stcs(reinterpret_cast<float2*>(dt), make_float2(dval[0], dval[1]));
        }
      } else {
#pragma unroll
        for (int c = 0; c < C; ++c)
          if (col0 + c < K) __stcs(dt + c, dval[c]);
      }
      dt += K;
      bool late = false;
      if constexpr (CL > 1) {
        const uint32_t bar = smem_addr(&s_bar[grp][cur]), par = (ph >> 1) & 1u;
        if (!mbar_try_wait_cluster(bar, par)) {
          const long long w0 = clock64();
          while (!late && !mbar_try_wait_cluster(bar, par))
            late = *(volatile int*)&s_abort || clock64() - w0 > kPruneWaitCycles;
        }
      }
      if (group_any(late)) {
        // (cluster exchange only) a wait ran out: the job group stops; its
        // own stores have landed by the end of the delay
        set_status(a.hdr, FV_ETIMEOUT, 5);
        *(volatile int*)&s_abort = 1;
        const long long w0 = clock64();
        while (clock64() - w0 < (1ll << 18)) {
        }
        live = false;
        break;
      }
    }
    if constexpr (LOOK_OUT) {
      if (live && t < T && !stop_before(t)) {
        look = 2 * look < T ? 2 * look : T;
        goto steps;
      }
    }
    if (!live) break;
    if (GIVE && gave) {
      gave = false;
      if (rank == 0 && gt == 0) {
        a.qlast[b] = -1;  // nothing to trace
        a.give_list[atomicAdd(a.give_count, 1)] = b;
      }
      continue;
    }
    if (BEAM && dead) {
      // the same in every CTA of the cluster, before anything of the step was
      // exchanged; the next job clears what this one read
      dead = false;
      group_any(false);
      continue;
    }
    if (rank == 0 && gw == 0) {
      // termination: q_{T-1} = lowest argmax_j delta_{T-1}[j], score = delta_{T-1}[q]
      const float* dl = sd + ((ph - 1u) & 1u) * KP;
      float v = dl[lane];
      int qi = lane;
#pragma unroll
      for (int k = 1; k < NW; ++k) {
        const float vk = dl[lane + 32 * k];
        if (vk > v) { v = vk; qi = lane + 32 * k; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int oq = __shfl_xor_sync(0xffffffffu, qi, o);
        if (ov > v || (ov == v && oq < qi)) { v = ov; qi = oq; }
      }
      if (lane == 0) {
        if (BEAM && !(v > -CUDART_INF_F)) set_status(a.hdr, FV_EINFEASIBLE, (uint32_t)b);
        a.qlast[b] = qi;
        a.scores[b] = dl[qi];
      }
    }
    if constexpr (BEAM && CL == 1) group_any(false);  // (the next job clears what this one read)
  }
  if constexpr (CL > 1) {
    // no CTA leaves while another may still write to it or read its barriers
    __syncwarp();
    if (!live && lane < CL) dsmem_st_u32(dsmem_addr(&s_stop[rank], lane), 1u);
    __syncwarp();
    cluster_sync_all();
    // where a wait ran out, a CTA may have left the steps before data that
    // was sent to it arrived: every copy of the cluster is on its way by now
    // and lands within the delay
    bool any = false;
#pragma unroll
    for (int r = 0; r < CL; ++r) any |= s_stop[r] != 0;
    if (any) {
      const long long w0 = clock64();
      while (clock64() - w0 < (1ll << 18)) {
      }
      __syncwarp();
      cluster_sync_all();
    }
  }
}

// ------------------------------------------------------------------ trace
// The path from the stored deltas: q_{t-1} = lowest argmax_i of
// fl(delta_{t-1}[i] + A[i][q_t]) -- only the path's own backpointers are
// ever computed.  A step waits for a column of logA that depends on the
// state before, so a sequence is cut into segments traced side by side: a
// segment's trace starts kTraceWarm steps after its end from the best state
// there (survivors of a Viterbi recursion meet within tens of steps), and a
// second kernel follows the segments from the last one, which starts at the
// known final state, and traces again from any end where the guess was not
// the path's state until it meets the written path.
constexpr int kTraceWarm = 24;

struct TraceArgs {
  const Job* jobs;
  const int32_t* order;
  int32_t begin, count, K, seg;  // seg: states per segment
  int32_t row, unit;             // BEAM: entries per row; at most this many table elements per step
  const int32_t* ids;            // BEAM: states of the entries
  const float* D;
  const float* AT;
  const int32_t* qlast;
  int32_t* paths;
  int32_t* guess;  // state assumed at each segment's end
  int64_t guess_cap;
  const WsHeader* hdr;
};
// TW warps of a CTA follow one chain, VPL rows of a column per thread; ROWS:
// AT is logA itself (K <= 128: it stays in L1 whatever the order).
template <int VPL, int TW, bool BEAM, bool ROWS>
struct Tracer {
  static constexpr int AH = VPL <= 8 ? 4 : 2;  // delta rows loaded ahead
  static constexpr int NT = 32 * TW;
  const float* D;     // delta rows, or the beams' scores
  const int32_t* ids;  // BEAM: their states (-1: no entry)
  const float* AT;
  int K, KD, tid;
  int N;  // entries of a row
  uint2* part;  // shared, [2][TW]: per warp (value, row) of a step, by turns
  int turn;
  struct Row {
    float d[VPL];
    int i[BEAM ? VPL : 1];
  };
  Row rows[AH];
  __device__ __forceinline__ void init(const TraceArgs& a, const Job& jb, uint2* part_) {
    D = a.D + jb.aux_off;
    if (BEAM) ids = a.ids + jb.aux_off;
    AT = a.AT;
    N = BEAM ? a.row : a.K;
    const int K_ = a.K;
    K = K_;
    KD = wide_lane_stride(K_);
    tid = threadIdx.x;
    part = part_;
    turn = 0;
  }
  __device__ __forceinline__ void load(int t, Row& x) {
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const int e = NT * k + tid;
      const bool in = t >= 0 && e < N;
      if constexpr (BEAM) {
        x.i[k] = in ? __ldcs(ids + (int64_t)t * N + e) : -1;
        if ((unsigned)x.i[k] >= (unsigned)K) x.i[k] = -1;
      }
      x.d[k] = in ? __ldcs(D + (int64_t)t * N + e) : -CUDART_INF_F;
    }
  }
  // rows t - 1, t - 2, ... for steps from state q_t downwards
  __device__ __forceinline__ void start(int t) {
#pragma unroll
    for (int k = 0; k < AH; ++k) load(t - 1 - k, rows[k]);
  }
  // lowest argmax over the threads' (value, row); 0 where every value is -inf
  __device__ __forceinline__ int lowest(float bv, int bi) {
    float v = __fadd_rn(bv, 0.f);  // (-0 as +0: they tie)
    float m = warp_max_f32(v);
    uint32_t r = __reduce_min_sync(0xffffffffu, v == m && v > -CUDART_INF_F ? (uint32_t)bi : 0xffffffffu);
    if constexpr (TW > 1) {
      if ((tid & 31) == 0) part[turn * TW + tid / 32] = make_uint2(__float_as_uint(m), r);
      __syncthreads();
#pragma unroll
      for (int w = 0; w < TW; ++w) {
        const uint2 x = part[turn * TW + w];
        const float y = __uint_as_float(x.x);
        if (w == 0 || y > m || (y == m && x.y < r)) {
          m = y;
          r = x.y;
        }
      }
      turn ^= 1;
    }
    return r < (uint32_t)K ? (int)r : 0;
  }
  // q_{t-1} from q_t; `x` holds delta_{t-1} and receives row t - 1 - AH
  __device__ __forceinline__ int step(int t, int q, Row& x) {
    const float* col = AT + (ROWS ? q : q * (int64_t)KD);
    float v[VPL];
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const int i = BEAM ? x.i[k] : NT * k + tid;
      v[k] = (BEAM ? i >= 0 : i < (ROWS ? K : KD)) ? __ldg(col + (ROWS ? i * K : i)) : -CUDART_INF_F;
    }
    float bv = -CUDART_INF_F;
    int bi = 0;
#pragma unroll
    for (int k = 0; k < VPL; ++k) pick(__fadd_rn(x.d[k], v[k]), x, k, bv, bi);
    load(t - 1 - AH, x);
    return lowest(bv, bi);
  }
  // (value, row) of entry k, if it comes before (bv, bi)
  __device__ __forceinline__ void pick(float c, const Row& x, int k, float& bv, int& bi) {
    if constexpr (BEAM) {
      // a row's entries come in any order
      if (x.i[k] >= 0 && (c > bv || (c == bv && x.i[k] < bi))) { bv = c; bi = x.i[k]; }
    } else {
      if (c > bv) { bv = c; bi = NT * k + tid; }
    }
  }
  // lowest argmax of delta_t
  __device__ __forceinline__ int best(int t) {
    Row x;
    load(t, x);
    float bv = -CUDART_INF_F;
    int bi = 0;
#pragma unroll
    for (int k = 0; k < VPL; ++k) pick(x.d[k], x, k, bv, bi);
    return lowest(bv, bi);
  }
  // from q_t down to state `to`; f(time, state) returns true to stop there
  template <typename F>
  __device__ __forceinline__ int run(int t, int to, int q, F f) {
    start(t);
    while (t > to) {
#pragma unroll
      for (int s = 0; s < AH; ++s) {
        if (t <= to) break;
        q = step(t, q, rows[s]);
        --t;
        if (f(t, q)) return q;
      }
    }
    return q;
  }
};

// first guess of a sequence: at least ceil(T / seg) apart, as a step has
// `unit` table elements or more
__device__ __forceinline__ int64_t guess_off(const TraceArgs& a, const Job& jb, int b) {
  return jb.aux_off / ((int64_t)a.unit * a.seg) + b;
}

template <int VPL, int TW, bool BEAM, bool ROWS>
__global__ void __launch_bounds__(32 * TW) prune_trace_kernel(TraceArgs a) {
  __shared__ uint2 part[2 * TW];
  if (a.hdr->status != 0) return;
  const int b = a.order[a.begin + blockIdx.x];
  const Job jb = a.jobs[b];
  const int T = jb.T, K = a.K;
  if (a.qlast[b] < 0) return;  // handed to another engine
  Tracer<VPL, TW, BEAM, ROWS> tr;
  tr.init(a, jb, part);
  int32_t* path = a.paths + jb.path_off;
  const bool lead = threadIdx.x == 0;
  // (a segment each, where the lengths here are no longer than the host's
  // that sized the grid)
  for (int64_t s = blockIdx.y; s * a.seg < T; s += gridDim.y) {
    const int lo = (int)s * a.seg;
    int q = a.qlast[b];
    q = (unsigned)q < (unsigned)K ? q : 0;
    int t = T - 1;  // q = q_t
    if (T - lo > a.seg) {
      const int hi = lo + a.seg;  // hi <= T - 1
      if (hi + kTraceWarm < T - 1) {
        t = hi + kTraceWarm;
        q = tr.best(t);
      }
      q = tr.run(t, hi, q, [](int, int) { return false; });
      t = hi;
      const int64_t g = guess_off(a, jb, b) + s;
      if (lead && g < a.guess_cap) a.guess[g] = q;
    } else if (lead) {
      path[t] = q;
    }
    tr.run(t, lo, q, [&](int u, int x) {
      if (lead) path[u] = x;
      return false;
    });
  }
}

template <int VPL, int TW, bool BEAM, bool ROWS>
__global__ void __launch_bounds__(32 * TW) prune_fix_kernel(TraceArgs a) {
  __shared__ uint2 part[2 * TW];
  if (a.hdr->status != 0) return;
  const int b = a.order[a.begin + blockIdx.x], lane = threadIdx.x & 31;
  const Job jb = a.jobs[b];
  if (a.qlast[b] < 0) return;
  const int K = a.K, nseg = (jb.T + a.seg - 1) / a.seg;
  int32_t* path = a.paths + jb.path_off;
  const int64_t g0 = guess_off(a, jb, b);
  auto sync = []() {
    if constexpr (TW > 1) __syncthreads();
    else __syncwarp();
  };
  for (int s1 = nseg - 2; s1 >= 0;) {
    // the highest of up to 32 segments s1, s1 - 1, ... whose end was guessed
    // wrong (every warp finds the same)
    const int s = s1 - lane;
    bool bad = false;
    if (s >= 0) bad = g0 + s >= a.guess_cap || a.guess[g0 + s] != __ldcg(path + (int64_t)(s + 1) * a.seg);
    const uint32_t m = __ballot_sync(0xffffffffu, bad);
    if (!m) {
      s1 -= 32;
      continue;
    }
    const int sb = s1 - (__ffs(m) - 1), lo = sb * a.seg, hi = lo + a.seg;
    Tracer<VPL, TW, BEAM, ROWS> tr;
    tr.init(a, jb, part);
    int q = __ldcg(path + hi);
    q = (unsigned)q < (unsigned)K ? q : 0;
    sync();
    tr.run(hi, lo, q, [&](int u, int x) {
      const bool same = __ldcg(path + u) == x;
      sync();
      if (!same && threadIdx.x == 0) path[u] = x;
      return same;
    });
    __threadfence_block();
    sync();
    s1 = sb - 1;
  }
}

int prune_pad(int K) { return K <= 256 ? 256 : K <= 512 ? 512 : K <= 1024 ? 1024 : K <= 2048 ? 2048 : 4096; }
// List lengths, from sweeps (us per step): K = 256, 4 / 6 entries: 1024
// sequences 4.47 / 4.32 (two columns per lane); K = 512, 8 / 12: one sequence
// 2.18 / 2.07; K = 1000, 8 / 12 / 16: 152 sequences 9.1 / 8.9 / 8.6.  A longer
// list lowers the cutoffs (fewer rows) but gathers more deltas.
int prune_list(int K) { return K <= 256 ? 6 : K <= 512 ? 12 : K <= 1024 ? 16 : 32; }
// the row copy, and in its place the row-pair copy of the engine that
// sequences are handed to once the others are traced
static size_t prune_copy_bytes(int K) {
  int kpm = 0, cols = 0;
  dense_stream_geometry(K, &kpm, &cols);
  const size_t rows = (size_t)K * prune_pad(K) * 4, pairs = (size_t)kpm * cols * 4;
  return align_up(rows > pairs ? rows : pairs);
}
// area: row copy, column-major copy, list values, cutoffs, list rows
size_t prune_area_bytes(int K) {
  if (K <= 128) return 0;  // (fv_small.cu needs none)
  const size_t KP = prune_pad(K), M = prune_list(K);
  return prune_copy_bytes(K) + align_up((size_t)K * wide_lane_stride(K) * 4) + align_up(KP * (M * 6 + 4));
}

template <int VPL>
static cudaError_t launch_prep_cfg(const float* logA, int K, float* A, float* at, float* val, uint16_t* row, float* cut,
                                   int32_t* stat, cudaStream_t st) {
  const size_t sm = 8 * (32 * VPL + 4) * sizeof(float);
  cudaError_t e =
      cudaFuncSetAttribute(prune_prep_kernel<VPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  prune_prep_kernel<VPL><<<prune_pad(K) / 8, 256, sm, st>>>(logA, K, prune_pad(K), prune_list(K), A, at, val, row,
                                                              cut, stat);
  return cudaGetLastError();
}

cudaError_t launch_prune_prep(const float* logA, int K, char* area, DenseArgs* a, cudaStream_t st) {
  const int KP = prune_pad(K), M = prune_list(K);
  float* copy = reinterpret_cast<float*>(area);
  area += prune_copy_bytes(K);
  float* at = reinterpret_cast<float*>(area);
  area += align_up((size_t)K * wide_lane_stride(K) * 4);
  float* val = reinterpret_cast<float*>(area);
  float* cut = val + (size_t)M * KP;
  uint16_t* row = reinterpret_cast<uint16_t*>(cut + KP);
  a->pr_A = copy;
  a->pr_val = val;
  a->pr_row = row;
  a->pr_cut = cut;
  a->wide_AT = at;
  if (K <= 256) return launch_prep_cfg<8>(logA, K, copy, at, val, row, cut, a->give_stat, st);
  if (K <= 512) return launch_prep_cfg<16>(logA, K, copy, at, val, row, cut, a->give_stat, st);
  if (K <= 1024) return launch_prep_cfg<32>(logA, K, copy, at, val, row, cut, a->give_stat, st);
  if (K <= 2048) return launch_prep_cfg<64>(logA, K, copy, at, val, row, cut, a->give_stat, st);
  return launch_prep_cfg<128>(logA, K, copy, at, val, row, cut, a->give_stat, st);
}

// Clusters (CTAs for CL = 1) of a configuration resident at once; 0 where the
// device does not take it.  A property of the kernel and the device, asked
// for once per device ordinal (a query and an attribute call cost several
// microseconds of a short decode).
template <int KP, int CL, int C, int G, bool RES, int M, bool BEAM>
static int prune_resident(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
  using Cfg = PruneCfg<KP, CL, C, G, RES, M, BEAM>;
  static_assert(Cfg::smem + 1024 <= 227 * 1024, "one CTA per SM");
  static_assert(Cfg::W == 1 || G <= 15, "a named barrier per job group");
  auto kern = prune_fwd_kernel<KP, CL, C, G, RES, M, BEAM>;
  static std::atomic<int> known[64];  // per device, plus one
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  const int nsm = device_sm_count();
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = CL;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg->gridDim = dim3(CL * nsm);
  cfg->blockDim = dim3(Cfg::NT);
  cfg->dynamicSmemBytes = Cfg::smem;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
  if (known[dev].load() > 0) return known[dev].load() - 1;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::smem);
  if (e == cudaSuccess && CL > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) {
    if (CL > 1) {
      e = cudaOccupancyMaxActiveClusters(&n, kern, cfg);
    } else {
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, Cfg::NT, Cfg::smem);
      n *= nsm;
    }
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  known[dev].store(n + 1);
  return n;
}

template <int KP, int CL, int C, int G, bool RES, int M, bool BEAM>
static cudaError_t launch_prune_cfg(const DenseArgs& a, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  const int resident = prune_resident<KP, CL, C, G, RES, M, BEAM>(&cfg, attr), jobs = a.order_count;
  if (resident < 1) return cudaErrorInvalidConfiguration;
  cfg.stream = st;
  cfg.gridDim = dim3(CL * (jobs < resident ? jobs : resident));
  return cudaLaunchKernelEx(&cfg, prune_fwd_kernel<KP, CL, C, G, RES, M, BEAM>, a);
}

// Configurations by state count and launch (GB300, us per step of the whole
// call, Dirichlet(1) weights; the slot engine of fv_dense.cu in brackets):
//   K <= 256, 2-CTA clusters, columns resident: two columns per lane and 8
//     jobs per cluster 1.28 / 2.12 / 3.75 at 1 / 608 / 1024 equal sequences
//     (2.29 / 6.78 / 11.6), four columns and 16 jobs 1.60 / 2.16 / 2.97.  Four
//     columns spend less per job step but more per step of a lone job, so
//     they are taken when the steps per SM outweigh the longest sequence
//     (1024 sequences of 500 .. 4000 steps, which don't: 7.7 against 8.4 ms).
//   K <= 512: one job per warp over 8-CTA clusters with resident columns
//     while its slots (8 jobs on each of 15 clusters) hold the launch: 2.07 /
//     2.46 at 1 / 64 sequences (3.47 / 4.27); then a CTA per job reading rows
//     through L2: two columns per lane up to a job per SM, 3.6 at 152 (8.05),
//     four columns and two CTAs per SM beyond, 4.8 at 304 (11.9).
//   K <= 1024: a CTA per job, 5.9 at 152 (26.6), bound by the L2 reads of its
//     rows (64 bytes per clock); half as many jobs take two CTAs each, 3.7 at
//     40 (10.7; four CTAs 4.1, eight 3.8).
//   K <= 2048: 4-CTA clusters, 5.1 at 1 .. 30 sequences (eight CTAs 5.3 up to
//     15 sequences); K <= 4096: 8-CTA clusters, 15 at a time, 8.7 at 8 (21.1 on
//     the whole-GPU engine of fv_wide.cu, which reads all of logA every step;
//     16-CTA clusters fit seven at a time and took 21.8).  512 columns per CTA,
//     two per lane (one per lane: 6.7 and 11.8).  List lengths 24 / 32 / 48 at
//     K = 4096, 8 sequences with Dirichlet(0.1) rows: 21.6 / 17.3 / 28.0 ms.
cudaError_t launch_prune_forward(const DenseArgs& a, int64_t sum_T, int max_T, cudaStream_t st) {
  const int jobs = a.order_count, nsm = device_sm_count();
  if (jobs <= 0) return cudaSuccess;
  if (a.K <= 256) {
    if (sum_T > 5ll * nsm * max_T) return launch_prune_cfg<256, 2, 4, 16, true, 6, false>(a, st);
    return launch_prune_cfg<256, 2, 2, 8, true, 6, false>(a, st);
  }
  if (a.K <= 512) {
    if (jobs <= 120) return launch_prune_cfg<512, 8, 2, 8, true, 12, false>(a, st);
    if (jobs <= nsm) return launch_prune_cfg<512, 1, 2, 1, false, 12, false>(a, st);
    return launch_prune_cfg<512, 1, 4, 1, false, 12, false>(a, st);
  }
  if (a.K <= 1024) {
    if (2 * jobs <= nsm) return launch_prune_cfg<1024, 2, 2, 1, false, 16, false>(a, st);
    return launch_prune_cfg<1024, 1, 4, 1, false, 16, false>(a, st);
  }
  if (a.K <= 2048) return launch_prune_cfg<2048, 4, 2, 1, false, 32, false>(a, st);
  return launch_prune_cfg<4096, 8, 2, 1, false, 32, false>(a, st);
}

// When a sequence is handed to the other engines.  Inputs whose bounds prune
// little (smooth position models, blocks of states, ties) make it read nearly
// every row for itself, where those engines share a row among the sequences
// of a cluster or of the GPU.  Measured (GB300, us per step of the launch):
//                  ordinary  ties  Gaussian band  all equal   other engine
//   K = 512,    64    2.8     4.1       7.3          8.1          4.1
//              152    3.0     5.0       9.2         11.3          7.7
//              400    8.0    14.6      28.3         35.4         15.2
//   K = 1000,   60    4.6    10.9      21.6         27.9         11.2
//              152    6.4    14.9      28.4         37.7         26.6
//   K = 1500,    4    4.7    11.9      20.0         30.0         11.2
//   K = 2048,    8    5.8    15.9      27.2         40.4         13.2
//   K = 4096,    8   11.8    37.3      55.0        100.6         20.1
// With the rule, us per step: K = 4096, 8 sequences of 600 steps, band 54 -> 22.6,
// all equal 99 -> 21.3 (the other engine alone 19.7); K = 1000, one of 1500,
// 18.4 -> 11.7 and 26.4 -> 10.8 (10.6); K = 512, 64 of 200, all equal 8.1 -> 4.8
// (4.1); 100 steps at K = 4096, all equal 91 -> 29: the shorter a sequence, the
// more of it is gone before the rule can tell.
// The constants are a line a + b rows through these (rows of the busiest
// warp) and the other engine's step; sequences have to lose 15%.  Where none
// is handed over the call pays launches that end at once (9 to 13 us), so it
// does without where that is more than a few percent of it: short calls, K
// <= 256 (all equal 16.9 against 13.6) and the few states where reading every
// row loses less than 30%.  Above K = 1024 the other engine waits for the whole
// GPU, so calls that share it do without too.
void prune_give(DenseArgs* a, int K, int jobs, int max_T, bool alone) {
  const int nsm = device_sm_count();
  a->give_a = a->give_b = 0.f;
  if (K <= 256 || max_T < (K <= 512 ? 128 : K <= 2048 ? 64 : 32) || (K > 1024 && !alone)) return;
  float ca, cb, there;
  if (K <= 512) {
    if (jobs <= 120) ca = 1.7f, cb = 0.0125f, there = 4.05f;
    else if (jobs <= nsm) ca = 1.7f, cb = 0.0185f, there = 7.7f;
    else ca = 1.2f, cb = 0.0225f, there = 5.8f;  // per 152 sequences
  } else if (K <= 1024) {
    if (2 * jobs <= nsm) ca = 1.5f, cb = 0.023f, there = 11.f;
    else ca = 2.5f, cb = 0.034f, there = 11.f + 15.6f * fminf(1.f, 2.f * (float)jobs / (float)nsm - 1.f);
  } else {
    // kWideLanes sequences at a time there, a cluster each here
    const int resident = K <= 2048 ? nsm / 4 - 2 : nsm / 8 - 4;
    const float turns = (float)((jobs + resident - 1) / resident);
    ca = (K <= 2048 ? 3.2f : 5.f) * turns;
    cb = (K <= 2048 ? 0.0175f : 5.25e-6f * (float)K) * turns;
    there = (5.5f + 0.0036f * (float)K) * (float)((jobs + kWideLanes - 1) / kWideLanes);
  }
  if (ca + cb * (float)K < 1.3f * there) return;
  a->give_a = ca / (1.15f * there);
  a->give_b = cb / (1.15f * there);
}

// States per segment of the trace: a few thousand segments over the launch,
// each several times the warm-up.
int prune_trace_seg(int64_t sum_T) {
  const int64_t s = (sum_T / 4096 + 15) / 16 * 16;
  return (int)(s < 48 ? 48 : s > 512 ? 512 : s);
}
// `unit`: table elements per step at least (the smallest K for delta rows,
// the beam table's row length)
size_t prune_guess_bytes(uint64_t aux_elems, int32_t n_seq, int64_t sum_T, int32_t unit) {
  const uint64_t per = (uint64_t)unit * (uint64_t)prune_trace_seg(sum_T);
  return sizeof(int32_t) * (size_t)(aux_elems / per + (uint64_t)n_seq + 1ull);
}

template <int VPL, int TW, bool BEAM, bool ROWS>
static cudaError_t launch_trace_cfg(TraceArgs t, int max_T, cudaStream_t st) {
  const dim3 grid(t.count, (max_T + t.seg - 1) / t.seg);
  if (grid.y == 1) t.seg = 0x7fffffff;  // one segment whatever the length on the device: no repair to launch
  prune_trace_kernel<VPL, TW, BEAM, ROWS><<<grid, 32 * TW, 0, st>>>(t);
  if (grid.y > 1) prune_fix_kernel<VPL, TW, BEAM, ROWS><<<t.count, 32 * TW, 0, st>>>(t);
  return cudaGetLastError();
}

template <bool BEAM>
static cudaError_t launch_trace(const TraceArgs& t, int n, int max_T, cudaStream_t st) {
  if (!BEAM && n <= 64) return launch_trace_cfg<2, 1, BEAM, true>(t, max_T, st);
  if (!BEAM && n <= 128) return launch_trace_cfg<4, 1, BEAM, true>(t, max_T, st);
  if (n <= 256) return launch_trace_cfg<8, 1, BEAM, false>(t, max_T, st);
  if (n <= 512) return launch_trace_cfg<16, 1, BEAM, false>(t, max_T, st);
  if (n <= 1024) return launch_trace_cfg<16, 2, BEAM, false>(t, max_T, st);
  if (n <= 2048) return launch_trace_cfg<16, 4, BEAM, false>(t, max_T, st);
  return launch_trace_cfg<16, 8, BEAM, false>(t, max_T, st);
}

cudaError_t launch_prune_trace(const DenseArgs& a, int32_t* guess, size_t guess_bytes, int64_t sum_T, int unit,
                               int max_T, int32_t* paths, cudaStream_t st) {
  if (a.order_count <= 0) return cudaSuccess;
  const bool beam = a.beam_B > 0;
  TraceArgs t;
  t.jobs = a.jobs;
  t.order = a.order;
  t.begin = a.order_begin;
  t.count = a.order_count;
  t.K = a.K;
  t.seg = prune_trace_seg(sum_T);
  // (grid.y is at most 65535)
  if (max_T / t.seg > 32768) t.seg = (max_T / 32768 + 1) * t.seg;
  t.row = a.beam_stride;
  t.unit = unit;
  t.ids = a.beam_id;
  t.D = beam ? a.beam_val : a.pr_D;
  t.AT = !beam && a.K <= 128 ? a.logA : a.wide_AT;
  t.qlast = a.qlast;
  t.paths = paths;
  t.guess = guess;
  t.guess_cap = (int64_t)(guess_bytes / sizeof(int32_t));
  t.hdr = a.hdr;
  return beam ? launch_trace<true>(t, a.beam_stride, max_T, st) : launch_trace<false>(t, a.K, max_T, st);
}

// Dynamic beams (P = 0) over the same step; `alone`: the call has the GPU to
// itself, so a launch may spread a sequence over more than one SM.
// Measured against fv_beam.cu, us per step of the whole call (GB300): K = 256,
// B = 64, 70 sequences 20.4 -> 2.9; K = 512, B = 128, 64 sequences 14.4 -> 4.8;
// K = 1024, B = 256, 40 sequences 27.7 -> 8.7, one sequence 8.7 -> 6.5.  At 1024
// < K <= 2048 a sequence takes a cluster of four CTAs (36 at a time; K = 2048,
// B = 256, one sequence 12.0 -> 10.2, 64 sequences 34.7 -> 21.8), so the launch
// is compared with one CTA per sequence on fv_beam.cu, whose step takes 3
// times as long or more; K = 4096 was no faster (one sequence 17.8 -> 21.5).
// Short calls stay there too, where the preparation of logA outweighs the
// steps: below 32 steps (48 from K = 1024) where fv_beam.cu would spread a
// sequence over a cluster (one sequence of 3 / 20 / 200 steps: K = 1024, B = 256,
// 51 / 185 / 1732 us there, 64 / 210 / 1390 here; K = 2048, B = 512, 72 / 302 / 2955
// against 103 / 362 / 1902), else below 8 (K = 1000, B = 16, 48 / 226 / 2135
// against 51 / 125 / 719).  Returns false where fv_beam.cu wins.
bool prune_beam_wins(int K, int64_t sum_T, int max_T, bool alone) {
  if (K >= 512 && max_T < (alone && K % 32 == 0 ? (K < 1024 ? 32 : 48) : 8)) return false;
  if (K <= 1024) return true;
  if (!alone || K > 2048) return false;
  const int64_t nsm = device_sm_count(), ncl = nsm / 4 - 2;
  const int64_t here = max_T > sum_T / ncl ? max_T : sum_T / ncl, there = max_T > sum_T / nsm ? max_T : sum_T / nsm;
  return here < 3 * there;
}

cudaError_t launch_prune_beam(const DenseArgs& a, bool alone, cudaStream_t st) {
  const int jobs = a.order_count, nsm = device_sm_count();
  if (jobs <= 0) return cudaSuccess;
  if (a.K <= 256) return launch_prune_cfg<256, 1, 1, 1, false, 6, true>(a, st);
  if (a.K <= 512) return launch_prune_cfg<512, 1, 2, 1, false, 12, true>(a, st);
  if (a.K <= 1024) {
    if (alone && 2 * jobs <= nsm) return launch_prune_cfg<1024, 2, 2, 1, false, 16, true>(a, st);
    return launch_prune_cfg<1024, 1, 4, 1, false, 16, true>(a, st);
  }
  return launch_prune_cfg<2048, 4, 2, 1, false, 32, true>(a, st);
}

}  // namespace fv
