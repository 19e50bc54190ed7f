// Calibration and selection of Sec. 3.4 - 3.7 (from s_bar to the index set I):
// one thread-block cluster of n = min(G, 8) CTAs per (sequence, layer).
//
// Phase 1, CTA r of the cluster works on groups g = r, r + n, ... (group r
// alone when G <= 8), one after the other:
//   (step path) AvgPool1D + group mean of the unpooled sums -> S[g, :] (Eqs.
//     3-4), four consecutive tokens per thread, the window's neighbours from
//     the adjacent lanes;
//   RankBin: the K equal-frequency bins of S[g, visual tokens] on
//     order-preserving keys, equal keys ordered by position: a 4096-bucket
//     histogram spread linearly over the row's key range gives every bucket's
//     first rank; a bucket whose ranks all lie in one bin sends its tokens
//     there, and the few tokens of the others are ranked pairwise by (key,
//     position).  Only when those hold more than 2048 tokens (many equal
//     scores) does an exact radix select over four 8-bit digits take over;
//   SpatialBin + joint histogram -> plug-in MI_g                        (Eq. 5);
//   phi_g = cos(current-frame row on the patch grid, m_g); m_g update    (Eq. 8).
// Phase 2, CTA r of the cluster works on tokens [r Lp / n, (r + 1) Lp / n):
//   MI EMA, min-max and softmax prior, lambda schedule                  (Eqs. 6-7);
//   s_bar, g*, Z = sum s_bar, the entropy H (Sec. 3.6) and x_t =
//     max(s_bar beta D, 0), with its bucket counted in the same pass: the
//     4096 buckets reach from a bound from the groups' largest S to below the
//     mean score (values outside fall into the end buckets), so no exchange of
//     the actual range is needed first;
//   global top-B with ties to the lower index (Sec. 3.7): every CTA sends its
//     128 coarse counts (32 buckets each) and its partial sums to its peers;
//     the coarse bucket that holds the B-th token is found on their sum, its
//     32 buckets are read from every peer, and the tokens of the bucket found
//     (at most 512) are sent to every peer and ranked pairwise by (key,
//     position).  Each CTA knows from the same counts how many tokens the
//     lower-ranked ones keep, so it writes its part of I without another
//     exchange.  A bucket with more tokens is split again over its own key
//     range until it fits or holds a single key (then ties are kept in
//     position order).
// Per-KV-head selection mode: in phase 2 CTA g works on its own row instead,
//   s_{g,t} = max(S[g,t] beta_g D_{g,t}, 0)^(1/T_g) with phi_g and the entropy of
//   S[g, .], and the same selection runs over that row alone.
//
// What a CTA tells its peers it writes into their shared memory before a
// cluster barrier, so that after the barrier every read but that of the 32
// buckets is local.
//
// What bounds it: latency.  A row's bytes (8 G per token) take microseconds at
// the memory rate; the time goes into some twenty phases between barriers.  A
// phase whose code a CTA runs once costs about 10 cycles per instruction
// (instruction fetch), so the token loops are kept small and not unrolled over
// tokens, scalar work is not repeated per boundary or bucket, and nothing that
// the loops use has its address taken (the refinement gets its view of the row
// by value: with closures over the kernel's variables every pass reloaded them
// from the stack, 40 thousand cycles against 14 in the pooling pass).
// Measured (events), one launch, 28 layers unless said: 14,000 tokens 47 -> 33 us
// (the kernel before: G CTAs of 1024 threads, a row's keys, cells and candidates
// on chip, whole histograms read from every peer), 56,096 tokens 213 -> 78, the
// same 14,000 with 28 groups 268 -> 140, 32 layers of 8 groups x 8,499 tokens
// 128 -> 40, 16 ragged sequences 917 -> 366, one layer of 568 tokens 32 -> 21.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"
#include "select.cuh"

namespace starkv {

namespace {

constexpr int kMaxTargets = 15;      // K - 1 with K <= 16
constexpr int kBuckets = 4096;       // buckets of the rank-bin and top-B histograms
constexpr int kFine = 32;            // buckets per coarse bucket (one per lane)
constexpr int kCoarse = kBuckets / kFine;
constexpr uint32_t kKeyMax = 0x7FFFFFFFu;   // largest descending key of a score
constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kPoolMax = kBuckets / 2;   // rank-bin candidates ranked pairwise ((key, position) pairs over the histogram)
constexpr int kCandMax = 512;        // top-B candidates ranked pairwise
// The top-B buckets span at least kTopOctaves octaves below a bound on the largest
// score, which holds all but a few scores of an ordinary row.  An attention sink lifts
// that bound far above all other scores; the span then goes on down to kMeanOctaves
// octaves below the mean score, w / L_p because softmax rows sum to 1: room for 99 %
// of the mass in the sink (7 octaves) and for beta and D.  Without that the B-th score
// falls into the last bucket with thousands of others, which takes a second
// histogram.  28 layers x 14,000 tokens with five tokens holding 90 to 99 %: 43 -> 39 us,
// as without a sink; 28 groups from 50 % on 147 -> 141, 56,000 tokens 86 -> 80.  A span wide
// enough for every row (28 octaves) makes ordinary rows 0.3 to 1 us slower, and the row's
// own smallest score costs another reduction (1 us).
constexpr int kTopOctaves = 14;
constexpr int kMeanOctaves = 10;
constexpr float kLn2 = 0.6931471805599453f;
constexpr size_t kSmemMax = 227 * 1024;
constexpr size_t kSmemTwo = 112 * 1024;   // two CTAs per SM

// Order-preserving map float -> uint32 (a < b  <=>  key(a) < key(b) for non-NaN).
__device__ __forceinline__ uint32_t order_key(float x) {
  const uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float order_value(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

// Descending key of a fused score x >= 0: a larger score has a smaller key.
__device__ __forceinline__ uint32_t desc_key(float x) { return kKeyMax - __float_as_uint(x); }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFullMask, v, o);
  return v;
}

// Sums of four values over the warp: lanes 8 k .. 8 k + 7 get value k's.
__device__ __forceinline__ float warp_sum4(float a, float b, float c, float d, int lane) {
  const bool hi = lane & 16, odd = lane & 8;
  float x = (hi ? c : a) + __shfl_xor_sync(kFullMask, hi ? a : c, 16);
  float y = (hi ? d : b) + __shfl_xor_sync(kFullMask, hi ? b : d, 16);
  x = (odd ? y : x) + __shfl_xor_sync(kFullMask, odd ? x : y, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(kFullMask, x, o);
  return x;
}

__device__ __forceinline__ int warp_incl_scan(int v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFullMask, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// One warp: the bin of a 256-bin histogram that holds rank `rank` (0-based)
// and the count of keys in lower bins; written by the lane that finds it.
__device__ void warp_find_256(const int* hist, int rank, int* digit, int* below) {
  const int lane = threadIdx.x & 31;
  const int4 q0 = reinterpret_cast<const int4*>(hist + lane * 8)[0];
  const int4 q1 = reinterpret_cast<const int4*>(hist + lane * 8)[1];
  const int v[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
  const int sum = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
  const int incl = warp_incl_scan(sum, lane);
  const int excl = incl - sum;
  if (rank >= excl && rank < incl) {
    int c = excl, d = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (d == i && rank >= c + v[i]) {
        c += v[i];
        d = i + 1;
      }
    *digit = lane * 8 + d;
    *below = c;
  }
}

struct CalShared {
  // ---- phase 1 (this CTA's current group)
  uint32_t kmin, kmax;             // key range of the MI span: the smallest key - 1 and the largest
  uint32_t smax;                   // the whole row's largest
  uint32_t slots;                  // boundary buckets so far: count in bits 24.., their tokens below
  int slot_off[kMaxTargets + 1];   // slot -> first entry of its candidates in the pool
  int slot_n[kMaxTargets + 1];     // slot -> tokens in its bucket
  int slot_rank[kMaxTargets + 1];  // slot -> rank of its bucket's first token
  int slot_cnt[kMaxTargets + 1];   // slot -> candidates placed so far
  int wsum[32];
  float red[4][32];
  // exact radix refinement (many equal scores)
  uint32_t prefix[kMaxTargets];    // boundary keys, built digit by digit
  int rem[kMaxTargets];            // rank of the boundary among the keys sharing its prefix
  int slot_of[kMaxTargets];        // boundary -> its slot, -1 when no bucket needs it
  int dig[kMaxTargets], below[kMaxTargets];
  int eqw[32][kMaxTargets];        // keys equal to each boundary before each warp's segment
  // ---- written by every CTA of the cluster
  float mi[kMaxGroups], phi[kMaxGroups];
  uint32_t gmax[kMaxGroups];
  float pz[kMaxCluster], pzl[kMaxCluster], pv[kMaxCluster];
  uint32_t psmax[kMaxCluster];
  uint32_t rlo[kMaxCluster], rhi[kMaxCluster];
  int4 coarse[kMaxCluster][kCoarse / 4];
  // ---- phase 2
  double mib_old[kMaxGroups];      // MI EMA before this step, per group
  float mib[kMaxGroups], w[kMaxGroups];
  float lam;
  int n_old;
  uint32_t blo;                    // first bucket's key and the bucket scale of the selection
  float bscale;
  uint32_t lo, hi;                 // key range of the bucket being split
  int ccnt;                        // candidates this CTA has sent
  int lowcnt;                      // kept candidates of the lower-ranked CTAs
  int segb[32], sege[32];          // per warp segment: tokens below, kept candidates or equal keys
  uint32_t tkey;
  int tpos;
};

constexpr size_t align16(size_t x) { return (x + 15) & ~size_t(15); }
constexpr size_t kCalSharedBytes = align16(sizeof(CalShared));
constexpr int kBucketTable = kBuckets;   // bytes: rank bin of each bucket, or 0x80 | slot
constexpr int kCandBytes = kCandMax * 8;

constexpr size_t fixed_bytes(int joint_cells, int patches) {   // K M^2, R C
  return kCalSharedBytes + static_cast<size_t>(kBuckets) * 4 + kCandBytes + align16(static_cast<size_t>(joint_cells) * 4) +
         align16(static_cast<size_t>(patches) * 4) + kBucketTable;
}
// Two CTAs without a row on chip fit an SM whatever the configuration (228 KB, of
// which each takes 1 KB more): the two-per-SM variant never runs alone.
static_assert(fixed_bytes(kMaxHist, kMaxGrid) + 1024 <= 114 * 1024, "two CTAs fit");

constexpr size_t kBytesPerToken = 4;   // a row's keys, then the CTA's fused scores

}  // namespace

// One group's row as the rank-bin passes read it.  Passed by value to the
// out-of-line refinement, so that no pass reads it back from the stack.
struct Row {
  const uint32_t* keys;   // on chip, or NULL: from S and the metadata
  const float* S;
  const uint32_t* meta;
  int Lp, R, C, M, cur_frame, mi_span;
  uint32_t inv_R, inv_C;
  uint32_t kmin;          // key range of the MI span and the bucket scale over it
  float binv;
  // key of a token of the MI span, else 0 (Sec. 3.4: the historical visual
  // tokens, or the newest frame's with mi_span 1)
  __device__ __forceinline__ uint32_t span_key(float s, uint32_t mt) const {
    const bool on = meta_visual(mt) && meta_row(mt) < R && meta_col(mt) < C &&
                    (mi_span == 0 || meta_frame(mt) == cur_frame);
    return on ? max(order_key(s), 1u) : 0u;
  }
  // SpatialBin: (floor(r M / R), floor(c M / C)), the quotients by multiplication
  __device__ __forceinline__ int cell(uint32_t mt) const {
    return static_cast<int>(__umulhi(meta_row(mt) * M, inv_R) * M + __umulhi(meta_col(mt) * M, inv_C));
  }
  __device__ __forceinline__ int bucket(uint32_t u) const {
    return min(kBuckets - 1, static_cast<int>(static_cast<float>(u - kmin) * binv));
  }
  __device__ __forceinline__ uint32_t key(int t) const { return keys ? keys[t] : span_key(S[t], meta[t]); }
};

// Exact rank bins of the boundary-bucket tokens by a radix select (four 8-bit
// digits) for every boundary at once, equal keys ordered by position; for rows
// whose boundary buckets hold too many tokens to rank pairwise.  Adds those
// tokens to the joint histogram.  Each warp walks its own contiguous segment,
// so that warp and lane order are position order.
template <int NT>
__device__ __noinline__ void refine_radix(CalShared& sh, int* hist, int* joint, const uint8_t* btab, int N, int K, Row row) {
  constexpr int NW = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = K - 1, MM = row.M * row.M;
  const int nslot = static_cast<int>(sh.slots >> 24);
  const int seg = ceil_div(row.Lp, NW * 32) * 32;
  const int s0 = min(row.Lp, warp * seg), s1 = min(row.Lp, s0 + seg);
  const unsigned lanes_below = (1u << lane) - 1u;
  if (tid < nt) {
    // boundary b = tid + 1 starts at rank ceil(b N / K); the slot that holds it, if any
    const int rb = static_cast<int>((static_cast<int64_t>(tid + 1) * N + K - 1) / K);
    int so = -1;
    for (int s = 0; s < nslot; ++s)
      if (rb > sh.slot_rank[s] && rb < sh.slot_rank[s] + sh.slot_n[s]) so = s;
    sh.slot_of[tid] = so;
    sh.rem[tid] = so >= 0 ? rb - sh.slot_rank[so] : 0;
    sh.prefix[tid] = 0;
  }
  __syncthreads();
  auto slot_key = [&](int t, uint32_t& u) {   // the token's slot, or -1
    u = row.key(t);
    if (u == 0u) return -1;
    const int v = btab[row.bucket(u)];
    return (v & 0x80) ? (v & 0x7F) : -1;
  };
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    const uint32_t hmask = pass == 0 ? 0u : (0xFFFFFFFFu << (shift + 8));
    for (int i = tid; i < nt * 256; i += NT) hist[i] = 0;
    __syncthreads();
    for (int t = s0 + lane; t < s1; t += 32) {
      uint32_t u;
      const int sl = slot_key(t, u);
      if (sl < 0) continue;
      for (int j = 0; j < nt; ++j)
        if (sh.slot_of[j] == sl && ((u ^ sh.prefix[j]) & hmask) == 0) atomicAdd(&hist[j * 256 + ((u >> shift) & 255)], 1);
    }
    __syncthreads();
    for (int j = warp; j < nt; j += NW)
      if (sh.slot_of[j] >= 0) warp_find_256(hist + j * 256, sh.rem[j], &sh.dig[j], &sh.below[j]);
    __syncthreads();
    if (tid < nt && sh.slot_of[tid] >= 0) {
      sh.prefix[tid] |= static_cast<uint32_t>(sh.dig[tid]) << shift;
      sh.rem[tid] -= sh.below[tid];
    }
    __syncthreads();
  }
  // equal keys before each warp's segment, per boundary
  for (int j = 0; j < nt; ++j) {
    int cnt = 0;
    if (sh.slot_of[j] >= 0)
      for (int t = s0 + lane; t < s1; t += 32) cnt += row.key(t) == sh.prefix[j];
    cnt = warp_sum(cnt);
    if (lane == 0) sh.eqw[warp][j] = cnt;
  }
  __syncthreads();
  if (tid < nt) {
    int run = 0;
    for (int w = 0; w < NW; ++w) {
      const int c = sh.eqw[w][tid];
      sh.eqw[w][tid] = run;
      run += c;
    }
  }
  __syncthreads();
  int eqrun[kMaxTargets];
#pragma unroll
  for (int j = 0; j < kMaxTargets; ++j) eqrun[j] = j < nt ? sh.eqw[warp][j] : 0;
  for (int base = s0; base < s1; base += 32) {
    const int t = base + lane;
    uint32_t u = 0;
    const int sl = t < s1 ? slot_key(t, u) : -1;
    int bin = 0;
    if (sl >= 0)   // boundaries at or below the bucket's first token
      bin = static_cast<int>(static_cast<uint32_t>(sh.slot_rank[sl]) * static_cast<uint32_t>(K) / static_cast<uint32_t>(N));
#pragma unroll
    for (int j = 0; j < kMaxTargets; ++j) {
      if (j >= nt) break;
      const uint32_t P = sh.prefix[j];
      const bool mine = sl >= 0 && sh.slot_of[j] == sl;
      const unsigned m = __ballot_sync(kFullMask, mine && u == P);
      if (mine) {
        if (u > P) ++bin;
        else if (u == P && eqrun[j] + __popc(m & lanes_below) >= sh.rem[j]) ++bin;
      }
      eqrun[j] += __popc(m);
    }
    if (sl >= 0) atomicAdd(&joint[bin * MM + row.cell(row.meta[t])], 1);
  }
}

// NT threads: 1024 (one CTA per SM) or 512 (two), 64 registers a thread either way.
template <bool FROM_RAW, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_calibrate(const __grid_constant__ SeqBatch b,
                                                             const __grid_constant__ KParams kp, DevState st,
                                                             int capl) {
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  CalShared& sh = *reinterpret_cast<CalShared*>(smem_raw);
  const int G = kp.G, K = kp.K, M = kp.M, R = kp.R, C = kp.C, MM = M * M, RC = R * C;
  int* hist = reinterpret_cast<int*>(smem_raw + kCalSharedBytes);
  uint2* clist = reinterpret_cast<uint2*>(hist + kBuckets);   // top-B candidates of the whole selection
  int* joint = reinterpret_cast<int*>(clist + kCandMax);
  float* cur = reinterpret_cast<float*>(joint + ((K * MM + 3) & ~3));
  uint8_t* btab = reinterpret_cast<uint8_t*>(cur + ((RC + 3) & ~3));
  uint32_t* keys = reinterpret_cast<uint32_t*>(btab + kBucketTable);   // [capl]

  const SeqView& sv = b.s[blockIdx.z];
  const int rank = blockIdx.x, ncta = gridDim.x;   // the cluster spans grid x
  const int ll = blockIdx.y, layer = b.layer0 + ll;
  const int Lp = sv.Lp;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sl = sv.slot * kp.n_layers + layer;
  const bool in_smem = Lp <= capl;
  // metadata row of group gi (the one shared row when meta_group_stride is 0)
  auto meta_of = [&](int gi) {
    return sv.meta + static_cast<int64_t>(layer) * sv.meta_layer_stride + gi * sv.meta_group_stride;
  };

  // block-wide counters, histograms and the current-frame row of the next group
  auto reset = [&]() {
    if (tid == 0) {
      sh.kmin = 0xFFFFFFFFu;
      sh.kmax = 0u;
      sh.smax = 0u;
      sh.slots = 0u;
    }
    if (tid <= kMaxTargets) sh.slot_cnt[tid] = 0;
    for (int i = tid; i < kBuckets / 4; i += NT) reinterpret_cast<int4*>(hist)[i] = make_int4(0, 0, 0, 0);
    for (int i = tid; i < (K * MM + 3) / 4; i += NT) reinterpret_cast<int4*>(joint)[i] = make_int4(0, 0, 0, 0);
    for (int i = tid; i < (RC + 3) / 4; i += NT) reinterpret_cast<float4*>(cur)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  };
  cluster_arrive();   // waited for before the first write into a peer's shared memory
  reset();
  // this CTA's groups' temporal EMA rows (state of the previous step, read
  // after phase 1) on their way into L2
  for (int gi = rank; gi < G; gi += ncta)
    for (int i = tid * 32; i < RC; i += NT * 32) prefetch_l2(st.m + static_cast<int64_t>(sl * G + gi) * RC + i);
  __syncthreads();
  // the set-up above overlaps the previous kernel's tail; its outputs are read below
  griddep_launch_dependents();
  griddep_wait();
  if (tid < G) sh.mib_old[tid] = st.mi_bar[sl * G + tid];
  if (tid == NT - 1) {   // step counter and lambda schedule
    const int n = st.n[sl];
    sh.n_old = n;
    float lam = 0.f;
    if (n >= kp.n_warmup)
      lam = kp.n_ramp <= 0 ? kp.lambda
                           : kp.lambda * fminf(1.f, static_cast<float>(n - kp.n_warmup) / kp.n_ramp);
    sh.lam = lam;
  }

  // the four block-wide sums of sh.red, in every warp
  auto sum4 = [&](float& a, float& b, float& c, float& d) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < NW; w += 8) v += sh.red[lane >> 3][w + (lane & 7)];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(kFullMask, v, o);
    a = __shfl_sync(kFullMask, v, 0);
    b = __shfl_sync(kFullMask, v, 8);
    c = __shfl_sync(kFullMask, v, 16);
    d = __shfl_sync(kFullMask, v, 24);
  };

  // ================= phase 1: groups rank, rank + ncta, ... =================
  const float pscale = static_cast<float>(G) / static_cast<float>(kp.H) / static_cast<float>(kp.pool);
  const int half = kp.pool >> 1;
  float* mrow = nullptr;   // the last group's m_g row and its update (0 none, 1 EMA, 2 first row),
  int mupd = 0;            // done while the phase-1 cluster barrier settles
  auto update_m = [&]() {
    const float rt = kp.rho_t;
    if (mupd == 0) return;
    for (int i0 = tid; i0 < RC; i0 += 4 * NT) {
      float old[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) old[k] = mupd == 1 && i0 + k * NT < RC ? mrow[i0 + k * NT] : 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = i0 + k * NT;
        if (i < RC) mrow[i] = mupd == 1 ? rt * old[k] + (1.f - rt) * cur[i] : cur[i];
      }
    }
  };
  for (int g = rank; g < G; g += ncta) {
    const uint32_t* meta = meta_of(g);
    float* S = sv.S + (static_cast<int64_t>(layer) * G + g) * Lp;
    const float* raw = FROM_RAW ? sv.s_raw + static_cast<int64_t>(ll * G + g) * raw_stride(Lp) : nullptr;
    // a pooling window wider than the neighbouring vectors: S first, from the
    // row staged in the key array when it fits
    const bool wide = FROM_RAW && half > 4;
    if (wide) {
      float* stage = reinterpret_cast<float*>(keys);
      if (in_smem) {
        for (int t = tid; t < Lp; t += NT) stage[t] = raw[t];
        __syncthreads();
      }
      for (int t = tid; t < Lp; t += NT) {
        float acc = 0.f;
        for (int u = max(0, t - half); u <= min(Lp - 1, t + half); ++u) acc += in_smem ? stage[u] : raw[u];
        S[t] = acc * pscale;
      }
      __syncthreads();
    }
    // ---- the row: pooling (Eqs. 3-4), the MI span's keys and their range,
    // the current frame on the patch grid.  Four consecutive tokens (a vector)
    // per lane; the window's neighbours come from the adjacent lanes, so that a
    // warp's first and last lane only carry theirs.  The next pass's loads are
    // in flight under this one's arithmetic (addresses clamped to the row
    // instead of guarded, so that nothing waits for them before).
    const bool pool_here = FROM_RAW && !wide;
    const int hw = pool_here ? 1 : 0, span = 32 - 2 * hw;   // vectors a warp works on per pass
    const float* src = pool_here ? raw : S;
    const bool src16 = (reinterpret_cast<uintptr_t>(src) & 15) == 0, s16 = (reinterpret_cast<uintptr_t>(S) & 15) == 0;
    const bool m16 = (reinterpret_cast<uintptr_t>(meta) & 15) == 0;
    const int nvec = (Lp + 3) >> 2;
    // fields of a metadata word compared in place
    const uint32_t row_end = static_cast<uint32_t>(R) << 10, frame_now = static_cast<uint32_t>(sv.cur_frame) << 20;
    const bool all_frames = kp.mi_span == 0;
    uint32_t kmn = 0xFFFFFFFFu, kmx = 0u;
    float smx = -3.4e38f;
    bool bad = false;   // a visual token outside the patch grid
    int v = warp * span + lane - hw;
    float4 s_next = make_float4(0.f, 0.f, 0.f, 0.f);
    uint4 m_next = make_uint4(0u, 0u, 0u, 0u);
    auto load = [&](int v) {
      const int t0 = 4 * max(0, min(nvec - 1, v));
      const bool whole = t0 + 3 < Lp;
      const int t1 = min(t0 + 1, Lp - 1), t2 = min(t0 + 2, Lp - 1), t3 = min(t0 + 3, Lp - 1);
      if (m16 && whole) m_next = *reinterpret_cast<const uint4*>(meta + t0);
      else m_next = make_uint4(meta[t0], meta[t1], meta[t2], meta[t3]);
      if (src16 && whole) s_next = *reinterpret_cast<const float4*>(src + t0);
      else s_next = make_float4(src[t0], src[t1], src[t2], src[t3]);
    };
    if (Lp > 0) load(v);
#pragma unroll 1
    for (int base = warp * span; base < nvec; base += NW * span) {
      float x[4] = {s_next.x, s_next.y, s_next.z, s_next.w};
      uint32_t mw[4] = {m_next.x, m_next.y, m_next.z, m_next.w};
      const int t0 = 4 * v;
      load(v + NW * span);
      // past the row's ends: zeros, and no visual token
      if (static_cast<uint32_t>(t0) + 3u >= static_cast<uint32_t>(Lp)) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (static_cast<uint32_t>(t0 + i) >= static_cast<uint32_t>(Lp)) {
            x[i] = 0.f;
            mw[i] = 0u;
          }
      }
      if (pool_here) {
        float o[4];
        if (half == 2) {   // the default window
          const float l2 = __shfl_up_sync(kFullMask, x[2], 1), l1 = __shfl_up_sync(kFullMask, x[3], 1);
          const float r1 = __shfl_down_sync(kFullMask, x[0], 1), r2 = __shfl_down_sync(kFullMask, x[1], 1);
          o[0] = (((l2 + l1) + x[0]) + x[1]) + x[2];
          o[1] = (((l1 + x[0]) + x[1]) + x[2]) + x[3];
          o[2] = (((x[0] + x[1]) + x[2]) + x[3]) + r1;
          o[3] = (((x[1] + x[2]) + x[3]) + r1) + r2;
        } else {   // up to four neighbours on each side, in tap order
          float y[12];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            y[i] = __shfl_up_sync(kFullMask, x[i], 1);
            y[4 + i] = x[i];
            y[8 + i] = __shfl_down_sync(kFullMask, x[i], 1);
            o[i] = 0.f;
          }
#pragma unroll
          for (int j = -4; j <= 4; ++j)
            if (j >= -half && j <= half)
#pragma unroll
              for (int i = 0; i < 4; ++i) o[i] += y[4 + i + j];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = o[i] * pscale;
      }
      if (lane >= hw && lane < 32 - hw && v < nvec) {
        if (pool_here) {
          if (s16 && t0 + 3 < Lp) {
            *reinterpret_cast<float4*>(S + t0) = make_float4(x[0], x[1], x[2], x[3]);
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (t0 + i < Lp) S[t0 + i] = x[i];
          }
        }
        // selects instead of branches: one rarely divergent branch per vector,
        // for the current frame's tokens
        uint32_t key[4];
        bool newest[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const bool vis = meta_visual(mw[i]);
          const bool in = vis && (mw[i] & 0xFFC00u) < row_end && (mw[i] & 0x3FFu) < static_cast<uint32_t>(C);
          bad |= vis && !in;
          newest[i] = in && (mw[i] & 0x7FF00000u) == frame_now;
          const bool on = all_frames ? in : newest[i];
          smx = fmaxf(smx, x[i]);
          // (the unpooled sums are sums of exponentials, so not negative)
          const uint32_t ok = pool_here ? __float_as_uint(x[i]) | 0x80000000u : max(order_key(x[i]), 1u);
          key[i] = on ? ok : 0u;
          kmn = min(kmn, key[i] - 1u);
          kmx = max(kmx, key[i]);
        }
        if (newest[0] || newest[1] || newest[2] || newest[3]) {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (newest[i]) atomicAdd(&cur[meta_row(mw[i]) * C + meta_col(mw[i])], x[i]);
        }
        if (in_smem) reinterpret_cast<uint4*>(keys)[v] = make_uint4(key[0], key[1], key[2], key[3]);
      }
      v += NW * span;
    }
    if (bad) atomicOr(st.err, kErrMeta);
    kmn = __reduce_min_sync(kFullMask, kmn);   // (the smallest key - 1)
    kmx = __reduce_max_sync(kFullMask, kmx);
    const uint32_t rmx = __reduce_max_sync(kFullMask, order_key(smx));
    if (lane == 0) {
      atomicMin(&sh.kmin, kmn);
      atomicMax(&sh.kmax, kmx);
      atomicMax(&sh.smax, rmx);
    }
    __syncthreads();
    const bool some = sh.kmax != 0u;   // the MI span holds a token
    // Sec. 3.4 RankBin: 4096 buckets spread linearly over the span's key range
    // (monotone in the key, so bucket order is key order)
    const Row row = {in_smem ? keys : nullptr, S, meta, Lp, R, C, M, sv.cur_frame, kp.mi_span, kp.inv_R, kp.inv_C,
                     sh.kmin + 1u, 4096.f / (static_cast<float>(sh.kmax - (sh.kmin + 1u)) + 1.f)};
    // every token of the MI span: f(token, key, metadata word).  A row that is
    // not on chip is read again from S, four tokens' loads at a time.
    auto each_span = [&](auto with_meta, auto&& f) {
      constexpr bool kMeta = decltype(with_meta)::value;
      if (in_smem) {
        uint32_t ma = kMeta && tid < Lp ? meta[tid] : 0u, mb = kMeta && tid + NT < Lp ? meta[tid + NT] : 0u;
#pragma unroll 1
        for (int t = tid; t < Lp; t += NT) {
          const uint32_t mc = kMeta && t + 2 * NT < Lp ? meta[t + 2 * NT] : 0u;   // two passes ahead
          const uint32_t key = keys[t];
          if (key != 0u) f(t, key, ma);
          ma = mb;
          mb = mc;
        }
      } else {
        for (int t0 = tid; t0 < Lp; t0 += 4 * NT) {
          float s[4];
          uint32_t m[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int t = t0 + k * NT;
            m[k] = t < Lp ? meta[t] : 0u;
            s[k] = t < Lp ? S[t] : 0.f;
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t key = row.span_key(s[k], m[k]);
            if (key != 0u) f(t0 + k * NT, key, m[k]);
          }
        }
      }
    };
    if (some) each_span(std::false_type(), [&](int, uint32_t u, uint32_t) { atomicAdd(&hist[row.bucket(u)], 1); });
    // ---- Sec. 3.5: the sums of phi_g = cos(current row, m_g)
    mrow = st.m + static_cast<int64_t>(sl * G + g) * RC;
    float dot = 0.f, ncur = 0.f, nm = 0.f;
    for (int i0 = tid; i0 < RC; i0 += 4 * NT) {
      float bm[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) bm[k] = i0 + k * NT < RC ? mrow[i0 + k * NT] : 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float a = i0 + k * NT < RC ? cur[i0 + k * NT] : 0.f;
        dot = fmaf(a, bm[k], dot);
        ncur = fmaf(a, a, ncur);
        nm = fmaf(bm[k], bm[k], nm);
      }
    }
    __syncthreads();
    float acc = 0.f;   // this thread's part of N MI_g
    int N = 0;
    if (some) {
      // ---- bucket table: the first rank of every bucket by a scan, then the
      // bin floor(rank K / N) of its first and last token.  One bin: every
      // token goes there.  Otherwise the bucket gets a slot and its tokens are
      // ranked among themselves.
      constexpr int kPer = kBuckets / NT;
      int h[kPer];
      int sum = 0;
      {
#pragma unroll
        for (int k = 0; k < kPer; k += 4) {
          const int4 q = reinterpret_cast<const int4*>(hist)[(tid * kPer + k) >> 2];
          h[k] = q.x;
          h[k + 1] = q.y;
          h[k + 2] = q.z;
          h[k + 3] = q.w;
          sum += (q.x + q.y) + (q.z + q.w);
        }
      }
      const int incl = warp_incl_scan(sum, lane);
      if (lane == 31) sh.wsum[warp] = incl;
      __syncthreads();
      const int wincl = warp_incl_scan(lane < NW ? sh.wsum[lane] : 0, lane);
      N = __shfl_sync(kFullMask, wincl, 31);
      int first = (warp ? __shfl_sync(kFullMask, wincl, warp - 1) : 0) + incl - sum;
      const float fN = static_cast<float>(N), kn = static_cast<float>(K) / fN;
      auto bin_of = [&](int r) {   // floor(r K / N): an estimate good to one, corrected in integers (r K < 2^28)
        int q = static_cast<int>(static_cast<float>(r) * kn);
        const int rk = r * K;
        q += (q + 1) * N <= rk;
        q -= q * N > rk;
        return q;
      };
      {
        uint32_t packed[kPer / 4];
        const int b0 = sum > 0 ? bin_of(first) : 0;
        if (sum == 0 || bin_of(first + sum - 1) == b0) {
#pragma unroll
          for (int k = 0; k < kPer / 4; ++k) packed[k] = static_cast<uint32_t>(b0) * 0x01010101u;
        } else {
#pragma unroll
          for (int k = 0; k < kPer / 4; ++k) packed[k] = 0u;
#pragma unroll
          for (int k = 0; k < kPer; ++k) {
            if (h[k] == 0) continue;
            uint32_t v = static_cast<uint32_t>(bin_of(first));
            if (bin_of(first + h[k] - 1) != static_cast<int>(v)) {
              const uint32_t a = atomicAdd(&sh.slots, (1u << 24) + static_cast<uint32_t>(h[k]));
              const int slot = static_cast<int>(a >> 24);   // at most K - 1 buckets hold a boundary
              sh.slot_off[slot] = static_cast<int>(a & 0xFFFFFFu);
              sh.slot_n[slot] = h[k];
              sh.slot_rank[slot] = first;
              v = 0x80u | static_cast<uint32_t>(slot);
            }
            packed[k >> 2] |= v << (8 * (k & 3));
            first += h[k];
          }
        }
#pragma unroll
        for (int k = 0; k < kPer / 4; ++k) reinterpret_cast<uint32_t*>(btab)[tid * (kPer / 4) + k] = packed[k];
      }
      __syncthreads();
      const int ncand = static_cast<int>(sh.slots & 0xFFFFFFu), nslot = static_cast<int>(sh.slots >> 24);
      const bool brute = ncand <= kPoolMax;
      // ---- joint histogram of the settled tokens; boundary-bucket tokens go
      // to their slot's (key, position) pool, over the histogram
      uint2* pool = reinterpret_cast<uint2*>(hist);
      each_span(std::true_type(), [&](int t, uint32_t u, uint32_t mt) {
        const int v = btab[row.bucket(u)];
        if (!(v & 0x80)) {
          atomicAdd(&joint[v * MM + row.cell(mt)], 1);
        } else if (brute) {
          const int s = v & 0x7F;
          pool[sh.slot_off[s] + atomicAdd(&sh.slot_cnt[s], 1)] = make_uint2(u, static_cast<uint32_t>(t));
        }
      });
      __syncthreads();
      if (brute) {
        // exact rank of each candidate inside its bucket by (key, position)
        for (int i = tid; i < ncand; i += NT) {
          int s = 0;
          while (s + 1 < nslot && sh.slot_off[s + 1] <= i) ++s;
          const uint2 me = pool[i];
          const uint32_t mt = meta[me.y];
          const int o = sh.slot_off[s], n = sh.slot_n[s];
          int r = sh.slot_rank[s];
          for (int j = o; j < o + n; ++j) {
            const uint2 p = pool[j];
            r += (p.x < me.x) || (p.x == me.x && p.y < me.y);
          }
          atomicAdd(&joint[bin_of(r) * MM + row.cell(mt)], 1);
        }
      } else {
        refine_radix<NT>(sh, hist, joint, btab, N, K, row);
      }
      __syncthreads();
      // ---- Eq. (5): plug-in MI (nats) from the joint histogram: a cell per
      // warp and pass, a bin per lane; bin b holds the ranks from ceil(b N / K)
      // to before ceil((b + 1) N / K)
      const uint32_t r0 = __umulhi(lane * N + K - 1, kp.inv_K), r1 = __umulhi((lane + 1) * N + K - 1, kp.inv_K);
      const float fb = static_cast<float>(r1 - r0);
#pragma unroll 1
      for (int c = warp; c < MM; c += NW) {
        const int n = lane < K ? joint[lane * MM + c] : 0;
        const float fn = static_cast<float>(n), fc = static_cast<float>(__reduce_add_sync(kFullMask, n));
        if (n > 0) acc += fn * logf(fn * fN / (fb * fc));
      }
    }
    // ---- MI_g and phi_g: one reduction of the four sums
    const float p4 = warp_sum4(acc, dot, ncur, nm, lane);
    if ((lane & 7) == 0) sh.red[lane >> 3][warp] = p4;
    __syncthreads();
    sum4(acc, dot, ncur, nm);
    const float mi = N > 0 ? acc / static_cast<float>(N) : 0.f;
    float phi = 0.f;
    mupd = 0;
    if (ncur > 0.f) {
      mupd = nm > 0.f ? 1 : 2;
      if (nm > 0.f) phi = dot / (sqrtf(ncur) * sqrtf(nm));
    }
    if (g == rank) cluster_wait();   // every CTA of the cluster runs: its shared memory may be written
    if (warp == 0 && lane < ncta) {
      dsmem_st_u32(dsmem_map(&sh.mi[g], lane), __float_as_uint(mi));
      dsmem_st_u32(dsmem_map(&sh.phi[g], lane), __float_as_uint(phi));
      dsmem_st_u32(dsmem_map(&sh.gmax[g], lane), sh.smax);
    }
    if (g + ncta < G) {   // the next group of this CTA starts from clean arrays
      update_m();
      __syncthreads();
      reset();
      __syncthreads();
    }
  }
  // every group's S row, MI_g and phi_g are written: the peers may read them
  // once the barrier completes; the last group's m_g (read by no peer) and the
  // top-B histogram's zeroing go in between
  cluster_arrive();
  update_m();
  for (int i = tid; i < kBuckets / 4; i += NT) reinterpret_cast<int4*>(hist)[i] = make_int4(0, 0, 0, 0);
  cluster_wait();

  // ================= phase 2 =================
  // global mode: CTA r scores and selects tokens [r Lp / ncta, (r + 1) Lp / ncta)
  // of s_bar; per-KV-head mode (one CTA per group): CTA g its own row S[g, .]
  const bool per_head = kp.per_head != 0;
  const int B = sv.budget;   // the same in every CTA of the cluster
  const uint32_t* meta = meta_of(per_head ? rank : 0);
  // (range boundaries on multiples of 4 tokens)
  auto split = [&](int r) {
    const int64_t t = (static_cast<int64_t>(r) * Lp / ncta + 3) & ~static_cast<int64_t>(3);
    return static_cast<int>(t < Lp ? t : Lp);
  };
  const int ta = per_head ? 0 : split(rank);
  const int nr = per_head ? Lp : split(rank + 1) - ta;
  // a token's S in every group (per-KV-head mode: in this CTA's) and its
  // metadata word; consecutive tokens on consecutive lanes
  const int g_lo = per_head ? rank : 0, g_n = per_head ? 1 : G;
  const float* S0 = sv.S + (static_cast<int64_t>(layer) * G + g_lo) * Lp + ta;
  const float g_scale = 1.f / static_cast<float>(g_n);
  struct Token {
    float q[4];   // S of the first four groups (more are read when the token is combined)
    uint32_t mt;
  };
  auto load_token = [&](int i) {   // (the address is clamped, so that nothing waits for a guard)
    Token k;
    const int ic = min(i, nr - 1);
    k.mt = meta[ta + ic];
#pragma unroll
    for (int j = 0; j < 4; ++j) k.q[j] = j < g_n ? S0[static_cast<int64_t>(j) * Lp + ic] : 0.f;
    return k;
  };
  Token cur_tok = {};
  if (tid < nr) cur_tok = load_token(tid);   // in flight under the prior
  // ---- Eqs. (6)-(7): MI EMA (double state), min-max, softmax prior; lambda
  // schedule.  The same arithmetic in every CTA; CTA 0 stores the new state.
  // warp 0, lane gg < G: group gg's MI and its EMA, then the min-max and the
  // softmax over the groups by warp reductions; last, the bucket range of the
  // selection: below a bound on x_t from the largest S and the largest factor
  static_assert(kMaxGroups <= 32, "one lane per group");
  if (warp == 0) {
    const int n = sh.n_old;
    const float mean = __fdividef(static_cast<float>(kp.w), static_cast<float>(Lp));   // of the scores, before beta and D
    const bool on = lane < G;
    float mf = 0.f;
    if (on) {
      const double mic = static_cast<double>(sh.mi[lane]);
      const double mib = n == 0 ? mic : kp.rho_mi * sh.mib_old[lane] + (1.0 - kp.rho_mi) * mic;
      mf = static_cast<float>(mib);
      sh.mib[lane] = mf;
      if (rank == 0) st.mi_bar[sl * G + lane] = mib;
    }
    const uint32_t ko = order_key(mf);
    const float lo = order_value(__reduce_min_sync(kFullMask, on ? ko : 0xFFFFFFFFu));
    const float hi = order_value(__reduce_max_sync(kFullMask, on ? ko : 0u));
    const float inv = 1.f / (((hi - lo) + kp.eps) * kp.tau);
    const float zmax = (hi - lo) * inv;   // the largest exponent (its lane's own expression)
    const float ex = on ? expf((mf - lo) * inv - zmax) : 0.f;
    if (on) sh.w[lane] = ex;
    const float exs = warp_sum(ex);
    if (on) sh.w[lane] = ex / exs;
    const bool mine = per_head ? lane == rank : on;
    const float shi = order_value(__reduce_max_sync(kFullMask, mine ? sh.gmax[lane] : 0u));
    if (lane == 0) {
      const float lam = sh.lam;
      // (values outside the span fall into the end buckets)
      float xhi = shi * ((1.f - lam) + lam * static_cast<float>(G));
      float xlo = fminf(xhi * (1.f / (1 << kTopOctaves)), mean * (1.f / (1 << kMeanOctaves)));
      if (!(xlo > 0.f && xhi < 3.0e38f)) {   // unusual scores: the whole range
        xlo = 0.f;
        xhi = 3.0e38f;
      }
      sh.blo = desc_key(xhi);
      sh.bscale = 4096.f / (static_cast<float>(__float_as_uint(xhi) - __float_as_uint(xlo)) + 1.f);
      sh.ccnt = 0;
      sh.lowcnt = 0;
      if (rank == 0) st.n[sl] = n + 1;
    }
  } else if (warp == 1) {
    sh.segb[lane] = sh.sege[lane] = 0;
  }
  __syncthreads();   // w, lambda and the buckets are read by every thread below
  float* score = sv.score + (static_cast<int64_t>(layer) * (per_head ? G : 1) + (per_head ? rank : 0)) * Lp + ta;
  // x_t of the range: on chip, or (a long row of the per-KV-head mode) in the
  // score row until the selection is done
  float* xs = nr <= capl ? reinterpret_cast<float*>(keys) : score;
  const float lam = sh.lam;
  uint32_t blo = sh.blo;
  float bscale = sh.bscale;
  auto sbucket = [&](uint32_t u) {   // monotone in the key
    const int bk = __float2int_rz(static_cast<float>(static_cast<int>(u) - static_cast<int>(blo)) * bscale);   // saturates
    return max(0, min(kBuckets - 1, bk));
  };
  // ---- one pass over the range: s_bar and its governing group g* (Eq. 4, the
  // lowest on ties; per-KV-head mode: S[g, t] and g itself); Z = sum s and sum s log2 s (Sec. 3.6, one
  // pass: H = -sum p log p / log L_p with p = s / (Z + eps), where the eps
  // inside the log changes H by less than L_p eps); the untempered fused score
  // x_t = max(s beta D, 0) (Eq. final_score with Eq. 9).  s_t = x_t^(1/T) is
  // increasing in x_t, so the top-B select ranks the keys of x_t.
  float z = 0.f, zl = 0.f, nvs = 0.f;   // counts below 2^24: exact in fp32
  uint32_t smx = 0u;   // the largest s (non-negative: its bits order like the values)
#pragma unroll 1
  for (int i = tid; i < nr; i += NT) {
    const Token next_tok = load_token(i + NT);
    const uint32_t mt = cur_tok.mt;
    float sb = cur_tok.q[0], best = sb;
    int gs = 0;
#pragma unroll
    for (int j = 1; j < 4; ++j)
      if (j < g_n) {
        sb += cur_tok.q[j];
        if (cur_tok.q[j] > best) {
          best = cur_tok.q[j];
          gs = j;
        }
      }
#pragma unroll 4
    for (int gg = 4; gg < g_n; ++gg) {
      const float q = S0[static_cast<int64_t>(gg) * Lp + i];
      sb += q;
      if (q > best) {
        best = q;
        gs = gg;
      }
    }
    sb *= g_scale;
    gs += g_lo;
    z += sb;
    smx = max(smx, __float_as_uint(fmaxf(sb, 0.f)));
    zl += sb > 0.f ? sb * lg2_approx(sb) : 0.f;
    const float beta = (1.f - lam) + lam * static_cast<float>(G) * sh.w[gs];
    // Eq. (9) and its variants, for every token; text takes D = 1
    const bool vis = meta_visual(mt);
    nvs += vis ? 1.f : 0.f;
    const float df = vis ? static_cast<float>(sv.cur_frame - meta_frame(mt)) : 0.f, ph = sh.phi[gs];
    float shape;
    if (kp.decay_mode == 1) shape = fmaxf(0.f, 1.f - kp.delta * (df * ph));
    else if (kp.decay_mode == 2) shape = powf(1.f + df * ph, -kp.delta);
    else shape = expf(-kp.delta * df * ph);
    const float d = vis ? kp.d_min + (1.f - kp.d_min) * shape : 1.f;
    const float x = fmaxf(sb * beta * d, 0.f) + 0.f;   // (no negative zero)
    xs[i] = x;
    if (B > 0) atomicAdd(&hist[sbucket(desc_key(x))], 1);
    cur_tok = next_tok;
  }
  // ---- this CTA's partial sums, to every peer
  const float p4 = warp_sum4(z, zl, nvs, 0.f, lane);
  smx = __reduce_max_sync(kFullMask, smx);
  if ((lane & 7) == 0) sh.red[lane >> 3][warp] = p4;
  if (lane == 0) sh.wsum[warp] = static_cast<int>(smx);
  __syncthreads();   // the histogram and x_t are complete, too
  if (warp == 0) {
    float none;
    sum4(z, zl, nvs, none);
    smx = __reduce_max_sync(kFullMask, lane < NW ? static_cast<uint32_t>(sh.wsum[lane]) : 0u);
    if (lane < ncta) {
      dsmem_st_u32(dsmem_map(&sh.pz[rank], lane), __float_as_uint(z));
      dsmem_st_u32(dsmem_map(&sh.pzl[rank], lane), __float_as_uint(zl));
      dsmem_st_u32(dsmem_map(&sh.pv[rank], lane), __float_as_uint(nvs));
      dsmem_st_u32(dsmem_map(&sh.psmax[rank], lane), smx);
    }
  }
  // ---- Sec. 3.7: top-B, ties to the lower index (global mode: over the
  // cluster; per-KV-head mode: over this CTA's row, block barriers only)
  const int r_lo = per_head ? rank : 0, r_n = per_head ? 1 : ncta, r_me = per_head ? 0 : rank;
  auto send_coarse = [&]() {   // 32-bucket counts of the histogram, to every CTA of the selection
#pragma unroll 1
    for (int c = warp; c < kCoarse; c += NW) {
      const int v = __reduce_add_sync(kFullMask, hist[c * kFine + lane]);
      if (lane < r_n) dsmem_st_u32(dsmem_map(reinterpret_cast<int*>(sh.coarse[r_me]) + c, r_lo + lane), static_cast<uint32_t>(v));
    }
  };
  if (B > 0) send_coarse();
  cluster_arrive();
  if (per_head) __syncthreads();   // the selection's own exchange; the partial sums are read at the end
  else cluster_wait();
  // the AEB signal of a row from its sums: the normalised entropy (Sec. 3.6)
  // or, with aeb_mode 1, the peak mass p_max = max s / (sum s + eps); T grows
  // with the entropy and falls with the peak mass
  auto entropy = [&](float Zr, float ZL2r, uint32_t smaxr) {   // ZL2r = sum s log2 s
    const float Ze = Zr + kp.eps_h;
    if (kp.aeb_mode == 1) return __uint_as_float(smaxr) / Ze;
    const float plogp = Zr > 0.f ? kLn2 * ZL2r / Ze - (Zr / Ze) * logf(Ze) : 0.f;
    return Lp > 1 ? -plogp / logf(static_cast<float>(Lp)) : 0.f;
  };
  auto temperature = [&](float sig) {
    return kp.t_min + (kp.t_max - kp.t_min) * (kp.aeb_mode == 1 ? 1.f - sig : sig);
  };
  float Hn = 0.f, T = 0.f, Z = 0.f;
  auto find_T = [&]() {
    float ZL = 0.f;
    uint32_t SM = 0u;
    for (int r = 0; r < r_n; ++r) {   // per-KV-head mode: this CTA's own row
      Z += sh.pz[r_lo + r];
      ZL += sh.pzl[r_lo + r];
      SM = max(SM, sh.psmax[r_lo + r]);
    }
    Hn = entropy(Z, ZL, SM);
    T = temperature(Hn);
  };
  auto write_stats = [&]() {   // by CTA 0's last warp
    if (rank != 0 || warp != NW - 1 || !sv.stats) return;
    float* stats = sv.stats + static_cast<int64_t>(layer) * STARKV_STATS_STRIDE(G);
    if (lane < G) {
      const float Hr = per_head ? entropy(sh.pz[lane], sh.pzl[lane], sh.psmax[lane]) : Hn;
      stats[8 + lane] = sh.mi[lane];
      stats[8 + G + lane] = sh.mib[lane];
      stats[8 + 2 * G + lane] = sh.w[lane];
      stats[8 + 3 * G + lane] = sh.phi[lane];
      stats[8 + 4 * G + lane] = Hr;
      stats[8 + 5 * G + lane] = per_head ? temperature(Hr) : T;
    }
    if (lane == 0) {
      float hs = Hn, ts = T, zs = Z, nvf = sh.pv[0];
      if (per_head) {
        hs = ts = zs = 0.f;
        for (int r = 0; r < G; ++r) {
          const float Hr = entropy(sh.pz[r], sh.pzl[r], sh.psmax[r]);
          hs += Hr;
          ts += temperature(Hr);
          zs += sh.pz[r];
        }
        hs *= 1.f / static_cast<float>(G);
        ts *= 1.f / static_cast<float>(G);
        zs *= 1.f / static_cast<float>(G);   // sum_t s_bar_t = mean over g of the row sums
      } else {
        for (int r = 1; r < ncta; ++r) nvf += sh.pv[r];
      }
      stats[0] = hs;
      stats[1] = ts;
      stats[2] = lam;
      stats[3] = static_cast<float>(sh.n_old);
      stats[4] = zs;
      stats[5] = nvf;
      stats[6] = static_cast<float>(B);
      stats[7] = 0.f;
    }
  };
  const int seg = ceil_div(nr, NW * 32) * 32;   // one contiguous segment per warp: warp and lane order are position order
  const int w0 = min(nr, warp * seg), w1 = min(nr, w0 + seg);
  if (B > 0) {
    uint32_t lo = 0u, hi = kKeyMax;   // keys still in question; those below lo are kept, above hi not
    int target = B - 1;               // rank of the B-th token among them
    int nlow = 0;                     // kept tokens of the lower-ranked CTAs, so far
    int bstar, rkb, ncb, coff, nown;
    bool ties = false;
    // The loop's cluster barriers, and the one after it, stand behind conditions on
    // ncb, lo and hi, which every CTA of the selection computes from the same
    // exchanged counts and key ranges: all take the same way.
    for (;;) {
      // every warp for itself: the coarse bucket of the target on the summed
      // counts (four per lane), then its 32 buckets (one per lane)
      int tot = 0, low = 0, q[4] = {0, 0, 0, 0}, ql[4] = {0, 0, 0, 0};
      for (int r = 0; r < r_n; ++r) {
        const int4 c4 = sh.coarse[r][lane];
        q[0] += c4.x;
        q[1] += c4.y;
        q[2] += c4.z;
        q[3] += c4.w;
        if (r < r_me) {
          ql[0] += c4.x;
          ql[1] += c4.y;
          ql[2] += c4.z;
          ql[3] += c4.w;
        }
      }
      tot = (q[0] + q[1]) + (q[2] + q[3]);
      const int incl = warp_incl_scan(tot, lane);
      int ex = incl - tot;
      const bool has = target >= ex && target < incl;
      int cb = 0;
      if (has) {
        if (target >= ex + q[0]) { ex += q[0]; low += ql[0]; cb = 1; }
        if (cb == 1 && target >= ex + q[1]) { ex += q[1]; low += ql[1]; cb = 2; }
        if (cb == 2 && target >= ex + q[2]) { ex += q[2]; low += ql[2]; cb = 3; }
      } else if (incl <= target) {
        low = (ql[0] + ql[1]) + (ql[2] + ql[3]);
      }
      const int src = __ffs(__ballot_sync(kFullMask, has)) - 1;
      cb = __shfl_sync(kFullMask, 4 * lane + cb, src);
      ex = __shfl_sync(kFullMask, ex, src);
      int f = 0, fl = 0, fo = 0;
#pragma unroll
      for (int r = 0; r < kMaxCluster; ++r)
        if (r < r_n) {
          const int v = r == r_me ? hist[cb * kFine + lane] : dsmem_ld_s32(dsmem_map(hist + cb * kFine + lane, r_lo + r));
          f += v;
          if (r < r_me) fl += v;
          if (r == r_me) fo = v;
        }
      const int fi = warp_incl_scan(f, lane);
      const int fx = ex + fi - f;
      const bool fhas = target >= fx && target < fx + f;
      const int fs = __ffs(__ballot_sync(kFullMask, fhas)) - 1;
      if (lane < fs) low += fl;
      nlow += __reduce_add_sync(kFullMask, low);
      bstar = cb * kFine + fs;
      ncb = __shfl_sync(kFullMask, f, fs);
      rkb = target - __shfl_sync(kFullMask, fx, fs);
      coff = __shfl_sync(kFullMask, fl, fs);
      nown = __shfl_sync(kFullMask, fo, fs);
      if (ncb <= kCandMax) break;
      // many tokens in the bucket: its exact key range, then its own buckets
      __syncthreads();
      if (tid == 0) {
        sh.lo = 0xFFFFFFFFu;
        sh.hi = 0u;
      }
      __syncthreads();
      uint32_t mn = 0xFFFFFFFFu, mx = 0u;
      for (int i = tid; i < nr; i += NT) {
        const uint32_t u = desc_key(xs[i]);
        if (u >= lo && u <= hi && sbucket(u) == bstar) {
          mn = min(mn, u);
          mx = max(mx, u);
        }
      }
      mn = __reduce_min_sync(kFullMask, mn);
      mx = __reduce_max_sync(kFullMask, mx);
      if (lane == 0) {
        atomicMin(&sh.lo, mn);
        atomicMax(&sh.hi, mx);
      }
      __syncthreads();
      if (warp == 0 && lane < r_n) {
        dsmem_st_u32(dsmem_map(&sh.rlo[r_me], r_lo + lane), sh.lo);
        dsmem_st_u32(dsmem_map(&sh.rhi[r_me], r_lo + lane), sh.hi);
      }
      if (per_head) __syncthreads();
      else cluster_sync();
      lo = 0xFFFFFFFFu;
      hi = 0u;
      for (int r = 0; r < r_n; ++r) {
        lo = min(lo, sh.rlo[r]);
        hi = max(hi, sh.rhi[r]);
      }
      if (lo == hi) {   // one key: its first rkb + 1 tokens in position order are kept
        ties = true;
        break;
      }
      target = rkb;
      blo = lo;
      bscale = 4096.f / (static_cast<float>(hi - lo) + 1.f);
      for (int i = tid; i < kBuckets / 4; i += NT) reinterpret_cast<int4*>(hist)[i] = make_int4(0, 0, 0, 0);
      __syncthreads();
      for (int i = tid; i < nr; i += NT) {
        const uint32_t u = desc_key(xs[i]);
        if (u >= lo && u <= hi) atomicAdd(&hist[sbucket(u)], 1);
      }
      __syncthreads();
      send_coarse();
      if (per_head) __syncthreads();
      else cluster_sync();
    }
    // ---- one pass over the warp's segment: tokens below the bucket counted,
    // the bucket's tokens sent to every CTA of the selection (each CTA's go
    // to their own place, known from the counts)
    int below = 0, eq = 0;
#pragma unroll 1
    for (int i0 = w0; i0 < w1; i0 += 32) {
      const int i = i0 + lane;
      if (i < w1) {
        const float x = xs[i];
        const uint32_t u = desc_key(x);
        if (u < lo) {
          ++below;
        } else if (u <= hi) {
          if (ties) {
            ++eq;
          } else {
            const int bk = sbucket(u);
            if (bk < bstar) {
              ++below;
            } else if (bk == bstar) {
              const int j = coff + atomicAdd(&sh.ccnt, 1);
              for (int r = 0; r < r_n; ++r) dsmem_st_v2(dsmem_map(clist + j, r_lo + r), u, static_cast<uint32_t>(ta + i));
            }
          }
        }
      }
    }
    below = __reduce_add_sync(kFullMask, below);
    eq = __reduce_add_sync(kFullMask, eq);
    if (lane == 0) {
      sh.segb[warp] = below;
      if (ties) sh.sege[warp] = eq;
    }
    const bool wait_peers = !per_head && !ties;
    if (wait_peers) cluster_arrive();
    find_T();   // while the candidates travel
    if (!per_head) write_stats();
    if (wait_peers) cluster_wait();
    else __syncthreads();
    uint32_t kT = lo, tT = 0u;   // kept: key below kT, or equal to it and (at position <= tT | among the first `quota`)
    int quota = 0;
    if (!ties) {
      // every candidate's rank by (key, position), in every CTA
      for (int i = tid; i < ncb; i += NT) {
        const uint2 me = clist[i];
        int r = 0;
        for (int j = 0; j < ncb; ++j) {
          const uint2 p = clist[j];
          r += (p.x < me.x) || (p.x == me.x && p.y < me.y);
        }
        if (r <= rkb) {   // kept (the order is by key, then position)
          const int i = static_cast<int>(me.y) - ta;
          if (i < 0) atomicAdd(&sh.lowcnt, 1);
          else if (i < nr) atomicAdd(&sh.sege[i / seg], 1);
          if (r == rkb) {
            sh.tkey = me.x;
            sh.tpos = static_cast<int>(me.y);
          }
        }
      }
      __syncthreads();
      kT = sh.tkey;
      tT = static_cast<uint32_t>(sh.tpos);
      nlow += sh.lowcnt;
    } else {
      quota = max(0, min(nown, rkb + 1 - coff));
      nlow += min(coff, rkb + 1);
    }
    // first output position of this warp's segment and, with ties, the equal
    // keys before it (a capped sum: the first `quota` of the CTA are kept)
    const int vb = lane < NW ? sh.segb[lane] : 0, ve = lane < NW ? sh.sege[lane] : 0;
    const int pb = __shfl_sync(kFullMask, warp_incl_scan(vb, lane) - vb, warp);
    const int pe = __shfl_sync(kFullMask, warp_incl_scan(ve, lane) - ve, warp);
    int pos = nlow + pb + (ties ? min(pe, quota) : pe), eqr = pe;
    int32_t* idx = sv.idx + (static_cast<int64_t>(layer) * (per_head ? G : 1) + (per_head ? rank : 0)) * B;
    const unsigned lanes_below = (1u << lane) - 1u;
    const float invT = 1.f / T;
#pragma unroll 1
    for (int i0 = w0; i0 < w1; i0 += 32) {
      const int i = i0 + lane;
      const float x = i < w1 ? xs[i] : 0.f;
      const uint32_t u = i < w1 ? desc_key(x) : 0xFFFFFFFFu;
      bool kept = u < kT;
      if (ties) {
        const unsigned me = __ballot_sync(kFullMask, u == kT);
        if (u == kT && eqr + __popc(me & lanes_below) < quota) kept = true;
        eqr += __popc(me);
      } else if (u == kT && static_cast<uint32_t>(ta + i) <= tT) {
        kept = true;
      }
      const unsigned mk = __ballot_sync(kFullMask, kept);
      if (kept) {
        const int p = pos + __popc(mk & lanes_below);
        if (p >= B) atomicOr(st.err, kErrIndex);   // cannot happen for a correct select
        else idx[p] = ta + i;
      }
      pos += __popc(mk);
      // s_t = x_t^(1/T) = 2^(log2(x_t) / T) (hardware exp2 / log2, relative error a few 1e-7)
      if (i < w1) score[i] = ex2_approx(invT * lg2_approx(x));
    }
  } else {
    find_T();
    if (!per_head) write_stats();
    const float invT = 1.f / T;
    for (int i = tid; i < nr; i += NT) score[i] = ex2_approx(invT * lg2_approx(xs[i]));
  }
  if (per_head) {
    cluster_wait();   // the peers' partial sums are here, and this CTA's have reached them
    write_stats();
  }
}

namespace {

int calibrate_capacity(size_t fixed, size_t smem) {
  if (fixed >= smem) return 0;
  return static_cast<int>(((smem - fixed) / kBytesPerToken) & ~size_t(15));
}

template <bool FROM_RAW, int NT>
cudaError_t launch(cudaLaunchConfig_t& cfg, const SeqBatch& b, const KParams& kp, const DevState& st, int capl) {
  cfg.blockDim = dim3(NT, 1, 1);
  return cudaLaunchKernelEx(&cfg, k_calibrate<FROM_RAW, NT>, b, kp, st, capl);
}

}  // namespace

cudaError_t select_configure() {
  const int bytes = static_cast<int>(kSmemMax);
  const void* fns[] = {reinterpret_cast<const void*>(k_calibrate<true, 512>), reinterpret_cast<const void*>(k_calibrate<true, 1024>),
                       reinterpret_cast<const void*>(k_calibrate<false, 512>), reinterpret_cast<const void*>(k_calibrate<false, 1024>)};
  for (const void* f : fns) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t calibrate_launch(const SeqBatch& b, const KParams& kp, const DevState& st, bool from_raw, int lp_max,
                             int num_sms, cudaStream_t stream) {
  const int ncta = std::min(kp.G, kMaxCluster);   // the per-KV-head mode has G <= kMaxCluster
  // More CTAs than SMs: 512 threads and at most half of the shared memory
  // each, so that two run on an SM and one's barriers hide under the other's
  // work.  Otherwise every CTA has an SM to itself and takes 1024 threads,
  // which halves its token loops.  32 sequences x 8 groups of 2,000 / 11,000 /
  // 30,000 / 56,000 tokens, two per SM and one: 27 / 42 / 83 / 134 us and 60 / 83 / 128 /
  // 203; on the largest patch grid and joint histogram, where two leave no room
  // for rows on chip: 38 / 57 / 95 / 152 and 72 / 95 / 150 / 218.
  const bool two = static_cast<int64_t>(ncta) * b.nlayers * b.nseq > num_sms;
  const size_t fixed = fixed_bytes(kp.K * kp.M * kp.M, kp.R * kp.C);
  const int cap = calibrate_capacity(fixed, two ? kSmemTwo : kSmemMax);
  // A row longer than the capacity is read again from S in every pass; only
  // the CTA's range of fused scores is then kept on chip.
  int capl = (lp_max + 15) & ~15;
  if (capl > cap) capl = cap;
  const size_t smem = fixed + static_cast<size_t>(capl) * kBytesPerToken;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ncta, b.nlayers, b.nseq);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ncta;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // set-up under the previous kernel's tail
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (from_raw) return two ? launch<true, 512>(cfg, b, kp, st, capl) : launch<true, 1024>(cfg, b, kp, st, capl);
  return two ? launch<false, 512>(cfg, b, kp, st, capl) : launch<false, 1024>(cfg, b, kp, st, capl);
}

}  // namespace starkv
