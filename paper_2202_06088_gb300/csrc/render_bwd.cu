// Fused adjoint of the VOctree renderer (Sec. 4.3 "Optimization": the
// derivatives of the volume-rendering loss with respect to the leaf
// coefficients, for SGD/Adam directly on the VOctree).
//
// No per-sample state is stored by the forward pass.  Each ray is replayed
// with the forward's traversal; per sample the kernel recomputes sigma,
// gamma, the harmonics and the colour, and forms
//   dL/dc_i     = w_i g
//   dL/dsigma_i = delta_i ( g . (T_{i+1} c_i - S_{>i}) + g_alpha T_final )
// where S_{>i} = C - sum_{j<=i} w_j c_j is the radiance still to come behind
// sample i (the back-to-front quantity, taken from the saved C without a
// reverse walk or a division) and T_final = exp(-tau) from the saved optical
// depth.  The chain continues through ReLU (zero slope at pre-activation <= 0),
// pi*sigmoid and d H / d gamma.  Gradients are scattered into an FP32
// record-layout buffer with 16-byte vector atomics.
#include <algorithm>

#include "neuvv_kernels.h"
#include "neuvv_ray.cuh"

namespace neuvv {

// Vector reduction into global memory.  No memory clobber: the kernel never
// reads the gradient buffer, so no load needs ordering against these adds.
__device__ __forceinline__ void red_add_v4(float *addr, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d));
}

// Per-ray replay state of the adjoint.
struct AdjState {
  float T;         // transmittance in front of the current sample
  float acc[3];    // sum_{j<=i} w_j c_j
  float C[3];      // saved colour
  float g[3];      // dL/dC
  float gA;        // dL/dalpha
  float T_final;   // exp(-tau)
  int count, target;
};

// A sample's share of the adjoint that only its own record and chord decide.
template <int DEG>
struct SampleTerms {
  Sample<DEG> s;
  float ex, al;  // exp(-sigma delta), 1 - exp(-sigma delta); 1 and 0 for zero density
};

// Evaluates one sample; false when it has zero density (no path from it to
// the loss).
template <int KP, int DEG, typename E, typename Rows>
__device__ __forceinline__ bool sample_terms(const BwdArgs &a, const Rows &rows, const float *Y, uint32_t leaf, float dt,
                                             SampleTerms<DEG> &m) {
  LeafRecord<KP, DEG, E> rec;
  rec.load(a.tr, leaf);
  eval_sample<KP, DEG, E, true>(a.tr, rows, Y, Loaded{}, rec, a.act, m.s);
  m.ex = 1.f;
  m.al = 0.f;
  if (!(m.s.sigma > 0.f)) {
    m.s.c[0] = m.s.c[1] = m.s.c[2] = 0.f;
    return false;
  }
  const float sd = m.s.sigma * dt;
  m.ex = __expf(-sd);
  m.al = alpha_of(sd);
  return true;
}

// Advances a ray's replay state over one sample (its terms al, ex and colour
// c): the sample's weight and dL/dsigma per unit chord.
__device__ __forceinline__ void replay_sample(AdjState &st, float al, float ex, const float c[3], float &wgt,
                                              float &dsig) {
  wgt = st.T * al;
  const float Tn = st.T * ex;
  dsig = st.gA * st.T_final;
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) {
    st.acc[ch] = fmaf(wgt, c[ch], st.acc[ch]);
    const float S_after = st.C[ch] - st.acc[ch];
    dsig = fmaf(st.g[ch], Tn * c[ch] - S_after, dsig);
  }
  st.T = Tn;
}

// Gradient factors of one sample: with them, dL/dw_sigma = dpre_s a(u),
// dL/dw_gamma = dpre_g b(u) and dL/dw_HH[ch][n,l,m] = R_nl(gamma) F[ch][l,m]
// with F[ch][l,m] = dz[ch] Y_lm.
template <int DEG>
__device__ __forceinline__ void factors_of(const BwdArgs &a, const Sample<DEG> &s, const float g[3], float wgt,
                                           float dsig, float dt, float dz[3], float &dpre_s, float &dpre_g) {
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) {
    const float dc = wgt * g[ch];
    dz[ch] = a.act == 0 ? dc * s.c[ch] * (1.f - s.c[ch]) : dc;
  }
  // dL/dgamma = sum_ch dz[ch] d z_ch / dgamma
  const float dgam = dz[0] * s.u[0] + dz[1] * s.u[1] + dz[2] * s.u[2];
  dpre_g = dgam * kPi * s.s_gamma * (1.f - s.s_gamma);
  dpre_s = s.pre_sigma > 0.f ? dsig * dt : 0.f;
}

// Scatters a leaf's gradient from its factors into its FP32 record with
// 16-byte vector atomics: the w_HH part in record order (channel, then idx
// ascending over n, l, m), one quad at a time, then w_sigma and w_gamma.
template <int KP, int DEG, typename Rows>
__device__ __forceinline__ void scatter_gradient(const BwdArgs &a, const Rows &rows, uint32_t leaf, const float *R,
                                                 const float *F, float dpre_s, float dpre_g) {
  constexpr int NY = (DEG + 1) * (DEG + 1);
  float *dst = a.grad + (size_t)leaf * a.grad_stride;
  float v[4];
  int j = 0;
#pragma unroll
  for (int ch = 0; ch < 3; ++ch)
#pragma unroll
    for (int n = 0; n <= DEG; ++n)
#pragma unroll
      for (int l = 0; l <= n; ++l)
#pragma unroll
        for (int m = -l; m <= l; ++m) {
          v[j & 3] = R[radial_index(n, l)] * F[ch * NY + l * l + l + m];
          if ((j & 3) == 3) red_add_v4(dst + 2 * KP + j - 3, v[0], v[1], v[2], v[3]);
          ++j;
        }
  if (j & 3) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k >= (j & 3)) v[k] = 0.f;
    red_add_v4(dst + 2 * KP + (j & ~3), v[0], v[1], v[2], v[3]);
  }
#pragma unroll
  for (int q = 0; q < KP / 4; ++q) {
    const float4 ra = rows.A4(q), rb = rows.B4(q);
    red_add_v4(dst + 4 * q, dpre_s * ra.x, dpre_s * ra.y, dpre_s * ra.z, dpre_s * ra.w);
    red_add_v4(dst + KP + 4 * q, dpre_g * rb.x, dpre_g * rb.y, dpre_g * rb.z, dpre_g * rb.w);
  }
  if (a.touched) {
    const unsigned int bit = 1u << (leaf & 31);
    unsigned int *word = a.touched + (leaf >> 5);
    if (!(__ldcg(word) & bit)) atomicOr(word, bit);
  }
}

// Gradient of one sample, scattered by its own thread (the plain kernel).
template <int KP, int DEG, typename E, typename Rows>
__device__ __forceinline__ void adjoint_sample(const BwdArgs &a, const Rows &rows, const float *Y, uint32_t leaf,
                                               float dt, AdjState &st) {
  constexpr int NY = (DEG + 1) * (DEG + 1);
  SampleTerms<DEG> m;
  if (!sample_terms<KP, DEG, E>(a, rows, Y, leaf, dt, m)) return;
  float wgt, dsig, dz[3], dpre_s, dpre_g;
  replay_sample(st, m.al, m.ex, m.s.c, wgt, dsig);
  factors_of<DEG>(a, m.s, st.g, wgt, dsig, dt, dz, dpre_s, dpre_g);
  float F[3 * NY];
#pragma unroll
  for (int ch = 0; ch < 3; ++ch)
#pragma unroll
    for (int k = 0; k < NY; ++k) F[ch * NY + k] = dz[ch] * Y[k];
  scatter_gradient<KP, DEG, Rows>(a, rows, leaf, m.s.R, F, dpre_s, dpre_g);
}

// Octahedral code of a unit direction (the direction divided by its L1 norm,
// the lower hemisphere folded over the diagonals of the square): two floats
// instead of three, exact to a few FP32 ulps of the direction (the decoder
// normalises, so the fast reciprocal's error of an ulp or two only scales
// the code).
__device__ __forceinline__ void oct_encode(const float d[3], float &e0, float &e1) {
  const float s = __fdividef(1.f, fabsf(d[0]) + fabsf(d[1]) + fabsf(d[2]));
  const float p = d[0] * s, q = d[1] * s;
  if (d[2] < 0.f) {
    e0 = copysignf(1.f - fabsf(q), p);
    e1 = copysignf(1.f - fabsf(p), q);
  } else {
    e0 = p;
    e1 = q;
  }
}
__device__ __forceinline__ void oct_decode(float e0, float e1, float d[3]) {
  const float z = 1.f - fabsf(e0) - fabsf(e1);
  float x = e0, y = e1;
  if (z < 0.f) {
    x = copysignf(1.f - fabsf(e1), e0);
    y = copysignf(1.f - fabsf(e0), e1);
  }
  const float il = 1.f / sqrtf(fmaf(x, x, fmaf(y, y, z * z)));
  d[0] = x * il;
  d[1] = y * il;
  d[2] = z * il;
}

// Adjoint of one batch of a packet's samples, called by the whole warp: lane j
// holds entry j (leaf, dt, the lane `owner` of its ray; has: a sample, valid:
// one whose leaf exists), a ray's entries in order.  Each entry is evaluated by its lane; each ray then
// runs its replay state over its own entries (at most target - count of them)
// and leaves every entry's weight and dL/dsigma in shared memory, from which
// the entry's lane forms the gradient factors.
//
// With kGather (leaf-major reduction) each sample takes the next position of
// its leaf's run (lanes of the batch that share a leaf take consecutive
// positions with one atomic), reserved before the sample is evaluated so that
// the atomic's round trip overlaps the evaluation, and leaves its factors
// (dpre_s, dpre_g, dz), its ray's frame coordinate u and the octahedral code
// of its unit direction there; a sample of zero density leaves a record marked
// kNoFactor.  No gradient atomics; the per-leaf sums are formed by
// leaf_reduce_kernel.
//
// Otherwise a warp-aggregated scatter: lanes whose samples share a leaf and a
// time (hence the basis rows a(u), b(u) and the hyper-angle, so the radial
// factors R_nl) add their factors dpre_s, dpre_g and F[ch][l,m] with shuffles,
// and the lowest lane of each such group scatters the group's gradient: one
// set of vector atomics per distinct (leaf, time) in the batch instead of one
// per sample.
// The records are read in place: staging them in shared memory a round ahead,
// as the forward does, measured 9.68 against 9.43 ms for the 8-view step (the
// copies' instructions, and two warps fewer per SM).
template <int KP, int DEG, typename E, bool kGather, typename Sh>
__device__ __forceinline__ void adjoint_batch(const BwdArgs &a, const Sh &sh, uint32_t leaf, float dt, int owner,
                                              bool has, bool valid, float t, AdjState &st) {
  constexpr int NY = (DEG + 1) * (DEG + 1);
  const int lane = threadIdx.x & 31;
  uint32_t base = 0u;
  if (kGather) {
    const unsigned grp = __match_any_sync(kFull, valid ? leaf : kEmpty);
    if (valid && lane == __ffs(grp) - 1) base = atomicAdd(a.gws.cur + leaf, (uint32_t)__popc(grp));
  }
  float dn[3], Y[NY];
  sh.get_dir(owner, dn);
  sh_real<DEG>(dn, Y);
  const SmemRows<KP> rows = sh.rows_of(owner);
  SampleTerms<DEG> m;
  m.al = 0.f;
  m.ex = 1.f;
  m.s.c[0] = m.s.c[1] = m.s.c[2] = 0.f;
  bool dense = false;
  if (valid) dense = sample_terms<KP, DEG, E>(a, rows, Y, leaf, dt, m);
  unsigned mine = sh.entries_of_lane(has, owner), kept = 0u;
  while (__any_sync(kFull, mine != 0u)) {
    const int j = mine ? __ffs(mine) - 1 : lane;
    const float al = __shfl_sync(kFull, m.al, j), ex = __shfl_sync(kFull, m.ex, j);
    float c[3];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) c[ch] = __shfl_sync(kFull, m.s.c[ch], j);
    if (mine) {
      mine &= mine - 1u;
      if (st.count < st.target) {
        ++st.count;
        kept |= 1u << j;
        float wgt, dsig;
        replay_sample(st, al, ex, c, wgt, dsig);
        sh.res[j] = make_float2(wgt, dsig);
      }
    }
  }
  kept = __reduce_or_sync(kFull, kept);
  const bool contrib = dense && ((kept >> lane) & 1u);
  float g[3];
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) g[ch] = __shfl_sync(kFull, st.g[ch], owner);
  const float to = __shfl_sync(kFull, t, owner);  // the entry's time
  __syncwarp();
  float dz[3] = {0.f, 0.f, 0.f}, dpre_s = 0.f, dpre_g = 0.f;
  if (contrib) {
    const float2 r = sh.res[lane];
    factors_of<DEG>(a, m.s, g, r.x, r.y, dt, dz, dpre_s, dpre_g);
  }
  if constexpr (kGather) {
    // the group again (recomputed rather than held through the evaluation)
    const unsigned grp = __match_any_sync(kFull, valid ? leaf : kEmpty);
    base = __shfl_sync(kFull, base, __ffs(grp) - 1);
    if (valid) {
      const uint32_t p = base + (uint32_t)__popc(grp & ((1u << lane) - 1u));
      // the count over the log bounds every run; this keeps a write inside the
      // workspace even if the log changed between the count and the replay
      if (p >= a.gws.cap_chunks * (uint32_t)(kLogRounds * 32)) {
        raise_status(a.tr, kStatusBadIndex);
      } else {
        float e0 = kNoFactor, e1 = 0.f;
        if (contrib) oct_encode(dn, e0, e1);
        float4 *f = a.gws.fac + 2 * (size_t)p;
        __stcs(f, make_float4(dpre_s, dpre_g, dz[0], dz[1]));
        __stcs(f + 1, make_float4(dz[2], to * (float)(a.tr.T - 1), e0, e1));
      }
    }
  } else {
    // lanes without a contribution get keys of their own (leaf ids are < 2^31)
    const unsigned long long key =
        contrib ? (((unsigned long long)leaf << 32) | __float_as_uint(to)) : (~0ull - (unsigned long long)lane);
    const unsigned grp = __match_any_sync(kFull, key);
    const bool leader = contrib && lane == __ffs(grp) - 1;
    float F[3 * NY];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch)
#pragma unroll
      for (int k = 0; k < NY; ++k) F[ch * NY + k] = dz[ch] * Y[k];
    const int gmax = (int)__reduce_max_sync(kFull, contrib ? (unsigned)__popc(grp) : 1u);
    unsigned rest = leader ? (grp & (grp - 1u)) : 0u;  // the leader's other members
    for (int it = 1; it < gmax; ++it) {
      const int src = rest ? __ffs(rest) - 1 : lane;
      rest &= rest - 1u;
      const bool add = src != lane;
      const float xs = __shfl_sync(kFull, dpre_s, src);
      const float xg = __shfl_sync(kFull, dpre_g, src);
      if (add) {
        dpre_s += xs;
        dpre_g += xg;
      }
#pragma unroll
      for (int k = 0; k < 3 * NY; ++k) {
        const float x = __shfl_sync(kFull, F[k], src);
        if (add) F[k] += x;
      }
    }
    if (leader) scatter_gradient<KP, DEG>(a, rows, leaf, m.s.R, F, dpre_s, dpre_g);
  }
  __syncwarp();  // the shared results are rewritten by the next batch
}

// Sets up the replay of ray i; false when the ray has nothing to replay.
__device__ __forceinline__ bool adjoint_setup(const BwdArgs &a, long long i, RayWalk &w, float dn[3], float &t,
                                              AdjState &st) {
  st.target = __ldcs(a.nseg + i);
  if (st.target <= 0) return false;
  float o[3], d[3];
  load_ray(a.rays, i, o, d, t);
  if (!walk_init(a.tr, o, d, w, dn)) return false;
  st.T = 1.f;
  st.count = 0;
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) {
    st.acc[ch] = 0.f;
    st.C[ch] = __ldcs(a.rgb + 3 * i + ch);
    st.g[ch] = __ldcs(a.grad_rgb + 3 * i + ch);
  }
  st.gA = a.grad_alpha ? __ldcs(a.grad_alpha + i) : 0.f;
  st.T_final = __expf(-__ldcs(a.tau + i));
  return true;
}

// One thread per ray (baseline); one loop over steps, as in integrate_ray.
template <int KP, int DEG, typename E>
__global__ void __launch_bounds__(256) render_bwd_plain_kernel(const __grid_constant__ BwdArgs a) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.rays.n) return;
  RayWalk w;
  float dn[3], t;
  AdjState st;
  if (!adjoint_setup(a, i, w, dn, t, st)) return;
  RayConst<KP, DEG> rc;
  ray_const_basis<KP, DEG>(a.tr, t * (float)(a.tr.T - 1), rc);
  sh_real<DEG>(dn, rc.Y);
  uint32_t leaf;
  float t0, dt;
  while (st.count < st.target && w.alive) {
    if (!walk_step(a.tr, w, leaf, t0, dt)) continue;
    ++st.count;
    adjoint_sample<KP, DEG, E>(a, RegRows<KP>{rc.a, rc.b}, rc.Y, leaf, dt, st);
  }
}

// Counting sort of the packets by their key (the first leaf they shade) into
// log.order, so that the adjoint runs the packets of all views that meet the
// same region of the tree close together in time: their leaf records and
// gradient rows are then shared in L2 instead of being fetched from and
// written back to DRAM once per view.
__device__ __forceinline__ int key_bin(uint32_t k, int shift) { return (int)min(k >> shift, (uint32_t)(kSortBins - 1)); }

__global__ void __launch_bounds__(256) key_hist_kernel(const SampleLog l, long long n_packets, int shift) {
  __shared__ uint32_t h[kSortBins];
  for (int b = threadIdx.x; b < kSortBins; b += blockDim.x) h[b] = 0;
  __syncthreads();
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n_packets;
       p += (long long)gridDim.x * blockDim.x)
    atomicAdd(&h[key_bin(__ldg(l.key + p), shift)], 1u);
  __syncthreads();
  for (int b = threadIdx.x; b < kSortBins; b += blockDim.x)
    if (h[b]) atomicAdd(&l.bins[b], h[b]);
}

// Exclusive prefix sum of the bin counts, in place (one block of 1024).
__global__ void __launch_bounds__(1024) key_scan_kernel(const SampleLog l) {
  __shared__ uint32_t part[1024];
  constexpr int kPer = kSortBins / 1024;
  const int t = threadIdx.x;
  uint32_t v[kPer], sum = 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    v[j] = l.bins[kPer * t + j];
    sum += v[j];
  }
  part[t] = sum;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    const uint32_t x = t >= off ? part[t - off] : 0u;
    __syncthreads();
    part[t] += x;
    __syncthreads();
  }
  uint32_t base = t ? part[t - 1] : 0u;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    l.bins[kPer * t + j] = base;
    base += v[j];
  }
}

// Each block places a contiguous range of kScatterPer packets: ranks within
// the block's share of a bin come from shared-memory counters, and one global
// add per (block, bin) reserves the share, so that a popular bin (all the
// packets that shade nothing share the last one) costs no global contention.
constexpr int kScatterThreads = 256, kScatterEach = 16, kScatterPer = kScatterThreads * kScatterEach;

__global__ void __launch_bounds__(kScatterThreads) key_scatter_kernel(const SampleLog l, long long n_packets,
                                                                      int shift) {
  __shared__ uint32_t cnt[kSortBins];
  for (int b = threadIdx.x; b < kSortBins; b += blockDim.x) cnt[b] = 0;
  __syncthreads();
  const long long first = (long long)blockIdx.x * kScatterPer;
  int bin[kScatterEach];
  uint32_t rank[kScatterEach];
#pragma unroll
  for (int k = 0; k < kScatterEach; ++k) {
    const long long p = first + (long long)k * kScatterThreads + threadIdx.x;
    bin[k] = p < n_packets ? key_bin(__ldg(l.key + p), shift) : -1;
    rank[k] = bin[k] >= 0 ? atomicAdd(&cnt[bin[k]], 1u) : 0u;
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kSortBins; b += blockDim.x)
    if (cnt[b]) cnt[b] = atomicAdd(&l.bins[b], cnt[b]);  // this block's first position in bin b
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kScatterEach; ++k)
    if (bin[k] >= 0) l.order[cnt[bin[k]] + rank[k]] = (uint32_t)(first + (long long)k * kScatterThreads + threadIdx.x);
}

// Region key of each packet for the forward's schedule (see
// launch_packet_order): the first leaf reached by the first of lanes 0, 8,
// 16, 24 whose ray enters the tree, kNoKey when none does.
__global__ void __launch_bounds__(256) packet_key_kernel(const __grid_constant__ DevTree tr, const DevRays rays,
                                                         const SampleLog l, long long n_packets) {
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n_packets) return;
  uint32_t key = kNoKey;
  for (int lane = 0; lane < 32 && key == kNoKey; lane += 8) {
    const long long i = (p << 5) + lane;
    if (i >= rays.n) break;
    float o[3], d[3], t, dn[3];
    load_ray(rays, i, o, d, t);
    RayWalk w;
    uint32_t leaf;
    float t0, dt;
    if (walk_init(tr, o, d, w, dn) && walk_next(tr, w, leaf, t0, dt)) key = leaf;
  }
  l.key[p] = key;
}

// Counting sort of the packets by their keys into l.order (bins of the
// leaf id's top bits).
static cudaError_t sort_packets_by_key(const SampleLog &l, long long n_packets, long long n_leaves, int num_sms,
                                       cudaStream_t s) {
  int bits = 0;
  while (bits < 32 && ((long long)1 << bits) <= n_leaves) ++bits;
  const int shift = bits > 12 ? bits - 12 : 0;
  const unsigned g = (unsigned)std::min<long long>((n_packets + 255) / 256, 4LL * num_sms);
  cudaError_t e = cudaMemsetAsync(l.bins, 0, kSortBins * sizeof(uint32_t), s);
  if (e != cudaSuccess) return e;
  key_hist_kernel<<<g, 256, 0, s>>>(l, n_packets, shift);
  key_scan_kernel<<<1, 1024, 0, s>>>(l);
  key_scatter_kernel<<<(unsigned)((n_packets + kScatterPer - 1) / kScatterPer), kScatterThreads, 0, s>>>(l, n_packets,
                                                                                                       shift);
  return cudaGetLastError();
}

cudaError_t launch_packet_order(const DevTree &tr, const DevRays &rays, const SampleLog &l, int num_sms,
                                cudaStream_t s) {
  const long long n_packets = (rays.n + 31) >> 5;
  if (n_packets == 0 || !l.n_chunks) return cudaSuccess;
  packet_key_kernel<<<(unsigned)((n_packets + 255) / 256), 256, 0, s>>>(tr, rays, l, n_packets);
  return sort_packets_by_key(l, n_packets, tr.n_leaves, num_sms, s);
}

// Walking adjoint of one packet (ray i of this lane, when live) that the
// segment log does not hold: the forward packet kernel's structure (walk steps
// and batches decoupled through the packet's ring), each ray's walk stopped at
// the forward's segment count.  Not inlined: its state does not add to the
// registers of the replay, which most packets take.
template <int KP, int DEG, typename E>
__device__ __noinline__ void adjoint_walk_packet(const BwdArgs &a, long long i, bool live) {
  extern __shared__ __align__(16) uint32_t smem[];
  const DevTree &tr = a.tr;
  const int lane = threadIdx.x & 31;
  const PacketShared<KP, 0> sh(smem);
  const PathRef pr{sh.path, sh.stride};
  RayWalk w;
  w.alive = false;
  AdjState st;
  st.count = st.target = 0;
  st.g[0] = st.g[1] = st.g[2] = 0.f;
  float dn[3], t = 0.f;
  live = live && adjoint_setup(a, i, w, dn, t, st);
  if (!__any_sync(kFull, live)) return;
  if (live) sh.put_ray(tr, dn, t * (float)(tr.T - 1), true);
  int walked = 0;  // segments found so far (the walk stops at the forward's count)
  bool walking = live && w.alive;
  int head = 0, count = 0;
  for (;;) {
    uint32_t leaf = 0u;
    float t0, dt = 0.f;
    bool found = false;
    if (walking) {
      found = walk_step<true>(tr, w, leaf, t0, dt, pr);
      walked += found ? 1 : 0;
      walking = w.alive && walked < st.target;
    }
    const unsigned finds = __ballot_sync(kFull, found);
    if (found) {
      const int slot = (head + count + __popc(finds & ((1u << lane) - 1u))) & (kRing - 1);
      sh.ring[slot] = make_uint4(leaf, __float_as_uint(dt), 0u, lane);
    }
    count += __popc(finds);
    if (count < kBatch && __any_sync(kFull, walking)) continue;
    if (count == 0) break;
    __syncwarp();
    const int batch = min(count, kBatch);
    const uint4 en = sh.ring[(head + lane) & (kRing - 1)];
    head += batch;
    count -= batch;
    adjoint_batch<KP, DEG, E, false>(a, sh, en.x, __uint_as_float(en.y), (int)en.w & 31, lane < batch, lane < batch, t,
                                     st);
  }
}

// One slot of a packet's logged round, as this lane reads it.
struct LogEntry {
  uint32_t leaf, chunk;
  float dt;
  int owner;
  bool has;  // a segment of a ray that is replayed
  __device__ __forceinline__ bool valid(const DevTree &tr) const { return has && leaf < (uint32_t)tr.n_leaves; }
};
// Walks a packet's chunks round by round (warp-uniform).
struct LogCursor {
  uint32_t chunk;
  int round = 0;
  __device__ __forceinline__ LogCursor(uint32_t head) : chunk(head) {}
  __device__ __forceinline__ LogEntry read(const SampleLog &l, unsigned rays) {
    LogEntry e{kEmpty, chunk, 0.f, 0, false};
    if (chunk >= l.n_chunks) return e;
    const size_t slot = ((size_t)chunk * kLogRounds + round) * 32 + (threadIdx.x & 31);
    const LogWord w = log_word(l, slot);
    e.leaf = w.leaf;
    e.dt = __ldcs(l.dt + slot);
    e.owner = w.lane;
    e.has = !w.empty && ((rays >> e.owner) & 1u);
    if (++round == kLogRounds) {
      round = 0;
      chunk = __ldg(l.next + chunk);
    }
    return e;
  }
};

// Packet adjoint: replays each packet's shading rounds from the forward's
// segment log when the log holds the packet (no walk); other packets (all of
// them without a log for these rays) take adjoint_walk_packet.  Records of up
// to 20 chunks, read in place, take 128 registers with at most 40 B of spills (K_pad
// 32 degree 1 and K_pad 16 degree 2 in FP32, 19 and 20 chunks: training steps as fast
// or up to 9 % faster than with 255, walked ones up to 4 % slower); larger ones take
// 255.
template <int KP, int DEG, typename E>
__global__ void __launch_bounds__(256, LeafRecord<KP, DEG, E>::kChunks <= 20 ? 2 : 1)
    render_bwd_packet_kernel(const __grid_constant__ BwdArgs a) {
  extern __shared__ __align__(16) uint32_t smem[];
  const DevTree &tr = a.tr;
  const int lane = threadIdx.x & 31;
  const PacketShared<KP, 0> sh(smem);
  // warp w adjoins packet w, or with a valid log in key order (the atomic
  // scatter) the w-th packet of that order
  const long long n_packets = (a.rays.n + 31) >> 5;
  const long long wp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (wp >= n_packets) return;
  const bool logged = a.log.n_chunks && log_matches(a.log, a.rays.n);
  const long long pk = logged && a.key_order ? (long long)min(__ldg(a.log.order + wp), (uint32_t)(n_packets - 1)) : wp;
  const long long pos = (pk << 5) + lane;  // position; the ray is pos, or perm[pos] in a permuted log
  // positions past the log's live rays hold rays that missed the tree
  if (logged && (pk << 5) >= ((long long)__ldg(a.log.header + 7) << 32 | __ldg(a.log.header + 6))) return;
  bool live = pos < a.rays.n;
  const long long i = live && logged && __ldg(a.log.header + 5) == 1u
                          ? (long long)min(__ldg(a.log.perm + pos), (uint32_t)(a.rays.n - 1))
                          : pos;
  const uint32_t head = logged ? __ldg(a.log.heads + pk) : kNoLog;  // warp-uniform
  if (head == kNoLog) {
    adjoint_walk_packet<KP, DEG, E>(a, i, live);
    return;
  }
  RayWalk w;
  AdjState st;
  st.count = st.target = 0;
  st.g[0] = st.g[1] = st.g[2] = 0.f;
  float dn[3], t = 0.f;
  live = live && adjoint_setup(a, i, w, dn, t, st);
  if (!__any_sync(kFull, live)) return;
  if (live) sh.put_ray(tr, dn, t * (float)(tr.T - 1), true);
  __syncwarp();
  // replay the forward's shading rounds from its log: no walk
  const unsigned rays = __ballot_sync(kFull, live);
  // the log is read one round ahead, and L2 asked for the next round's records
  // (3.28 -> 3.13 ms for the replay of the 8-view step)
  LogCursor cur(head);
  LogEntry now = cur.read(a.log, rays), next;
  while (__any_sync(kFull, live && st.count < st.target)) {
    if (now.chunk >= a.log.n_chunks) {  // the chain's end: a log that does not belong to these rays
      raise_status(tr, kStatusBadIndex);
      break;
    }
    next = cur.read(a.log, rays);
    if (next.valid(tr)) LeafRecord<KP, DEG, E>::prefetch_l2(tr, next.leaf);
    const bool valid = now.valid(tr);
    if (now.has && !valid) raise_status(tr, kStatusBadIndex);
    // chunks with room in the workspace: factors to the leaf's run; others: atomics
    if (now.chunk < a.gws.cap_chunks)
      adjoint_batch<KP, DEG, E, true>(a, sh, now.leaf, now.dt, now.owner, now.has, valid, t, st);
    else
      adjoint_batch<KP, DEG, E, false>(a, sh, now.leaf, now.dt, now.owner, now.has, valid, t, st);
    now = next;
  }
}

// ---------------------------------------------------------------------------
// Leaf-major reduction of the gradient factors.
// ---------------------------------------------------------------------------

// Counts, per leaf, the samples that the replay will leave in the workspace:
// every slot of the chunks below the workspace's capacity, read in order (the
// forward leaves kEmpty in slots without a segment), when the log was written
// by a forward over these rays.  The 32 slots of a warp are one shading
// round of one packet: lanes that share a leaf add to its count with one
// atomic.  A packet whose log ran out of chunks is walked by the replay, so
// its counted samples only leave unused room at the end of their runs.
__global__ void __launch_bounds__(256) leaf_count_kernel(const __grid_constant__ BwdArgs a) {
  if (!log_matches(a.log, a.rays.n)) return;
  const unsigned long long used = *a.log.counter;  // chunks the forward handed out
  const long long chunks = (long long)min(used, (unsigned long long)min(a.log.n_chunks, a.gws.cap_chunks));
  const long long n_slots = chunks * kLogRounds * 32;
  const uint32_t n_leaves = (uint32_t)a.tr.n_leaves;
  const int lane = threadIdx.x & 31;
  const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * 32 < n_slots; w += warps) {
    const uint32_t word = __ldcs(a.log.leaf + w * 32 + lane);
    const uint32_t leaf = a.log.lane ? word : word >> 5;
    const bool has = word != kEmpty && leaf < n_leaves;
    const unsigned grp = __match_any_sync(0xFFFFFFFFu, has ? leaf : kEmpty);
    if (has && lane == __ffs(grp) - 1) atomicAdd(a.gws.off + leaf, (uint32_t)__popc(grp));
  }
}

// One thread per leaf: sums the factors of the leaf's samples, whose records
// lie one after another in the leaf's run.  Samples of
// one frame coordinate u share the basis rows a(u), b(u) and the radial
// factors R_nl(gamma(u)), so they are summed first (dpre_s, dpre_g and
// F[ch][l,m] = sum dz[ch] Y_lm) and expanded into the record when u changes:
// dL/dw_sigma += a(u) sum dpre_s, dL/dw_gamma += b(u) sum dpre_g,
// dL/dw_HH[ch][n,l,m] += R_nl F[ch][l,m].  The record accumulates in shared
// memory; the block then adds its records (consecutive leaves, consecutive
// in memory) to the gradient buffer with coalesced 16-byte accesses, and sets
// the touched bits.
template <int KP, int DEG>
__host__ __device__ constexpr int reduce_pitch() { return (2 * KP + 3 * n_hh(DEG)) | 1; }

template <int KP, int DEG, typename E>
__device__ __forceinline__ void leaf_flush(const DevTree &tr, const LeafRecord<KP, DEG, E> &rec, float u,
                                           float ps, float pg, const float *F, float *acc) {
  constexpr int NY = (DEG + 1) * (DEG + 1);
  RayConst<KP, DEG> rc;
  ray_const_basis<KP, DEG>(tr, u, rc);
  const RegRows<KP> rows{rc.a, rc.b};
  const float pgam = pre_gamma_of<KP>(rows, rec);
  float sg, cg, R[(DEG + 1) * (DEG + 2) / 2];
  sincospif(sigmoidf_fast(pgam), &sg, &cg);
  hh_radial<DEG, false>(cg, sg, tr.hh_norm, R, nullptr);
#pragma unroll
  for (int k = 0; k < KP; ++k) {
    acc[k] = fmaf(ps, rc.a[k], acc[k]);
    acc[KP + k] = fmaf(pg, rc.b[k], acc[KP + k]);
  }
  int j = 0;
#pragma unroll
  for (int ch = 0; ch < 3; ++ch)
#pragma unroll
    for (int n = 0; n <= DEG; ++n)
#pragma unroll
      for (int l = 0; l <= n; ++l)
#pragma unroll
        for (int m = -l; m <= l; ++m) {
          acc[2 * KP + j] = fmaf(R[radial_index(n, l)], F[ch * NY + l * l + l + m], acc[2 * KP + j]);
          ++j;
        }
}


// With Adam (ad.on, Sec. 4.3 "Optimization"), the block's finished records
// are not added to the gradient buffer: each warp takes rows of the block in
// turn, a lane a 4-entry quad of the row, and applies the Adam step to the
// leaf's FP32 master, m and v and writes its storage record (BF16 rounded,
// FP8 re-encoded with the row's group scales from warp reductions).  A leaf
// whose touched bit was set before the call also takes what the atomic
// scatter left in its gradient row, which is then cleared; the caller clears
// the touched bitmap afterwards.
template <int KP, int DEG, typename E>
__global__ void __launch_bounds__(128) leaf_reduce_kernel(const __grid_constant__ BwdArgs a,
                                                          const __grid_constant__ AdamArgs ad) {
  constexpr int NY = (DEG + 1) * (DEG + 1);
  constexpr int LEN = 2 * KP + 3 * n_hh(DEG), PITCH = reduce_pitch<KP, DEG>(), Q4 = (LEN + 3) / 4;
  extern __shared__ float acc_s[];  // [blockDim][PITCH], then one flag per thread
  int *has = reinterpret_cast<int *>(acc_s + blockDim.x * PITCH);
  const DevTree &tr = a.tr;
  const long long first = (long long)blockIdx.x * blockDim.x;
  const long long leaf = first + threadIdx.x;
  float *acc = acc_s + threadIdx.x * PITCH;
  uint32_t lo = 0, hi = 0;
  bool before = false;  // Adam: touched before this kernel (the atomic scatter left a part in the row)
  if (leaf < tr.n_leaves) {
    lo = __ldg(a.gws.off + leaf);
    hi = min(__ldg(a.gws.cur + leaf), __ldg(a.gws.off + leaf + 1));
    lo = min(lo, hi);
    if (ad.on && a.touched) before = (a.touched[leaf >> 5] >> (leaf & 31)) & 1u;
  }
  if (lo < hi || before)  // only rows the epilogue may read
    for (int j = 0; j < LEN; ++j) acc[j] = 0.f;
  bool got = false;  // a sample of nonzero density reached the leaf
  if (lo < hi) {
    LeafRecord<KP, DEG, E> rec;
    rec.load_gamma(tr, (uint32_t)leaf);
    float F[3 * NY];
#pragma unroll
    for (int k = 0; k < 3 * NY; ++k) F[k] = 0.f;
    float ps = 0.f, pg = 0.f;
    // The run is taken one group at a time (consecutive records of one frame
    // coordinate u), each group's sums expanded once at its end: the lanes
    // of a warp expand together, once per group of the lane with the most
    // groups, rather than whenever any lane's next record changes u.
    const float4 *f = a.gws.fac + 2 * (size_t)lo;
    float4 c0 = __ldg(f), c1 = __ldg(f + 1);  // the current record
    float4 n0 = c0, n1 = c1;                  // the one after it
    if (lo + 1 < hi) {
      n0 = __ldg(f + 2);
      n1 = __ldg(f + 3);
    }
    f += 4;
    uint32_t p = lo;
    while (p < hi) {
      const float u = c1.y;
      bool any = false;
      for (;;) {
        if (c1.z != kNoFactor) {
          any = true;
          ps += c0.x;
          pg += c0.y;
          const float dz[3] = {c0.z, c0.w, c1.x};
          float dn[3];
          oct_decode(c1.z, c1.w, dn);
          float Y[NY];
          sh_real<DEG>(dn, Y);
#pragma unroll
          for (int ch = 0; ch < 3; ++ch)
#pragma unroll
            for (int k = 0; k < NY; ++k) F[ch * NY + k] = fmaf(dz[ch], Y[k], F[ch * NY + k]);
        }
        ++p;
        const bool same = p < hi && n1.y == u;
        c0 = n0;
        c1 = n1;
        if (p + 1 < hi) {
          n0 = __ldg(f);
          n1 = __ldg(f + 1);
          f += 2;
        }
        if (!same) break;
      }
      if (any) {
        leaf_flush<KP, DEG, E>(tr, rec, u, ps, pg, F, acc);
#pragma unroll
        for (int k = 0; k < 3 * NY; ++k) F[k] = 0.f;
        ps = pg = 0.f;
        got = true;
      }
    }
  }
  has[threadIdx.x] = (got ? 1 : 0) | (before ? 2 : 0);
  if (a.touched && !ad.on) {
    const unsigned bits = __ballot_sync(0xFFFFFFFFu, got);
    if ((threadIdx.x & 31) == 0 && bits) atomicOr(a.touched + (leaf >> 5), bits);
  }
  __syncthreads();
  const int rows_here = (int)min((long long)blockDim.x, tr.n_leaves - first);
  if (!ad.on) {
    // add the block's records to the gradient buffer, 16 bytes per thread
    for (int q = threadIdx.x; q < rows_here * Q4; q += blockDim.x) {
      const int r = q / Q4, v = q - r * Q4;
      if (!has[r]) continue;
      const float *src = acc_s + r * PITCH + 4 * v;
      float4 *dst = reinterpret_cast<float4 *>(a.grad + (size_t)(first + r) * a.grad_stride) + v;
      float4 g = *dst;
      g.x += src[0];
      if (4 * v + 1 < LEN) g.y += src[1];
      if (4 * v + 2 < LEN) g.z += src[2];
      if (4 * v + 3 < LEN) g.w += src[3];
      *dst = g;
    }
    return;
  }
  // each warp takes kER rows of the block together (r, r + nw, ...: their
  // loads in flight at once), a lane one 4-entry quad of each
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const float lr_c1 = ad.lr / ad.c1, inv_c2 = 1.f / ad.c2;
  float *__restrict__ mst = ad.master;
  float *__restrict__ mom = ad.m;
  float *__restrict__ vel = ad.v;
  constexpr int QR = (Q4 + 31) / 32;  // quads of a row per lane
  constexpr int kER = 4;
  for (int r0 = threadIdx.x >> 5; r0 < rows_here; r0 += kER * nw) {
    int rr[kER], h[kER], any = 0;
#pragma unroll
    for (int e = 0; e < kER; ++e) {
      rr[e] = r0 + e * nw;
      h[e] = rr[e] < rows_here ? has[rr[e]] : 0;
      any |= h[e];
    }
    if (!any) continue;  // the same for the whole warp
    float4 g[kER][QR], w[kER][QR], m[kER][QR], v[kER][QR];
#pragma unroll
    for (int e = 0; e < kER; ++e)
#pragma unroll
      for (int k = 0; k < QR; ++k) {
        const int q = lane + 32 * k;
        if (!h[e] || q >= Q4) continue;
        const size_t row = (size_t)(first + rr[e]) * a.grad_stride;
        const float *src = acc_s + rr[e] * PITCH + 4 * q;
        g[e][k] = make_float4(src[0], 4 * q + 1 < LEN ? src[1] : 0.f, 4 * q + 2 < LEN ? src[2] : 0.f,
                              4 * q + 3 < LEN ? src[3] : 0.f);
        if (h[e] & 2) {
          float4 *gp = reinterpret_cast<float4 *>(a.grad + row) + q;
          const float4 x = *gp;
          g[e][k].x += x.x;
          g[e][k].y += x.y;
          g[e][k].z += x.z;
          g[e][k].w += x.w;
          *gp = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        w[e][k] = __ldcs(reinterpret_cast<const float4 *>(mst + row) + q);
        m[e][k] = __ldcs(reinterpret_cast<const float4 *>(mom + row) + q);
        v[e][k] = __ldcs(reinterpret_cast<const float4 *>(vel + row) + q);
      }
#pragma unroll
    for (int e = 0; e < kER; ++e) {
      if (!h[e]) continue;
      const size_t row = (size_t)(first + rr[e]) * a.grad_stride;
      float mx0 = 0.f, mx1 = 0.f, mx2 = 0.f;  // FP8: largest magnitudes of w_sigma, w_gamma, w_hh
      float wq[QR][4];
#pragma unroll
      for (int k = 0; k < QR; ++k) {
        const int q = lane + 32 * k;
        if (q >= Q4) continue;
        float gs[4] = {g[e][k].x, g[e][k].y, g[e][k].z, g[e][k].w};
        float ws[4] = {w[e][k].x, w[e][k].y, w[e][k].z, w[e][k].w};
        float ms[4] = {m[e][k].x, m[e][k].y, m[e][k].z, m[e][k].w};
        float vs[4] = {v[e][k].x, v[e][k].y, v[e][k].z, v[e][k].w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int j = 4 * q + c;
          if (j >= LEN) continue;  // padding stays zero
          adam_entry(gs[c], ad.b1, ad.b2, lr_c1, inv_c2, ad.eps, ws[c], ms[c], vs[c]);
          const float aw = fabsf(ws[c]);
          if (j < KP) mx0 = fmaxf(mx0, aw);
          else if (j < 2 * KP) mx1 = fmaxf(mx1, aw);
          else mx2 = fmaxf(mx2, aw);
        }
        __stcs(reinterpret_cast<float4 *>(mst + row) + q, make_float4(ws[0], ws[1], ws[2], ws[3]));
        __stcs(reinterpret_cast<float4 *>(mom + row) + q, make_float4(ms[0], ms[1], ms[2], ms[3]));
        __stcs(reinterpret_cast<float4 *>(vel + row) + q, make_float4(vs[0], vs[1], vs[2], vs[3]));
#pragma unroll
        for (int c = 0; c < 4; ++c) wq[k][c] = ws[c];
        if (ad.dt == kBF16) {
          unsigned short *st = static_cast<unsigned short *>(ad.storage) + (size_t)(first + rr[e]) * ad.storage_stride;
          const unsigned int lo16 = f32_to_bf16_rne(ws[0]) | ((unsigned int)f32_to_bf16_rne(ws[1]) << 16);
          const unsigned int hi16 = f32_to_bf16_rne(ws[2]) | ((unsigned int)f32_to_bf16_rne(ws[3]) << 16);
          __stcs(reinterpret_cast<uint2 *>(st + 4 * q), make_uint2(lo16, hi16));
        }
      }
      if (ad.dt == kFP8) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          mx0 = fmaxf(mx0, __shfl_xor_sync(0xFFFFFFFFu, mx0, o));
          mx1 = fmaxf(mx1, __shfl_xor_sync(0xFFFFFFFFu, mx1, o));
          mx2 = fmaxf(mx2, __shfl_xor_sync(0xFFFFFFFFu, mx2, o));
        }
        const int p[3] = {fp8_scale_exp(mx0), fp8_scale_exp(mx1), fp8_scale_exp(mx2)};
        unsigned char *rec = static_cast<unsigned char *>(ad.storage) + (size_t)(first + rr[e]) * ad.storage_stride;
        if (lane == 0)
          *reinterpret_cast<uint4 *>(rec) = make_uint4(__float_as_uint(ldexpf(1.f, p[0])),
                                                       __float_as_uint(ldexpf(1.f, p[1])),
                                                       __float_as_uint(ldexpf(1.f, p[2])), 0u);
#pragma unroll
        for (int k = 0; k < QR; ++k) {
          const int q = lane + 32 * k;
          if (q >= Q4) continue;
          unsigned int word = 0;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int j = 4 * q + c;
            if (j >= LEN) continue;
            const int pe = j < KP ? p[0] : (j < 2 * KP ? p[1] : p[2]);
            word |= (unsigned int)__nv_cvt_float_to_fp8(ldexpf(wq[k][c], -pe), __NV_SATFINITE, __NV_E4M3) << (8 * c);
          }
          *reinterpret_cast<unsigned int *>(rec + 16 + 4 * q) = word;
        }
      }
    }
  }
}

template <int KP, int DEG>
__host__ __device__ constexpr size_t reduce_smem_bytes(int block) {
  return (size_t)block * (reduce_pitch<KP, DEG>() * sizeof(float) + sizeof(int));
}

template <int KP, int DEG, typename E>
static cudaError_t bwd_one(bool packet, const BwdArgs &a, const LaunchCfg &cfg, cudaStream_t s, const AdamArgs *adam,
                           bool *fused) {
  if (fused) *fused = false;
  if (a.rays.n == 0) return cudaSuccess;
  const long long blocks = (a.rays.n + cfg.block - 1) / cfg.block;
  if (!packet) {
    render_bwd_plain_kernel<KP, DEG, E><<<(unsigned)blocks, cfg.block, 0, s>>>(a);
  } else {
    const size_t sm = smem_bytes(cfg.block, KP, 0, path_words(a.tr));
    if (sm > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(render_bwd_packet_kernel<KP, DEG, E>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (e != cudaSuccess) return e;
    }
    const long long nl = a.tr.n_leaves;
    const bool gather = a.log.n_chunks && a.gws.cap_chunks && nl > 0;
    // The atomic scatter takes the packets in key order, so that the views'
    // packets over one region run together and share records and gradient
    // lines in L2.  The leaf-major reduction takes them in ray order (the
    // views one after another): a leaf's run then holds each view's samples
    // together, and the per-leaf pass expands one group of equal u at a time
    // (6.4-6.5 against 6.7 ms for the 8-view call).
    BwdArgs b = a;
    b.key_order = gather ? 0 : 1;
    if (a.log.n_chunks && b.key_order) {
      // packets in key order (a permutation whatever the log holds; the
      // adjoint uses it only when the log belongs to these rays)
      cudaError_t e = sort_packets_by_key(a.log, (a.rays.n + 31) >> 5, a.tr.n_leaves, cfg.num_sms, s);
      if (e != cudaSuccess) return e;
    }
    if (gather) {
      // samples per leaf counted over the log, scanned into the first
      // position of each leaf's run; the replay advances a copy of them
      cudaError_t e = cudaMemsetAsync(a.gws.off, 0, (size_t)(nl + 1) * sizeof(uint32_t), s);
      if (e != cudaSuccess) return e;
      leaf_count_kernel<<<(unsigned)(16 * cfg.num_sms), 256, 0, s>>>(a);
      if ((e = launch_exclusive_scan(a.gws.off, nl, a.gws.part, cfg.num_sms, s)) != cudaSuccess) return e;
      e = cudaMemcpyAsync(a.gws.cur, a.gws.off, (size_t)(nl + 1) * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
      if (e != cudaSuccess) return e;
    }
    render_bwd_packet_kernel<KP, DEG, E><<<(unsigned)blocks, cfg.block, sm, s>>>(b);
    if (gather) {
      // the per-leaf sums over each leaf's run
      AdamArgs ad{};
      if (adam && adam->on) ad = *adam;
      constexpr int kReduceBlock = 64;
      const size_t rsm = reduce_smem_bytes<KP, DEG>(kReduceBlock);
      if (rsm > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(leaf_reduce_kernel<KP, DEG, E>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rsm);
        if (e != cudaSuccess) return e;
      }
      leaf_reduce_kernel<KP, DEG, E><<<(unsigned)((nl + kReduceBlock - 1) / kReduceBlock), kReduceBlock, rsm, s>>>(a,
                                                                                                                 ad);
      if (ad.on) {
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (a.touched && (e = cudaMemsetAsync(a.touched, 0, (size_t)((nl + 31) / 32) * 4, s)) != cudaSuccess)
          return e;
        if (fused) *fused = true;
      }
    }
  }
  return cudaGetLastError();
}

template <typename E>
static cudaError_t bwd_dispatch(int KP, int DEG, bool packet, const BwdArgs &a, const LaunchCfg &cfg, cudaStream_t s,
                                const AdamArgs *adam, bool *fused) {
  switch (KP * 10 + DEG) {
    case 81: return bwd_one<8, 1, E>(packet, a, cfg, s, adam, fused);
    case 82: return bwd_one<8, 2, E>(packet, a, cfg, s, adam, fused);
    case 83: return bwd_one<8, 3, E>(packet, a, cfg, s, adam, fused);
    case 161: return bwd_one<16, 1, E>(packet, a, cfg, s, adam, fused);
    case 162: return bwd_one<16, 2, E>(packet, a, cfg, s, adam, fused);
    case 163: return bwd_one<16, 3, E>(packet, a, cfg, s, adam, fused);
    case 321: return bwd_one<32, 1, E>(packet, a, cfg, s, adam, fused);
    case 322: return bwd_one<32, 2, E>(packet, a, cfg, s, adam, fused);
    case 323: return bwd_one<32, 3, E>(packet, a, cfg, s, adam, fused);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_render_bwd(int KP, int DEG, DType dt, bool packet, const BwdArgs &a, const LaunchCfg &cfg,
                              cudaStream_t s, const AdamArgs *adam, bool *fused) {
  if (dt == kF32) return bwd_dispatch<float>(KP, DEG, packet, a, cfg, s, adam, fused);
  if (dt == kBF16) return bwd_dispatch<__nv_bfloat16>(KP, DEG, packet, a, cfg, s, adam, fused);
  if (KP == 8 && DEG == 2) return bwd_one<8, 2, Fp8E4M3>(packet, a, cfg, s, adam, fused);
  if (KP == 16 && DEG == 3) return bwd_one<16, 3, Fp8E4M3>(packet, a, cfg, s, adam, fused);
  return cudaErrorInvalidValue;
}

}  // namespace neuvv
