// Rays through one VOctree (Sec. 4.3 "Rendering"; Eq. volume-rendering): the
// integrator of one thread per ray (the plain kernel), and the packets' ring and
// batch shading shared by the packet forward, the adjoint and composition.
#pragma once

#include "neuvv_kernels.h"

namespace neuvv {

struct RayResult {
  float C[3];    // premultiplied colour, sum w_i c_i
  float A;       // alpha, sum w_i
  float dnum;    // sum w_i t_mid,i (world distance from the ray origin)
  float tau;     // sum sigma_i delta_i
  int nseg;      // composited segments
};

// One ray given in the tree's own frame, composited front to back up to and
// including the segment that brings the transmittance below t_stop.  u: frame
// coordinate.  One loop over walk steps with the sample inside it: lanes of a
// warp keep stepping together and meet at the loop's head, where a search for
// the next segment nested in a loop over segments made each lane wait for the
// slowest search of every segment (1080p view of a depth-8 shell, 500,000 leaves,
// K_pad 8 BF16: 0.86 of the time before the mirrored walk against 1.11 nested).
template <int KP, int DEG, typename E>
__device__ __forceinline__ void integrate_ray(const DevTree &tr, const float o[3],
                                              const float d[3], float u, float t_stop, int act, RayResult &res) {
  res.C[0] = res.C[1] = res.C[2] = 0.f;
  res.A = res.dnum = res.tau = 0.f;
  res.nseg = 0;
  RayWalk w;
  float dn[3];
  if (!walk_init(tr, o, d, w, dn)) return;
  RayConst<KP, DEG> rc;
  ray_const_basis<KP, DEG>(tr, u, rc);
  sh_real<DEG>(dn, rc.Y);
  float T = 1.f;
  uint32_t leaf;
  float t0, dt;
  while (w.alive) {
    if (!walk_step(tr, w, leaf, t0, dt)) continue;
    LeafRecord<KP, DEG, E> rec;
    rec.load(tr, leaf);
    Sample<DEG> s;
    eval_sample<KP, DEG, E>(tr, rc, rec, act, s);
    res.nseg += 1;
    if (s.sigma > 0.f) {
      const float sd = s.sigma * dt;
      const float e = __expf(-sd);
      const float wgt = T * alpha_of(sd);
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) res.C[ch] = fmaf(wgt, s.c[ch], res.C[ch]);
      res.A += wgt;
      res.dnum = fmaf(wgt, w.t_base + fmaf(0.5f, dt, t0), res.dnum);
      res.tau += sd;
      T *= e;
      if (T < t_stop) break;
    }
  }
}

// ---------------------------------------------------------------------------
// Packets: the 32 rays of a warp walk independently, and the segments they
// find wait in one ring of the warp.  A batch of up to 32 waiting segments is
// evaluated one per lane whichever rays they belong to -- a sample is some
// six hundred instructions, and packets of uneven or incoherent rays would
// run them with few lanes active if each lane shaded its own ray's segments
// only -- and each ray then composites its own entries of the batch in order.
// Against a queue per ray, lanes active per instruction, walk included: 1080p view
// 21.7 -> 26.6 of 32; 262,144 rays in drawn order 5.2 -> 13.2 in the forward and
// 5.7 -> 25.4 in the adjoint, training step 3.25 -> 1.24 ms.
// ---------------------------------------------------------------------------
constexpr unsigned kFull = 0xFFFFFFFFu;

// Whether a segment log was written by a forward over n rays.
__device__ __forceinline__ bool log_matches(const SampleLog &l, long long n) {
  return __ldg(l.header + 4) == 1u && __ldg(l.header) == l.n_chunks && __ldg(l.header + 1) == (uint32_t)kLogRounds &&
         __ldg(l.header + 2) == (uint32_t)(n & 0xFFFFFFFFll) && __ldg(l.header + 3) == (uint32_t)(n >> 32) &&
         __ldg(l.header + 9) == l.layout();
}
// Leaf and lane of a slot of the log.
struct LogWord {
  uint32_t leaf;
  int lane;
  bool empty;
};
__device__ __forceinline__ LogWord log_word(const SampleLog &l, size_t slot) {
  const uint32_t w = __ldcs(l.leaf + slot);
  if (l.lane) return LogWord{w, (int)__ldcs(l.lane + slot) & 31, w == kEmpty};
  return LogWord{w >> 5, (int)(w & 31u), w == kEmpty};
}

// Asynchronous 16-byte copy from global to shared memory (past L1), and the
// wait for this thread's copies.
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Pointers into a packet kernel's dynamic shared memory (kPacketWords); CHUNKS:
// 16-byte chunks of the records that are staged (0: none are).
template <int KP, int CHUNKS>
struct PacketShared {
  static constexpr bool kStaged = CHUNKS > 0;
  static constexpr int kPitch = stage_pitch(CHUNKS);
  uint4 *ring;      // [kRing] leaf, chord, distance of its middle, lane of the ray
  uint4 *stage;     // [32][kPitch] records of a batch
  unsigned *own;    // [32] entries of the batch that belong to each lane's ray
  float2 *res;      // [32] per entry of the batch (the adjoint)
  float *dn, *rows; // unit direction and basis rows of lane 0's ray; next lane +1, next value +stride
  uint32_t *path;   // this thread's descent path, next level +stride
  int stride;
  __device__ __forceinline__ explicit PacketShared(uint32_t *smem) {
    const int B = blockDim.x, w0 = threadIdx.x & ~31;
    ring = reinterpret_cast<uint4 *>(smem) + 2 * w0;
    uint32_t *p = smem + 4 * kRing / 32 * B;
    stage = reinterpret_cast<uint4 *>(p) + kPitch * w0;
    p += 4 * kPitch * B;
    own = p + w0;
    res = reinterpret_cast<float2 *>(p + B) + w0;
    dn = reinterpret_cast<float *>(p + 3 * B) + w0;
    rows = reinterpret_cast<float *>(p + 6 * B) + w0;
    path = p + (6 + 2 * KP) * B + threadIdx.x;
    stride = B;
  }
  // Starts copying the records of a batch (lane j: entry j's leaf; count
  // entries) into the staging area.  A group of kGroup lanes takes one record,
  // a lane a chunk, so a warp's load covers whole lines (each lane reading its
  // own record 16 bytes at a time touches 32 lines per load; those wavefronts
  // kept L1 at 56 % of its peak in the 1080p forward, against 18 % now).  The
  // copies run while the rays walk on.  Lanes without an entry pass leaf 0.
  static constexpr int kGroup = CHUNKS > 16 ? 32 : (CHUNKS > 8 ? 16 : 8);
  __device__ __forceinline__ void stage_records(const void *base, uint32_t rec_bytes, uint32_t leaf, int count) const {
    const int lane = threadIdx.x & 31, c = lane % kGroup, r0 = lane / kGroup;
    constexpr int kPer = 32 / kGroup;  // records per step
    const char *src = static_cast<const char *>(base) + 16 * c;
    uint4 *dst = stage + r0 * kPitch + c;
#pragma unroll
    for (int k0 = 0; k0 < kGroup; k0 += 4) {
      if (k0 * kPer >= count) break;  // uniform; at most 4 steps past a short batch
#pragma unroll
      for (int k = k0; k < k0 + 4; ++k) {
        const uint32_t lf = __shfl_sync(kFull, leaf, k * kPer + r0);
        if (c < CHUNKS) cp_async16(dst + k * kPer * kPitch, src + (unsigned long long)lf * rec_bytes);
      }
    }
  }
  // Waits for the staged records (all lanes' copies).
  __device__ __forceinline__ void staged_wait() const {
    cp_async_wait();
    __syncwarp();
  }
  __device__ __forceinline__ const uint4 *staged_record() const { return stage + (threadIdx.x & 31) * kPitch; }
  // This thread's ray, for the batch evaluation (any lane may shade it).
  __device__ __forceinline__ void put_ray(const DevTree &tr, const float d[3], float u, bool with_rows) const {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 3; ++k) dn[k * stride + lane] = d[k];
    if (with_rows) rows_to_smem<KP>(tr, u, rows + lane, stride);
  }
  __device__ __forceinline__ void get_dir(int lane, float d[3]) const {
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] = dn[k * stride + lane];
  }
  __device__ __forceinline__ SmemRows<KP> rows_of(int lane) const { return SmemRows<KP>{rows + lane, stride}; }
  // Entries of the batch that belong to this lane's ray, as a mask (entry j
  // of `owner` in lane j when has).  Collected with shared-memory atomics: a
  // match over the warp took some 5 % of a call whose packets are coherent (1080p
  // view of a depth-7 solid, K_pad 8 BF16, 1.02 -> 0.95 of the time with a queue per
  // ray; density alone 1.05 -> 0.91; depth-8 shell 0.85 -> 0.82).
  __device__ __forceinline__ unsigned entries_of_lane(bool has, int owner) const {
    const int lane = threadIdx.x & 31;
    own[lane] = 0u;
    __syncwarp();
    if (has) atomicOr(own + owner, 1u << lane);
    __syncwarp();
    return own[lane];
  }
};

// What a batch is shaded from: kShadeTree (the tree's records), kShadeSlice (a
// time slice), kShadeEdit (the tree's records with appearance edits) or
// kShadeAlpha (density only: the w_sigma part of each record is read, colour
// is neither evaluated nor written; alpha, depth, tau and nseg are those of
// the full render) or kShadePick (density only: the leaf at which the ray's
// opacity first reaches t_stop, in RayAccum::nseg).
constexpr int kShadeTree = 0, kShadeSlice = 1, kShadeEdit = 2, kShadeAlpha = 3, kShadePick = 4;
__host__ __device__ constexpr bool density_only(int shade) { return shade == kShadeAlpha || shade == kShadePick; }
template <int KP, int DEG, typename E, int kShade>
__host__ __device__ constexpr int shade_chunks() {
  // slice rows are small, and a density-only batch reads few chunks: in place
  return kShade == kShadeSlice || density_only(kShade) ? 0 : stage_chunks<KP, DEG, E>();
}
struct Shading {
  int act;
  float t_stop;
  const float *slice;  // kShadeSlice: [n_leaves][slice_stride]
  int slice_stride;
  const float *edits;  // kShadeEdit: [n_leaves][8], blended by edit_beta
  float edit_beta;
};

// A ray's composited sums.
struct RayAccum {
  float T = 1.f, C[3] = {0.f, 0.f, 0.f}, A = 0.f, dnum = 0.f, tau = 0.f;
  int nseg = 0;
  bool dead = false;  // ended early: its waiting entries are dropped
  __device__ __forceinline__ float depth() const { return A >= 1e-4f ? dnum / A : INFINITY; }
};

// Shades one batch of a packet's ring, called by the whole warp: lane j holds
// entry j (en; has: one of the batch) and evaluates it, whichever ray it
// belongs to; each ray then composites its own entries, oldest first, into acc
// (the values of an entry that compositing needs come by shuffle from its
// lane).  t: the time of this lane's ray.  Returns the mask of the entries
// this lane's ray composited.
// The records are read from the staging area (Sh::kStaged) or in place.
template <int KP, int DEG, typename E, int kShade, typename Sh>
__device__ __forceinline__ unsigned shade_batch(const DevTree &tr, const Sh &sh, const Shading &p,
                                                const uint4 en, bool has, float t, RayAccum &acc) {
  const int lane = threadIdx.x & 31, owner = (int)en.w & 31;
  const float to = kShade == kShadeEdit ? __shfl_sync(kFull, t, owner) : 0.f;
  float sd = 0.f, al = 0.f, ex = 1.f, col[3] = {0.f, 0.f, 0.f};
  if (has) {
    const uint32_t leaf = en.x;
    float sigma, dn[3], Y[(DEG + 1) * (DEG + 1)];
    if (!density_only(kShade)) {
      sh.get_dir(owner, dn);
      sh_real<DEG>(dn, Y);
    }
    if constexpr (kShade == kShadeSlice) {
      shade_slice<DEG>(p.slice, p.slice_stride, leaf, Y, p.act, sigma, col);
    } else if constexpr (density_only(kShade)) {
      LeafRecord<KP, DEG, E> rec;
      rec.load_sigma(tr, leaf);
      sigma = fmaxf(pre_sigma_of<KP>(sh.rows_of(owner), rec), 0.f);
    } else {
      LeafRecord<KP, DEG, E> rec;
      Sample<DEG> s;
      s.c[0] = s.c[1] = s.c[2] = 0.f;
      if constexpr (Sh::kStaged) {
        eval_sample<KP, DEG, E>(tr, sh.rows_of(owner), Y, FromShared{sh.staged_record()}, rec, p.act, s);
      } else {
        rec.load(tr, leaf);
        eval_sample<KP, DEG, E>(tr, sh.rows_of(owner), Y, Loaded{}, rec, p.act, s);
      }
      sigma = s.sigma;
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) col[ch] = s.c[ch];
      if constexpr (kShade == kShadeEdit) {
        // appearance edit of the voxel, active from its time t_d on
        const float4 e0 = __ldg(reinterpret_cast<const float4 *>(p.edits) + 2 * (size_t)leaf);
        const float4 e1 = __ldg(reinterpret_cast<const float4 *>(p.edits) + 2 * (size_t)leaf + 1);
        if (to >= e1.x) {
          if (e0.w >= 0.f) sigma = e0.w;
          col[0] = fmaf(p.edit_beta, e0.x - col[0], col[0]);
          col[1] = fmaf(p.edit_beta, e0.y - col[1], col[1]);
          col[2] = fmaf(p.edit_beta, e0.z - col[2], col[2]);
        }
      }
    }
    if constexpr (kShade == kShadePick) {
      sd = sigma;
    } else if (sigma > 0.f) {
      sd = sigma * __uint_as_float(en.y);
      ex = __expf(-sd);
      al = alpha_of(sd);
    } else {  // no contribution: weight 0, colour unused
      col[0] = col[1] = col[2] = 0.f;
    }
  }
  unsigned mine = sh.entries_of_lane(has, owner), kept = 0u;
  if (acc.dead) mine = 0u;
  if constexpr (kShade == kShadePick) {
    while (__any_sync(kFull, mine != 0u)) {
      const int j = mine ? __ffs(mine) - 1 : lane;
      const float x_sigma = __shfl_sync(kFull, sd, j), x_dt = __shfl_sync(kFull, __uint_as_float(en.y), j);
      const uint32_t x_leaf = __shfl_sync(kFull, en.x, j);
      if (mine) {
        mine &= mine - 1u;
        acc.tau = fmaf(x_sigma, x_dt, acc.tau);
        if (-expm1f(-acc.tau) >= p.t_stop) {
          acc.nseg = (int)x_leaf;
          acc.dead = true;
          mine = 0u;
        }
      }
    }
    return 0u;
  }
  while (__any_sync(kFull, mine != 0u)) {
    const int j = mine ? __ffs(mine) - 1 : lane;
    const float x_al = __shfl_sync(kFull, al, j), x_ex = __shfl_sync(kFull, ex, j);
    const float x_sd = __shfl_sync(kFull, sd, j), x_tm = __shfl_sync(kFull, __uint_as_float(en.z), j);
    float x_c[3] = {0.f, 0.f, 0.f};
    if (!density_only(kShade)) {
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) x_c[ch] = __shfl_sync(kFull, col[ch], j);
    }
    if (mine) {
      mine &= mine - 1u;
      kept |= 1u << j;
      ++acc.nseg;
      const float wgt = acc.T * x_al;
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) acc.C[ch] = fmaf(wgt, x_c[ch], acc.C[ch]);
      acc.A += wgt;
      acc.dnum = fmaf(wgt, x_tm, acc.dnum);
      acc.tau += x_sd;
      acc.T *= x_ex;
      if (acc.T < p.t_stop) {
        acc.dead = true;
        mine = 0u;
      }
    }
  }
  return kept;
}

__device__ __forceinline__ float depth_of(const RayResult &r) { return r.A >= 1e-4f ? r.dnum / r.A : INFINITY; }

}  // namespace neuvv
