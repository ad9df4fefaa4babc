// One ray through one VOctree: the forward integrator shared by the render and
// compose kernels (Sec. 4.3 "Rendering"; Eq. volume-rendering).
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

// Composites front to back along a started walk, stopping after the segment
// that brings the transmittance below t_stop.  dn: unit direction in the
// tree's frame (the view direction of the harmonics); u: frame coordinate;
// t_base + dist_scale * t converts a walk distance t to the caller's frame.
template <int KP, int DEG, typename E>
__device__ __forceinline__ void integrate_walk(const DevTree &tr, RayWalk &w,
                                               const float dn[3], float u, float t_stop, int act, float t_base,
                                               float dist_scale, RayResult &res) {
  RayConst<KP, DEG> rc;
  ray_const_basis<KP, DEG>(tr, u, rc);
  sh_real<DEG>(dn, rc.Y);
  float T = 1.f;
  uint32_t leaf;
  float t0, dt;
  while (walk_next(tr, w, leaf, t0, dt)) {
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
      res.dnum = fmaf(wgt, fmaf(dist_scale, fmaf(0.5f, dt, t0), t_base), res.dnum);
      res.tau += sd;
      T *= e;
      if (T < t_stop) break;
    }
  }
}

__device__ __forceinline__ void clear(RayResult &res) {
  res.C[0] = res.C[1] = res.C[2] = 0.f;
  res.A = 0.f;
  res.dnum = 0.f;
  res.tau = 0.f;
  res.nseg = 0;
}

// One ray given in the tree's own frame (render kernels).
template <int KP, int DEG, typename E>
__device__ __forceinline__ void integrate_ray(const DevTree &tr, const float o[3],
                                              const float d[3], float u, float t_stop, int act, RayResult &res) {
  clear(res);
  RayWalk w;
  float dn[3];
  if (!walk_init(tr, o, d, w, dn)) return;
  integrate_walk<KP, DEG, E>(tr, w, dn, u, t_stop, act, w.t_base, 1.f, res);
}

// ---------------------------------------------------------------------------
// Packets: the 32 rays of a warp walk independently, and the segments they
// find wait in one ring of the warp.  A batch of up to 32 waiting segments is
// evaluated one per lane whichever rays they belong to -- a sample is some
// six hundred instructions, and packets of uneven or incoherent rays would
// run them with few lanes active if each lane shaded its own ray's segments
// only -- and each ray then composites its own entries of the batch in order.
// ---------------------------------------------------------------------------
constexpr unsigned kFull = 0xFFFFFFFFu;

// Pointers into a packet kernel's dynamic shared memory (kPacketWords).
template <int KP>
struct PacketShared {
  uint4 *ring;      // [kRing] leaf, chord, distance of its middle, lane of the ray
  unsigned *own;    // [32] entries of the batch that belong to each lane's ray
  float2 *res;      // [32] per entry of the batch (the adjoint)
  float *dn, *rows; // unit direction and basis rows of lane 0's ray; next lane +1, next value +stride
  uint32_t *path;   // this thread's descent path, next level +stride
  int stride;
  __device__ __forceinline__ explicit PacketShared(uint32_t *smem) {
    const int B = blockDim.x, w0 = threadIdx.x & ~31;
    ring = reinterpret_cast<uint4 *>(smem) + 2 * w0;
    uint32_t *p = smem + 4 * kRing / 32 * B;
    own = p + w0;
    res = reinterpret_cast<float2 *>(p + B) + w0;
    dn = reinterpret_cast<float *>(p + 3 * B) + w0;
    rows = reinterpret_cast<float *>(p + 6 * B) + w0;
    path = p + (6 + 2 * KP) * B + threadIdx.x;
    stride = B;
  }
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
  // of `owner` in lane j when has).
  __device__ __forceinline__ unsigned entries_of_lane(bool has, int owner) const {
    const int lane = threadIdx.x & 31;
    const unsigned grp = __match_any_sync(kFull, has ? owner : 32 + lane);
    own[lane] = 0u;
    __syncwarp();
    if (has && lane == __ffs(grp) - 1) own[owner] = grp;
    __syncwarp();
    return own[lane];
  }
};

__device__ __forceinline__ float depth_of(const RayResult &r) { return r.A >= 1e-4f ? r.dnum / r.A : INFINITY; }

}  // namespace neuvv
