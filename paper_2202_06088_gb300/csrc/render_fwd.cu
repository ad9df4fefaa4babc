// Forward render and trace kernels (Sec. 4.3 "Rendering").
//
// render_plain_kernel  : one thread per ray, child table read from global
//                        memory -- the baseline single-view path.
// render_packet_kernel : one thread per ray with warps as 32-ray packets;
//                        walking and shading decoupled through one ring of
//                        found segments per packet; descents restart at the
//                        lowest common ancestor of successive cells.
#include "neuvv_kernels.h"
#include "neuvv_ray.cuh"

namespace neuvv {

// Blocks of 128 threads that an SM must hold.  Two record shapes end a few
// registers above what one block more allows (171 of 168, 130 of 128).
template <int KP, int DEG, typename E>
constexpr int plain_min_blocks() {
  if (KP == 8 && DEG == 3 && sizeof(E) == 4) return 3;
  return KP == 32 && DEG == 1 && sizeof(E) == 2 ? 4 : 0;
}
template <int KP, int DEG, typename E>
constexpr int plain_max_threads() { return plain_min_blocks<KP, DEG, E>() ? 128 : 256; }

template <int KP, int DEG, typename E>
__global__ void __launch_bounds__(plain_max_threads<KP, DEG, E>(), plain_min_blocks<KP, DEG, E>())
    render_plain_kernel(const __grid_constant__ FwdArgs a) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.rays.n) return;
  float o[3], d[3], t;
  load_ray(a.rays, i, o, d, t);
  RayResult r;
  integrate_ray<KP, DEG, E>(a.tr, o, d, t * (float)(a.tr.T - 1), a.t_stop, a.act, r);
  a.out.rgb[3 * i + 0] = r.C[0];
  a.out.rgb[3 * i + 1] = r.C[1];
  a.out.rgb[3 * i + 2] = r.C[2];
  a.out.alpha[i] = r.A;
  if (a.out.depth) a.out.depth[i] = depth_of(r);
  if (a.out.tau) a.out.tau[i] = r.tau;
  if (a.out.nseg) a.out.nseg[i] = r.nseg;
}

// Outputs and the segment log are written once and read by later launches:
// stores with the evict-first (streaming) policy.
__device__ __forceinline__ void write_miss(const DevOut &out, long long i) {
  if (out.rgb) {
    __stcs(out.rgb + 3 * i + 0, 0.f);
    __stcs(out.rgb + 3 * i + 1, 0.f);
    __stcs(out.rgb + 3 * i + 2, 0.f);
  }
  __stcs(out.alpha + i, 0.f);
  if (out.depth) __stcs(out.depth + i, INFINITY);
  if (out.tau) __stcs(out.tau + i, 0.f);
  if (out.nseg) __stcs(out.nseg + i, 0);
}

// Packet forward kernel: one thread per ray, so each warp is a packet of 32
// consecutive rays (an 8x4 pixel tile when the caller orders rays that way).
// Walking and shading are decoupled: in every iteration of one warp-uniform
// loop each lane takes at most one walk step, and the occupied-leaf segments
// found join the packet's ring.  Once kBatch segments wait, or no ray can step
// any further, the warp shades a batch of up to 32 of them, one per lane
// whichever rays they belong to, and each ray composites its own entries in
// order (a shuffle of the seven values that compositing needs per entry).
// Shading rounds therefore run full even where the packet's rays are uneven:
// one long ray among finished ones shades up to 32 of its own segments at once.
// Descents restart at the lowest common ancestor of successive cells (path per
// thread in shared memory); basis rows and directions live in shared memory.
// CHUNKS: chunks of the records that are staged (0: read in place).
template <int KP, int DEG, typename E, int kShade, int CHUNKS>
__device__ __forceinline__ void packet_forward(const FwdArgs &a, long long pk, int split, int part, long long n_live) {
  extern __shared__ __align__(16) uint32_t smem[];
  const DevTree &tr = a.tr;
  const int lane = threadIdx.x & 31;
  using Shared = PacketShared<KP, CHUNKS>;
  const Shared sh(smem);
  const PathRef pr{sh.path, sh.stride};
  // the warp holds 32 >> split of the packet's rays, in its first lanes
  const long long pos = (pk << 5) + (part << (5 - split)) + lane;
  // i: the ray (its data and outputs); pos: its position (packet pos >> 5, lane)
  const bool live = lane < (32 >> split) && pos < n_live;
  const long long i = live && a.perm ? (long long)min(__ldg(a.perm + pos), (uint32_t)(a.rays.n - 1)) : pos;
  float t = 0.f;
  RayWalk w;
  w.alive = false;
  bool hit = false;
  if (live) {
    float o[3], d[3], dn[3];
    load_ray(a.rays, i, o, d, t);
    hit = walk_init(tr, o, d, w, dn);
    if (hit) sh.put_ray(tr, dn, t * (float)(tr.T - 1), kShade != kShadeSlice);
    else if (kShade == kShadePick) __stcs(a.out.nseg + i, -1);
    else write_miss(a.out, i);
  }
  if (a.log.n_chunks && lane == 0) {
    a.log.key[pk] = kNoKey;
    a.log.heads[pk] = kNoLog;  // until the packet's first chunk
  }
  if (!__any_sync(kFull, hit)) return;  // the whole packet missed the tree
  const Shading shading{a.act, a.t_stop, a.slice, a.slice_stride, a.edits, a.edit_beta};
  RayAccum acc;
  if (kShade == kShadePick) acc.nseg = -1;
  bool walking = hit && w.alive;
  int head = 0, count = 0;  // the ring's oldest entry and length (warp-uniform)
  uint4 en = make_uint4(0u, 0u, 0u, 0u);  // this lane's entry of the batch to shade next
  bool has = false, pending = false;
  // segment log of this packet (warp-uniform state): current chunk and round
  bool logging = a.log.n_chunks != 0;
  uint32_t chunk = kNoLog;
  int round = kLogRounds;
  for (;;) {
    uint32_t leaf = 0u;
    float t0 = 0.f, dt = 0.f;
    bool found = false;
    if (walking) {
      found = walk_step<true>(tr, w, leaf, t0, dt, pr);
      walking = w.alive;
    }
    const unsigned finds = __ballot_sync(kFull, found);
    if (found) {
      const int slot = (head + count + __popc(finds & ((1u << lane) - 1u))) & (kRing - 1);
      sh.ring[slot] = make_uint4(leaf, __float_as_uint(dt), __float_as_uint(w.t_base + fmaf(0.5f, dt, t0)), lane);
      if (!Shared::kStaged) {  // the record is read when the segment's batch comes: ask L2 for it now
        if (kShade == kShadeSlice) slice_prefetch_l2(a.slice, a.slice_stride, DEG, leaf);
        else if (density_only(kShade)) LeafRecord<KP, DEG, E>::prefetch_sigma_l2(tr, leaf);
        else LeafRecord<KP, DEG, E>::prefetch_l2(tr, leaf);
      }
    }
    count += __popc(finds);
    if (count < kBatch && __any_sync(kFull, walking)) continue;
    // the next batch: with staging its records are on their way while the
    // rays walk on, and it is shaded when the one after it is complete
    __syncwarp();
    const int batch = min(count, kBatch);
    const bool next_has = lane < batch;
    const uint4 next_en = sh.ring[(head + lane) & (kRing - 1)];
    if (!Shared::kStaged) {
      en = next_en;
      has = next_has;
      pending = batch > 0;
    }
    unsigned kept = 0u;
    if (pending) {
      if (Shared::kStaged) sh.staged_wait();
      kept = shade_batch<KP, DEG, E, kShade>(tr, sh, shading, en, has, t, acc);
      if (acc.dead) walking = false;  // early termination: what still waits is dropped
    if (logging) {
      if (round == kLogRounds) {  // next chunk: one counter add per 8 rounds
        if (chunk == kNoLog) {  // the packet's sort key: the smallest leaf of its first round
          const uint32_t k = __reduce_min_sync(kFull, has ? en.x : kNoKey);
          if (lane == 0) a.log.key[pk] = k;
        }
        uint32_t nc = kNoLog;
        if (lane == 0) {
          const unsigned long long c = atomicAdd(a.log.counter, 1ull);
          if (c < a.log.n_chunks) {
            nc = (uint32_t)c;
            a.log.next[nc] = kNoLog;  // the chain's end until another chunk follows
            if (chunk == kNoLog) a.log.heads[pk] = nc;
            else a.log.next[chunk] = nc;
          } else {
            a.log.heads[pk] = kNoLog;  // out of room: the adjoint walks this packet
          }
        }
        nc = __shfl_sync(kFull, nc, 0);
        logging = nc != kNoLog;
        chunk = nc;
        round = 0;
      }
      if (logging) {
        // the entries that were composited (a ray that ended drops its later ones)
        const bool keep = (__reduce_or_sync(kFull, kept) >> lane) & 1u;
        const size_t slot = ((size_t)chunk * kLogRounds + round) * 32 + lane;
        __stcs(a.log.leaf + slot, !keep ? kEmpty : (a.log.lane ? en.x : (en.x << 5 | (en.w & 31u))));
        __stcs(a.log.dt + slot, keep ? __uint_as_float(en.y) : 0.f);
        if (a.log.lane) a.log.lane[slot] = (uint8_t)en.w;
        ++round;
      }
    }
    }
    if (batch == 0) break;
    head += batch;
    count -= batch;
    if (Shared::kStaged) {
      __syncwarp();  // every lane has read its staged record
      en = next_en;
      has = next_has;
      pending = true;
      sh.stage_records(tr.rec, LeafRecord<KP, DEG, E>::stride_bytes(tr), has ? en.x : 0u, batch);
    }
  }
  // slots that hold no segment read kEmpty, so that the log can be read slot
  // by slot: the rounds of the last chunk that the packet did not reach
  if (logging && chunk != kNoLog)
    for (int r = round; r < kLogRounds; ++r) a.log.leaf[((size_t)chunk * kLogRounds + r) * 32 + lane] = kEmpty;
  if (!hit) return;
  if (kShade == kShadePick) {
    __stcs(a.out.nseg + i, acc.nseg);
    return;
  }
  if (kShade != kShadeAlpha) {
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) __stcs(a.out.rgb + 3 * i + ch, acc.C[ch]);
  }
  __stcs(a.out.alpha + i, acc.A);
  if (a.out.depth) __stcs(a.out.depth + i, acc.depth());
  if (a.out.tau) __stcs(a.out.tau + i, acc.tau);
  if (a.out.nseg) __stcs(a.out.nseg + i, acc.nseg);
}

// Packet forward kernel.  With a work counter the grid is persistent: each
// warp takes the next 32-ray packet from the counter when it finishes one, so
// a long ray holds up only its own warp, not the other warps of its block.
// Registers: those that packet_min_blocks leaves a block of 256 threads, and 96
// for a density-only shading.  Held to 64 that one spilled the walk's state;
// with 80 the larger K_pad were slower, with 128 the smaller.  Two 1280 x 720
// views of density alone, with 64 -> 96, against the kernel before batches
// (128): depth-8 shell of 500,000 leaves K_pad 16 FP32 degree 3 1.05 -> 0.80, K_pad 8
// BF16 0.91 -> 0.87; depth-7 solid of 160,000 1.32 -> 0.99 and 1.06 -> 1.02.
template <int KP, int DEG, typename E, int kShade>
constexpr int packet_registers() { return density_only(kShade) ? 96 : (packet_min_blocks<KP, DEG, E>() == 2 ? 128 : 255); }
template <int KP, int DEG, typename E, int kShade, int CHUNKS>
__global__ void __maxnreg__((packet_registers<KP, DEG, E, kShade>()))
    render_packet_kernel(const __grid_constant__ FwdArgs a) {
  // one packet per warp of the grid, or (with a work counter) packets pulled
  // one after another until the counter passes the last
  const int lane = threadIdx.x & 31;
  const long long n_live = a.n_live ? (long long)__ldg(a.n_live) : a.rays.n;
  const uint32_t n_first = a.list ? __ldg(a.counts) : 0u;
  const long long n_packets = (n_live + 31) >> 5;
  const long long n_parts = a.list ? (long long)n_first + __ldg(a.counts + 1) : n_packets << a.split;
  if (a.log.n_chunks && blockIdx.x == 0 && threadIdx.x == 0) {
    a.log.header[0] = a.log.n_chunks;
    a.log.header[1] = kLogRounds;
    a.log.header[2] = (uint32_t)(a.rays.n & 0xFFFFFFFFll);
    a.log.header[3] = (uint32_t)(a.rays.n >> 32);
    a.log.header[4] = 1u;
    a.log.header[5] = a.perm ? 1u : 0u;
    a.log.header[9] = a.log.layout();
    if (!a.n_live) {
      a.log.header[6] = (uint32_t)(n_live & 0xFFFFFFFFll);
      a.log.header[7] = (uint32_t)(n_live >> 32);
    }
  }
  long long k = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (a.work) {
    unsigned long long q = 0;
    if (lane == 0) q = atomicAdd(a.work, 1ull);
    k = (long long)__shfl_sync(kFull, q, 0);
  }
  while (k < n_parts) {
    long long pk = k >> a.split;
    int split = a.split, part = (int)(k & ((1 << a.split) - 1));
    if (a.order) {
      pk = (long long)min(__ldg(a.order + k), (uint32_t)(n_packets - 1));
    } else if (a.list) {
      const uint32_t v = __ldg(a.list + (k < n_first ? k : kQueueEntries - 1 - (k - n_first)));
      pk = v & 0xFFFFFu;
      split = (int)(v >> 20) & 3;
      part = (int)(v >> 24);
    }
    packet_forward<KP, DEG, E, kShade, CHUNKS>(a, pk, split, part, n_live);
    __syncwarp();
    if (!a.work) break;
    unsigned long long q = 0;
    if (lane == 0) q = atomicAdd(a.work, 1ull);
    k = (long long)__shfl_sync(kFull, q, 0);
  }
}

// ---------------------------------------------------------------------------
// Triage of a forward call of more packets than warps are resident.  Most
// rays of a view miss the tree (72 % of the 8-view step's), and a packet
// that missed cost the packet kernel a trip to the work counter and to its
// rays; and a single long packet taken late kept a few SMs busy after the
// others had finished (SMs active for 77 % of a 1080p view's time).
// ---------------------------------------------------------------------------

// Packets as given: writes the outputs of packets whose rays all miss the
// box and lists the parts the others are run in.  A packet's work is estimated
// from one point of each of its rays (a different fraction of the way through
// the box for each lane): the brick-map cells that hold something, per ray, as
// 32 such points see them.  Packets of `quarter` or more are run in four
// parts, from `half` in two, these at the front of list (counts[0]) and so
// first; the others whole, from its end backwards (counts[1]).
__global__ void __launch_bounds__(256) triage_packets_kernel(const __grid_constant__ DevTree tr, const DevRays rays,
                                                             const DevOut out, float half, float quarter,
                                                             uint32_t *list, uint32_t *counts) {
  __shared__ int parts[8];  // parts of each of the block's packets (0: none)
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  bool hit = false;
  float cells = 0.f;
  if (i < rays.n) {
    float o[3], d[3], t, s_in, s_out;
    load_ray(rays, i, o, d, t);
    hit = ray_meets_box(tr, o, d, s_in, s_out);
    if (hit) {
      // bit-reversed lane: neighbouring rays look at distant depths
      const float s = fmaf(((float)(__brev((unsigned)lane) >> 27) + 0.5f) * (1.f / 32.f), s_out - s_in, s_in);
      const int Lc = tr.brick_level, mask = (1 << tr.depth) - 1;
      uint32_t idx = 0u;
      float len2 = 0.f;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float g = (fmaf(s, d[a], o[a]) - tr.bmin[a]) * tr.scale[a], e = (s_out - s_in) * d[a] * tr.scale[a];
        idx = (idx << Lc) | (uint32_t)(min(max((int)g, 0), mask) >> kBrickShift);
        len2 = fmaf(e, e, len2);
      }
      if ((__ldg(tr.coarse + idx) >> 28) != kCoarseEmpty) cells = sqrtf(len2) * (1.f / (32 << kBrickShift));
    }
  }
  const unsigned hits = __ballot_sync(kFull, hit);
  if (!hits && i < rays.n) write_miss(out, i);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cells += __shfl_xor_sync(kFull, cells, o);
  if (lane == 0) parts[wid] = !hits ? 0 : (cells >= quarter ? 4 : (cells >= half ? 2 : 1));
  __syncthreads();
  if (wid == 0) {
    // the block's packets in order, one add per count and block
    const int p = lane < 8 ? parts[lane] : 0;
    int incl = p > 1 ? p : 0;
    const unsigned whole = __ballot_sync(kFull, p == 1);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(kFull, incl, 7);
    uint32_t bf = 0u, bl = 0u;
    if (lane == 0) {
      if (total) bf = atomicAdd(counts, (uint32_t)total);
      if (whole) bl = atomicAdd(counts + 1, (uint32_t)__popc(whole));
    }
    bf = __shfl_sync(kFull, bf, 0) + (uint32_t)incl - (uint32_t)p;
    bl = __shfl_sync(kFull, bl, 0) + (uint32_t)__popc(whole & ((1u << lane) - 1u));
    const uint32_t pk = blockIdx.x * 8 + lane;
    if (p == 1) list[kQueueEntries - 1 - bl] = part_entry(pk, 0, 0);
    for (int k = 0; k < p && p > 1; ++k) list[bf + k] = part_entry(pk, p == 4 ? 2 : 1, k);
  }
}

// Calls with a segment log (whose permutation the adjoint follows): packets
// are formed from the rays that meet the box, listed block by block in the
// given order; the others' outputs are written here and they are listed from
// the end of miss_list.  262,144 rays in drawn order: step 1378 -> 1284 us; the
// 8-view step (16.6 M rays, 72 % of them misses) 9.35 -> 9.21 ms.
constexpr int kTriageBlock = 1024;
__global__ void __launch_bounds__(kTriageBlock) triage_rays_kernel(const __grid_constant__ DevTree tr, const DevRays rays,
                                                                   const DevOut out, uint32_t *hit_list,
                                                                   uint32_t *miss_list, uint32_t *n_live,
                                                                   uint32_t *n_miss) {
  __shared__ uint32_t sum[kTriageBlock / 32], base_hit, base_miss;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = i < rays.n;
  bool hit = false;
  if (in) {
    float o[3], d[3], t;
    load_ray(rays, i, o, d, t);
    float s_in, s_out;
    hit = ray_meets_box(tr, o, d, s_in, s_out);
    if (!hit) write_miss(out, i);
  }
  const unsigned hits = __ballot_sync(kFull, hit);
  if (lane == 0) sum[wid] = (uint32_t)__popc(hits);
  __syncthreads();
  if (wid == 0) {
    const uint32_t own = sum[lane];
    uint32_t incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    sum[lane] = incl - own;
    if (lane == 31) {
      const uint32_t rays_here = (uint32_t)min(rays.n - (long long)blockIdx.x * blockDim.x, (long long)kTriageBlock);
      base_hit = incl ? atomicAdd(n_live, incl) : 0u;
      base_miss = rays_here > incl ? atomicAdd(n_miss, rays_here - incl) : 0u;
    }
  }
  __syncthreads();
  if (!in) return;
  const uint32_t before = sum[wid] + (uint32_t)__popc(hits & ((1u << lane) - 1u));  // hits before this ray in the block
  if (hit) hit_list[base_hit + before] = (uint32_t)i;
  else miss_list[rays.n - 1 - (base_miss + (threadIdx.x - before))] = (uint32_t)i;
}

cudaError_t launch_triage_rays(const DevTree &tr, const DevRays &rays, const DevOut &out, uint32_t *hits,
                               uint32_t *misses, uint32_t *n_live, uint32_t *n_miss, cudaStream_t s) {
  triage_rays_kernel<<<(unsigned)((rays.n + kTriageBlock - 1) / kTriageBlock), kTriageBlock, 0, s>>>(
      tr, rays, out, hits, misses, n_live, n_miss);
  return cudaGetLastError();
}

// Bricks per ray, per packet of a resident warp's share, from which a packet
// counts as long (see packet_launch).  Measured us, caches flushed between passes,
// of a 1080p view / an FP8 view of 1283 x 717 / a slice and its 1080p view / an
// edited 720p frame: 0.25: 598 / 335 / 724 / 594; 0.4: 570 / 305 / 668 / 561; 0.65:
// 622 / 299 / 727 / 564; 1.0: 665 / 307 / 754 / 585; without triage 658 / 415 / 752 /
// 665.
constexpr float kLongShare = 0.4f;

// Launches a packet forward of any shading.  Without a log each packet is run
// in two or four parts while the parts stay within four per resident warp (up
// to two packets per warp in halves, up to one in quarters), on a plain grid without
// counter or triage: these calls are bound by the latency of their longest
// packet (a 128 x 128 view: 78 us whole, 49 in four parts).  A log's layout is by
// whole packets, so calls with one run them whole, on a plain grid up to one
// packet per resident warp.  Above: a persistent grid on the work counter, after
// the triage that the call allows: of rays with a log in which the packets are
// taken as given (n < 2^32), of packets without a log on the trees that gain from
// it (triage_gains; already at 2.5 packets per warp: a 480 x 400 view of a depth-8
// shell 189 us with the list, 273 without).
template <int KP, int DEG, typename E, int kShade, int CHUNKS = shade_chunks<KP, DEG, E, kShade>()>
static cudaError_t packet_launch(FwdArgs a, const LaunchCfg &cfg, cudaStream_t s) {
  if (a.rays.n == 0) return cudaSuccess;
  const long long n_packets = (a.rays.n + 31) >> 5;
  const int warps = cfg.block / 32;
  const size_t sm = smem_bytes(cfg.block, KP, CHUNKS, path_words(a.tr));
  if constexpr (CHUNKS > 0)
    if (!stage_fits(cfg.block, sm)) return packet_launch<KP, DEG, E, kShade, 0>(a, cfg, s);
  const auto kernel = render_packet_kernel<KP, DEG, E, kShade, CHUNKS>;
  cudaError_t e;
  if (sm > 48 * 1024 &&
      (e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)) != cudaSuccess)
    return e;
  int per_sm = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, cfg.block, sm)) != cudaSuccess) return e;
  const long long want = (long long)(per_sm > 0 ? per_sm : 1) * cfg.num_sms;  // resident blocks
  const long long resident = want * warps;
  if (!a.log.n_chunks)
    while (a.split < kMaxSplit && (n_packets << (a.split + 1)) <= 4 * resident) ++a.split;
  long long grid = ((n_packets << a.split) + warps - 1) / warps;
  if (grid <= want || a.split) a.work = nullptr;
  if (a.work) {
    grid = want;
    if ((e = cudaMemsetAsync(a.work, 0, 2 * sizeof(unsigned long long), s)) != cudaSuccess) return e;
    if (a.log.n_chunks && !a.order && !a.perm && a.rays.n <= 0xFFFFFFFFll) {
      a.perm = a.log.perm;
      a.n_live = a.log.header + 6;
      if ((e = launch_triage_rays(a.tr, a.rays, a.out, a.log.perm, a.log.perm, a.log.header + 6, a.log.header + 8, s)) !=
          cudaSuccess)
        return e;
    } else if (!a.log.n_chunks && a.queue && n_packets <= kQueuePackets) {
      // a packet is long when its work is a notable part of an average warp's
      // share, which grows with the packets per resident warp
      uint32_t *counts = reinterpret_cast<uint32_t *>(a.work + 1);
      const float half = kLongShare * (float)n_packets / (float)resident;
      triage_packets_kernel<<<(unsigned)((a.rays.n + 255) / 256), 256, 0, s>>>(a.tr, a.rays, a.out, half, 2.f * half,
                                                                               a.queue, counts);
      a.list = a.queue;
      a.counts = counts;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  // packets past the live rays are not run: no chunk, no key
  if (a.n_live && (e = cudaMemsetAsync(a.log.heads, 0xFF, (size_t)((char *)(a.log.key + n_packets) - (char *)a.log.heads),
                                       s)) != cudaSuccess)
    return e;
  kernel<<<(unsigned)grid, cfg.block, sm, s>>>(a);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(256) trace_kernel(const __grid_constant__ TraceArgs a) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.rays.n) return;
  float o[3], d[3], t;
  load_ray(a.rays, i, o, d, t);
  RayWalk w;
  float dn[3];
  int c = 0;
  if (walk_init(a.tr, o, d, w, dn)) {
    uint32_t leaf;
    float t0, dt;
    while (w.alive) {  // one loop over steps, as in integrate_ray (nested: 2.6 times as long on a shell)
      if (!walk_step(a.tr, w, leaf, t0, dt)) continue;
      if (c < a.max_out) {
        a.leaf[i * a.max_out + c] = (int)leaf;
        a.t0[i * a.max_out + c] = w.t_base + t0;
        a.t1[i * a.max_out + c] = w.t_base + (t0 + dt);
      }
      ++c;
    }
  }
  for (int k = c; k < a.max_out; ++k) {
    a.leaf[i * a.max_out + k] = -1;
    a.t0[i * a.max_out + k] = 0.f;
    a.t1[i * a.max_out + k] = 0.f;
  }
  a.count[i] = c;
}

template <int KP, int DEG, typename E>
static cudaError_t fwd_one(bool packet, const FwdArgs &a, const LaunchCfg &cfg, cudaStream_t s) {
  if (packet) return packet_launch<KP, DEG, E, kShadeTree>(a, cfg, s);
  if (a.rays.n == 0) return cudaSuccess;
  render_plain_kernel<KP, DEG, E><<<(unsigned)((a.rays.n + cfg.block - 1) / cfg.block), cfg.block, 0, s>>>(a);
  return cudaGetLastError();
}

#define NEUVV_DISPATCH_KD(FN, ...)                                              \
  switch (KP * 10 + DEG) {                                                       \
    case 81: return FN<8, 1, E>(__VA_ARGS__);                                   \
    case 82: return FN<8, 2, E>(__VA_ARGS__);                                   \
    case 83: return FN<8, 3, E>(__VA_ARGS__);                                   \
    case 161: return FN<16, 1, E>(__VA_ARGS__);                                 \
    case 162: return FN<16, 2, E>(__VA_ARGS__);                                 \
    case 163: return FN<16, 3, E>(__VA_ARGS__);                                 \
    case 321: return FN<32, 1, E>(__VA_ARGS__);                                 \
    case 322: return FN<32, 2, E>(__VA_ARGS__);                                 \
    case 323: return FN<32, 3, E>(__VA_ARGS__);                                 \
    default: return cudaErrorInvalidValue;                                      \
  }

template <typename E>
static cudaError_t fwd_dispatch(int KP, int DEG, bool packet, const FwdArgs &a, const LaunchCfg &cfg, cudaStream_t s) {
  NEUVV_DISPATCH_KD(fwd_one, packet, a, cfg, s)
}

cudaError_t launch_render_fwd(int KP, int DEG, DType dt, bool packet, const FwdArgs &a, const LaunchCfg &cfg,
                              cudaStream_t s) {
  if (dt == kF32) return fwd_dispatch<float>(KP, DEG, packet, a, cfg, s);
  if (dt == kBF16) return fwd_dispatch<__nv_bfloat16>(KP, DEG, packet, a, cfg, s);
  // FP8 storage is built for the two record shapes of the workloads only
  if (KP == 8 && DEG == 2) return fwd_one<8, 2, Fp8E4M3>(packet, a, cfg, s);
  if (KP == 16 && DEG == 3) return fwd_one<16, 3, Fp8E4M3>(packet, a, cfg, s);
  return cudaErrorInvalidValue;
}

// Time slice of one leaf whose record is loaded: density and hyper angle from
// the basis rows at frame coordinate u (Eq. project-sigma, Eq. project-gamma),
// the radial factors R_nl(gamma) by the Gegenbauer recurrence, then
// s[ch][l,m] = sum_{n >= l} w[ch][n,l,m] R_nl (Eq. HH-color-2 with gamma
// fixed), written as one slice row of NV float4.
template <int KP, int DEG, typename E>
__device__ __forceinline__ void slice_row(const DevTree &tr, const RegRows<KP> &rows, const LeafRecord<KP, DEG, E> &rec,
                                          float4 *dst) {
  constexpr int NY = (DEG + 1) * (DEG + 1), NV = slice_min_stride(DEG) / 4;
  float out[NV * 4];
#pragma unroll
  for (int k = 0; k < NV * 4; ++k) out[k] = 0.f;
  out[0] = fmaxf(pre_sigma_of<KP>(rows, rec), 0.f);
  const float pg = pre_gamma_of<KP>(rows, rec);
  float sg, cg, R[(DEG + 1) * (DEG + 2) / 2];
  sincospif(sigmoidf_fast(pg), &sg, &cg);
  hh_radial<DEG, false>(cg, sg, tr.hh_norm, R, nullptr);
#pragma unroll
  for (int ch = 0; ch < 3; ++ch)
#pragma unroll
    for (int l = 0; l <= DEG; ++l)
#pragma unroll
      for (int m = -l; m <= l; ++m) {
        float acc = 0.f;
#pragma unroll
        for (int n = l; n <= DEG; ++n) acc = fmaf(rec.hh(ch, hh_index(n, l, m)), R[radial_index(n, l)], acc);
        out[4 + ch * NY + l * l + l + m] = acc * rec.scale_hh();
      }
#pragma unroll
  for (int i = 0; i < NV; ++i) dst[i] = make_float4(out[4 * i], out[4 * i + 1], out[4 * i + 2], out[4 * i + 3]);
}

// Time slice, one thread per leaf, records read from global memory (any
// record and row size).
template <int KP, int DEG, typename E>
__global__ void __launch_bounds__(256) slice_kernel(const __grid_constant__ DevTree tr, float u, float *slice,
                                                    int stride) {
  const long long leaf = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (leaf >= tr.n_leaves) return;
  RayConst<KP, DEG> rc;
  ray_const_basis<KP, DEG>(tr, u, rc);
  LeafRecord<KP, DEG, E> rec;
  rec.load(tr, (uint32_t)leaf);
  slice_row<KP, DEG, E>(tr, RegRows<KP>{rc.a, rc.b}, rec, reinterpret_cast<float4 *>(slice + (size_t)leaf * stride));
}

// Bulk copies between global and shared memory through the TMA unit.
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Waits until the mbarrier's phase `parity` completes, for at most `limit`
// polls; false on time-out.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int limit) {
  for (int k = 0; k < limit; ++k) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

constexpr int kSliceTile = 64;    // leaves per tile (one per thread)
// Polls of the wait that lets a tile's copy in flight land after the tile's
// own wait gave up (the block must not exit while the copy writes into its
// shared memory).
constexpr int kSliceDrainPolls = 1 << 22;

// Time slice with TMA staging: a block takes tiles of kSliceTile consecutive
// leaves; one thread loads the tile's records (consecutive in memory) into
// shared memory with a single bulk copy completed on an mbarrier, every
// thread turns its record into its slice row in a shared output tile, and one
// bulk copy stores the tile's rows (consecutive in memory when the row
// stride is the minimal one).  A wait that does not complete within the
// tree's poll limit flags kStatusTimeout; the whole block then waits (again
// bounded) for its copy in flight to land and ends.
template <int KP, int DEG, typename E>
__global__ void __launch_bounds__(kSliceTile) slice_tma_kernel(const __grid_constant__ DevTree tr, float u,
                                                               float *slice, int rec_bytes) {
  constexpr int NV = slice_min_stride(DEG) / 4;
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ __align__(8) unsigned long long bar;
  uint4 *in = reinterpret_cast<uint4 *>(sm);
  float4 *out = reinterpret_cast<float4 *>(sm + (size_t)kSliceTile * rec_bytes);
  const uint32_t bar_a = smem_addr(&bar);
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  RayConst<KP, DEG> rc;
  ray_const_basis<KP, DEG>(tr, u, rc);
  const RegRows<KP> rows{rc.a, rc.b};
  const long long n_tiles = (tr.n_leaves + kSliceTile - 1) / kSliceTile;
  uint32_t parity = 0;
  for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, parity ^= 1u) {
    const long long first = tile * kSliceTile;
    const int count = (int)min((long long)kSliceTile, tr.n_leaves - first);
    if (threadIdx.x == 0) {
      const uint32_t bytes = (uint32_t)count * (uint32_t)rec_bytes;
      const char *src = static_cast<const char *>(tr.rec) + (size_t)first * rec_bytes;
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_a), "r"(bytes) : "memory");
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(in)),
          "l"(src), "r"(bytes), "r"(bar_a)
          : "memory");
    }
    // one decision for the block, so that no thread leaves while others sync
    if (!__syncthreads_and(mbar_wait(bar_a, parity, tr.wait_polls))) {
      if (threadIdx.x == 0) raise_status(tr, kStatusTimeout);
      mbar_wait(bar_a, parity, kSliceDrainPolls);
      if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
      return;
    }
    if ((int)threadIdx.x < count) {
      LeafRecord<KP, DEG, E> rec;
      rec.load_shared(in + (size_t)threadIdx.x * (rec_bytes / 16));
      slice_row<KP, DEG, E>(tr, rows, rec, out + (size_t)threadIdx.x * NV);
    }
    // the rows become visible to the bulk copy (async proxy), then one store
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(slice + (size_t)first * NV * 4),
                   "r"(smem_addr(out)), "r"((uint32_t)count * NV * 16)
                   : "memory");
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      // the output tile and the input buffer are reused by the next tile
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");  // stores complete
}

template <int KP, int DEG, typename E>
static cudaError_t slice_one(const DevTree &tr, float u, float *slice, int stride, int rec_bytes, int num_sms,
                             cudaStream_t s) {
  if (tr.n_leaves == 0) return cudaSuccess;
  if (stride == slice_min_stride(DEG) && rec_bytes % 16 == 0) {
    const size_t sm = (size_t)kSliceTile * (rec_bytes + slice_min_stride(DEG) * 4);
    cudaError_t e;
    if (sm > 48 * 1024 &&
        (e = cudaFuncSetAttribute(slice_tma_kernel<KP, DEG, E>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sm)) != cudaSuccess)
      return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, slice_tma_kernel<KP, DEG, E>, kSliceTile, sm)) !=
        cudaSuccess)
      return e;
    const long long tiles = (tr.n_leaves + kSliceTile - 1) / kSliceTile;
    long long grid = (long long)(per_sm > 0 ? per_sm : 1) * num_sms;
    if (grid > tiles) grid = tiles;
    slice_tma_kernel<KP, DEG, E><<<(unsigned)grid, kSliceTile, sm, s>>>(tr, u, slice, rec_bytes);
    return cudaGetLastError();
  }
  slice_kernel<KP, DEG, E><<<(unsigned)((tr.n_leaves + 255) / 256), 256, 0, s>>>(tr, u, slice, stride);
  return cudaGetLastError();
}

cudaError_t launch_slice(int KP, int DEG, DType dt, const DevTree &tr, float u, float *slice, int stride,
                         int rec_bytes, int num_sms, cudaStream_t s) {
#define NEUVV_SLICE_KD(E)                                   \
  switch (KP * 10 + DEG) {                                  \
    case 81: return slice_one<8, 1, E>(tr, u, slice, stride, rec_bytes, num_sms, s);   \
    case 82: return slice_one<8, 2, E>(tr, u, slice, stride, rec_bytes, num_sms, s);   \
    case 83: return slice_one<8, 3, E>(tr, u, slice, stride, rec_bytes, num_sms, s);   \
    case 161: return slice_one<16, 1, E>(tr, u, slice, stride, rec_bytes, num_sms, s); \
    case 162: return slice_one<16, 2, E>(tr, u, slice, stride, rec_bytes, num_sms, s); \
    case 163: return slice_one<16, 3, E>(tr, u, slice, stride, rec_bytes, num_sms, s); \
    case 321: return slice_one<32, 1, E>(tr, u, slice, stride, rec_bytes, num_sms, s); \
    case 322: return slice_one<32, 2, E>(tr, u, slice, stride, rec_bytes, num_sms, s); \
    case 323: return slice_one<32, 3, E>(tr, u, slice, stride, rec_bytes, num_sms, s); \
    default: return cudaErrorInvalidValue;                  \
  }
  if (dt == kF32) NEUVV_SLICE_KD(float)
  if (dt == kBF16) NEUVV_SLICE_KD(__nv_bfloat16)
#undef NEUVV_SLICE_KD
  if (KP == 8 && DEG == 2) return slice_one<8, 2, Fp8E4M3>(tr, u, slice, stride, rec_bytes, num_sms, s);
  if (KP == 16 && DEG == 3) return slice_one<16, 3, Fp8E4M3>(tr, u, slice, stride, rec_bytes, num_sms, s);
  return cudaErrorInvalidValue;
}

// Packet render of a slice: the packet forward with the slice shader (the
// basis-row part of its shared memory is laid out for K_pad = 8 and unused;
// the storage type only sets the register budget, 128 per thread).
template <int DEG>
static cudaError_t render_slice_one(const FwdArgs &a, const LaunchCfg &cfg, cudaStream_t s) {
  return packet_launch<8, DEG, __nv_bfloat16, kShadeSlice>(a, cfg, s);
}

cudaError_t launch_render_slice(int DEG, const FwdArgs &a, const LaunchCfg &cfg, cudaStream_t s) {
  if (DEG == 1) return render_slice_one<1>(a, cfg, s);
  if (DEG == 2) return render_slice_one<2>(a, cfg, s);
  if (DEG == 3) return render_slice_one<3>(a, cfg, s);
  return cudaErrorInvalidValue;
}

// Terminating voxel of each ray (Sec. 5 "Appearance editing"): the leaf of the
// segment at which 1 - exp(-sum sigma delta) of the unedited render first
// reaches the threshold; -1 when it never does.  The density-only packet
// forward with the threshold in the place of the early stop.
template <int KP, int DEG, typename E>
static cudaError_t pick_one(FwdArgs a, float threshold, int *leaf_out, const LaunchCfg &cfg, cudaStream_t s) {
  a.t_stop = threshold;
  a.out = DevOut{nullptr, nullptr, nullptr, nullptr, leaf_out};
  return packet_launch<KP, DEG, E, kShadePick>(a, cfg, s);
}

cudaError_t launch_pick(int KP, int DEG, DType dt, const FwdArgs &a, float threshold, int *leaf_out,
                        const LaunchCfg &cfg, cudaStream_t s) {
#define NEUVV_PICK_KD(E)                                   \
  switch (KP * 10 + DEG) {                                 \
    case 81: return pick_one<8, 1, E>(a, threshold, leaf_out, cfg, s);   \
    case 82: return pick_one<8, 2, E>(a, threshold, leaf_out, cfg, s);   \
    case 83: return pick_one<8, 3, E>(a, threshold, leaf_out, cfg, s);   \
    case 161: return pick_one<16, 1, E>(a, threshold, leaf_out, cfg, s); \
    case 162: return pick_one<16, 2, E>(a, threshold, leaf_out, cfg, s); \
    case 163: return pick_one<16, 3, E>(a, threshold, leaf_out, cfg, s); \
    case 321: return pick_one<32, 1, E>(a, threshold, leaf_out, cfg, s); \
    case 322: return pick_one<32, 2, E>(a, threshold, leaf_out, cfg, s); \
    case 323: return pick_one<32, 3, E>(a, threshold, leaf_out, cfg, s); \
    default: return cudaErrorInvalidValue;                 \
  }
  if (dt == kF32) NEUVV_PICK_KD(float)
  if (dt == kBF16) NEUVV_PICK_KD(__nv_bfloat16)
#undef NEUVV_PICK_KD
  if (KP == 8 && DEG == 2) return pick_one<8, 2, Fp8E4M3>(a, threshold, leaf_out, cfg, s);
  if (KP == 16 && DEG == 3) return pick_one<16, 3, Fp8E4M3>(a, threshold, leaf_out, cfg, s);
  return cudaErrorInvalidValue;
}

// Painting: the colours of the rays that picked each leaf are summed (with
// their count) into accum [n_leaves][4], then every leaf with a count gets
// the mean colour, sigma_d and t_d in its edit record [n_leaves][8].
__global__ void __launch_bounds__(256) paint_accum_kernel(const int *leaf, const float *color, long long n,
                                                          long long n_leaves, float *accum) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int l = leaf[i];
  if (l < 0 || l >= n_leaves) return;
  atomicAdd(accum + 4 * (size_t)l + 0, color[3 * i + 0]);
  atomicAdd(accum + 4 * (size_t)l + 1, color[3 * i + 1]);
  atomicAdd(accum + 4 * (size_t)l + 2, color[3 * i + 2]);
  atomicAdd(accum + 4 * (size_t)l + 3, 1.f);
}

__global__ void __launch_bounds__(256) paint_finish_kernel(const float *accum, long long n_leaves, float sigma_d,
                                                           float t_d, float *edits) {
  const long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= n_leaves) return;
  const float4 s = reinterpret_cast<const float4 *>(accum)[l];
  if (s.w > 0.f) {
    float4 *e = reinterpret_cast<float4 *>(edits) + 2 * l;
    e[0] = make_float4(s.x / s.w, s.y / s.w, s.z / s.w, sigma_d);
    e[1] = make_float4(t_d, 0.f, 0.f, 0.f);
  }
}

cudaError_t launch_paint(const int *leaf, const float *color, long long n, long long n_leaves, float *accum,
                         float sigma_d, float t_d, float *edits, cudaStream_t s) {
  if (n > 0) paint_accum_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(leaf, color, n, n_leaves, accum);
  if (n_leaves > 0)
    paint_finish_kernel<<<(unsigned)((n_leaves + 255) / 256), 256, 0, s>>>(accum, n_leaves, sigma_d, t_d, edits);
  return cudaGetLastError();
}

// Density-only packet render (alpha, depth, tau and nseg of the full render,
// no colour): one packet per warp of a full grid, no work counter, so it may
// run beside other calls on the same tree.  Built for the two record shapes
// of the workloads (K_pad 8 with degree 2, K_pad 16 with degree 3), as are
// the renders with appearance edits.
cudaError_t launch_render_alpha(int KP, int DEG, DType dt, const FwdArgs &a, const LaunchCfg &cfg, cudaStream_t s) {
  if (a.work || a.log.n_chunks) return cudaErrorInvalidValue;
  if (KP == 8 && DEG == 2) {
    if (dt == kF32) return packet_launch<8, 2, float, kShadeAlpha>(a, cfg, s);
    if (dt == kBF16) return packet_launch<8, 2, __nv_bfloat16, kShadeAlpha>(a, cfg, s);
    return packet_launch<8, 2, Fp8E4M3, kShadeAlpha>(a, cfg, s);
  }
  if (KP == 16 && DEG == 3) {
    if (dt == kF32) return packet_launch<16, 3, float, kShadeAlpha>(a, cfg, s);
    if (dt == kBF16) return packet_launch<16, 3, __nv_bfloat16, kShadeAlpha>(a, cfg, s);
    return packet_launch<16, 3, Fp8E4M3, kShadeAlpha>(a, cfg, s);
  }
  return cudaErrorNotSupported;
}

cudaError_t launch_render_edit(int KP, int DEG, DType dt, const FwdArgs &a, const LaunchCfg &cfg, cudaStream_t s) {
  if (KP == 8 && DEG == 2) {
    if (dt == kF32) return packet_launch<8, 2, float, kShadeEdit>(a, cfg, s);
    if (dt == kBF16) return packet_launch<8, 2, __nv_bfloat16, kShadeEdit>(a, cfg, s);
  }
  if (KP == 16 && DEG == 3) {
    if (dt == kF32) return packet_launch<16, 3, float, kShadeEdit>(a, cfg, s);
    if (dt == kBF16) return packet_launch<16, 3, __nv_bfloat16, kShadeEdit>(a, cfg, s);
  }
  return cudaErrorNotSupported;
}

// Segment log decoder: ray i's composited segments are the slots of its
// packet's chunks that hold a leaf and name its lane, in slot order, nseg[i]
// of them.  count[i] = -1 when the ray's packet is not in the log (no log, a log
// of other rays, or a packet that did not fit); chunk links are checked
// against the log's size.  packed, wide: the two views of the buffer, of which
// the header names the one the forward wrote.
__global__ void __launch_bounds__(256) log_read_kernel(const SampleLog packed, const SampleLog wide, long long n,
                                                        const int *nseg, int max_out, int *leaf, float *chord,
                                                        int *count) {
  const long long pos = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (pos >= n) return;
  int c = -1;
  const bool is_wide = wide.n_chunks && __ldg(wide.header + 9) == wide.layout();
  const SampleLog &l = is_wide ? wide : packed;
  const bool valid = l.n_chunks && log_matches(l, n);
  // the ray at this position (its outputs are written at the ray's index)
  const long long i = valid && __ldg(l.header + 5) == 1u ? (long long)min(__ldg(l.perm + pos), (uint32_t)(n - 1)) : pos;
  if (valid) {
    uint32_t chunk = __ldg(l.heads + (pos >> 5));
    const int want = __ldg(nseg + i);
    if (want == 0) {
      c = 0;
    } else if (chunk != kNoLog) {
      c = 0;
      for (uint32_t guard = 0; c < want && guard < l.n_chunks; ++guard) {
        if (chunk >= l.n_chunks) {
          c = -1;
          break;
        }
        for (int k = 0; k < kLogRounds * 32 && c < want; ++k) {
          const size_t slot = (size_t)chunk * kLogRounds * 32 + k;
          const LogWord w = log_word(l, slot);
          if (w.empty || w.lane != (int)(pos & 31)) continue;
          if (c < max_out) {
            leaf[i * max_out + c] = (int)w.leaf;
            chord[i * max_out + c] = __ldg(l.dt + slot);
          }
          ++c;
        }
        if (c < want) chunk = __ldg(l.next + chunk);
      }
    }
  }
  for (int k = c < 0 ? 0 : c; k < max_out; ++k) {
    leaf[i * max_out + k] = -1;
    chord[i * max_out + k] = 0.f;
  }
  count[i] = c;
}

cudaError_t launch_log_read(const SampleLog &packed, const SampleLog &wide, long long n_rays, const int *nseg,
                            int max_out, int *leaf, float *chord, int *count, cudaStream_t s) {
  if (n_rays == 0) return cudaSuccess;
  log_read_kernel<<<(unsigned)((n_rays + 255) / 256), 256, 0, s>>>(packed, wide, n_rays, nseg, max_out, leaf,
                                                                  chord, count);
  return cudaGetLastError();
}

cudaError_t launch_trace(const TraceArgs &a, cudaStream_t s) {
  if (a.rays.n == 0) return cudaSuccess;
  const long long blocks = (a.rays.n + 127) / 128;
  trace_kernel<<<(unsigned)blocks, 128, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace neuvv
