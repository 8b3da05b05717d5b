// gg_flow.cu -- every projected-Jacobi sweep of a step in one launch, ordered by data
// instead of by launches or grid barriers.
//
// What bounds a sweep as a launch of its own: 4.2 us at 4,096 spheres and 5.0 at 262,144
// with a fifth of them in contact, whatever the bytes -- a launch (0.9 us) and a chain of
// four dependent loads (counts, partner ids, partners' estimates, bodies) -- and, where
// every sphere is in contact, the re-reading of the records (48 bytes per contact and
// sweep: normal, impulse in and out).  Here a block loads the contact records of its spheres once, keeps them in
// shared memory for all I sweeps, impulses included, and what a sweep moves through L2 is
// 16 bytes out per sphere that other blocks' spheres touch and 16 bytes in per such contact.
// Measured (sweep stage of a step, 20 iterations, us): 4,096 spheres 84 -> 48, 16,384
// 82 -> 49, 262,144 with a fifth in contact 100 -> 72, all in contact 184 -> 125, 64
// environments of 1.86M spheres 1804 -> 915.  A sweep then takes 1.5 us at 4,096 spheres
// (two block barriers, the exchange between the dies 0.45 us, the shared-memory latency of
// two dependent stages) and 4.5 us at 1,700 spheres a block (shared-memory bandwidth);
// taking the records up costs about 10 to 25 us a step.
//
// Order.  Sweep s of sphere i needs U^s of its partners.  Estimates that another block needs
// are published as one 128-bit store {x, y, z, tag}, the tag naming launch and iteration
// (the fourth component of U, n / m, does not change during the sweeps and is folded into
// each contact's effective mass beforehand), and a reader polls until the tag is the one it
// needs; 128-bit relaxed accesses of one location are single-copy atomic, so no flag, fence
// or barrier is involved.  Two slots by iteration parity suffice: i overwrites U^s with
// U^{s+2} only after reading U^{s+1} of every partner, which each partner publishes only
// after it has read U^s_i -- because contact lists are symmetric.  They are unless detection
// cut one short (a latched capacity or bucket flag) or a sphere is larger than the cells
// allow (the lists' symmetry sum is not zero then); in those cases, and where a block's
// lists would not fit its shared memory, the launch runs the plain sweeps with a grid barrier
// between them, like k_pja_fused.  Those take 1.5 to 1.8 times as long as split launches (a
// packed bed of 400,000 spheres 412 us a step and 279, of a million 1,435 and 797), so where
// most spheres get them the launch tells the host, which goes over to the fastest split set if
// the autotuner had chosen (a bed tuned while it was falling).  A wait is bounded (wait_cycles), latches kFlagTimeout and
// makes every later wait return at once.
//
// All blocks are resident (cooperative launch, one block per SM, no more blocks than the
// spheres can keep busy).  A batch is swept in
// ranges of whole environments that fit the chip, one after another with no barrier between
// them.  Within a range the 32-sphere tiles that have contacts are shared out in order, an
// equal part of the contacts to every block, so that most partners are the block's own.
//
// Same arithmetic and the same per-sphere summation order as the per-launch sweeps, so
// positions, velocities and wrenches are bit-identical (an impulse that is zero may read
// back with the other sign).
#include <algorithm>

#include "gg_device.cuh"
#include "gg_internal.h"
#include "gg_sweep.cuh"

namespace gg {

namespace {

constexpr int kFlowThreads = 1024;
constexpr int kFlowWarps = kFlowThreads / 32;
constexpr int kEarly = 2;              // records with other blocks' spheres whose estimates a thread asks for ahead
// cost of a 32-sphere tile beside its contacts, in contacts (0 and 32 measure the same but for a
// batch, 420 us of sweeps with 0 and 404 with 16; at 64 a pile of 262,144 no longer fits)
constexpr uint32_t kTileWeight = 16;
constexpr uint32_t kBytesPerCost = 24; // ... and no less than its lists and estimates take in shared memory over this
// least work worth a block of its own (sweep stage at 1,000, 4,096 and 16,384 spheres: 47, 47 and
// 49 us, with 320 47, 47 and 47, with 1,280 51, 51 and 51; fewer blocks leave more of the chip
// to other streams)
constexpr uint32_t kMinWork = 640;
constexpr uint32_t kTileMax = 32u * (kMaxK + kMaxKb) + kTileWeight;  // most a tile costs
constexpr uint32_t kNone = 0xffffffffu;
constexpr uint32_t kAsymmetric = kFlagPPOverflow | kFlagBucketBound | kFlagListBound | kFlagDebugCheck;

#define GG_LD_TAGGED(name, order)                                                                                  \
  __device__ __forceinline__ float4 name(const float4 *p) {                                                        \
    float4 v;                                                                                                      \
    asm volatile("{\n\t.reg .b128 t;\n\t.reg .b64 lo, hi;\n\tld." order                                            \
                 ".gpu.global.b128 t, [%4];\n\tmov.b128 {lo, hi}, t;\n\t"                                          \
                 "mov.b64 {%0, %1}, lo;\n\tmov.b64 {%2, %3}, hi;\n\t}"                                             \
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)                                                      \
                 : "l"(p)                                                                                          \
                 : "memory");                                                                                      \
    return v;                                                                                                      \
  }
GG_LD_TAGGED(ld_tagged, "relaxed")
GG_LD_TAGGED(ld_tagged_acquire, "acquire")
#undef GG_LD_TAGGED

__device__ __forceinline__ void st_tagged(float4 *p, float x, float y, float z, uint32_t tag) {
  asm volatile(
      "{\n\t.reg .b128 t;\n\t.reg .b64 lo, hi;\n\tmov.b64 lo, {%1, %2};\n\tmov.b64 hi, {%3, %4};\n\t"
      "mov.b128 t, {lo, hi};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
      "f"(x), "f"(y), "f"(z), "f"(__uint_as_float(tag))
      : "memory");
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Bounded waits of one thread: `dead` once a wait of this launch gave up.
struct Waits {
  bool dead;
  // poll number `polls` of a wait that began at t0 has failed; false: give up
  __device__ __forceinline__ bool again(const StepArgs &a, uint32_t &polls, long long &t0) {
    if (dead) return false;
    if ((++polls & 255u) == 0u) {
      const long long t = clock64();
      if (polls == 256u) t0 = t;
      volatile uint32_t *ab = &a.ctrl->bar_abort;
      if (*ab || t - t0 > a.wait_cycles) {
        atomicOr(&a.ctrl->status, kFlagTimeout);
        atomicExch(&a.ctrl->bar_abort, 1u);
        dead = true;
        return false;
      }
    }
    return true;
  }
};

__device__ __forceinline__ float4 wait_tagged(const StepArgs &a, const float4 *p, float4 v, uint32_t tag, Waits &w) {
  uint32_t polls = 0;
  long long t0 = 0;
  while (__float_as_uint(v.w) != tag && w.again(a, polls, t0)) v = ld_tagged(p);
  return v;
}
__device__ __forceinline__ void wait_word(const StepArgs &a, const uint32_t *p, uint32_t v, Waits &w) {
  uint32_t polls = 0;
  long long t0 = 0;
  while (ld_acquire(p) != v && w.again(a, polls, t0)) {
  }
}

// Mass-split inverse mass of a free body at a contact (as in pja_particle).
__device__ __forceinline__ float body_inv(const StepArgs &a, const DevBody &B, uint32_t gb, float4 nn, float rx, float ry,
                                          float rz) {
  if (!B.is_free) return 0.f;
  const float cx = ry * nn.z - rz * nn.y, cy = rz * nn.x - rx * nn.z, cz = rx * nn.y - ry * nn.x;
  const float t0 = B.R[0] * cx + B.R[3] * cy + B.R[6] * cz;
  const float t1 = B.R[1] * cx + B.R[4] * cy + B.R[7] * cz;
  const float t2 = B.R[2] * cx + B.R[5] * cy + B.R[8] * cz;
  return (float)a.ncb[gb] * (1.0f / B.mass + t0 * t0 / B.inertia[0] + t1 * t1 / B.inertia[1] + t2 * t2 / B.inertia[2]);
}

__device__ __forceinline__ float3 point_velocity(float3 V, float3 W, float rx, float ry, float rz) {
  return make_float3(V.x + (W.y * rz - W.z * ry), V.y + (W.z * rx - W.x * rz), V.z + (W.x * ry - W.y * rx));
}

// Twist of free body `fid` for sweep s: the step's own for the first, then as published.
template <bool FREE>
__device__ __forceinline__ void free_twist(const StepArgs &a, const DevBody &B, uint32_t fid, uint32_t s, uint32_t tag,
                                           Waits &w, float3 *V, float3 *W) {
  if (!FREE || s == 0) {
    *V = make_float3(B.v[0], B.v[1], B.v[2]);
    *W = make_float3(B.w[0], B.w[1], B.w[2]);
    return;
  }
  // published as the angular half, a fence, then the linear half with the tag: acquired by
  // loads of the size of that store (polling four bytes of it would be a race in the memory
  // model), so that the angular half may be read after it.  (A relaxed poll and a fence: eight
  // steps of a 37,224-sphere excavation 1,504 us instead of 1,427; a tag in both halves 1,438.)
  const float4 *p = a.ftw + ((size_t)fid * 2 + (s & 1u)) * 2;
  float4 v = ld_tagged_acquire(p);
  uint32_t polls = 0;
  long long t0 = 0;
  while (__float_as_uint(v.w) != tag && w.again(a, polls, t0)) v = ld_tagged_acquire(p);
  const float4 o = __ldcg(p + 1);
  *V = make_float3(v.x, v.y, v.z);
  *W = make_float3(o.x, o.y, o.z);
}

// An impulse on a free body's contact, for the body's block: stored, then counted.
__device__ __forceinline__ void hand_over(const StepArgs &a, uint32_t fid, size_t o, size_t KbN, float3 l) {
  a.blam[o] = l.x;
  a.blam[o + KbN] = l.y;
  a.blam[o + 2 * KbN] = l.z;
  __threadfence();
  atomicAdd(&a.farr[fid], 1u);
}

// Lists that may be asymmetric, or more spheres or contacts than fit: the plain sweeps with grid barriers (as in k_pja_fused),
// free bodies updated by the last blocks in between.
__device__ __forceinline__ void barrier_sweeps(const StepArgs &a, uint32_t iters, uint32_t G, uint32_t p0, uint32_t p1) {
  const Tape none{};
  const uint32_t stride = G * kFlowThreads;
  const size_t n = a.n, KbN = (size_t)a.Kb * n;
  if (blockIdx.x < G)
    for (uint32_t i = p0 + blockIdx.x * kFlowThreads + threadIdx.x; i < p1; i += stride) {
      const uint32_t cc = a.ccount[i];
      if (!(cc & 0xffffu)) {  // (left out by the contact build, but a cut list elsewhere may name it)
        const float4 b = base_velocity(a, a.vel_id[i]);
        a.U[0][i] = make_float4(b.x, b.y, b.z, 0.f);
      }
      for (uint32_t c = 0; c < (cc & 0xffu); ++c) a.clam[(size_t)c * n + i] = no_impulse(a.cj[(size_t)c * n + i]);
      for (uint32_t c = 0; c < 3 * ((cc >> 8) & 0xffu); ++c) a.blam[(size_t)(c % 3) * KbN + (size_t)(c / 3) * n + i] = 0.f;
    }
  grid_barrier(a.ctrl, a.wait_cycles);
  for (uint32_t it = 0; it < iters; ++it) {
    if (blockIdx.x < G)
      for (uint32_t i = p0 + blockIdx.x * kFlowThreads + threadIdx.x; i < p1; i += stride)
        pja_particle<false, true>(a, i, (int)(it & 1), none, (int)it);
    if (a.F) {
      grid_barrier(a.ctrl, a.wait_cycles);
      if (blockIdx.x >= G) {
        const uint32_t fid = blockIdx.x - G, gb = a.fgb[fid];
        if (gb != 0xffffffffu) free_update<kFlowThreads, true>(a, fid, gb);
      }
    }
    if (it + 1 < iters) grid_barrier(a.ctrl, a.wait_cycles);
  }
}

// The block of one free body: after each sweep, once every contact of the body has handed
// its impulse over, the body's update; then its twist for the next sweep.
__device__ __forceinline__ void free_block(const StepArgs &a, uint32_t fid, uint32_t iters, uint32_t tag0, Waits &wt) {
  const uint32_t gb = a.fgb[fid];
  if (gb == 0xffffffffu) return;
  const uint32_t cnt = a.fcount[fid];
  for (uint32_t s = 0; s < iters; ++s) {
    if (threadIdx.x == 0) {
      wait_word(a, a.farr + fid, cnt * (s + 1u), wt);  // (all of them: none is handed over twice before the next twist)
    }
    __syncthreads();
    free_update<kFlowThreads, true>(a, fid, gb);  // (thread 0 sets the body's twist)
    if (threadIdx.x == 0 && s + 1 < iters) {
      const DevBody &B = a.bodies[gb];
      float4 *p = a.ftw + ((size_t)fid * 2 + ((s + 1u) & 1u)) * 2;
      __stcg(p + 1, make_float4(B.w[0], B.w[1], B.w[2], 0.f));
      __threadfence();
      st_tagged(p, B.v[0], B.v[1], B.v[2], tag0 + s + 1u);
    }
    __syncthreads();
  }
}

// What a block keeps in dynamic shared memory (byte offsets: a word each, where pointers
// would take two registers).  Its spheres have places 32 t + lane, t the position of their
// tile among the block's.
//
// A pair whose spheres are both in the block is one record, worked on once a sweep: the
// impulse on its second sphere is the exact negative of that on the first (every product
// and sum of the update is odd in velocity, normal and impulse).  Records: "near" ones of
// such pairs, "far" ones whose partner is another block's sphere or a body, both in chunks
// of 32 (N, L, then words; no bank conflicts), near chunks from `rec` up, far chunks from
// `top` down; and those that do not fit, in global memory.  A sphere's contacts are listed
// by references in contact order, row c of tile t in ref[(row[t] + c) 32 + lane]: the byte
// offset of the record's impulse and whether it counts with the other sign.
extern __shared__ __align__(16) char s_pool[];
template <typename T>
__device__ __forceinline__ T &at(uint32_t off, uint32_t i) {
  return reinterpret_cast<T *>(s_pool + off)[i];
}
struct Block {
  uint32_t nt;      // tiles; their indices (u32, ascending) at offset 0
  uint32_t row;     // u16 [nt] first row of references
  uint32_t cnt;     // u8 [32 nt] contacts, kFar
  uint32_t ref;     // u32 [32 rows]
  uint32_t U;       // float4 [32 nt] velocity estimate, n / m
  uint32_t base;    // float4 [32 nt] velocity before impulses, 1 / m (0: computed from global memory)
  uint32_t rec, top;
};
constexpr uint32_t kFar = 0x80u;            // the sphere has partners in other blocks
constexpr uint32_t kNearChunk = 1152;       // 32 x (N 16, L 16, places 4)
constexpr uint32_t kFarChunk = 1280;        // 32 x (N 16, L 16, place and flags 4, id 4)
constexpr uint32_t kBody = 0x10000u, kFree = 0x20000u, kNear = 0x40000u;  // flags of a far / memory record
// references: the impulse's offset, or with kMem the record's index in memory
constexpr uint32_t kSign = 0x80000000u, kMem = 0x40000000u;
// (while records are made) not resolved: the rest is the partner's place times 16, an offset
// that is aligned and inside the pool should a list ever name a sphere that does not name it
constexpr uint32_t kOpen = 0x20000000u;
constexpr uint32_t kRefBits = 0x1fffffffu;

__device__ __forceinline__ uint32_t open_ref(uint32_t place) { return kOpen | place << 4; }

__device__ __forceinline__ uint32_t near_at(const Block &k, uint32_t r) { return k.rec + (r >> 5) * kNearChunk + (r & 31u) * 16u; }
__device__ __forceinline__ uint32_t far_at(const Block &k, uint32_t r) { return k.top - ((r >> 5) + 1u) * kFarChunk + (r & 31u) * 16u; }
__device__ __forceinline__ uint32_t near_word(const Block &k, uint32_t r) { return k.rec + (r >> 5) * kNearChunk + 1024u + (r & 31u) * 4u; }
__device__ __forceinline__ uint32_t far_word(const Block &k, uint32_t r) { return k.top - ((r >> 5) + 1u) * kFarChunk + 1024u + (r & 31u) * 4u; }
__device__ __forceinline__ size_t scratch(const StepArgs &a) { return (size_t)blockIdx.x * a.flow_region; }
__device__ __forceinline__ size_t body_scratch(const StepArgs &a) { return (size_t)blockIdx.x * a.flow_bodies; }

__device__ __forceinline__ uint32_t place_id(uint32_t o) { return at<uint32_t>(0, o >> 5) * 32u + (o & 31u); }

// Place of sphere j among the block's, kNone if it is another block's.
__device__ __forceinline__ uint32_t place_of(const Block &k, uint32_t j, uint32_t p0, uint32_t p1) {
  const uint32_t t = j >> 5, head = at<uint32_t>(0, 0);
  if (j < p0 || j >= p1) return kNone;  // (a tile at a range's end holds spheres of the next one)
  if (t < head || t > at<uint32_t>(0, k.nt - 1u)) return kNone;
  uint32_t lo = t - head;                            // the tile's position if no empty tile lies in between
  if (!(lo < k.nt && at<uint32_t>(0, lo) == t)) {
    lo = 0;
    for (uint32_t hi = k.nt; lo < hi;) {
      const uint32_t mid = (lo + hi) >> 1;
      if (at<uint32_t>(0, mid) < t) lo = mid + 1;
      else hi = mid;
    }
    if (!(lo < k.nt && at<uint32_t>(0, lo) == t)) return kNone;
  }
  return lo * 32u + (j & 31u);
}

struct Sweep {
  uint32_t s;               // iteration
  uint32_t tag, pub;        // tag of U^s, tag under which U^{s+1} is published
};

// A contact's update: the impulse on the sphere with estimate ui against uj.
__device__ __forceinline__ float4 update(const StepArgs &a, float4 nn, float4 la, float4 ui, float4 uj) {
  const float3 l = pja_project(make_float3(la.x, la.y, la.z), make_float3(ui.x - uj.x, ui.y - uj.y, ui.z - uj.z),
                               make_float3(nn.x, nn.y, nn.z), nn.w, la.w, a.mu);
  return make_float4(l.x, l.y, l.z, la.w);
}

// The partner's estimate of a far record, asked for (`v`) and then waited for.
__device__ __forceinline__ float4 ask(const StepArgs &a, uint32_t of, uint32_t id, const Sweep &w) {
  if (of & kBody) return a.flow_b[body_scratch(a) + id];
  return ld_tagged((w.s ? a.T[w.s & 1u] : a.U[0]) + id);
}
template <bool FREE>
__device__ __forceinline__ float4 answer(const StepArgs &a, uint32_t of, uint32_t id, float4 v, const Sweep &w, Waits &wt) {
  if (!(of & kBody)) return w.s ? wait_tagged(a, a.T[w.s & 1u] + id, v, w.tag, wt) : v;
  if (!FREE || !(of & kFree)) return v;
  const DevBody &B = a.bodies[__float_as_uint(v.w) >> 3];
  float3 V, W;
  free_twist<true>(a, B, B.fid, w.s, w.tag, wt, &V, &W);
  const float3 ub = point_velocity(V, W, v.x, v.y, v.z);
  return make_float4(ub.x, ub.y, ub.z, 0.f);
}
// A free body's impulse goes to the body's block.
__device__ __forceinline__ void give(const StepArgs &a, uint32_t of, uint32_t id, float4 l) {
  const uint32_t gbk = __float_as_uint(a.flow_b[body_scratch(a) + id].w);
  hand_over(a, a.bodies[gbk >> 3].fid, (size_t)(gbk & 7u) * a.n + place_id(of & 0xffffu), (size_t)a.Kb * a.n,
            make_float3(l.x, l.y, l.z));
}

// Impulse behind a reference (its sign apart).
__device__ __forceinline__ float4 referred(const StepArgs &a, uint32_t r) {
  if (r & kMem) return a.flow_l[scratch(a) + (r & ~(kMem | kSign))];
  return at<float4>(r & kRefBits, 0);
}
// Sum of a sphere's impulses in contact order, kGroup of them fetched together.
constexpr uint32_t kGroup = 4;
__device__ __forceinline__ float3 sum_impulses(const StepArgs &a, uint32_t ref, uint32_t cnt) {
  float3 S = make_float3(0.f, 0.f, 0.f);
#pragma unroll 1
  for (uint32_t c = 0; c < cnt; c += kGroup) {
    uint32_t r[kGroup];
    float4 l[kGroup];
#pragma unroll
    for (uint32_t q = 0; q < kGroup; ++q)
      if (c + q < cnt) r[q] = at<uint32_t>(ref, 32u * (c + q));
#pragma unroll
    for (uint32_t q = 0; q < kGroup; ++q)
      if (c + q < cnt) l[q] = referred(a, r[q]);
#pragma unroll
    for (uint32_t q = 0; q < kGroup; ++q) {
      if (c + q >= cnt) break;
      const float sg = (r[q] & kSign) ? -1.f : 1.f;
      S.x = __fmaf_rn(sg, l[q].x, S.x);
      S.y = __fmaf_rn(sg, l[q].y, S.y);
      S.z = __fmaf_rn(sg, l[q].z, S.z);
    }
  }
  return S;
}
__device__ __forceinline__ uint32_t refs_of(const Block &k, uint32_t o) {
  return k.ref + 128u * at<uint16_t>(k.row, o >> 5) + 4u * (o & 31u);
}

// Every sweep of the block's spheres (nl near, nr far records and nm in memory).
template <bool FREE>
__device__ __forceinline__ void sweeps(const StepArgs &a, const Block &k, uint32_t iters, uint32_t nl, uint32_t nr, uint32_t nm,
                                       uint32_t tag0, uint32_t out0, Waits &wt) {
  const uint32_t tid = threadIdx.x;
  Sweep w;
  for (uint32_t s = 0; s < iters; ++s) {
    w.s = s;
    w.tag = tag0 + s;
    w.pub = out0 + s + 1u;
    // other blocks' estimates are asked for first and used last
    float4 early[kEarly];
#pragma unroll
    for (int q = 0; q < kEarly; ++q) {
      const uint32_t r = (uint32_t)q * kFlowThreads + tid;
      if (r < nr) early[q] = ask(a, at<uint32_t>(far_word(k, r), 0), at<uint32_t>(far_word(k, r) + 128u, 0), w);
    }
#pragma unroll 1
    for (uint32_t r = tid; r < nl; r += kFlowThreads) {
      const uint32_t op = at<uint32_t>(near_word(k, r), 0), e = near_at(k, r);
      at<float4>(e + 512u, 0) =
          update(a, at<float4>(e, 0), at<float4>(e + 512u, 0), at<float4>(k.U, op & 0xffffu), at<float4>(k.U, op >> 16));
    }
#pragma unroll 1
    for (uint32_t r = tid; r < nr; r += kFlowThreads) {
      const uint32_t of = at<uint32_t>(far_word(k, r), 0), id = at<uint32_t>(far_word(k, r) + 128u, 0), e = far_at(k, r);
      float4 uj = early[0];
      if (r >= kFlowThreads) uj = r < 2u * kFlowThreads ? early[1] : ask(a, of, id, w);
      uj = answer<FREE>(a, of, id, uj, w, wt);
      const float4 l = update(a, at<float4>(e, 0), at<float4>(e + 512u, 0), at<float4>(k.U, of & 0xffffu), uj);
      at<float4>(e + 512u, 0) = l;
      if (FREE && (of & kFree)) give(a, of, id, l);
    }
#pragma unroll 1
    for (uint32_t m = tid; m < nm; m += kFlowThreads) {
      const uint2 r = a.flow_r[scratch(a) + m];
      const float4 nn = a.flow_n[scratch(a) + m], la = a.flow_l[scratch(a) + m];
      const float4 uj = (r.x & kNear) ? at<float4>(k.U, r.y) : answer<FREE>(a, r.x, r.y, ask(a, r.x, r.y, w), w, wt);
      const float4 l = update(a, nn, la, at<float4>(k.U, r.x & 0xffffu), uj);
      a.flow_l[scratch(a) + m] = l;
      if (FREE && (r.x & kFree)) give(a, r.x, r.y, l);
    }
    __syncthreads();
    // new estimates: the impulses of each sphere summed in contact order
#pragma unroll 1
    for (uint32_t o = tid; o < 32u * k.nt; o += kFlowThreads) {
      const uint32_t cf = at<uint8_t>(k.cnt, o), cnt = cf & 0x7fu;
      if (!cnt) continue;
      const uint32_t i = place_id(o);
      const float uw = at<float4>(k.U, o).w;
      const float4 base = k.base ? at<float4>(k.base, o) : base_velocity(a, a.vel_id[i]);
      const float3 S = sum_impulses(a, refs_of(k, o), cnt);
      const float4 un = make_float4(base.x + base.w * S.x, base.y + base.w * S.y, base.z + base.w * S.z, uw);
      if (s + 1u < iters) {
        if (cf & kFar) st_tagged(a.T[(s + 1u) & 1u] + i, un.x, un.y, un.z, w.pub);
        at<float4>(k.U, o) = un;
      } else {
        a.U[iters & 1u][i] = un;
      }
    }
    __syncthreads();
  }
  // the impulses, for the readbacks and the wrenches
  const size_t n = a.n;
#pragma unroll 1
  for (uint32_t o = tid; o < 32u * k.nt; o += kFlowThreads) {
    const uint32_t cnt = at<uint8_t>(k.cnt, o) & 0x7fu;
    if (!cnt) continue;
    const uint32_t ref = refs_of(k, o);
    const uint32_t i = place_id(o), npp = a.ccount[i] & 0xffu;
#pragma unroll 1
    for (uint32_t c = 0; c < cnt; ++c) {
      const uint32_t r = at<uint32_t>(ref, 32u * c);
      const float sg = (r & kSign) ? -1.f : 1.f;
      const float4 l = referred(a, r);
      if (c < npp) {
        a.clam[(size_t)c * n + i] = make_float4(sg * l.x, sg * l.y, sg * l.z, 0.f);
      } else {
        float *d = a.blam + (size_t)(c - npp) * n + i;
        const size_t plane = (size_t)a.Kb * n;
        d[0] = sg * l.x;
        d[plane] = sg * l.y;
        d[2 * plane] = sg * l.z;
      }
    }
  }
}

// A record without its place: normal and bias, zero impulse and effective mass, of sphere
// i's contact c (uw: its n / m).  Partner: the place of a near one, the id of a far one, or
// for a body contact the slot of its point in flow_b (kinematic: the point's velocity;
// free: lever arm and body).
template <bool FREE>
__device__ __forceinline__ void fill_record(const StepArgs &a, const Block &k, uint32_t i, uint32_t c, float uw, uint32_t flags,
                                            uint32_t code, float4 *N, float4 *L) {
  const size_t n = a.n;
  float4 nn;
  float ow;
  if (!(flags & kBody)) {
    nn = a.cn[(size_t)c * n + i];
    ow = (flags & kNear) ? at<float4>(k.U, code).w : a.U[0][code].w;
  } else {
    const size_t o = (size_t)c * n + i;
    uint32_t gb = a.bj[o];
    if (!GG_GUARD(a.ctrl, gb < a.n_envs * a.maxb)) gb = 0;
    const DevBody &B = a.bodies[gb];
    const float4 xc = a.bxc[o];
    nn = a.bn[o];
    const float rx = xc.x - B.p[0], ry = xc.y - B.p[1], rz = xc.z - B.p[2];
    ow = FREE ? body_inv(a, B, gb, nn, rx, ry, rz) : 0.f;
    float4 rb = make_float4(rx, ry, rz, __uint_as_float(gb << 3 | c));
    if (!FREE || !(flags & kFree)) {
      const float3 ub = point_velocity(make_float3(B.v[0], B.v[1], B.v[2]), make_float3(B.w[0], B.w[1], B.w[2]), rx, ry, rz);
      rb = make_float4(ub.x, ub.y, ub.z, 0.f);
    }
    a.flow_b[body_scratch(a) + code] = rb;
  }
  *N = make_float4(nn.x, nn.y, nn.z, a.ab * nn.w);
  *L = make_float4(0.f, 0.f, 0.f, 1.0f / (uw + ow));
}

__device__ __forceinline__ uint2 block_scan2(uint2 v, uint2 *total, uint2 *ws) {
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  const uint2 inc = make_uint2(warp_incl_scan(v.x), warp_incl_scan(v.y));
  if (lane == 31) ws[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    const uint2 s = lane < kFlowWarps ? ws[lane] : make_uint2(0u, 0u);
    const uint2 si = make_uint2(warp_incl_scan(s.x), warp_incl_scan(s.y));
    if (lane < kFlowWarps) ws[lane] = make_uint2(si.x - s.x, si.y - s.y);
    if (lane == 31) ws[kFlowWarps] = si;
  }
  __syncthreads();
  *total = ws[kFlowWarps];
  return make_uint2(ws[wid].x + inc.x - v.x, ws[wid].y + inc.y - v.y);
}

// The block's share of a range's tiles, found from the per-tile contact counts.
struct Share {
  uint2 pre;           // (tiles with contacts, their cost) before the thread's own tiles
  uint32_t ta, tb;     // the thread's own tiles ...
  uint32_t own;        // ... and their cost
  uint32_t lo, hi;     // the block's window of the cost prefix
};
__host__ __device__ __forceinline__ uint32_t tile_cost(uint32_t v) {
  const uint32_t c = (v & 0xffffu) + kTileWeight, b = (4u + 2u + 32u + 512u + 128u * (v >> 16)) / kBytesPerCost + 1u;
  return v ? (c > b ? c : b) : 0u;
}

// f(tile, tiles with contacts before, its count word) for the thread's tiles that are in
// the block's window.
template <typename Fn>
__device__ __forceinline__ void each_tile(const StepArgs &a, const Share &h, uint32_t t0, uint32_t t1, Fn f) {
  uint2 q = h.pre;
  if (q.y >= h.hi || q.y + h.own <= h.lo) return;
#pragma unroll 1
  for (uint32_t t = h.ta; t < h.tb; t += 4) {
    const uint4 v4 = *reinterpret_cast<const uint4 *>(a.tile_work + t);
    const uint32_t v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) {
      if (t + u < t0 || t + u >= t1 || !v[u]) continue;
      if (q.y >= h.lo && q.y < h.hi) f(t + u, q.x, v[u]);
      q.x += 1u;
      q.y += tile_cost(v[u]);
    }
  }
}

template <bool FREE>
__global__ void __launch_bounds__(kFlowThreads, 1) k_flow(const __grid_constant__ StepArgs a, uint32_t iters, uint32_t pool_bytes) {
  pdl_enter();
  __shared__ uint2 s_ws[kFlowWarps + 1];
  __shared__ uint32_t s_c0, s_c1, s_rows;   // tiles before the block's first and last, its rows of references
  __shared__ uint32_t s_all, s_nl, s_nr;    // records handed out (near | far << 16), and taken, of either kind
  __shared__ uint32_t s_nm, s_nb;           // records in memory, with bodies
  __shared__ uint32_t s_plain[kFlowMaxWaves / 32u];
  const uint32_t G = gridDim.x - (FREE ? a.F : 0u);
  const uint32_t out0 = *a.epoch;
  // ranges that get the plain sweeps: all of them when a list may be asymmetric
  const uint32_t sym = a.flow == kFlowCheck ? a.list_sym[(threadIdx.x & 31u) * kSymStride] : 0u;
  const bool asym = ((a.ctrl->status & kAsymmetric) | __reduce_add_sync(0xffffffffu, sym)) != 0u;
  // (a phantom participant, for tests of the bounded waits: tags that nothing writes)
  const uint32_t tag0 = out0 + (a.ctrl->bar_extra ? 0x40000000u : 0u);
  Waits wt{false};
  const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5;
  if (tid < kFlowMaxWaves / 32u) s_plain[tid] = 0u;
  const size_t n = a.n;
  for (uint32_t wave = 0; wave < a.n_waves && !asym; ++wave) {
    const uint32_t p0 = a.n_waves == 1 ? 0u : a.wave_off[wave], p1 = a.n_waves == 1 ? a.n : a.wave_off[wave + 1];
    if (p0 >= p1) continue;
    // ---- the block's tiles: an equal share of the range's cost
    const uint32_t t0 = p0 >> 5, t1 = (p1 + 31u) >> 5, ts = t0 & ~3u;
    const uint32_t per = ((t1 - ts + kFlowThreads - 1u) / kFlowThreads + 3u) & ~3u;
    Share h;
    h.ta = min(ts + tid * per, t1);
    h.tb = min(h.ta + per, t1);
    if (tid == 0) {
      s_c0 = kNone;
      s_c1 = s_rows = s_all = s_nl = s_nr = s_nm = s_nb = 0;
    }
    uint2 sum = make_uint2(0u, 0u);
#pragma unroll 2
    for (uint32_t t = h.ta; t < h.tb; t += 4) {
      const uint4 v4 = *reinterpret_cast<const uint4 *>(a.tile_work + t);
      const uint32_t v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
      for (uint32_t u = 0; u < 4; ++u) {
        if (t + u < t0 || t + u >= t1) continue;
        sum.x += v[u] ? 1u : 0u;
        sum.y += tile_cost(v[u]);
      }
    }
    uint2 tot;
    h.pre = block_scan2(sum, &tot, s_ws);
    h.own = sum.y;
    const uint32_t W = tot.y;
    const uint32_t Gw = min(G, max(1u, W / kMinWork));
    // no share costs more than W / Gw + kTileMax: its lists fit the shared memory, its records
    // the references' range (every block sees the same totals)
    static_assert(kFlowRecords >= 227u * 1024u / kBytesPerCost, "as many records as a share that fits can have");
    if ((W / Gw + kTileMax) * kBytesPerCost + 256u > pool_bytes) {
      if (tid == 0) s_plain[wave >> 5] |= 1u << (wave & 31u);
      __syncthreads();
      continue;
    }
    if (FREE && blockIdx.x >= G) {
      free_block(a, blockIdx.x - G, iters, out0, wt);
      return;
    }
    if (W == 0 || blockIdx.x >= Gw) {
      __syncthreads();
      continue;
    }
    h.lo = (uint32_t)((uint64_t)W * blockIdx.x / Gw);
    h.hi = (uint32_t)((uint64_t)W * (blockIdx.x + 1u) / Gw);
    {
      uint32_t cf = kNone, cl = 0, rw = 0;
      each_tile(a, h, t0, t1, [&](uint32_t, uint32_t c, uint32_t v) {
        cf = min(cf, c);
        cl = c + 1u;
        rw += v >> 16;
      });
      if (cl) {
        atomicMin(&s_c0, cf);
        atomicMax(&s_c1, cl);
        atomicAdd(&s_rows, rw);
      }
    }
    __syncthreads();
    const uint32_t c0 = s_c0;
    Block k;
    k.nt = s_c1 ? s_c1 - c0 : 0u;
    if (!k.nt) {
      __syncthreads();
      continue;
    }
    k.row = 4u * k.nt;
    k.cnt = k.row + 2u * k.nt;
    k.ref = (k.cnt + 32u * k.nt + 15u) & ~15u;
    k.U = k.ref + 128u * s_rows;
    k.rec = k.U + 512u * k.nt;
    k.top = pool_bytes;
    each_tile(a, h, t0, t1, [&](uint32_t t, uint32_t c, uint32_t) { at<uint32_t>(0, c - c0) = t; });
    __syncthreads();
    if (tid == 0) s_rows = 0;
    __syncthreads();
    // ---- spheres and their contacts' places: a warp takes up a tile, a lane a sphere; a
    // record's slot keeps which contact it is until the next stage
    for (uint32_t t = wid; t < k.nt; t += kFlowWarps) {
      const uint32_t o = 32u * t + lane, i = at<uint32_t>(0, t) * 32u + lane;
      const bool own = i >= p0 && i < p1;
      const uint32_t cc = own ? a.ccount[i] : 0u, npp = cc & 0xffu, cnt = npp + ((cc >> 8) & 0xffu);
      at<float4>(k.U, o) = cnt ? a.U[0][i] : make_float4(0.f, 0.f, 0.f, 0.f);
      const uint32_t most = __reduce_max_sync(0xffffffffu, cnt);
      uint32_t row = 0;
      if (lane == 0) row = atomicAdd(&s_rows, most);
      row = __shfl_sync(0xffffffffu, row, 0);
      if (lane == 0) at<uint16_t>(k.row, t) = (uint16_t)row;
      // the partners first, several loads in flight, then their places row by row
#pragma unroll 4
      for (uint32_t c = 0; c < npp; ++c) at<uint32_t>(k.ref, (row + c) * 32u + lane) = a.cj[(size_t)c * n + i];
      uint32_t far = 0, nn = 0, nf = 0;   // near and far records of the tile
#pragma unroll 1
      for (uint32_t c = 0; c < most; ++c) {
        bool near = false;
        if (c < npp) {
          uint32_t code = at<uint32_t>(k.ref, (row + c) * 32u + lane);
          if (!GG_GUARD(a.ctrl, code < a.n)) code = i;
          const uint32_t pl = place_of(k, code, p0, p1);
          if (pl == kNone) far = kFar;
          else at<uint32_t>(k.ref, (row + c) * 32u + lane) = open_ref(pl);
          near = pl != kNone && pl > o;
          nf += pl == kNone ? 1u : 0u;
        } else if (c < cnt) {
          nf += 1u;
        }
        nn += near ? 1u : 0u;
      }
      // their slots, a lane's side by side (the slot keeps which contact it is until the next stage)
      const uint32_t in = warp_incl_scan(nn | nf << 16), sum2 = __shfl_sync(0xffffffffu, in, 31);
      uint32_t got = 0;
      if (lane == 0) got = atomicAdd(&s_all, sum2);
      got = __shfl_sync(0xffffffffu, got, 0);
      const uint32_t el = (got & 0xffffu) + (sum2 & 0xffffu), er = (got >> 16) + (sum2 >> 16);
      const bool fits = k.rec + ((el + 31u) >> 5) * kNearChunk + ((er + 31u) >> 5) * kFarChunk <= k.top;
      if (fits && lane == 0) {
        atomicMax(&s_nl, el);
        atomicMax(&s_nr, er);
      }
      uint32_t rn = (got & 0xffffu) + (in & 0xffffu) - nn, rf = (got >> 16) + (in >> 16) - nf;
#pragma unroll 1
      for (uint32_t c = 0; c < cnt; ++c) {
        uint32_t code = c < npp ? at<uint32_t>(k.ref, (row + c) * 32u + lane) : 0u;   // partner
        uint32_t word = o, kc = c;                                                    // place and flags, contact of its kind
        const bool local = c < npp && (code & kOpen);
        if (local) code = (code & kRefBits) >> 4;
        if (local && code < o) continue;
        if (c >= npp) {
          kc = c - npp;
          code = atomicAdd(&s_nb, 1u);
          word |= kBody | (FREE && a.bodies[a.bj[(size_t)kc * n + i]].is_free ? kFree : 0u);
        }
        uint32_t ref;
        if (fits) {
          const uint32_t r = local ? rn++ : rf++;
          const uint32_t e = local ? near_at(k, r) : far_at(k, r), wd = local ? near_word(k, r) : far_word(k, r);
          at<uint32_t>(wd, 0) = local ? (o | code << 16) : word;
          if (!local) at<uint32_t>(wd + 128u, 0) = code;
          ref = e + 512u;
          at<uint32_t>(ref, 0) = kc;
        } else {
          const uint32_t m = atomicAdd(&s_nm, 1u);
          a.flow_r[scratch(a) + m] = make_uint2(word | (local ? kNear : 0u), code);
          ref = kMem | m;
          a.flow_l[scratch(a) + m] = make_float4(__uint_as_float(kc), 0.f, 0.f, 0.f);
        }
        at<uint32_t>(k.ref, (row + c) * 32u + lane) = ref;
      }
      at<uint8_t>(k.cnt, o) = (uint8_t)(cnt | far);
    }
    __syncthreads();
    // ---- the records themselves, a thread each; and a near pair's second sphere learns
    // where its record is
    const uint32_t nl = s_nl, nr = s_nr, nm = s_nm;
    auto resolve = [&](uint32_t o, uint32_t p, uint32_t ref) {
      const uint32_t pc = at<uint8_t>(k.cnt, p) & 0x7fu, pr = refs_of(k, p);
#pragma unroll 2
      for (uint32_t d = 0; d < pc; ++d)
        if (at<uint32_t>(pr, 32u * d) == open_ref(o)) at<uint32_t>(pr, 32u * d) = ref | kSign;
    };
#pragma unroll 1
    for (uint32_t r = tid; r < nl; r += kFlowThreads) {
      const uint32_t op = at<uint32_t>(near_word(k, r), 0), o = op & 0xffffu, e = near_at(k, r);
      float4 N, L;
      fill_record<FREE>(a, k, place_id(o), at<uint32_t>(e + 512u, 0), at<float4>(k.U, o).w, kNear, op >> 16, &N, &L);
      at<float4>(e, 0) = N;
      at<float4>(e + 512u, 0) = L;
      resolve(o, op >> 16, e + 512u);
    }
#pragma unroll 1
    for (uint32_t r = tid; r < nr; r += kFlowThreads) {
      const uint32_t of = at<uint32_t>(far_word(k, r), 0), id = at<uint32_t>(far_word(k, r) + 128u, 0), e = far_at(k, r);
      float4 N, L;
      fill_record<FREE>(a, k, place_id(of & 0xffffu), at<uint32_t>(e + 512u, 0), at<float4>(k.U, of & 0xffffu).w, of, id, &N, &L);
      at<float4>(e, 0) = N;
      at<float4>(e + 512u, 0) = L;
    }
#pragma unroll 1
    for (uint32_t m = tid; m < nm; m += kFlowThreads) {
      const uint2 r = a.flow_r[scratch(a) + m];
      const uint32_t o = r.x & 0xffffu;
      float4 N, L;
      fill_record<FREE>(a, k, place_id(o), __float_as_uint(a.flow_l[scratch(a) + m].x), at<float4>(k.U, o).w, r.x, r.y, &N, &L);
      a.flow_n[scratch(a) + m] = N;
      a.flow_l[scratch(a) + m] = L;
      if (r.x & kNear) resolve(o, r.y, kMem | m);
    }
    // what is left of the shared memory takes the velocities before impulses
    const uint32_t end = k.rec + ((nl + 31u) >> 5) * kNearChunk, low = k.top - ((nr + 31u) >> 5) * kFarChunk;
    k.base = end + 512u * k.nt <= low ? end : 0u;
    if (k.base)
      for (uint32_t o = tid; o < 32u * k.nt; o += kFlowThreads)
        if (at<uint8_t>(k.cnt, o)) at<float4>(k.base, o) = base_velocity(a, a.vel_id[place_id(o)]);
    __syncthreads();
    sweeps<FREE>(a, k, iters, nl, nr, nm, tag0, out0, wt);
    __syncthreads();
  }
  __syncthreads();
  if (a.flow_told && blockIdx.x == 0 && tid == 0) {  // the host chooses another set when it next steps
    uint32_t plain = 0;
    for (uint32_t wave = 0; wave < a.n_waves; ++wave)
      if (asym || (s_plain[wave >> 5] >> (wave & 31u) & 1u)) plain += a.wave_off[wave + 1] - a.wave_off[wave];
    if (plain > a.n / 2u) *(volatile uint32_t *)a.flow_told = 1u;
  }
  for (uint32_t wave = 0; wave < a.n_waves; ++wave)
    if (asym || (s_plain[wave >> 5] >> (wave & 31u) & 1u)) barrier_sweeps(a, iters, G, a.wave_off[wave], a.wave_off[wave + 1]);
}

template <bool FREE>
int flow_setup_for(uint32_t *pool) {
  cudaFuncAttributes at{};
  int dev = 0, optin = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaFuncGetAttributes(&at, k_flow<FREE>) != cudaSuccess)
    return 0;
  *pool = ((uint32_t)optin - (uint32_t)at.sharedSizeBytes) & ~255u;
  if (cudaFuncSetAttribute(k_flow<FREE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*pool) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_flow<FREE>, kFlowThreads, *pool) != cudaSuccess)
    return 0;
  return per;
}

}  // namespace

int flow_setup(bool free, uint32_t *pool) {
  const int per = free ? flow_setup_for<true>(pool) : flow_setup_for<false>(pool);
  if (!per) (void)cudaGetLastError();
  return per;
}

// A settled bed costs 3.5 to 3.8 a sphere (three contacts, a tile's weight, tiles of uneven
// lists); with a margin for denser ones that is 302,000 spheres on 152 SMs.  (Sweep stage of
// a batch of 1.64 million spheres, 2.7 contacts each, with 3.6, 4.2, 6.3 and 8.4: 870, 799, 948
// and 930 us: too large a range does not fit, too small a one pays the load more often.)
constexpr double kSettledCost = 4.2;
uint32_t flow_range(uint32_t grid, uint32_t pool) {
  return (uint32_t)(grid * (double)((pool - 256u) / kBytesPerCost - kTileMax) / kSettledCost);
}

// (With all 152 blocks at any size, two simulations in two streams took turns: 4,096 spheres
// 62 us a step alone and 88 for a step of both, now 68; 1,000 spheres 60, 84 and now 65.)
uint32_t flow_blocks(uint32_t most) {
  constexpr uint32_t kCrowded = 32u * 8u;  // contacts of a tile: above a dense packing's six a sphere
  return (uint32_t)(((uint64_t)most / 32u + 1u) * tile_cost(kCrowded | 12u << 16) / kMinWork) + 1u;
}

// A block's share costs at most W / Gw + one tile (W the range's cost, Gw = min(grid, W /
// kMinWork) the blocks that share it); its lists take at most kBytesPerCost bytes per cost
// and it has at most as many records as its cost, 40 bytes each and two chunks for rounding.
FlowScratch flow_scratch(const StepArgs &a, uint32_t most, uint32_t grid, uint32_t pool) {
  const uint64_t per = a.K + a.Kb, tile = tile_cost((uint32_t)(32u * per | per << 16));
  const uint64_t g = std::max(1u, grid), W = ((uint64_t)most / 32u + 2u) * tile;
  const uint64_t share = std::max(std::min<uint64_t>(W, 2u * kMinWork - 1u), W / g) + tile;
  const bool on_chip = share * (kBytesPerCost + 40u) + 256u + kNearChunk + kFarChunk <= pool;
  FlowScratch f;
  f.blocks = (uint32_t)std::min(g, std::max<uint64_t>(1u, W / kMinWork));
  f.records = on_chip ? 0u : (uint32_t)std::min<uint64_t>(share, kFlowRecords);
  f.bodies = (uint32_t)std::min({share, (uint64_t)kFlowRecords, (uint64_t)most * a.Kb});
  return f;
}

cudaError_t enqueue_flow(const StepArgs &a, const LaunchShape &ls, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ls.flow_grid);
  cfg.blockDim = dim3(kFlowThreads);
  cfg.dynamicSmemBytes = ls.flow_pool;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, a.F ? k_flow<true> : k_flow<false>, a, ls.iters, ls.flow_pool);
}

}  // namespace gg
