// gg_sweep.cuh -- the projected-Jacobi update of one particle and of one free body, and the
// grid barrier: shared by the per-launch sweeps (gg_kernels.cu) and the one-launch
// dataflow sweeps (gg_flow.cu), so that both compile the same arithmetic.
#pragma once
#include "gg_device.cuh"

namespace gg {

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Fixed-order sum of 6 floats over the block, result valid in thread 0.
template <int NT>
__device__ __forceinline__ void block_sum6(float v[6]) {
  __shared__ float sm[NT / 32][6];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 6; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < 6; ++k) sm[wid][k] = v[k];
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      float s = sm[0][k];
      for (int w = 1; w < NT / 32; ++w) s += sm[w][k];
      v[k] = s;
    }
  }
}

__device__ __forceinline__ void flag(DevCtrl *c, uint32_t f) { atomicOr(&c->status, f); }

// a contact's record before its first update: no impulse, the partner's id
__device__ __forceinline__ float4 no_impulse(uint32_t j) { return make_float4(0.f, 0.f, 0.f, __uint_as_float(j)); }

// v + dt g (the velocity before contact impulses), with 1/m in w; the fused multiply-add is
// spelled out, so that a hoisted product cannot round differently in one of the callers
__device__ __forceinline__ float4 base_velocity(const StepArgs &a, float4 v) {
  return make_float4(__fmaf_rn(a.dt, a.g[0], v.x), __fmaf_rn(a.dt, a.g[1], v.y), __fmaf_rn(a.dt, a.g[2], v.z), v.w);
}

// One Jacobi update of particle i: U[s] -> U[s^1] (s: double-buffer index).
// TAPE: also keep the iterates in tape slot it + 1 (it = iteration number).
// LDCG: read the velocity estimates through L2 only (the fused kernel reads, within
// one launch, estimates that other SMs wrote in the previous iteration).
// PRE: load the records of slots 0 and 1 together with the counts (below).
template <bool TAPE, bool LDCG, bool PRE = false>
__device__ __forceinline__ void pja_particle(const StepArgs &a, uint32_t i, int s, const Tape &tp, int it) {
  const float4 *__restrict__ Uin = a.U[s];
  const float4 *__restrict__ cn = a.cn;
  float4 *__restrict__ clam = a.clam;
  const size_t n = a.n;
  const uint32_t cc = a.ccount[i];
  const uint32_t npp = cc & 0xffu, nbc = (cc >> 8) & 0xffu;
  const float4 ui = LDCG ? __ldcg(Uin + i) : Uin[i];
  const float4 base = base_velocity(a, a.vel_id[i]);
  float sx = 0.f, sy = 0.f, sz = 0.f;
  const size_t KN = (size_t)a.K * n;
  const float mu = a.mu, ab = a.ab;
  const float pw = a.lit ? 0.f : 1.f;  // partner's share of the effective mass (exact 0 or 1)
  // one contact update (Alg. 1 with the accumulated clamp): new impulse stored (and taped)
  auto update = [&](size_t o, const float4 &nn, const float4 &la, const float4 &uj) {
    const float3 l = pja_project(make_float3(la.x, la.y, la.z), make_float3(ui.x - uj.x, ui.y - uj.y, ui.z - uj.z), make_float3(nn.x, nn.y, nn.z),
                                 ab * nn.w, 1.0f / (ui.w + pw * uj.w), mu);
    clam[o] = make_float4(l.x, l.y, l.z, la.w);
    if (TAPE) {
      float *h = tp.lamh + (size_t)(it + 1) * 3 * KN;
      h[o] = l.x;
      h[o + KN] = l.y;
      h[o + 2 * KN] = l.z;
    }
    return l;
  };
  auto gather = [&](uint32_t j) { return LDCG ? __ldcg(Uin + j) : Uin[j]; };
  // PRE: the records of slots 0 and 1 are loaded together with the counts (those rows
  // exist for every particle; a particle with fewer contacts does not use them), so for
  // most particles the partner gathers are the second dependent load, not the third.
  // That pays on settled beds streaming from DRAM (1M spheres: 35.1 -> 33.6 us per
  // sweep) and costs where most spheres have no contact (the collapsing column: their
  // unused records are 64 bytes of extra reads each, 3.2 -> 3.6 us), so the serpentine
  // launch shapes, which the autotuner picks for the former, use it.
  // (Loading only the partner ids of slots 0 and 1 early was measured too: slower on
  // every workload, 64 registers with spills.)
  const bool two = PRE && a.K > 1;
  float4 pn0 = make_float4(0.f, 0.f, 0.f, 0.f), pn1 = pn0, pl0 = pn0, pl1 = pn0;
  if (PRE) {
    pn0 = cn[i];
    pl0 = clam[i];
    if (two) {
      pn1 = cn[n + i];
      pl1 = clam[n + i];
    }
  }
  // two contacts per round: both rounds' loads issue before either update is stored;
  // the impulses are still added in contact order
  uint32_t c = 0;
  if (two && npp >= 2) {
    uint32_t j0 = __float_as_uint(pl0.w), j1 = __float_as_uint(pl1.w);
    if (!GG_GUARD(a.ctrl, j0 < a.n && j1 < a.n)) j0 = j1 = i;  // debug build: never gather out of range
    const float4 u0 = gather(j0), u1 = gather(j1);
    const float3 l0 = update(i, pn0, pl0, u0);
    const float3 l1 = update(n + i, pn1, pl1, u1);
    sx += l0.x;
    sy += l0.y;
    sz += l0.z;
    sx += l1.x;
    sy += l1.y;
    sz += l1.z;
    c = 2;
  }
  for (; c + 1 < npp; c += 2) {
    const size_t o0 = (size_t)c * n + i, o1 = o0 + n;
    const float4 n0 = cn[o0], n1 = cn[o1];
    const float4 la0 = clam[o0], la1 = clam[o1];
    uint32_t j0 = __float_as_uint(la0.w), j1 = __float_as_uint(la1.w);
    if (!GG_GUARD(a.ctrl, j0 < a.n && j1 < a.n)) j0 = j1 = i;  // debug build: never gather out of range
    const float4 u0 = gather(j0), u1 = gather(j1);
    const float3 l0 = update(o0, n0, la0, u0);
    const float3 l1 = update(o1, n1, la1, u1);
    sx += l0.x;
    sy += l0.y;
    sz += l0.z;
    sx += l1.x;
    sy += l1.y;
    sz += l1.z;
  }
  if (c < npp) {
    const size_t o = (size_t)c * n + i;
    const bool pre = PRE && c == 0;
    const float4 lam = pre ? pl0 : clam[o];
    uint32_t j = __float_as_uint(lam.w);
    if (!GG_GUARD(a.ctrl, j < a.n)) j = i;
    const float4 nn = pre ? pn0 : cn[o];
    const float3 l = update(o, nn, lam, gather(j));
    sx += l.x;
    sy += l.y;
    sz += l.z;
  }
  const size_t KbN = (size_t)a.Kb * n;
  for (uint32_t c = 0; c < nbc; ++c) {
    const size_t o = (size_t)c * n + i;
    const uint32_t gbo = a.bj[o];
    if (!GG_GUARD(a.ctrl, gbo < a.n_envs * a.maxb)) continue;
    const DevBody &B = a.bodies[gbo];
    const float4 nn = a.bn[o];
    const float4 xc = a.bxc[o];
    const float3 lam = make_float3(a.blam[o], a.blam[o + KbN], a.blam[o + 2 * KbN]);
    const float rx = xc.x - B.p[0], ry = xc.y - B.p[1], rz = xc.z - B.p[2];
    // (LDCG: a free body's twist changes within the launch)
    auto tw = [&](const float *p) { return LDCG ? __ldcg(p) : *p; };
    const float bw0 = tw(B.w), bw1 = tw(B.w + 1), bw2 = tw(B.w + 2);
    const float ubx = tw(B.v) + (bw1 * rz - bw2 * ry);
    const float uby = tw(B.v + 1) + (bw2 * rx - bw0 * rz);
    const float ubz = tw(B.v + 2) + (bw0 * ry - bw1 * rx);
    float invb = 0.f;
    if (B.is_free) {  // n_b (1/M + (a x n) . I_w^-1 (a x n)), mass split over the body's contacts
      const float cx = ry * nn.z - rz * nn.y, cy = rz * nn.x - rx * nn.z, cz = rx * nn.y - ry * nn.x;
      const float t0 = B.R[0] * cx + B.R[3] * cy + B.R[6] * cz;
      const float t1 = B.R[1] * cx + B.R[4] * cy + B.R[7] * cz;
      const float t2 = B.R[2] * cx + B.R[5] * cy + B.R[8] * cz;
      invb = (float)a.ncb[gbo] * (1.0f / B.mass + t0 * t0 / B.inertia[0] + t1 * t1 / B.inertia[1] +
                                      t2 * t2 / B.inertia[2]);
    }
    const float w = 1.0f / (ui.w + invb);
    const float3 u = make_float3(ui.x - ubx, ui.y - uby, ui.z - ubz);
    const float3 l = pja_project(lam, u, make_float3(nn.x, nn.y, nn.z), a.ab * nn.w, w, a.mu);
    a.blam[o] = l.x;
    a.blam[o + KbN] = l.y;
    a.blam[o + 2 * KbN] = l.z;
    if (TAPE) {
      float *h = tp.blamh + (size_t)(it + 1) * 3 * KbN;
      h[o] = l.x;
      h[o + KbN] = l.y;
      h[o + 2 * KbN] = l.z;
    }
    sx += l.x;
    sy += l.y;
    sz += l.z;
  }
  const float4 un = make_float4(base.x + base.w * sx, base.y + base.w * sy, base.z + base.w * sz, ui.w);
  a.U[s ^ 1][i] = un;
  if (TAPE) tp.Uh[(size_t)(it + 1) * n + i] = un;
}

// Grid-wide barrier of a cooperative launch (all blocks resident).  The wait is
// bounded: past `limit` SM cycles it latches kFlagTimeout and sets bar_abort, after
// which every later barrier returns at once, so the kernel always finishes.
__device__ __forceinline__ void grid_barrier(DevCtrl *c, long long limit) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile uint32_t *vgen = &c->bar_gen;
    volatile uint32_t *vab = &c->bar_abort;
    const uint32_t gen = *vgen;
    __threadfence();
    const uint32_t arrived = atomicAdd(&c->bar_count, 1u);
    if (arrived == gridDim.x - 1 + c->bar_extra) {
      atomicExch(&c->bar_count, 0u);
      __threadfence();
      atomicAdd(&c->bar_gen, 1u);
    } else if (!*vab) {
      const long long t0 = clock64();
      while (*vgen == gen) {
        if (*vab) break;
        if (clock64() - t0 > limit) {
          atomicOr(&c->status, kFlagTimeout);
          atomicExch(&c->bar_abort, 1u);
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
  }
  __syncthreads();
}

__device__ __forceinline__ float free_inv_mass(const DevBody &B, float3 r, float3 n) {
  const float cx = r.y * n.z - r.z * n.y, cy = r.z * n.x - r.x * n.z, cz = r.x * n.y - r.y * n.x;
  const float t0 = B.R[0] * cx + B.R[3] * cy + B.R[6] * cz;
  const float t1 = B.R[1] * cx + B.R[4] * cy + B.R[7] * cz;
  const float t2 = B.R[2] * cx + B.R[5] * cy + B.R[8] * cz;
  return 1.0f / B.mass + t0 * t0 / B.inertia[0] + t1 * t1 / B.inertia[1] + t2 * t2 / B.inertia[2];
}

// After each sweep, one block of kFreeThreads threads per free body: update its corner
// contacts (against the twist of this iteration), sum every impulse it received in a fixed
// order, and set its twist for the next iteration (Newton-Euler, gyroscopic term dropped).
// LDCG: read the particles' impulses through L2 (written by other SMs of the same launch).
// NT: threads of the block (those past kFreeThreads only add zeros to the sums).
constexpr int kFreeThreads = 256;

template <int NT, bool LDCG>
__device__ __forceinline__ void free_update(const StepArgs &a, uint32_t fid, uint32_t gb) {
  DevBody &B = a.bodies[gb];
  const uint32_t e = gb / a.maxb;
  const float nb = (float)a.ncb[gb];
  const float3 V = make_float3(B.v[0], B.v[1], B.v[2]), W = make_float3(B.w[0], B.w[1], B.w[2]);
  float v[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  CornerContact *cc = a.fcc + (size_t)fid * 8 * a.maxb;
  const uint32_t t0 = threadIdx.x < kFreeThreads ? threadIdx.x : 0x40000000u;  // past every loop's end
  for (uint32_t t = t0; t < 8 * a.maxb; t += kFreeThreads) {
    CornerContact c = cc[t];
    if (!c.valid) continue;
    const DevBody &O = a.bodies[e * a.maxb + c.o];
    const float3 r = make_float3(c.xc[0] - B.p[0], c.xc[1] - B.p[1], c.xc[2] - B.p[2]);
    const float3 ro = make_float3(c.xc[0] - O.p[0], c.xc[1] - O.p[1], c.xc[2] - O.p[2]);
    const float3 ub = make_float3(V.x + W.y * r.z - W.z * r.y, V.y + W.z * r.x - W.x * r.z, V.z + W.x * r.y - W.y * r.x);
    const float3 uo = make_float3(O.v[0] + O.w[1] * ro.z - O.w[2] * ro.y, O.v[1] + O.w[2] * ro.x - O.w[0] * ro.z,
                                  O.v[2] + O.w[0] * ro.y - O.w[1] * ro.x);
    const float3 nn = make_float3(c.n[0], c.n[1], c.n[2]);
    const float w = 1.0f / (nb * free_inv_mass(B, r, nn));
    const float3 l = pja_project(make_float3(c.lam[0], c.lam[1], c.lam[2]),
                                 make_float3(ub.x - uo.x, ub.y - uo.y, ub.z - uo.z), nn, a.ab * c.psi, w, a.mu);
    cc[t].lam[0] = l.x;
    cc[t].lam[1] = l.y;
    cc[t].lam[2] = l.z;
    v[0] += l.x;
    v[1] += l.y;
    v[2] += l.z;
    v[3] += r.y * l.z - r.z * l.y;
    v[4] += r.z * l.x - r.x * l.z;
    v[5] += r.x * l.y - r.y * l.x;
  }
  const size_t n = a.n, KbN = (size_t)a.Kb * n;
  const uint32_t cnt = min(a.fcount[fid], a.Lcap);
  const uint32_t *lst = a.flist + (size_t)fid * a.Lcap;
  for (uint32_t t = t0; t < cnt; t += kFreeThreads) {
    const uint32_t code = lst[t];
    const size_t o = (size_t)(code % a.Kb) * n + code / a.Kb;
    const float fx = -(LDCG ? __ldcg(a.blam + o) : a.blam[o]), fy = -(LDCG ? __ldcg(a.blam + o + KbN) : a.blam[o + KbN]),
                fz = -(LDCG ? __ldcg(a.blam + o + 2 * KbN) : a.blam[o + 2 * KbN]);
    const float4 xc = a.bxc[o];
    const float rx = xc.x - B.p[0], ry = xc.y - B.p[1], rz = xc.z - B.p[2];
    v[0] += fx;
    v[1] += fy;
    v[2] += fz;
    v[3] += ry * fz - rz * fy;
    v[4] += rz * fx - rx * fz;
    v[5] += rx * fy - ry * fx;
  }
  block_sum6<NT>(v);
  if (threadIdx.x == 0) {
    const float im = 1.0f / B.mass;
    // I_w^-1 L = R diag(1/I) R^T L
    const float t0 = (B.R[0] * v[3] + B.R[3] * v[4] + B.R[6] * v[5]) / B.inertia[0];
    const float t1 = (B.R[1] * v[3] + B.R[4] * v[4] + B.R[7] * v[5]) / B.inertia[1];
    const float t2 = (B.R[2] * v[3] + B.R[5] * v[4] + B.R[8] * v[5]) / B.inertia[2];
    B.v[0] = B.own_v[0] + a.dt * a.g[0] + im * v[0];
    B.v[1] = B.own_v[1] + a.dt * a.g[1] + im * v[1];
    B.v[2] = B.own_v[2] + a.dt * a.g[2] + im * v[2];
    B.w[0] = B.own_w[0] + (B.R[0] * t0 + B.R[1] * t1 + B.R[2] * t2);
    B.w[1] = B.own_w[1] + (B.R[3] * t0 + B.R[4] * t1 + B.R[5] * t2);
    B.w[2] = B.own_w[2] + (B.R[6] * t0 + B.R[7] * t1 + B.R[8] * t2);
  }
}

}  // namespace gg
