// p2g.cu -- particle-to-grid transfer of the free-motion solve (Eq. (6),
// MLS-MPM with quadratic B-splines) fused with contact registration
// (Sec. V-B: one contact point per particle inside a rigid geometry, at the
// start of the substep).
//
// A warp stages 32 or 96 particles in shared memory and three nine-lane
// walkers go through them in cell order, each lane summing three nodes of the
// current cell's stencil in registers (details at p2g_walk_block).
//
// The Kirchhoff stress comes precomputed from the previous G2P, so no SVD
// runs here.
#include "kernels.h"

namespace mpmcr {

namespace {

// Whether body b may hold a point of the box with centre c and half extents
// h. The signed distance is 1-Lipschitz, so a body whose distance at c exceeds
// the half diagonal holds none. A body inside the ball of radius b.bound
// around its origin is at least |c - p| - bound away from c, so the ball is
// tried first (with slack, so it only rejects bodies the distance would
// reject too) and the signed distance, whose branch differs between the
// lanes' primitives, is evaluated only for the bodies that it leaves.
__device__ __forceinline__ bool box_may_touch(const DevBody& b, float c0, float c1, float c2,
                                              float h0, float h1, float h2) {
  const float thr = sqrtf(h0 * h0 + h1 * h1 + h2 * h2) * 1.001f + 1e-6f;
  const float r0 = c0 - b.p[0], r1 = c1 - b.p[1], r2 = c2 - b.p[2];
  const float lim = (b.bound + thr) * 1.0001f + 1e-5f;  // inf for an unbounded body
  if (r0 * r0 + r1 * r1 + r2 * r2 > lim * lim) return false;
  float nrm[3];
  return body_sdf(b, c0, c1, c2, nrm) <= thr;
}

// Nine lanes per particle, three particles at a time: the lanes of a third of
// the warp (a walker) own the nine node rows (cy, cz) of the current cell's
// stencil and hold the row's three nodes' sums in registers. The warp first
// stages its particles in shared memory, per unit mass: b = v (+ h f_ext / m)
// + A f and A = -dx (C - h 4/dx^2 (V/m) tau), f the particle's position in its
// base cell, so that the node at offset c receives w m and w m (b - A c), the
// APIC momentum m v + (m C - h 4/dx^2 V tau)(x_j - x_p). Each walker then goes
// through its share of the particles in cell order: a particle costs four
// broadcast loads and two of its lanes' own weights for three nodes each,
// where a lane per node needs five loads for one, and no shuffles.
// When the walker enters another cell it adds the sums to the grid (one
// red.global.add.v4.f32 per node); moving to the next cell along x it adds
// only the column that it leaves and keeps the two that the cells share.
//
// Order: each 32 staged particles are put in shared memory grouped by their
// current cell (not by the cell that the step's sort saw), so that particles
// that have crossed a cell face since then do not cut the walk into runs of
// one. On lattice layers that lie on cell faces that alone took a lane-per-node
// gather over runs of equal cells from 259 to 450 us within the ten substeps
// of one step (4M particles in 32 objects).
//
// Staging: the raw planes of all the warp's sets are copied into shared memory
// asynchronously, 16 bytes per lane, before anything waits, and turned into
// records in place: one exposed memory latency per warp instead of two per 32
// particles (long-scoreboard stalls 2.6 -> 0.9 cycles per issued instruction).
//
// Bound by shared-memory traffic and instruction issue together (1M elastic
// particles at 8 per cell: the L1's data path 81% busy, 66% of the issue slots,
// 1,084 instructions per 32 particles) and, near one particle per cell, by the
// walkers' cell changes and the reductions too (1M sand: 1,779 instructions, 60%,
// L2 42%; 270-290 G red.v4/s measured on GB300, 0.9 per clock and SM: why columns
// shared by cells adjacent in x are kept). Measured per launch, against the better of
// the lane-per-node gather into a shared window and the scatter with a shuffle
// pre-reduction that it replaces: 1M elastic particles at 8 per cell 73 -> 51
// us, 4M in 32 objects 395 -> 231 us, 1M sand at one per cell 126 -> 94 us,
// 250,000 sand at four per cell 30.5 -> 22.5 us, 8,000 particles 12.0 -> 8.9 us.
// A node takes more, smaller sums than from a window per block, which rounds a
// little more: ten substeps of elastic particles in flight were 1.02 (1M) to 1.07
// times (36,000 on a sparse grid) as far from 64 bits in v and C. The grid update's
// single rounding and G2P's differences take off more than that (0.93 to 1.00 of
// the error with the window and the sums over v_i; sand the same with all).
//
// Rounds: a warp that takes three sets gives each walker a set of its own and
// cuts fewer cells between walkers; with few particles one set per warp spreads
// the work over more SMs and shortens each warp's chain. us per launch with one
// and with three sets: elastic at 8 per cell 79,507 13.3 and 16.4, 125,000 13.7 and
// 14.8, 157,464 14.6 and 14.1, 250,047 24.7 and 23.0, 1M 59.5 and 51.6; sand at 4 per
// cell 160,000 18.2 and 20.7, 250,000 22.4 and 22.7; at one per cell 250,000 27.1 and
// 29.7, 1M 79.6 and 78.4. The line is where the denser one crosses.
constexpr int kWalkOneRound = 160000;  // fewer particles than this: one set per warp
constexpr int kWalkThreads = 32;  // a warp per block: blocks spread evenly, and nothing is shared
constexpr int kRawPlanes = 21;  // x, v, C, tau as copied from the particle planes

// One set of 32 staged particles. It arrives as raw planes and is turned into
// records in place. 728 words: the walkers' sets start 24 banks apart.
struct __align__(16) WalkSet {
  union {
    struct {
      float4 row[4][33];  // (b, key), (A00 A10 A01 A11), (A02 A12 A20 A21), (A22, m wx)
      float wy[3][33], wz[3][33];
    };
    struct {
      float raw[kRawPlanes][32];
      uint16_t grp[32];
    };
  };
};
static_assert(sizeof(WalkSet) == 728 * 4, "WalkSet layout");

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}

// Copies the raw planes of the 32 particles from i0 (a multiple of 32) into
// `set`, 16 bytes per lane and copy: eight lanes per plane. The planes are
// padded to a multiple of 32 particles, so the last set may read past n.
__device__ __forceinline__ void copy_set(const Particles& P, int i0, WalkSet& set, int lane) {
  const int sub = lane >> 3, seg = 4 * (lane & 7);
  const float* src = P.plane(sub) + i0 + seg;
  float* dst = &set.raw[sub][seg];
#pragma unroll
  for (int j = 0; j < 5; ++j) {  // planes 4 j + sub: x, v, C (0-14), then tau (planes 24-29)
    const int skip = 4 * j + sub >= 15 ? 9 : 0;
    cp_async16(dst + 4 * j * 32, src + (long long)(4 * j + skip) * P.stride);
  }
  if (sub == 0) cp_async16(dst + 20 * 32, src + 29LL * P.stride);
  if (sub == 1 && seg < 16) cp_async16(set.grp + 2 * seg, P.grp + i0 + 2 * seg);
}

// One contact registration pass over the 32 particles [first, first + 32) of
// the warp: one contact per (particle, body) pair with the particle strictly
// inside, appended with one atomic per warp and body.
__device__ __forceinline__ void register_contacts(const P2GArgs& a, unsigned cand, int i,
                                                  bool valid, int lane) {
  float xp[3] = {0.f, 0.f, 0.f}, vp[3] = {0.f, 0.f, 0.f};
  if (valid) {
#pragma unroll
    for (int c = 0; c < 3; ++c) { xp[c] = a.P.x(c)[i]; vp[c] = a.P.v(c)[i]; }
  }
  for (int b = 0; b < a.nb; ++b) {
    if (!((cand >> b) & 1u)) continue;
    float nrm[3] = {0.f, 0.f, 1.f};
    float phi = 1.0f;
    if (valid) {
      phi = body_sdf(a.bodies[b], xp[0], xp[1], xp[2], nrm);
      // near the surface the sign and the depth come from FP64
      if (phi < 1e-6f + 1e-6f * (fabsf(xp[0]) + fabsf(xp[1]) + fabsf(xp[2])))
        phi = (float)body_sdf_f64(a.bodies[b], xp[0], xp[1], xp[2]);
    }
    const bool hit = valid && phi < 0.0f;
    const unsigned mask = __ballot_sync(0xffffffffu, hit);
    if (mask == 0u) continue;
    const int leader = __ffs(mask) - 1;
    int slot0 = 0;
    if (lane == leader) slot0 = atomicAdd(a.C.count, __popc(mask));
    slot0 = __shfl_sync(0xffffffffu, slot0, leader);
    if (hit) {
      const int slot = slot0 + __popc(mask & ((1u << lane) - 1u));
      if (slot < a.C.cap) {
        const DevBody& bd = a.bodies[b];
        float vr[3];
        body_velocity(bd, xp[0], xp[1], xp[2], vr);
        const float vn0 = nrm[0] * (vp[0] - vr[0]) + nrm[1] * (vp[1] - vr[1]) + nrm[2] * (vp[2] - vr[2]);
        const float phi0 = -phi;
        const float n0 = normal_impulse(phi0, bd.k, bd.d, a.h, vn0);
        a.C.xp[slot] = make_float4(xp[0], xp[1], xp[2], phi0);
        a.C.nrm[slot] = make_float4(nrm[0], nrm[1], nrm[2], n0);
        a.C.bias[slot] = make_float4(-vr[0], -vr[1], -vr[2], 0.f);
        a.C.id[slot] = make_int2((int)a.P.pid[i], b);
      } else {
        atomicOr(a.status, kStCapacity);
      }
    }
  }
}

// ROUNDS staged sets of 32 particles per warp: three (a walker's own 32 each)
// or one (a third of the 32 each).
template <int ROUNDS, bool kDense>
__device__ __forceinline__ void p2g_walk_block(const P2GArgs& a, int block) {
  extern __shared__ float4 s_dyn[];
  const GridDev& g = a.g;
  const int lane = threadIdx.x;
  const int first = block * 32 * ROUNDS;
  if (first >= a.n) return;
  WalkSet* S = reinterpret_cast<WalkSet*>(s_dyn);
  // all of the warp's particles are on their way before anything waits
#pragma unroll
  for (int it = 0; it < ROUNDS; ++it)
    if (first + it * 32 < a.n) copy_set(a.P, first + it * 32, S[it], lane);

  const float h = a.h;
  const float dinv = 4.0f * g.inv_dx * g.inv_dx;

  // this lane's walker (3: idle) and node row
  const int walker = lane / 9;
  const int row = lane - 9 * walker;
  const int cy = row % 3, cz = row / 3;
  // the walker's slots: 32 of its own set, or a third of the only one (whose
  // slot 32 is empty); slots without a particle hold no weight and key -1
  constexpr int kSteps = ROUNDS == 1 ? 11 : 32;
  const WalkSet& W = S[ROUNDS == 1 ? 0 : min(walker, ROUNDS - 1)];
  const int w_begin = ROUNDS == 1 ? min(walker, 2) * kSteps : 0;

  // ---- staging
  int marked = -1;  // the block (and neighbours) that the warp marked last
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
  int lo[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, hi[3] = {-0x7fffffff, -0x7fffffff, -0x7fffffff};
#pragma unroll 1
  for (int it = 0; it < ROUNDS; ++it) {
    const int i = first + it * 32 + lane;
    const float x0 = S[it].raw[0][lane], x1 = S[it].raw[1][lane], x2 = S[it].raw[2][lane];
    float vv[3], Cp[9], tau[6];
#pragma unroll
    for (int c = 0; c < 3; ++c) vv[c] = S[it].raw[3 + c][lane];
#pragma unroll
    for (int c = 0; c < 9; ++c) Cp[c] = S[it].raw[6 + c][lane];
#pragma unroll
    for (int c = 0; c < 6; ++c) tau[c] = S[it].raw[15 + c][lane];
    const int grp = S[it].grp[lane];
    __syncwarp();  // (the records overwrite the raw planes)
    Stencil st;
    stencil(g, x0, x1, x2, st);
    const bool inside = stencil_inside(g, st);
    const bool valid = i < a.n && inside;
    DevGroup gr = DevGroup{};
    if (valid) gr = a.groups[grp];
    int key = -1 - lane;
    if (i < a.n && !inside) atomicOr(a.status, kStOutOfDomain);
    if (valid) {
      key = node_index<true>(g, st.base[0], st.base[1], st.base[2]);  // (the grid's, also when sparse)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        lo[c] = min(lo[c], st.base[c]);
        hi[c] = max(hi[c], st.base[c]);
      }
    }
    // the 4^3 blocks that the set's stencils reach (a sparse grid marked its
    // blocks before P2G): per block of base nodes, the neighbours that the
    // particles beyond its middle reach along each axis. Marked once per set:
    // byte stores at every cell change queued up in L2 (1M particles at 8 per
    // cell: 59 against 51 us)
    if (kDense) {
      unsigned left = __ballot_sync(0xffffffffu, valid);
      while (left) {
        const int b = __shfl_sync(0xffffffffu, key >> 6, __ffs(left) - 1);
        const bool mine = valid && (key >> 6) == b;
        const bool rx = __any_sync(0xffffffffu, mine && (key & 2)), ry = __any_sync(0xffffffffu, mine && (key & 8)),
                   rz = __any_sync(0xffffffffu, mine && (key & 32));
        const int seen = b * 8 + rx + 2 * ry + 4 * rz;
        if (seen != marked && lane < 8 && (rx || !(lane & 1)) && (ry || !(lane & 2)) && (rz || !(lane & 4)))
          a.G.mark[b + (lane & 1) + ((lane >> 1) & 1) * g.nbx + (lane >> 2) * (g.nbx * g.nby)] = 1;
        marked = seen;
        left &= ~__ballot_sync(0xffffffffu, mine);
      }
    }
    // slots of equal cells together, cells in the order of their first particle
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    const int leader = __ffs(peers) - 1;
    const unsigned below = (1u << lane) - 1u;
    int start = valid && lane == leader ? __popc(peers) : 0;
    {
      int incl = start;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      start = __shfl_sync(0xffffffffu, incl - start, leader);
    }
    const unsigned vmask = __ballot_sync(0xffffffffu, valid);
    const int p = valid ? start + __popc(peers & below) : __popc(vmask) + __popc(~vmask & below);
    if (ROUNDS == 1 && lane == 0) {
      S[it].row[0][32] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
      S[it].row[3][32] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (!valid) {
      S[it].row[0][p] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
      S[it].row[1][p] = S[it].row[2][p] = S[it].row[3][p] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int c = 0; c < 3; ++c) S[it].wy[c][p] = S[it].wz[c][p] = 0.f;
      continue;
    }
    const float sc = h * dinv * gr.vol_m;
    const float tf[9] = {tau[0], tau[3], tau[4], tau[3], tau[1], tau[5], tau[4], tau[5], tau[2]};
    float A[9];
#pragma unroll
    for (int c = 0; c < 9; ++c) A[c] = -g.dx * (Cp[c] - sc * tf[c]);
    if (a.fext) {  // cloth: + h f / m, the force planes left zero for the next substep
      const float hm = h * gr.inv_m;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        vv[c] = fmaf(hm, a.fext[c * a.fext_stride + i], vv[c]);
        a.fext[c * a.fext_stride + i] = 0.f;
      }
    }
    float b[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
      b[c] = fmaf(A[3 * c], st.fx[0], fmaf(A[3 * c + 1], st.fx[1], fmaf(A[3 * c + 2], st.fx[2], vv[c])));
    S[it].row[0][p] = make_float4(b[0], b[1], b[2], __int_as_float(key));
    S[it].row[1][p] = make_float4(A[0], A[3], A[1], A[4]);
    S[it].row[2][p] = make_float4(A[2], A[5], A[6], A[7]);
    S[it].row[3][p] = make_float4(A[8], gr.mass * st.w[0][0], gr.mass * st.w[0][1], gr.mass * st.w[0][2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      S[it].wy[c][p] = st.w[1][c];
      S[it].wz[c][p] = st.w[2][c];
    }
  }
  __syncwarp();

  // ---- the walk
  const float2 ny = make_float2(-(float)cy, -(float)cy), nz = make_float2(-(float)cz, -(float)cz);
  const float2 n2 = make_float2(-2.f, -2.f);
  // sums of the row's three nodes: mass, (x, y), z momentum
  float m0 = 0.f, m1 = 0.f, m2 = 0.f, z0 = 0.f, z1 = 0.f, z2 = 0.f;
  float2 p0 = make_float2(0.f, 0.f), p1 = p0, p2 = p0;
  int cur = -2;        // the walker's cell (-2: none yet, -1: no particles left)
  int node = 0, l0 = 0;    // the row's first node; the cell along x in its block
  const int yb = g.nbx * kBlockNodes, zb = g.nby * yb;  // nodes from a block to the next along y, z
  // the row's nodes cell along x l0, l0 + 1, l0 + 2: the block's nodes are
  // consecutive, the next block's start 60 nodes further on
  auto add_first = [&]() {
    red_add_v4(a.G.mp + (kDense ? node : g.slot[node >> 6] * kBlockNodes + (node & 63)), m0, p0.x, p0.y, z0);
  };
  auto add_others = [&]() {
    int n1 = node + (l0 == 3 ? 61 : 1), n2 = node + (l0 >= 2 ? 62 : 2);
    if (!kDense) {
      n1 = g.slot[n1 >> 6] * kBlockNodes + (n1 & 63);
      n2 = g.slot[n2 >> 6] * kBlockNodes + (n2 & 63);
    }
    red_add_v4(a.G.mp + n1, m1, p1.x, p1.y, z1);
    red_add_v4(a.G.mp + n2, m2, p2.x, p2.y, z2);
  };
  const bool worker = walker < 3;
#pragma unroll 1
  for (int t = 0; t < kSteps; ++t) {
    const int p = w_begin + t;
    const float4 q0 = W.row[0][p], q1 = W.row[1][p], q2 = W.row[2][p], q3 = W.row[3][p];
    const float wyz = W.wy[cy][p] * W.wz[cz][p];
    const int key = __float_as_int(q0.w);
    if (key != cur) {
      const bool slide = key == cur + 1 && l0 < 3;  // the next cell along x: two columns are kept
      if (cur >= 0 && worker) {
        add_first();
        if (!slide) add_others();
      }
      m0 = slide ? m1 : 0.f;
      p0.x = slide ? p1.x : 0.f;
      p0.y = slide ? p1.y : 0.f;
      z0 = slide ? z1 : 0.f;
      m1 = slide ? m2 : 0.f;
      p1.x = slide ? p2.x : 0.f;
      p1.y = slide ? p2.y : 0.f;
      z1 = slide ? z2 : 0.f;
      m2 = z2 = 0.f;
      p2 = make_float2(0.f, 0.f);
      const int ly = ((key >> 2) & 3) + cy, lz = ((key >> 4) & 3) + cz;
      l0 = key & 3;
      node = (key & ~60) + ((ly & 3) << 2) + ((lz & 3) << 4) + (ly >= 4 ? yb : 0) + (lz >= 4 ? zb : 0);
      cur = key;
    }
    // b - A c at the row's first node, then along x
    const float2 Axy = make_float2(q1.x, q1.y);
    const float2 v0 = __ffma2_rn(make_float2(q1.z, q1.w), ny,
                                 __ffma2_rn(make_float2(q2.x, q2.y), nz, make_float2(q0.x, q0.y)));
    const float u0 = fmaf(q2.w, ny.x, fmaf(q3.x, nz.x, q0.z));
    const float2 v1 = __fadd2_rn(v0, make_float2(-Axy.x, -Axy.y));
    const float u1 = u0 - q2.z;
    const float2 v2 = __ffma2_rn(Axy, n2, v0);
    const float u2 = fmaf(q2.z, -2.f, u0);
    const float w0 = wyz * q3.y, w1 = wyz * q3.z, w2 = wyz * q3.w;
    m0 += w0;
    m1 += w1;
    m2 += w2;
    p0 = __ffma2_rn(make_float2(w0, w0), v0, p0);
    p1 = __ffma2_rn(make_float2(w1, w1), v1, p1);
    p2 = __ffma2_rn(make_float2(w2, w2), v2, p2);
    z0 = fmaf(w0, u0, z0);
    z1 = fmaf(w1, u1, z1);
    z2 = fmaf(w2, u2, z2);
  }
  if (cur >= 0 && worker) {
    add_first();
    add_others();
  }

  // ---- contact registration: bodies that may hold a particle of this warp
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    lo[c] = __reduce_min_sync(0xffffffffu, lo[c]);
    hi[c] = __reduce_max_sync(0xffffffffu, hi[c]);
  }
  bool cand_b = false;
  if (hi[0] >= lo[0] && lane < a.nb) {
    const float c0 = g.ox + g.dx * (0.5f * (lo[0] + hi[0]) + 1.0f);
    const float c1 = g.oy + g.dx * (0.5f * (lo[1] + hi[1]) + 1.0f);
    const float c2 = g.oz + g.dx * (0.5f * (lo[2] + hi[2]) + 1.0f);
    const float h0 = 0.5f * g.dx * (hi[0] - lo[0] + 1), h1 = 0.5f * g.dx * (hi[1] - lo[1] + 1),
                h2 = 0.5f * g.dx * (hi[2] - lo[2] + 1);
    cand_b = box_may_touch(a.bodies[lane], c0, c1, c2, h0, h1, h2);
  }
  const unsigned cand = __ballot_sync(0xffffffffu, cand_b);
  if (cand) {
#pragma unroll 1
    for (int it = 0; it < ROUNDS; ++it) {
      const int i = first + it * 32 + lane;
      bool valid = false;
      if (i < a.n) {
        Stencil st;
        stencil(g, a.P.x(0)[i], a.P.x(1)[i], a.P.x(2)[i], st);
        valid = stencil_inside(g, st);
      }
      register_contacts(a, cand, i, valid, lane);
    }
  }
}

template <int ROUNDS, bool kDense>
__global__ void __launch_bounds__(kWalkThreads, 24) k_p2g_w(P2GArgs a) {
  chain_begin();
  if (a.in_flight && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(a.in_flight, 1);
  p2g_walk_block<ROUNDS, kDense>(a, blockIdx.x);
}

template <int ROUNDS>
__global__ void __launch_bounds__(kWalkThreads, 24) k_p2g_w_batch(const P2GArgs* __restrict__ args,
                                                                 const int2* __restrict__ work) {
  __shared__ P2GArgs s_a;
  chain_begin();
  const int2 wk = work[blockIdx.x];
  load_args(args + wk.x, s_a);
  __syncthreads();
  p2g_walk_block<ROUNDS, true>(s_a, wk.y);  // (batches take dense grids)
}

template <int ROUNDS>
constexpr size_t walk_smem() { return sizeof(WalkSet) * ROUNDS; }

template <int ROUNDS>
void launch_walk(const P2GArgs& a, cudaStream_t s) {
  const int per_block = kWalkThreads * ROUNDS;
  const int nblk = (a.n + per_block - 1) / per_block;
  if (a.g.slot)
    launch_chained(k_p2g_w<ROUNDS, false>, dim3(nblk), kWalkThreads, walk_smem<ROUNDS>(), s, a);
  else
    launch_chained(k_p2g_w<ROUNDS, true>, dim3(nblk), kWalkThreads, walk_smem<ROUNDS>(), s, a);
}

template <class K>
cudaError_t prepare_kernel(K k, size_t smem) {
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  return e;
}

template <int ROUNDS>
cudaError_t prepare_walk() {
  cudaError_t e = prepare_kernel(k_p2g_w<ROUNDS, true>, walk_smem<ROUNDS>());
  if (e == cudaSuccess) e = prepare_kernel(k_p2g_w<ROUNDS, false>, walk_smem<ROUNDS>());
  if (e == cudaSuccess) e = prepare_kernel(k_p2g_w_batch<ROUNDS>, walk_smem<ROUNDS>());
  return e;
}

}  // namespace

cudaError_t p2g_prepare() {
  cudaError_t e = prepare_walk<1>();
  if (e == cudaSuccess) e = prepare_walk<3>();
  return e;
}

int p2g_block_particles(long long n) { return kWalkThreads * (n < kWalkOneRound ? 1 : 3); }

void launch_p2g_batch(const P2GArgs* args, const int2* work, int n_work, long long n, cudaStream_t s) {
  if (n_work <= 0) return;
  if (n < kWalkOneRound)
    launch_chained(k_p2g_w_batch<1>, dim3(n_work), kWalkThreads, walk_smem<1>(), s, args, work);
  else
    launch_chained(k_p2g_w_batch<3>, dim3(n_work), kWalkThreads, walk_smem<3>(), s, args, work);
}

void launch_p2g(const P2GArgs& a, cudaStream_t s) {
  if (a.n <= 0) return;
  if (a.n < kWalkOneRound)
    launch_walk<1>(a, s);
  else
    launch_walk<3>(a, s);
}

}  // namespace mpmcr
