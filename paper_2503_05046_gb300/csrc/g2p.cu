// g2p.cu -- grid-to-particle transfer with the constitutive update (Sec. V-A
// op (3), MLS-MPM): v_p = sum_i w v_i, C_p = (4/dx^2) sum_i w v_i (x_i - x_p)^T,
// x_p += h v_p, F_p <- (I + h C_p) F_p, then the Drucker-Prager return map for
// sand, fused with the stress update: the Kirchhoff stress of the new F is
// stored for the next P2G (elastic: a polynomial of F^T F - I; sand: one SVD per
// particle and substep serves both the plasticity and the stress). One thread per
// particle; particle planes are read and written with coalesced loads and stores,
// grid velocities are gathered from L2.
//
// Block 0 also closes the substep: it records the contact / active-block
// counts for diagnostics and resets the per-substep counters, the solve's
// barrier word, so the next substep needs no memset.
#include "kernels.h"

namespace mpmcr {

namespace {

// 128 threads, eight blocks per SM for a dense grid (64 registers, 16 B spilled),
// six for a sparse one. 1M elastic particles 47.5 us per launch, 4M mixed 235, 1M
// sand scooped 87.9; with seven blocks 51.2, 246 and 90.4. On a sparse grid 79,000
// particles 14.2 and 1M 56.0; with eight blocks 15.3 and 54.2, with seven 14.9 and
// 57.0. Bound by the latency of the gathers; the 216 B per
// particle that the planes move take 32 us at HBM's rate. (1M elastic 66 us with
// the decomposition for every particle.)
constexpr int kThreads = 128;

// Block `block` of G2P over one scene's particles, blockDim.x particles (a
// thread block of the single-scene launch, or a work item of the batched one).
template <bool kDense>
__device__ __forceinline__ void g2p_block(const G2PArgs& a, int block) {
  const GridDev& g = a.g;
  if (block == 0) {
    if (threadIdx.x == 0) {
      const int count = *a.C.count;
      const int nc = count < a.C.cap ? count : a.C.cap;
      a.stats->last_contacts = nc;
      atomicMax(&a.stats->contacts_max, nc);
      atomicAdd(&a.stats->contacts_total, (unsigned long long)nc);
      atomicAdd(&a.stats->substeps, 1);
      const int n_act = *a.G.n_act;
      atomicMax(&a.stats->active_blocks_max, n_act);
      a.stats->last_active = n_act;
      *a.C.count = 0;
      *a.G.n_act = 0;
      *a.G.n_cnodes = 0;
      *a.G.pstar2 = 0.0;
      if (a.in_flight) atomicSub(a.in_flight, 1);
    }
    if (threadIdx.x < 2) a.bar[threadIdx.x] = 0u;  // the solve's 64-bit barrier counter
  }
  const int i = block * (int)blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  const float xp[3] = {a.P.x(0)[i], a.P.x(1)[i], a.P.x(2)[i]};
  Stencil s;
  stencil(g, xp[0], xp[1], xp[2], s);
  if (!stencil_inside(g, s)) return;  // reported by P2G
  // dense node address = ax[cx] + ay[cy] + az[cz] (block-major: each axis
  // contributes its block and its cell within the block)
  int ax[3], ay[3], az[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int ix = s.base[0] + c, iy = s.base[1] + c, iz = s.base[2] + c;
    ax[c] = (ix >> 2) * kBlockNodes + (ix & 3);
    ay[c] = (iy >> 2) * (g.nbx * kBlockNodes) + ((iy & 3) << 2);
    az[c] = (iz >> 2) * (g.nbx * g.nby * kBlockNodes) + ((iz & 3) << 4);
  }
  // x and y components go in pairs (paired FP32 ops): v_xy, and the x, y
  // rows of B = sum w v (x_i - x_p)^T as (B_xx, B_yx), (B_xy, B_yy), (B_xz, B_yz)
  // Velocities are gathered as differences to the centre node's: the weights add
  // up to one and to no moment, so v_p = v_c + sum w (v_i - v_c) and B is the same
  // sum over the differences, but the sums round at the scale of the velocity's
  // variation over three cells, not of the velocity, and the weights' own
  // roundings meet the variation alone. Ten substeps of elastic particles in flight
  // against 64 bits, of v and C, against the sums over v_i: 1M 0.92 of their error,
  // 97,000 0.92, 36,000 on a sparse grid 0.94, 343,000 for three substeps 0.78.
  // A row's nodes lie in one block or two: a sparse grid's table is read for the
  // first and the last (for each of three, 1M elastic particles took 59.6 us).
  struct Row {
    int first, last;  // the storage blocks' row starts
  };
  auto row_of = [&](int cy, int cz) {
    Row r = {0, 0};
    if (!kDense) {
      const int iy = s.base[1] + cy, iz = s.base[2] + cz, in = ((iz & 3) << 4) + ((iy & 3) << 2);
      const int* slot = g.slot + ((iz >> 2) * g.nby + (iy >> 2)) * g.nbx;
      r.first = slot[s.base[0] >> 2] * kBlockNodes + in;
      r.last = slot[(s.base[0] + 2) >> 2] * kBlockNodes + in;
    }
    return r;
  };
  // (the solve before writes v: no read-only load)
  auto load = [&](const Row& r, int cx, int cy, int cz) {
    const int ix = s.base[0] + cx;
    return a.G.v[kDense ? az[cz] + ay[cy] + ax[cx]
                        : ((ix ^ s.base[0]) >> 2 ? r.last : r.first) + (ix & 3)];
  };
  float4 vc = load(row_of(1, 1), 1, 1, 1);
  // (a velocity beyond FP32 stays one: it is added to the sums, not taken off
  // the others', and C has no value)
  const bool finite = fabsf(vc.x) + fabsf(vc.y) + fabsf(vc.z) < INFINITY;
  const float4 v_centre = vc;
  if (!finite) vc.x = vc.y = vc.z = 0.f;
  const float2 ncxy = make_float2(-vc.x, -vc.y);
  float2 vxy = make_float2(0.f, 0.f), B0 = vxy, B1 = vxy, B2 = vxy;
  float vz = 0.f, Bz0 = 0.f, Bz1 = 0.f, Bz2 = 0.f;
  // weights and weighted offsets along x; a row's sums take them alone, and its
  // y and z weight and offsets once
  const float wx[3] = {s.w[0][0], s.w[0][1], s.w[0][2]};
  const float wd[3] = {wx[0] * ((0.f - s.fx[0]) * g.dx), wx[1] * ((1.f - s.fx[0]) * g.dx),
                       wx[2] * ((2.f - s.fx[0]) * g.dx)};
  auto dup = [](float f) { return make_float2(f, f); };
#pragma unroll
  for (int cz = 0; cz < 3; ++cz) {
    const float dz = (cz - s.fx[2]) * g.dx;
#pragma unroll
    for (int cy = 0; cy < 3; ++cy) {
      const float dy = (cy - s.fx[1]) * g.dx;
      const float wyz = s.w[1][cy] * s.w[2][cz];
      // the row's sums of w_x (v - v_c) and of w_x (v - v_c) (x_i - x_p)
      const Row row = row_of(cy, cz);
      float2 Sxy, Txy;
      float Sz, Tz;
#pragma unroll
      for (int cx = 0; cx < 3; ++cx) {
        if (cx == 1 && cy == 1 && cz == 1) continue;  // (the centre itself)
        const float4 v = load(row, cx, cy, cz);
        const float2 dxy = __fadd2_rn(make_float2(v.x, v.y), ncxy);
        const float dvz = v.z - vc.z;
        if (cx == 0) {
          Sxy = __fmul2_rn(dup(wx[0]), dxy);
          Txy = __fmul2_rn(dup(wd[0]), dxy);
          Sz = wx[0] * dvz;
          Tz = wd[0] * dvz;
        } else {
          Sxy = __ffma2_rn(dup(wx[cx]), dxy, Sxy);
          Txy = __ffma2_rn(dup(wd[cx]), dxy, Txy);
          Sz = fmaf(wx[cx], dvz, Sz);
          Tz = fmaf(wd[cx], dvz, Tz);
        }
      }
      const float wy = wyz * dy, wz = wyz * dz;
      vxy = __ffma2_rn(dup(wyz), Sxy, vxy);
      B0 = __ffma2_rn(dup(wyz), Txy, B0);
      B1 = __ffma2_rn(dup(wy), Sxy, B1);
      B2 = __ffma2_rn(dup(wz), Sxy, B2);
      vz = fmaf(wyz, Sz, vz);
      Bz0 = fmaf(wyz, Tz, Bz0);
      Bz1 = fmaf(wy, Sz, Bz1);
      Bz2 = fmaf(wz, Sz, Bz2);
    }
  }
  const float vp[3] = {vxy.x + v_centre.x, vxy.y + v_centre.y, vz + v_centre.z};
  const float Bm[9] = {B0.x, B1.x, B2.x, B0.y, B1.y, B2.y, Bz0, Bz1, Bz2};
  const float dinv = finite ? 4.0f * g.inv_dx * g.inv_dx : NAN;
  const float h = a.h;
  float C[9], F[9], Fn[9];
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    C[c] = dinv * Bm[c];
    F[c] = a.P.F(c)[i];
  }
  const DevGroup gr = a.groups[a.P.grp[i]];
  float tau[6];
  if (gr.model == MPM_CLOTH) {
    // the mesh carries the cloth's elasticity: F stays, no stress
#pragma unroll
    for (int c = 0; c < 9; ++c) Fn[c] = F[c];
#pragma unroll
    for (int c = 0; c < 6; ++c) tau[c] = 0.f;
  } else {
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c)
        Fn[3 * r + c] =
            F[3 * r + c] + h * (C[3 * r] * F[c] + C[3 * r + 1] * F[3 + c] + C[3 * r + 2] * F[6 + c]);
    constitutive_update(gr, Fn, tau);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    a.P.v(c)[i] = vp[c];
    a.P.x(c)[i] = xp[c] + h * vp[c];
  }
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    a.P.C(c)[i] = C[c];
    a.P.F(c)[i] = Fn[c];
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) a.P.tau(c)[i] = tau[c];
}

// kDense: a dense grid's node addresses (no block-table lookup)
template <bool kDense>
__global__ void __launch_bounds__(kThreads, kDense ? 8 : 6) k_g2p(G2PArgs a) {
  chain_begin();
  g2p_block<kDense>(a, blockIdx.x);
}

// Batched: thread block b is block work[b].y of scene work[b].x
__global__ void __launch_bounds__(512, 2) k_g2p_batch(const G2PArgs* __restrict__ args,
                                                      const int2* __restrict__ work) {
  __shared__ G2PArgs s_a;
  chain_begin();
  const int2 wk = work[blockIdx.x];
  load_args(args + wk.x, s_a);
  __syncthreads();
  g2p_block<true>(s_a, wk.y);  // (batches take dense grids)
}

}  // namespace

void launch_g2p(const G2PArgs& a, cudaStream_t s) {
  const int blocks = a.n > 0 ? (a.n + kThreads - 1) / kThreads : 1;
  if (a.g.slot)
    launch_chained(k_g2p<false>, dim3(blocks), kThreads, 0, s, a);
  else
    launch_chained(k_g2p<true>, dim3(blocks), kThreads, 0, s, a);
}

void launch_g2p_batch(const G2PArgs* args, const int2* work, int n_work, int threads,
                      cudaStream_t s) {
  if (n_work > 0) launch_chained(k_g2p_batch, dim3(n_work), threads, 0, s, args, work);
}

}  // namespace mpmcr
