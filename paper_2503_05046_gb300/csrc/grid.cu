// grid.cu -- the active-block list and the grid update of the free-motion
// solve (Sec. V-A op (2): v* = p / m + h g on every node with mass), with the
// domain walls held at zero velocity.
//
// Only 4^3 blocks marked by P2G are swept. The update also clears the P2G
// accumulator it consumed, so the accumulator is all zero between substeps
// and no separate clearing pass is needed.
//
// A block-sparse grid (GridDev::slot) stores only the substep's active
// blocks: before P2G the blocks of the particles' stencils are marked and
// compacted, and entry t of the active list gets storage block t (the slot
// table maps the grid block to it; the previous substep's entries are unmapped
// first, so unmapped blocks read -1). Blocks beyond the pool share its spare
// block and the substep reports a capacity error.
#include "kernels.h"

namespace mpmcr {

namespace {

// Compaction of one scene's block marks into its active-block list, the
// threads striding by `stride` from `start` (taken warp-aligned).
__device__ __forceinline__ void compact_range(uint8_t* __restrict__ mark, int start, int stride,
                                              int n_blocks, int* __restrict__ act,
                                              int* __restrict__ n_act,
                                              int* __restrict__ slot_tab = nullptr, int pool = 0,
                                              uint32_t* __restrict__ status = nullptr) {
  const int lane = threadIdx.x & 31;
  for (int base = start & ~31; base < n_blocks; base += stride) {
    const int b = base + lane;
    const bool on = b < n_blocks && mark[b] != 0;
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (m == 0u) continue;
    int slot0 = 0;
    if (lane == 0) slot0 = atomicAdd(n_act, __popc(m));
    slot0 = __shfl_sync(0xffffffffu, slot0, 0);
    if (on) {
      const int t = slot0 + __popc(m & ((1u << lane) - 1u));
      act[t] = b;
      mark[b] = 0;
      if (slot_tab) {
        slot_tab[b] = t < pool ? t : pool;  // beyond the pool: the spare block
        if (t >= pool) atomicOr(status, kStCapacity);
      }
    }
  }
}

// Sparse grids, before P2G: unmap the previous substep's blocks, then mark
// the blocks of every particle's stencil (the nodes P2G, the solve and G2P
// of this substep touch).
__global__ void k_mark_sparse(GridDev g, Particles P, int n, uint8_t* mark, const int* act,
                              const int* n_mapped, int* slot_tab) {
  chain_begin();
  const int stride = gridDim.x * blockDim.x;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  const int nm = *n_mapped;
  for (int t = tid; t < nm; t += stride) slot_tab[act[t]] = -1;
  for (int i = tid; i < n; i += stride) {
    Stencil st;
    stencil(g, P.x(0)[i], P.x(1)[i], P.x(2)[i], st);
    if (!stencil_inside(g, st)) continue;  // reported by P2G
    const int bx0 = st.base[0] >> 2, by0 = st.base[1] >> 2, bz0 = st.base[2] >> 2;
    const int bx1 = (st.base[0] + 2) >> 2, by1 = (st.base[1] + 2) >> 2, bz1 = (st.base[2] + 2) >> 2;
    for (int bz = bz0; bz <= bz1; ++bz)
      for (int by = by0; by <= by1; ++by)
        for (int bx = bx0; bx <= bx1; ++bx) mark[(bz * g.nby + by) * g.nbx + bx] = 1;
  }
}

__global__ void k_compact_sparse(uint8_t* __restrict__ mark, int n_blocks, int* __restrict__ act,
                                 int* __restrict__ n_act, int* __restrict__ slot_tab, int pool,
                                 uint32_t* __restrict__ status) {
  chain_begin();
  compact_range(mark, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, n_blocks,
                act, n_act, slot_tab, pool, status);
}

// The grid update of one node: cell `cell` of grid block `blk`, stored at
// `node`. Returns m |v*|^2 of a free node.
__device__ __forceinline__ float update_node(const GridDev& g, const GridArrays& G, float h, int blk,
                                             int cell, int node) {
  const float4 mp = G.mp[node];
  float4 vs = make_float4(0.f, 0.f, 0.f, 0.f);
  const int bx = blk % g.nbx, by = (blk / g.nbx) % g.nby, bz = blk / (g.nbx * g.nby);
  const int i = bx * 4 + (cell & 3), j = by * 4 + ((cell >> 2) & 3), k = bz * 4 + (cell >> 4);
  const bool wall = i < g.bc || j < g.bc || k < g.bc || i >= g.rx - g.bc || j >= g.ry - g.bc ||
                    k >= g.rz - g.bc;
  float p2 = 0.f;
  if (mp.x > 0.0f) {
    // p / m + h g with one rounding: the quotient's remainder goes with h g
    const float inv_m = 1.0f / mp.x;
    auto vstar = [&](float p, float hg) {
      const float q = p * inv_m;
      return fabsf(q) < INFINITY ? q + fmaf(fmaf(-q, mp.x, p), inv_m, hg) : q;
    };
    vs.x = wall ? 0.0f : vstar(mp.y, h * g.gx);
    vs.y = wall ? 0.0f : vstar(mp.z, h * g.gy);
    vs.z = wall ? 0.0f : vstar(mp.w, h * g.gz);
    vs.w = mp.x;
    if (!wall) p2 = mp.x * (vs.x * vs.x + vs.y * vs.y + vs.z * vs.z);
  }
  G.mp[node] = make_float4(0.f, 0.f, 0.f, 0.f);
  G.vs[node] = vs;
  // .w flags a Dirichlet node for the contact solve
  G.v[node] = make_float4(vs.x, vs.y, vs.z, wall ? 1.f : 0.f);
  G.vlo[node] = make_float4(0.f, 0.f, 0.f, 0.f);
  return p2;
}

// Adds the threads' sums of m |v*|^2 over free nodes (the momentum norm of
// Alg. 1) to the substep's.
__device__ __forceinline__ void add_momentum_norm(const GridArrays& G, float p2) {
  __shared__ double s_p2[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) p2 += __shfl_xor_sync(0xffffffffu, p2, o);
  if ((threadIdx.x & 31) == 0) s_p2[threadIdx.x >> 5] = (double)p2;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += s_p2[w];
    if (sum != 0.0) atomicAdd(G.pstar2, sum);
  }
}

// The grid update of a dense grid straight from P2G's marks: warp `first` of
// `n_warps` takes blocks first, first + n_warps, ..., 32 marks at a time (so
// that neighbouring blocks, which are active together, go to different warps),
// appends its marked blocks to the active list and updates their 64 nodes. One
// launch instead of a compaction and an update; G2P closes the substep's count.
__device__ __forceinline__ void grid_dense_range(const GridDev& g, const GridArrays& G, float h,
                                                 int first, int n_warps) {
  const int lane = threadIdx.x & 31;
  const int n_blocks = g.nbx * g.nby * g.nbz;
  float p2 = 0.f;
  for (int base = first; base < n_blocks; base += 32 * n_warps) {
    const int b = base + lane * n_warps;
    const bool on = b < n_blocks && G.mark[b] != 0;
    unsigned left = __ballot_sync(0xffffffffu, on);
    if (left == 0u) continue;
    int slot0 = 0;
    if (lane == 0) slot0 = atomicAdd(G.n_act, __popc(left));
    slot0 = __shfl_sync(0xffffffffu, slot0, 0);
    if (on) {
      G.act[slot0 + __popc(left & ((1u << lane) - 1u))] = b;
      G.mark[b] = 0;
    }
    for (; left; left &= left - 1u) {
      const int blk = base + (__ffs(left) - 1) * n_warps;
      p2 += update_node(g, G, h, blk, lane, blk * kBlockNodes + lane);
      p2 += update_node(g, G, h, blk, 32 + lane, blk * kBlockNodes + 32 + lane);
    }
  }
  add_momentum_norm(G, p2);
}

__global__ void __launch_bounds__(256) k_grid_update_dense(GridDev g, GridArrays G, float h) {
  chain_begin();
  grid_dense_range(g, G, h, (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5),
                   (int)(gridDim.x * (blockDim.x >> 5)));
}

// The grid update of nodes t = start, start + stride, ... of the active
// blocks' nodes; `first`: the thread that notes the mapped list's length.
__device__ __forceinline__ void grid_update_range(const GridDev& g, const GridArrays& G, float h,
                                                  long long start, long long stride, bool first) {
  const int n_act = *G.n_act;
  if (first && g.slot) *G.n_mapped = n_act;  // the list the slot table now holds
  const long long total = (long long)active_with_storage(g, n_act) * kBlockNodes;
  float p2 = 0.f;
  for (long long t = start; t < total; t += stride) {
    const int cell = (int)(t & 63);
    p2 += update_node(g, G, h, G.act[t >> 6], cell,
                      active_storage_block(g, G.act, (int)(t >> 6)) * kBlockNodes + cell);
  }
  add_momentum_norm(G, p2);
}

__global__ void __launch_bounds__(256) k_grid_update(GridDev g, GridArrays G, float h) {
  chain_begin();
  grid_update_range(g, G, h, (long long)blockIdx.x * blockDim.x + threadIdx.x,
                    (long long)gridDim.x * blockDim.x, blockIdx.x == 0 && threadIdx.x == 0);
}

// Batched: thread block b is slice work[b].y of work[b].x's scene; a scene's
// n_slices blocks go over its marks together
__global__ void __launch_bounds__(256) k_grid_update_batch(const GridBatchArgs* __restrict__ args,
                                                           const int2* __restrict__ work) {
  __shared__ GridBatchArgs s_a;
  chain_begin();
  const int2 wk = work[blockIdx.x];
  load_args(args + wk.x, s_a);
  __syncthreads();
  const int warps = blockDim.x >> 5;
  grid_dense_range(s_a.g, s_a.G, s_a.h, wk.y * warps + (int)(threadIdx.x >> 5), s_a.n_slices * warps);
}

}  // namespace

void launch_grid(const GridDev& g, const GridArrays& G, float h, int num_sms, cudaStream_t s) {
  const int n_blocks = g.nbx * g.nby * g.nbz;
  if (g.slot) {  // (compacted before P2G)
    launch_chained(k_grid_update, dim3(num_sms * 8), 256, 0, s, g, G, h);
    return;
  }
  // a warp per two blocks of the domain, up to eight thread blocks per SM
  int tb = (n_blocks + 15) / 16;
  tb = tb > num_sms * 8 ? num_sms * 8 : tb;
  launch_chained(k_grid_update_dense, dim3(tb), 256, 0, s, g, G, h);
}

void launch_sparse_map(const GridDev& g, const GridArrays& G, const Particles& P, int n,
                       int* slot_tab, uint32_t* status, int num_sms, cudaStream_t s) {
  const int n_blocks = g.nbx * g.nby * g.nbz;
  const int pb = (n + 255) / 256;
  launch_chained(k_mark_sparse, dim3(pb < num_sms * 8 ? (pb > 0 ? pb : 1) : num_sms * 8), 256, 0, s, g, P,
                 n, G.mark, G.act, G.n_mapped, slot_tab);
  int cb = (n_blocks + 255) / 256;
  cb = cb > num_sms * 8 ? num_sms * 8 : cb;
  launch_chained(k_compact_sparse, dim3(cb), 256, 0, s, G.mark, n_blocks, G.act, G.n_act, slot_tab,
                 g.pool_blocks, status);
}

void launch_grid_batch(const GridBatchArgs* args, const int2* work, int n_work, cudaStream_t s) {
  if (n_work <= 0) return;
  launch_chained(k_grid_update_batch, dim3(n_work), 256, 0, s, args, work);
}

}  // namespace mpmcr
