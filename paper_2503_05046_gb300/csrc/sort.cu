// sort.cu -- particle ordering by grid block (Sec. V-A: particles sorted by
// cell so that particles writing the same grid nodes are processed together;
// the order is computed once per time step and reused by its N substeps).
//
// Key: Morton code of the 4^3 block holding the particle's B-spline base
// node (bits above an axis's own block count left out), so that a run of
// consecutive particles covers a compact box of blocks, followed by the base
// cell within the block (x fastest), so that a warp's particles of one cell are
// adjacent. Sort: stable LSD radix sort, the key's bits split evenly over as few
// passes of up to 8 bits as they need (a 128^3 grid has 15 + 6 bits: three
// passes of 7; 320 x 184 x 64 has 17 + 6: three of 8). A pass is three launches:
// tile histograms (the first one also forms the keys), a prefix sum along each
// digit's row of tiles, and a stable scatter that adds the digits' starts itself
// and ranks a warp's keys by votes on the digit's bits. The permutation is then
// applied to every particle plane at once.
//
// Bound by latency below about 1M particles (each launch is a few microseconds),
// above by the permutation (1.0 GB at 4M: 153 us at the copy rate). Against one
// warp per tile of 1,024 keys, three scan launches per pass and a load-store
// chain over the planes in the permutation, a step of no substeps: 16,000
// particles 145 -> 83 us, 79,000 189 -> 98, 1M 267 -> 166, 4M 526 -> 344 (about
// 50 of each are the call).
//
// Up to 8,192 particles one thread block sorts in shared memory: the same radix
// sort with 6-bit digits, two launches in place of ten (8,192 particles: 32 to
// 40 us by bits, the tiled sort 32 to 34; 5,000: 23 to 28; 1,000: 13). A bitonic
// network over (key, index) pairs, with a barrier for each of its 91 stages,
// took 74 us for 8,000.
#include "kernels.h"

namespace mpmcr {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxBins = 256;

constexpr int kSmallSortMax = 8192;      // particles sorted by one thread block
constexpr int kSmallSortThreads = 1024;
constexpr int kSmallSortWarps = kSmallSortThreads / 32;
constexpr int kSmallBits = 6;
constexpr int kSmallBins = 1 << kSmallBits;
constexpr int kSmallRounds = kSmallSortMax / kSmallSortThreads;
// two key and two index buffers, and a counter per digit and warp
// (rows one longer than the warps, so that a warp's digits lie in different banks)
constexpr int kSmallRow = kSmallSortWarps + 1;
constexpr size_t kSmallSortSmem =
    kSmallSortMax * 2 * (sizeof(uint32_t) + sizeof(uint16_t)) + kSmallBins * kSmallRow * sizeof(int);

// the sort key of a particle at (x, y, z)
__device__ __forceinline__ uint32_t sort_key(const GridDev& g, float x, float y, float z) {
  // the base node of the particle's stencil, as P2G computes it
  Stencil st;
  stencil(g, x, y, z, st);
  const int lim[3] = {g.nbx - 1, g.nby - 1, g.nbz - 1};
  uint32_t b[3], c[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int base = st.base[a];
    int blk = base >> 2;  // arithmetic shift: floor division for negatives
    c[a] = (uint32_t)(base & 3);
    if (blk < 0) { blk = 0; c[a] = 0; }
    if (blk > lim[a]) { blk = lim[a]; c[a] = 3; }
    b[a] = (uint32_t)blk;
  }
  // bit i of each axis that has one, x lowest
  uint32_t key = 0u;
  int pos = 0;
  for (int i = 0; i < g.morton_bits; ++i) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if ((lim[a] >> i) != 0) key |= ((b[a] >> i) & 1u) << pos++;
  }
  // cell within the block, x fastest (the order of P2G's walk), when it fits
  if (g.sort_cell_bits) key = (key << 6) | (c[2] << 4) | (c[1] << 2) | c[0];
  return key;
}

// The lanes of the warp whose digit (of `bits` bits) is this lane's. A vote per
// bit, not __match_any_sync: that one occupies its SM for about 64 cycles.
__device__ __forceinline__ unsigned same_digit(int d, int bits) {
  unsigned peers = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    if (b < bits) {
      const unsigned set = __ballot_sync(0xffffffffu, (d >> b) & 1);
      peers &= (d >> b) & 1 ? set : ~set;
    }
  }
  return peers;
}

// Up to kSmallSortMax particles in one thread block: `rounds` keys per thread,
// a warp's keys consecutive; the permutation goes to vals.
__device__ __forceinline__ void sort_small(const SortArgs& a) {
  extern __shared__ uint32_t s_sort[];
  uint32_t* in = s_sort;
  uint32_t* out = in + kSmallSortMax;
  int* cnt = reinterpret_cast<int*>(out + kSmallSortMax);  // [digit][warp]
  uint16_t* idx_in = reinterpret_cast<uint16_t*>(cnt + kSmallBins * kSmallRow);
  uint16_t* idx_out = idx_in + kSmallSortMax;
  __shared__ int s_warp[kSmallSortWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rounds = (a.n + kSmallSortThreads - 1) / kSmallSortThreads;
  const int first = warp * 32 * rounds + lane;
  for (int r = 0; r < rounds; ++r) {
    const int i = first + 32 * r;
    in[i] = i < a.n ? sort_key(a.g, a.src.x(0)[i], a.src.x(1)[i], a.src.x(2)[i]) : ~0u;
    idx_in[i] = (uint16_t)i;
  }
  const unsigned below = (1u << lane) - 1u;
  // (the padding's keys have every bit set: they sort behind the particles)
  for (int shift = 0; shift < a.bits; shift += kSmallBits) {
    for (int i = tid; i < kSmallBins * kSmallRow; i += kSmallSortThreads) cnt[i] = 0;
    __syncthreads();
    int rank[kSmallRounds];
#pragma unroll
    for (int r = 0; r < kSmallRounds; ++r) {
      if (r < rounds) {
        const int d = (in[first + 32 * r] >> shift) & (kSmallBins - 1);
        const unsigned peers = same_digit(d, kSmallBits);
        int* c = cnt + d * kSmallRow + warp;
        const int seen = *c;
        rank[r] = seen + __popc(peers & below);
        __syncwarp();
        if ((peers & below) == 0u) *c = seen + __popc(peers);
        __syncwarp();
      }
    }
    __syncthreads();
    // exclusive prefix sum over (digit, warp): two counters per thread
    {
      int* c = cnt + (2 * tid / kSmallSortWarps) * kSmallRow + 2 * tid % kSmallSortWarps;
      const int c0 = c[0], c1 = c[1];
      int x = c0 + c1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) s_warp[warp] = x;
      __syncthreads();
      int t = s_warp[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += y;
      }
      const int before = __shfl_sync(0xffffffffu, t, warp > 0 ? warp - 1 : 0);
      const int start = (warp > 0 ? before : 0) + x - c0 - c1;
      c[0] = start;
      c[1] = start + c0;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSmallRounds; ++r) {
      if (r < rounds) {
        const uint32_t key = in[first + 32 * r];
        const int d = (key >> shift) & (kSmallBins - 1);
        const int pos = cnt[d * kSmallRow + warp] + rank[r];
        out[pos] = key;
        idx_out[pos] = idx_in[first + 32 * r];
      }
    }
    __syncthreads();
    uint32_t* k = in;
    in = out;
    out = k;
    uint16_t* x = idx_in;
    idx_in = idx_out;
    idx_out = x;
  }
  for (int i = tid; i < a.n; i += kSmallSortThreads) a.vals[0][i] = idx_in[i];
}

__global__ void __launch_bounds__(kSmallSortThreads) k_sort_small(SortArgs a) {
  chain_begin();
  sort_small(a);
}

// Histogram of digit `pass` over tile `tile` (a.rounds x 32 keys per warp); the
// first pass forms the keys.
__device__ __forceinline__ void sort_hist(const SortArgs& a, int pass, int tile) {
  __shared__ int h[kMaxBins];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  h[tid] = 0;
  __syncthreads();
  const int first = (tile * kWarps + warp) * 32 * a.rounds + lane;
  const int shift = pass * a.digit, mask = (1 << a.digit) - 1;
  const uint32_t* in = a.keys[pass & 1];
  for (int r = 0; r < a.rounds; ++r) {
    const int i = first + 32 * r;
    if (i < a.n) {
      uint32_t key;
      if (pass == 0) {
        key = sort_key(a.g, a.src.x(0)[i], a.src.x(1)[i], a.src.x(2)[i]);
        a.keys[0][i] = key;
      } else {
        key = in[i];
      }
      atomicAdd(h + ((key >> shift) & mask), 1);
    }
  }
  __syncthreads();
  if (tid <= mask) a.hist[(size_t)tid * a.n_tiles + tile] = h[tid];
}

// Exclusive prefix sum along digit `d`'s row of tiles, its total behind the rows.
__device__ __forceinline__ void sort_rows(const SortArgs& a, int d) {
  __shared__ int s_warp[kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (d >= 1 << a.digit) return;
  uint32_t* row = a.hist + (size_t)d * a.n_tiles;
  int carry = 0;
  for (int base = 0; base < a.n_tiles; base += 4 * kThreads) {
    int v[4], sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = base + 4 * tid + k;
      v[k] = i < a.n_tiles ? (int)row[i] : 0;
      sum += v[k];
    }
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      before += w < warp ? s_warp[w] : 0;
      total += s_warp[w];
    }
    int start = carry + before + x - sum;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = base + 4 * tid + k;
      if (i < a.n_tiles) row[i] = (uint32_t)start;
      start += v[k];
    }
    carry += total;
    __syncthreads();
  }
  if (tid == 0) a.hist[(size_t)(1 << a.digit) * a.n_tiles + d] = (uint32_t)carry;
}

// Stable scatter of tile `tile` by digit `pass`.
__device__ __forceinline__ void sort_scatter(const SortArgs& a, int pass, int tile) {
  constexpr int kRounds = kSortRoundsMax;
  __shared__ int cnt[kWarps][kMaxBins];
  __shared__ int s_warp[kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int shift = pass * a.digit, bins = 1 << a.digit, mask = bins - 1;
  const int first = (tile * kWarps + warp) * 32 * a.rounds + lane;
  const unsigned below = (1u << lane) - 1u;
  for (int d = lane; d < bins; d += 32) cnt[warp][d] = 0;
  // where this tile's keys of digit `tid` go: the digits before it, the tiles
  // before this one
  int total = 0, row = 0;
  if (tid < bins) {
    total = (int)a.hist[(size_t)bins * a.n_tiles + tid];
    row = (int)a.hist[(size_t)tid * a.n_tiles + tile];
  }
  int x = total;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  int start = row + x - total;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) start += w < warp ? s_warp[w] : 0;
  // ranks within the warp
  uint32_t key[kRounds];
  int rank[kRounds];
#pragma unroll
  for (int r = 0; r < kRounds; ++r)
    if (r < a.rounds) {
      const int i = first + 32 * r;
      key[r] = i < a.n ? a.keys[pass & 1][i] : ~0u;
    }
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    if (r < a.rounds) {
      // (lanes behind the last particle have a digit of all ones and are the
      // last of its lanes: they take no rank from a particle)
      const int d = (key[r] >> shift) & mask;
      const unsigned peers = same_digit(d, a.digit);
      const int seen = cnt[warp][d];
      rank[r] = seen + __popc(peers & below);
      __syncwarp();
      if ((peers & below) == 0u) cnt[warp][d] = seen + __popc(peers);
      __syncwarp();
    }
  }
  __syncthreads();
  if (tid < bins) {
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const int c = cnt[w][tid];
      cnt[w][tid] = start;
      start += c;
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int i = first + 32 * r;
    if (r < a.rounds && i < a.n) {
      const int pos = cnt[warp][(key[r] >> shift) & mask] + rank[r];
      a.vals[(pass + 1) & 1][pos] = pass == 0 ? (uint32_t)i : a.vals[pass & 1][i];
      if (pass + 1 < a.passes) a.keys[(pass + 1) & 1][pos] = key[r];
    }
  }
}

__global__ void __launch_bounds__(kThreads) k_sort_hist(SortArgs a, int pass) {
  chain_begin();
  sort_hist(a, pass, blockIdx.x);
}
__global__ void __launch_bounds__(kThreads) k_sort_rows(SortArgs a) {
  chain_begin();
  sort_rows(a, blockIdx.x);
}
__global__ void __launch_bounds__(kThreads) k_sort_scatter(SortArgs a, int pass) {
  chain_begin();
  sort_scatter(a, pass, blockIdx.x);
}

// Batched: thread block b is tile work[b].y of scene work[b].x, or digit
// blockIdx.y of scene blockIdx.x. A scene whose keys need fewer passes than the
// batch's most takes narrower digits.
__global__ void __launch_bounds__(kThreads) k_sort_hist_batch(const SortArgs* __restrict__ args,
                                                              const int2* __restrict__ work, int pass) {
  __shared__ SortArgs s_a;
  chain_begin();
  const int2 wk = work[blockIdx.x];
  load_args(args + wk.x, s_a);
  __syncthreads();
  sort_hist(s_a, pass, wk.y);
}
__global__ void __launch_bounds__(kThreads) k_sort_rows_batch(const SortArgs* __restrict__ args) {
  __shared__ SortArgs s_a;
  chain_begin();
  load_args(args + blockIdx.x, s_a);
  __syncthreads();
  if (s_a.n > 0) sort_rows(s_a, blockIdx.y);
}
__global__ void __launch_bounds__(kThreads) k_sort_scatter_batch(const SortArgs* __restrict__ args,
                                                                 const int2* __restrict__ work, int pass) {
  __shared__ SortArgs s_a;
  chain_begin();
  const int2 wk = work[blockIdx.x];
  load_args(args + wk.x, s_a);
  __syncthreads();
  sort_scatter(s_a, pass, wk.y);
}

__device__ __forceinline__ void permute_one(const Particles& src, const Particles& dst,
                                            const uint32_t* perm, int i) {
  // every plane's load before the first store: the compiler may not move a
  // load of src above a store to dst
  const uint32_t j = perm[i];
  float v[kParticlePlanes];
#pragma unroll
  for (int k = 0; k < kParticlePlanes; ++k) v[k] = src.plane(k)[j];
  const uint32_t pid = src.pid[j];
  const uint16_t grp = src.grp[j];
#pragma unroll
  for (int k = 0; k < kParticlePlanes; ++k) dst.plane(k)[i] = v[k];
  dst.pid[i] = pid;
  dst.grp[i] = grp;
}

__global__ void k_permute(Particles src, Particles dst, const uint32_t* perm, int n) {
  chain_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) permute_one(src, dst, perm, i);
}

__global__ void __launch_bounds__(kThreads) k_permute_batch(const SortArgs* __restrict__ args,
                                                            const int2* __restrict__ work) {
  __shared__ SortArgs s_a;
  chain_begin();
  const int2 wk = work[blockIdx.x];
  load_args(args + wk.x, s_a);
  __syncthreads();
  for (int r = 0; r < s_a.rounds; ++r) {
    const int i = (wk.y * s_a.rounds + r) * kThreads + (int)threadIdx.x;
    if (i < s_a.n) permute_one(s_a.src, s_a.dst, s_a.vals[s_a.passes & 1], i);
  }
}

// Records of W floats between particle planes and id order, a warp's 32
// particles at a time: through shared memory, so that a record's words are
// written (or read) by neighbouring lanes. With a lane to a record each of its W
// stores touched 32 sectors: all four arrays of 1M particles of random ids out
// 191 -> 98 us and in (the stress had a launch of its own) 109 -> 79, 4M
// 1228 -> 575 and 442 -> 367 (a call's 15 us included).
constexpr int kIdThreads = 256;

template <int W>
__device__ __forceinline__ void put_records(float* s, const float* v, unsigned id, int cnt, float* out) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll
  for (int c = 0; c < W; ++c) s[lane * W + c] = v[c];
  __syncwarp();
#pragma unroll
  for (int k = 0; k < W; ++k) {
    const int w = k * 32 + lane, rec = w / W;
    const size_t rid = __shfl_sync(0xffffffffu, id, rec);
    if (rec < cnt) out[W * rid + (w - rec * W)] = s[w];
  }
}

template <int W>
__device__ __forceinline__ void get_records(float* s, float* v, unsigned id, int cnt, const float* in) {
  const int lane = threadIdx.x & 31;
  float t[W];
#pragma unroll
  for (int k = 0; k < W; ++k) {
    const int w = k * 32 + lane, rec = w / W;
    const size_t rid = __shfl_sync(0xffffffffu, id, rec);
    t[k] = rec < cnt ? in[W * rid + (w - rec * W)] : 0.f;
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k < W; ++k) s[k * 32 + lane] = t[k];
  __syncwarp();
#pragma unroll
  for (int c = 0; c < W; ++c) v[c] = s[lane * W + c];
}

__global__ void __launch_bounds__(kIdThreads) k_to_id(Particles P, int n, float* __restrict__ ox,
                                                      float* __restrict__ ov, float* __restrict__ oC,
                                                      float* __restrict__ oF) {
  __shared__ float s_rec[kIdThreads / 32][32 * 9];
  const int i = blockIdx.x * kIdThreads + threadIdx.x;
  float* s = s_rec[threadIdx.x >> 5];
  const int cnt = min(n - (i & ~31), 32);  // this warp's particles
  if (cnt <= 0) return;
  const int j = min(i, n - 1);
  const unsigned id = P.pid[j];
  float x[3], v[3], C[9], F[9];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    x[c] = ox ? P.x(c)[j] : 0.f;
    v[c] = ov ? P.v(c)[j] : 0.f;
  }
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    C[c] = oC ? P.C(c)[j] : 0.f;
    F[c] = oF ? P.F(c)[j] : 0.f;
  }
  if (ox) put_records<3>(s, x, id, cnt, ox);
  if (ov) put_records<3>(s, v, id, cnt, ov);
  if (oC) put_records<9>(s, C, id, cnt, oC);
  if (oF) put_records<9>(s, F, id, cnt, oF);
}

// With iF also the stress that belongs to it.
__global__ void __launch_bounds__(kIdThreads) k_from_id(Particles P, int n, const float* __restrict__ ix,
                                                        const float* __restrict__ iv,
                                                        const float* __restrict__ iC,
                                                        const float* __restrict__ iF,
                                                        const DevGroup* __restrict__ groups) {
  __shared__ float s_rec[kIdThreads / 32][32 * 9];
  const int i = blockIdx.x * kIdThreads + threadIdx.x;
  float* s = s_rec[threadIdx.x >> 5];
  const int cnt = min(n - (i & ~31), 32);
  if (cnt <= 0) return;
  const bool mine = i < n;
  const int j = min(i, n - 1);
  const unsigned id = P.pid[j];
  float r[9];
  if (ix) {
    get_records<3>(s, r, id, cnt, ix);
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (mine) P.x(c)[i] = r[c];
  }
  if (iv) {
    get_records<3>(s, r, id, cnt, iv);
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (mine) P.v(c)[i] = r[c];
  }
  if (iC) {
    get_records<9>(s, r, id, cnt, iC);
#pragma unroll
    for (int c = 0; c < 9; ++c)
      if (mine) P.C(c)[i] = r[c];
  }
  if (iF) {
    get_records<9>(s, r, id, cnt, iF);
    float t[6];
    if (mine) {
#pragma unroll
      for (int c = 0; c < 9; ++c) P.F(c)[i] = r[c];
      kirchhoff(groups[P.grp[i]], r, t);
#pragma unroll
      for (int c = 0; c < 6; ++c) P.tau(c)[i] = t[c];
    }
  }
}

__global__ void k_stress(Particles P, int n, const DevGroup* __restrict__ groups) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float F[9], t[6];
#pragma unroll
  for (int c = 0; c < 9; ++c) F[c] = P.F(c)[i];
  kirchhoff(groups[P.grp[i]], F, t);
#pragma unroll
  for (int c = 0; c < 6; ++c) P.tau(c)[i] = t[c];
}

int rounds_of(int n) { return n > 1 << 19 ? kSortRoundsMax : kSortRoundsMin; }

SortArgs sort_args(const GridDev& g, const Particles& src, const Particles& dst, int n,
                   const SortBuffers& sb) {
  SortArgs a;
  a.g = g;
  a.src = src;
  a.dst = dst;
  a.n = n;
  a.bits = sort_key_bits(g);
  a.passes = (a.bits + 7) / 8;
  a.digit = (a.bits + a.passes - 1) / a.passes;
  a.rounds = rounds_of(n);
  a.n_tiles = (n + kThreads * a.rounds - 1) / (kThreads * a.rounds);
  for (int k = 0; k < 2; ++k) {
    a.keys[k] = sb.keys[k];
    a.vals[k] = sb.vals[k];
  }
  a.hist = sb.hist;
  return a;
}

}  // namespace

int sort_key_bits(const GridDev& g) {
  int bits = 0;
  for (int nb : {g.nbx, g.nby, g.nbz})
    for (int lim = nb - 1; lim; lim >>= 1) ++bits;
  bits += g.sort_cell_bits ? 6 : 0;
  return bits > 0 ? bits : 1;
}

cudaError_t sort_prepare() {
  return cudaFuncSetAttribute(k_sort_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kSmallSortSmem);
}

// (tiles of the fewest rounds)
int sort_max_tiles(int n) { return n > 0 ? (n - 1) / (kThreads * kSortRoundsMin) + 1 : 1; }

// digits x tiles, and a total per digit
int sort_hist_len(int n) { return kMaxBins * (sort_max_tiles(n) + 1); }

void launch_sort(const GridDev& g, const Particles& src, const Particles& dst, int n,
                 SortBuffers& sb, cudaStream_t s) {
  if (n <= 0) return;
  const SortArgs a = sort_args(g, src, dst, n, sb);
  int out = 0;
  if (n <= kSmallSortMax) {
    launch_chained(k_sort_small, dim3(1), kSmallSortThreads, kSmallSortSmem, s, a);
  } else {
    for (int p = 0; p < a.passes; ++p) {
      launch_chained(k_sort_hist, dim3(a.n_tiles), kThreads, 0, s, a, p);
      launch_chained(k_sort_rows, dim3(1 << a.digit), kThreads, 0, s, a);
      launch_chained(k_sort_scatter, dim3(a.n_tiles), kThreads, 0, s, a, p);
    }
    out = a.passes & 1;
  }
  launch_chained(k_permute, dim3((n + kThreads - 1) / kThreads), kThreads, 0, s, src, dst, sb.vals[out], n);
}

// a batch's scenes: every one takes the passes of the one with the most
void sort_batch_args(SortArgs* args, int n_scenes) {
  int passes = 1;
  for (int i = 0; i < n_scenes; ++i)
    if (args[i].passes > passes) passes = args[i].passes;
  for (int i = 0; i < n_scenes; ++i) {
    args[i].passes = passes;
    args[i].digit = (args[i].bits + passes - 1) / passes;
  }
}

SortArgs make_sort_args(const GridDev& g, const Particles& src, const Particles& dst, int n,
                        const SortBuffers& sb) {
  return sort_args(g, src, dst, n, sb);
}

void launch_sort_batch(const SortArgs* args, int n_scenes, int passes, const int2* work, int n_work,
                       cudaStream_t s) {
  if (n_work <= 0) return;
  for (int p = 0; p < passes; ++p) {
    launch_chained(k_sort_hist_batch, dim3(n_work), kThreads, 0, s, args, work, p);
    launch_chained(k_sort_rows_batch, dim3(n_scenes, kMaxBins), kThreads, 0, s, args);
    launch_chained(k_sort_scatter_batch, dim3(n_work), kThreads, 0, s, args, work, p);
  }
  launch_chained(k_permute_batch, dim3(n_work), kThreads, 0, s, args, work);
}

void launch_to_id_order(const Particles& P, int n, float* ox, float* ov, float* oC, float* oF,
                        cudaStream_t s) {
  if (n <= 0) return;
  k_to_id<<<(n + kIdThreads - 1) / kIdThreads, kIdThreads, 0, s>>>(P, n, ox, ov, oC, oF);
}

void launch_from_id_order(const Particles& P, int n, const float* ix, const float* iv, const float* iC,
                          const float* iF, const DevGroup* groups, cudaStream_t s) {
  if (n <= 0) return;
  k_from_id<<<(n + kIdThreads - 1) / kIdThreads, kIdThreads, 0, s>>>(P, n, ix, iv, iC, iF, groups);
}

void launch_stress_from_F(const Particles& P, int n, const DevGroup* groups, cudaStream_t s) {
  if (n <= 0) return;
  k_stress<<<(n + 255) / 256, 256, 0, s>>>(P, n, groups);
}

}  // namespace mpmcr
